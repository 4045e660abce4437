"""What the GEMM waits for after a failed wait (csrc/gemm_drain.h), against a model of its ring's barriers:
every copy that either CTA of a pair issued has landed, and no wait is for one that never comes (no GPU
needed)."""
import ctypes
import itertools

import pytest
from host_build import host_lib


class Drain(ctypes.Structure):
    _fields_ = [("uses", ctypes.c_uint32), ("fix", ctypes.c_int), ("block", ctypes.c_uint32)]


class Barrier:
    """Transaction barrier of one stage: a phase completes once the leader has arrived and the expected
    halves have landed."""

    def __init__(self):
        self.phase, self.arrived, self.tx = 0, False, 0

    def add(self, arrive=False, expect=0, landed=0):
        self.arrived |= arrive
        self.tx += expect - landed
        if self.arrived and self.tx == 0:
            self.phase, self.arrived = self.phase + 1, False


@pytest.fixture(scope="module")
def drain(tmp_path_factory):
    lib = host_lib(tmp_path_factory.mktemp("drain"), """
#include "gemm_drain.h"
extern "C" vp::StageDrain drain(unsigned a, unsigned b, unsigned s, unsigned n) { return vp::stage_drain(a, b, s, n); }""")
    lib.drain.restype = Drain
    return lib.drain


@pytest.mark.parametrize("stages", [5, 7])
def test_drain_covers_every_issued_copy(drain, stages):
    for leader, peer in itertools.product(range(4 * stages), repeat=2):
        if abs(leader - peer) > stages:  # a use begins only after the MMAs of the one before
            continue
        for s in range(stages):
            mine, theirs = range(s, leader, stages), range(s, peer, stages)
            if abs(len(mine) - len(theirs)) > 1:
                continue
            d = drain(leader, peer, s, stages)
            # Copies landed so far: all uses but the last, and of the last none, one half or what was issued.
            last = max(len(mine), len(theirs)) - 1
            assert d.uses == last + 1
            if last < 0:
                continue
            assert d.block == s + last * stages
            bar = Barrier()
            for _ in range(last):
                bar.add(arrive=True, expect=2)
                bar.add(landed=2)
            halves = (len(mine) > last) + (len(theirs) > last)
            if len(mine) > last:
                bar.add(arrive=True, expect=2)
            for early in range(halves + 1):  # halves that land before the drain's correction
                b = Barrier()
                b.__dict__.update(bar.__dict__)
                b.add(landed=early) if early else None
                if d.fix > 0:
                    b.add(arrive=True, expect=1)
                if d.fix < 0:
                    b.add(landed=1)
                if early < halves:
                    assert b.phase < d.uses, "the wait would end with a copy in flight"
                    b.add(landed=halves - early)
                assert b.phase == d.uses, "the wait would be for a copy that never comes"

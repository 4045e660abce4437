"""The hand-over of surrogate heads' vectors between the warps of the cheap-heads kernel (csrc/heads_vec.h),
gone through in random interleavings: no warp writes an entry that another may still read (no GPU needed)."""
import random

from host_build import host_lib

WARPS = 3  # of each of the two groups; eight in the kernel


def conflicts(entry, heads, seed):
    """Steps of each warp, for the n-th head of its group's list: write its part of entry(g, n, head), arrive
    and wait for the group's n-th hand-over, read the whole entry once per tile.  Counts the writes to an
    entry that another warp has begun to read for a head and not finished with."""
    rng = random.Random(seed)
    at = {(g, w): (0, "write") for g in range(2) for w in range(WARPS)}
    arrived = [[0] * (len(heads[g]) + 1) for g in range(2)]
    reading = {}  # warp -> entry
    bad = 0
    while at:
        g, w = rng.choice(sorted(at))
        n, step = at[g, w]
        if n == len(heads[g]):
            del at[g, w]
        elif step == "write":
            e = entry(g, n, heads[g][n])
            bad += sum(r == e for other, r in reading.items() if other != (g, w))
            arrived[g][n] += 1
            at[g, w] = (n, "wait")
        elif step == "wait" and arrived[g][n] == WARPS:
            reading[g, w] = entry(g, n, heads[g][n])
            at[g, w] = (n, "read")
        elif step == "read":
            del reading[g, w]
            at[g, w] = (n + 1, "write")
    return bad


def test_no_entry_is_written_while_another_warp_reads_it(tmp_path):
    lib = host_lib(tmp_path, """
#include "heads_vec.h"
extern "C" int entry(int g, unsigned n) { return vp::vec_entry(g, n); }""")
    # Heads by slot: the same ones in both groups, some in one only, the same head for several tiles is one entry.
    lists = [([0, 1, 2, 3], [0, 1, 2, 3]), ([0], [0]), ([0, 2, 5], [1, 2, 4, 5]), ([7], [6, 7])]
    for i, heads in enumerate(lists):
        for seed in range(200):
            assert conflicts(lambda g, n, h: lib.entry(g, n), heads, seed) == 0, (i, seed)
    assert len({lib.entry(g, n) for g in range(2) for n in range(2)}) == 4
    # What the entries avoid: one per head, shared by the groups, and one per group.
    assert any(conflicts(lambda g, n, h: h, lists[0], seed) for seed in range(200))
    assert any(conflicts(lambda g, n, h: g, lists[0], seed) for seed in range(200))

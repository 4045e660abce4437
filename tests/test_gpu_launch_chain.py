"""The overlapped launches of a layer and of a stack give what the same call gives on an idle GPU: called
again and again on one workspace with other weights, modes and tokens written by kernels just before on the
same stream; on two streams at once; captured into a graph and replayed.

Bits are compared, except with merged tokens: their members are summed in the order of atomics, so a
merged token's mean may differ in its last fp32 bits and each block's stored value by a bf16 step."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import synth
from helpers import BF16_STEP, compare
from paper_2609_23733_gb300 import binding as vpb

pytestmark = pytest.mark.gpu

H, VIEW, GRID = 16, 261, 16
BLOCKS = {"layer": 1, "stack": 3, "merge": 2}


class Call:
    """One call with its own buffers; ``put(i)`` enqueues kernels that write the i-th weights, modes and
    tokens into them."""

    def __init__(self, kind, seed, views):
        self.kind, self.L, self.N = kind, BLOCKS[kind], views * VIEW
        g = synth.rng(seed)
        qk = synth.make_qk_norm_weights(g)
        self.sets = []
        for i in range(2):
            w = [vpb.to_device(synth.make_layer_weights(g, block=kind != "layer", bias_std=0.05, norm_jitter=0.1))
                 for _ in range(self.L)]
            modes = np.stack([np.roll(synth.forced_mix(H, (0.25, 0.5, 0.0)[(l + i) % 3]), 5 * i + l)
                              for l in range(self.L)]).astype(np.int32)
            self.sets.append((w, torch.from_numpy(modes).cuda(),
                              vpb.bf16_from_bits(synth.make_tokens(seed + 10 + i, self.N))))
        w, modes, x = self.sets[0]
        self.w = [{k: torch.empty_like(t) for k, t in d.items()} for d in w]
        self.force, self.x = torch.empty_like(modes), torch.empty_like(x)
        self.assign = torch.zeros(self.N, dtype=torch.int32, device="cuda")
        self.dm = vpb.dims(self.N, H)
        self.ws = vpb.workspace(self.dm, {"layer": vpb.VP_WS_LAYER, "stack": vpb.VP_WS_STACK,
                                          "merge": vpb.VP_WS_STACK_MERGE}[kind])
        self.modes = torch.empty(self.L, H, dtype=torch.int32, device="cuda")
        self.s = torch.empty(self.L, H, device="cuda")
        self.s_attn = torch.empty(self.L, H, device="cuda")
        self.out = torch.empty_like(x)
        self.qk_w = vpb.to_device(qk)
        self.qk = vpb.qk_options(self.qk_w, 1e-6, True, VIEW, 5, GRID, 100.0)
        self.merge = vpb.merge_options(4, VIEW, 5, assign_out=self.assign) if kind == "merge" else None
        self.layers = None if kind == "layer" else [
            vpb.layer_weights(d, merge=self.merge if l == 0 else None) for l, d in enumerate(self.w)]

    def put(self, i):
        w, modes, x = self.sets[i]
        torch.add(modes, 0, out=self.force)
        torch.add(x, 0, out=self.x)
        for src, dst in zip(w, self.w):
            # last, those that kernels read ahead of their wait
            for k in sorted(src, key=lambda k: k in ("w_qkv", "w_fc1", "w_fc2", "ln1_g", "ln1_b", "b_qkv")):
                torch.add(src[k], 0, out=dst[k])

    def run(self):
        if self.kind == "layer":
            d = self.w[0]
            vpb.vp_moh_global_attention(self.dm, self.x, d["w_qkv"], d["b_qkv"], d["w_o"], d["b_o"],
                                        vpb.router_weights(d), vpb.surrogate_weights(d), self.force, self.out, None,
                                        None, self.s, self.modes, self.ws, qk=self.qk, s_attn_out=self.s_attn)
        else:
            vpb.vp_global_stack(self.dm, self.x, self.layers, self.force, self.modes, self.s, 1e-6, self.ws,
                                s_attn_out=self.s_attn)

    def results(self):
        y = self.out if self.kind == "layer" else self.x
        return [t.clone() for t in (y, self.modes, self.s, self.s_attn, self.assign)]

    def alone(self):
        """The results of both sets on an idle GPU."""
        out = []
        for i in range(2):
            self.put(i)
            torch.cuda.synchronize()
            self.run()
            torch.cuda.synchronize()
            out.append(self.results())
        assert vpb.vp_read_device_error(self.ws) == 0
        assert not torch.equal(out[0][0], out[1][0])
        return out

    def check(self, got, want):
        assert torch.equal(got[1], want[1]) and torch.equal(got[4], want[4])
        if self.kind != "merge":
            for a, b in zip(got, want):
                assert torch.equal(a, b), float((a.float() - b.float()).abs().max())
        else:
            compare(got[0].float().cpu().numpy(), want[0].float().cpu().numpy(), rel=self.L * BF16_STEP)


@pytest.mark.parametrize("kind,views", [("layer", 5), ("layer", 21), ("stack", 4), ("merge", 4)])
def test_calls_behind_one_another_on_one_workspace(kind, views):
    c = Call(kind, 3, views)
    want = c.alone()
    order = [0, 1, 1, 0, 1, 0, 0, 1]
    got = []
    for i in order:  # nothing waits in between
        c.put(i)
        c.run()
        got.append(c.results())
    torch.cuda.synchronize()
    assert vpb.vp_read_device_error(c.ws) == 0
    for i, g in zip(order, got):
        c.check(g, want[i])


@pytest.mark.parametrize("kind", list(BLOCKS))
def test_two_streams_at_once(kind):
    calls = [Call(kind, 20, 4), Call(kind, 40, 4)]
    want = [c.alone() for c in calls]
    streams = [torch.cuda.Stream() for _ in calls]
    torch.cuda.synchronize()
    got = [[], []]
    for i in (0, 1, 0, 1):
        for j, (c, s) in enumerate(zip(calls, streams)):
            with torch.cuda.stream(s):
                c.put(i)
                c.run()
                got[j].append((i, c.results()))
    torch.cuda.synchronize()
    for j, c in enumerate(calls):
        assert vpb.vp_read_device_error(c.ws) == 0
        for i, g in got[j]:
            c.check(g, want[j][i])


@pytest.mark.parametrize("kind", list(BLOCKS))
def test_captured_and_replayed(kind):
    c = Call(kind, 60, 4)
    want = c.alone()
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        c.run()
    for i in (0, 1, 1, 0):
        with torch.cuda.stream(s):
            c.put(i)
            graph.replay()
            got = c.results()
        torch.cuda.synchronize()
        c.check(got, want[i])
    assert vpb.vp_read_device_error(c.ws) == 0

"""vp_linear where its tiling can go wrong: edges of the 256 x 256 pair tiles, one round and several,
a last round that is cut into half-width tiles, both epilogue widths, the residual in place."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2609_23733_gb300 import binding as vpb

pytestmark = pytest.mark.gpu

# (M, N, K): a single ragged tile; tile edges; one full round of pairs and two; 172 tiles (the last
# 20 cut); a cut tile whose second half is past N; 137 + tiles with ragged columns.
SHAPES = [(1, 8, 8), (256, 256, 64), (257, 264, 72), (19456, 256, 64), (19456, 512, 64),
          (10992, 1024, 64), (2700, 1096, 136), (9000, 1000, 64)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual", "in_place"])
def test_linear_tiles(M, N, K, epilogue):
    g = synth.rng(M + 7 * N + K)
    a = synth.f32_to_bf16_bits(g.standard_normal((M, K), dtype=np.float32))
    w = synth.f32_to_bf16_bits(g.standard_normal((N, K), dtype=np.float32) / np.sqrt(K))
    bias = g.standard_normal(N).astype(np.float32)
    A, W = oracle.bf16_bits_to_f64(a), oracle.bf16_bits_to_f64(w)
    want = A @ W.T + bias
    dev = {"A": vpb.bf16_from_bits(a), "W": vpb.bf16_from_bits(w), "bias": torch.from_numpy(bias).cuda()}
    kw = {}
    if epilogue == "gelu":
        want = oracle.gelu(want)
        kw["act"] = vpb.VP_ACT_GELU
    elif epilogue != "bias":
        scale = (1 + 0.1 * g.standard_normal(N)).astype(np.float32)
        r = synth.f32_to_bf16_bits(g.standard_normal((M, N), dtype=np.float32))
        want = want * scale + oracle.bf16_bits_to_f64(r)
        kw["scale"], kw["residual"] = torch.from_numpy(scale).cuda(), vpb.bf16_from_bits(r)
        if epilogue == "in_place":
            kw["out"] = kw["residual"]
    got = vpb.vp_linear(dev["A"], dev["W"], dev["bias"], **kw)
    torch.cuda.synchronize()
    got = oracle.bf16_bits_to_f64(vpb.bits_from_bf16(got))
    # bf16 rounding of the result (2^-9 relative) and fp32 accumulation, K terms of |a| |w|; the
    # GELU's erf adds 1.5e-7 |x|.
    tol = 2.0 ** -8 * np.abs(want) + 2.0 ** -23 * (K + 8) * (np.abs(A) @ np.abs(W).T + np.abs(bias) + 4)
    assert np.all(np.abs(got - want) <= tol), float((np.abs(got - want) / tol).max())

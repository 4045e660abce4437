"""The router around the token counts where its splits change (a CTA of the key sweep per 256 tokens
up to 4,864, then one wave), with and without biases, against the oracle on the same QKV."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2609_23733_gb300 import binding as vpb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [4864, 4865, 5001, 12289])
@pytest.mark.parametrize("H,bias_std", [(16, 0.0), (5, 0.2)])
def test_router_splits(N, H, bias_std):
    g = synth.rng(N + H)
    w = synth.make_layer_weights(g, D=H * 64, H=H, bias_std=bias_std)
    bits = synth.f32_to_bf16_bits(g.standard_normal((N, 3, H, 64), dtype=np.float32) + 0.3)
    if bias_std == 0.0:
        w.pop("r_bW"), w.pop("r_bU")
    dw = vpb.to_device(w)
    dm = vpb.dims(N, H)
    ws = vpb.workspace(dm, vpb.VP_WS_ROUTER)
    s, modes = torch.zeros(H, device="cuda"), torch.zeros(H, dtype=torch.int32, device="cuda")
    q_pool, ctx, mean_v = (torch.zeros(H, 64, device="cuda") for _ in range(3))
    r = torch.zeros(H, N, device="cuda")
    vpb.vp_router(dm, vpb.bf16_from_bits(bits), vpb.router_weights(dw), None, s, modes, q_pool, ctx, mean_v, r, ws)
    torch.cuda.synchronize()
    assert vpb.vp_read_device_error(ws) == 0
    lw = oracle.load_layer(w)
    qkv = oracle.bf16_bits_to_f64(bits)
    for h in range(H):
        b = (lw["r_bW"][h], lw["r_bU"][h]) if bias_std else (None, None)
        _, want = oracle.attention_pool(qkv[:, 0, h], lw["r_W"][h], lw["r_U"][h], lw["r_w"][h], *b)
        # fp32 sums of N weights in (0, 1] and values of order 1, weights good to 1e-6 relative.
        np.testing.assert_allclose(q_pool[h].cpu().numpy(), want, rtol=0, atol=1e-5)
        rv = oracle.routing_vector(want, qkv[:, 1, h], 1 / 8)
        np.testing.assert_allclose(r[h].cpu().numpy(), rv, rtol=1e-4)
        np.testing.assert_allclose(s[h].item(), rv.max(), rtol=1e-4)
        np.testing.assert_allclose(ctx[h].cpu().numpy(), rv @ qkv[:, 2, h], rtol=0, atol=2e-5)
        np.testing.assert_allclose(mean_v[h].cpu().numpy(), qkv[:, 2, h].mean(0), rtol=0, atol=1e-5)

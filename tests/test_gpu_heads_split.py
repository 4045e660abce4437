"""Head attention around the sizes where its work is cut another way: at most one group of 384 query
rows per SM or more (3,456 tokens at 16 heads), 40 or 41 key tiles (2,560 tokens), surrogate items
handed out one by one or in batches (1,216 items), one token; against the oracle on the same QKV."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import compare
from paper_2609_23733_gb300 import binding as vpb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,n_mean,n_sur", [
    (1, 16, 5, 5), (65, 3, 1, 1), (385, 16, 0, 0), (2560, 16, 4, 9), (2561, 16, 4, 9), (3456, 16, 0, 15),
    (3457, 16, 1, 2), (5001, 1, 0, 0), (12289, 16, 2, 12), (12289, 16, 1, 13)])
def test_heads_where_the_work_is_cut_another_way(N, H, n_mean, n_sur):
    g = synth.rng(N + H + n_mean)
    w = synth.make_layer_weights(g, D=H * 64, H=H, bias_std=0.1)
    bits = synth.f32_to_bf16_bits(g.standard_normal((N, 3, H, 64), dtype=np.float32))
    ctx, mean_v = (0.3 * g.standard_normal((H, 64)).astype(np.float32) for _ in range(2))
    order = g.permutation(H).astype(np.int32)
    dm = vpb.dims(N, H)
    ws = vpb.workspace(dm, vpb.VP_WS_ROUTER)
    y = torch.full((N, H * 64), float("nan"), dtype=torch.bfloat16, device="cuda")
    s_attn = torch.full((H,), float("nan"), device="cuda")
    dw = vpb.to_device(w)
    vpb.vp_head_attention(dm, vpb.bf16_from_bits(bits), torch.from_numpy(order).cuda(),
                          torch.tensor([0, n_mean, n_mean + n_sur, H], dtype=torch.int32, device="cuda"),
                          torch.from_numpy(ctx).cuda(), torch.from_numpy(mean_v).cuda(),
                          vpb.surrogate_weights(dw), y, ws, s_attn=s_attn)
    torch.cuda.synchronize()
    assert vpb.vp_read_device_error(ws) == 0
    got = y.float().cpu().numpy().reshape(N, H, 64)
    assert np.all(np.isfinite(got))
    lw = oracle.load_layer(w)
    qkv = oracle.bf16_bits_to_f64(bits)
    rows = np.unique(np.concatenate([np.arange(0, N, max(1, N // 61)), [N - 1]]))
    full = order[n_mean + n_sur:]
    for i, h in enumerate(order):
        q, k, v = (qkv[:, j, h] for j in range(3))
        if i < n_mean:
            want = np.tile(mean_v[h].astype(np.float64), (len(rows), 1))
        elif i < n_mean + n_sur:
            c = ctx[h].astype(np.float64)
            z = np.concatenate([v[rows], np.tile(c, (len(rows), 1))], axis=1)
            gm, dl = (oracle.surrogate_mlp(z, lw[f"s_{m}1_w"][h], lw[f"s_{m}1_b"][h],
                                                 lw[f"s_{m}2_w"][h], lw[f"s_{m}2_b"][h]) for m in "gd")
            want = c + oracle.sigmoid(gm) * dl
        else:
            want = oracle.full_attention(q, k, v, rows)
        # The parity bar for bf16 outputs, and a bf16 step where a value is large.
        compare(got[rows, h], want, rel=2.0 ** -7, what=f"head {h}")
    # Rows of 64-term fp32 scores; the largest entry is good to the bar of the saliency test.
    for h in full[:2] if N <= 4096 else []:
        np.testing.assert_allclose(s_attn[int(h)].item(),
                                   oracle.max_attention_saliency(qkv[:, 0, h], qkv[:, 1, h]), rtol=1e-3)

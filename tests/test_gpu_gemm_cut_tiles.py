"""vp_linear where a cut tile's second half lies past N (0 < N % 256 <= 128 in a last round that is cut), and
the merge metric's projection in that regime (64 columns, LayerNorm folded in); against float64.  The
regimes follow from the SM count and are asserted."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2609_23733_gb300 import binding as vpb
from test_gpu_gemm_tiles import test_linear_tiles as check_linear

pytestmark = pytest.mark.gpu


def _pairs():
    return max(1, torch.cuda.get_device_properties(0).multi_processor_count // 2)


def _cut_past_n(M, N):
    """Whether a launch of M x N cuts a tile whose second half holds no column (launch_linear's rule)."""
    m_tiles, n_tiles, pairs = -(-M // 256), -(-N // 256), _pairs()
    tiles = m_tiles * n_tiles
    left = tiles % pairs
    narrow = 2 * tiles <= pairs
    return not narrow and 0 < left and 2 * left <= pairs and 0 < N % 256 <= 128


def _rows(N):
    """The smallest M, less a ragged edge, of more than one round with such a cut."""
    m = next(m for m in range(1, 10_000) if m * -(-N // 256) > _pairs() and _cut_past_n(256 * m, N))
    return 256 * m - 17


@pytest.mark.parametrize("N,K", [(64, 1024), (8, 72), (1096, 136)])
@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual", "in_place"])
def test_linear_with_a_cut_half_past_the_columns(N, K, epilogue):
    M = _rows(N)
    assert _cut_past_n(M, N)
    check_linear(M, N, K, epilogue)


def test_merge_metric_with_a_cut_half_past_the_columns():
    H, P, stride = 8, 261, 10
    views = -(-(_pairs() + 3) * 256 // P)
    N, D = views * P, 64 * H
    assert _cut_past_n(N, 64)
    g = synth.rng(7)
    w = synth.make_layer_weights(g, D=D, H=H, block=True, bias_std=0.05, norm_jitter=0.1)
    bits = synth.make_tokens(7, N, D)
    dw = vpb.to_device(w)
    assign = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    dm = vpb.dims(N, H)
    ws = vpb.workspace(dm, vpb.VP_WS_STACK_MERGE)
    modes, s = torch.zeros(1, H, dtype=torch.int32, device="cuda"), torch.zeros(1, H, device="cuda")
    vpb.vp_global_stack(dm, vpb.bf16_from_bits(bits), [vpb.layer_weights(dw, None, vpb.merge_options(stride, P, 5, assign))],
                        torch.zeros(1, H, dtype=torch.int32, device="cuda"), modes, s, 1e-6, ws)
    torch.cuda.synchronize()
    assert vpb.vp_read_device_error(ws) == 0
    lw = oracle.load_layer(w)
    xt = oracle.layer_norm(oracle.bf16_bits_to_f64(bits), lw["ln1_g"], lw["ln1_b"], 1e-6)
    row_of, dst_tok = oracle.destinations(N, P, 5, stride)
    want, scores = oracle.match(oracle.key_metric(xt, lw), row_of, dst_tok)
    got = assign.cpu().numpy().astype(np.int64)
    src = np.nonzero(row_of < 0)[0]
    assert np.array_equal(got[row_of >= 0], want[row_of >= 0])
    # The library's head-mean key weights and metric rows are bf16 (2^-9 relative each): 2e-2 of cosine.
    best = scores[src].max(axis=1)
    assert np.all(scores[src, got[src]] >= best - 2e-2)
    second = np.partition(scores[src], -2, axis=1)[:, -2]
    clear = best - second > 4e-2
    assert clear.sum() >= 100
    assert np.array_equal(got[src][clear], want[src][clear])
    # The last rows of the projection, which the cut tiles hold, are among the clear ones.
    assert np.any(clear & (src >= (N // 256) * 256 - 256))

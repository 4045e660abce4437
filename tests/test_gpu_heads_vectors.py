"""Surrogate heads with items handed out one by one, where a CTA meets many heads (1,216 items of 32 heads over
the SMs), so that the entries for a head's vectors are taken in turn; against the oracle."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

from test_gpu_heads_split import test_heads_where_the_work_is_cut_another_way as check_heads  # noqa: E402


@pytest.mark.parametrize("N,H,n_mean,n_sur", [(4864, 32, 0, 32), (2305, 32, 1, 31)])
def test_heads_vectors_taken_in_turn(N, H, n_mean, n_sur):
    check_heads(N, H, n_mean, n_sur)

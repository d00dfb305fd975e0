"""Scores of fp32 inputs at the edges of the 128-token tiles (needs a B200)."""
import numpy as np
import pytest
import torch

from helpers import check_scores, oracle_scores

pytestmark = pytest.mark.gpu

# A logit is a sum of 128 products of N(0, 1) x N(0, 2) numbers, scaled by D^-1/2: |logit| < 16 here, its
# fp32 rounding (and that of the normaliser) below 2^-23 * 16 = 2e-6, and exp doubles no relative error.
TOL = 1e-5


@pytest.mark.parametrize("B,L,H,D,N", [(1, 1, 1, 64, 1), (1, 2, 3, 128, 127), (1, 2, 2, 64, 128), (1, 1, 2, 128, 129),
                                       (1, 2, 2, 64, 193), (1, 1, 2, 128, 257), (2, 1, 3, 64, 385),
                                       (1, 10, 20, 64, 65), (1, 5, 40, 128, 40)])   # the last two: items > SMs
@pytest.mark.parametrize("given_lse", [False, True])
def test_fp32_scores_at_tile_edges(B, L, H, D, N, given_lse):
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(N * 7 + D)
    # token-major storage seen through [B, L, H, N, D] strides
    q = torch.randn(B, L, N, H, D, device="cuda", generator=g).transpose(2, 3)
    k = (torch.randn(B, L, N, H, D, device="cuda", generator=g) * 2).transpose(2, 3)
    scale = np.full(L, 0.5 / np.sqrt(D), np.float32)
    lse = None
    if given_lse:
        x = torch.matmul(q.double(), k.double().transpose(-1, -2)) * float(scale[0])
        x.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
        lse = torch.logsumexp(x, -1).float().contiguous()
    s = Session(B, L, H, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=L)
    s.scores.fill_(float("nan"))
    got = s.score(q, k, lse=lse).cpu().numpy()
    for (b, l), ref in oracle_scores(q, k, scale).items():
        check_scores(got[b, l], ref, TOL)
    np.testing.assert_array_equal(got, s.score(q, k, lse=lse).cpu().numpy())   # bitwise reproducible

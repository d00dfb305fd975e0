"""Long segments whose sort is split over a cluster of four CTAs (up to 37 segments), two (up to 74, above 8192 scores) or none, bit for bit
against the oracle (needs a B200)."""
import numpy as np
import pytest
import torch

from helpers import oracle_select
from test_gpu_select_edges import _scores

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,N", [(1, 1, 4097), (1, 37, 4224), (1, 38, 4097), (1, 38, 8193), (2, 37, 8700), (1, 75, 8200), (1, 2, 16384), (1, 40, 16383)])
@pytest.mark.parametrize("kind", ["ties", "wide", "halves", "zero"])
def test_split_sort(B, L, N, kind):
    from paper_2412_03409_b200.session import Session
    scores = np.stack([np.zeros((L, N), np.float32) if kind == "zero" else _scores(kind, L, N, 7 * b + N) for b in range(B)])
    budget = max(L, int(0.3 * L * N))
    s = Session(B, L, 1, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    s.search(budget, scores=torch.from_numpy(scores).cuda())
    for b, (order, cum, res) in enumerate(oracle_select(scores, [budget] * B)):
        np.testing.assert_array_equal(s.order[b].cpu().numpy(), order)
        np.testing.assert_array_equal(s.cum[b].cpu().numpy().view(np.uint64), cum)
        np.testing.assert_array_equal(s.len[b].cpu().numpy(), res.len)
    assert s.status.cpu().tolist() == [0] * B


@pytest.mark.parametrize("value,place,code", [(2.0 ** 21, 16000, "DEV_RANGE"), (2.0 ** 9, None, "DEV_RANGE"), (-1.0, 9000, "DEV_BAD_SCORE"),
                                              (float("nan"), 100, "DEV_BAD_SCORE"), (1.0, None, "DEV_OK")])
@pytest.mark.parametrize("L", [3, 60])
def test_split_sort_reports(value, place, code, L):
    """A bad score, a weight of 2^53 or a total that reaches it only over all CTAs (16384 of 2^41) is reported."""
    from paper_2412_03409_b200 import api
    from paper_2412_03409_b200.session import Session
    scores = torch.ones(1, L, 16384, device="cuda")
    if place is None:
        scores[0, 1] = value
    else:
        scores[0, 1, place] = value
    s = Session(1, L, 1, 64, 16384, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    s.search(100 * L, scores=scores)
    assert s.status.tolist() == [getattr(api, code)]

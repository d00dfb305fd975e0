"""Long segments whose sort is split over a cluster of four CTAs (as many as run at once, 33 on a B200), two (up to 74, above 8192
scores) or none, bit for bit against the oracle (needs a B200)."""
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


@pytest.mark.parametrize("N", [4300, 8193, 12000])
def test_clusters_of_a_second_wave_are_not_made(N):
    """A few segments more than clusters that run at once do not take twice the time."""
    from paper_2412_03409_b200.session import Session
    times = []
    for L in (33, 34, 37):
        scores = torch.rand(1, L, N, device="cuda")
        s = Session(1, L, 1, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
        lens = torch.full((L,), 9, dtype=torch.int32, device="cuda")
        runs = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(10):
                s.apply_lengths(lens, scores=scores)
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        times.append(sorted(runs[2:])[5])
    assert max(times[1:]) < 1.5 * times[0], times    # (1.04 to 1.31 measured; 1.17 to 1.9 in two waves)


@pytest.mark.parametrize("L,N", [(33, 4097), (34, 4097), (33, 9000), (34, 9000), (35, 8192)])
def test_at_the_number_of_clusters(L, N):
    from paper_2412_03409_b200.session import Session
    scores = _scores("ties", L, N, N)
    s = Session(1, L, 1, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    s.search(int(0.3 * L * N), scores=torch.from_numpy(scores[None]).cuda())
    (order, cum, res), = oracle_select(scores[None], [int(0.3 * L * N)])
    np.testing.assert_array_equal(s.order[0].cpu().numpy(), order)
    np.testing.assert_array_equal(s.cum[0].cpu().numpy().view(np.uint64), cum)
    np.testing.assert_array_equal(s.len[0].cpu().numpy(), res.len)

"""Selection, bit for bit against the oracle, where the radix sort and the search change their ways (needs a B200)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from helpers import oracle_select

pytestmark = pytest.mark.gpu


def _scores(kind, L, N, seed):
    rng = np.random.default_rng(seed)
    if kind == "ties":        # few distinct values, zeros of both signs among them
        s = rng.integers(0, 5, (L, N)).astype(np.float32) / 4
        s[rng.random((L, N)) < 0.1] = -0.0
    elif kind == "wide":      # the whole exponent range, subnormals included, that keeps the total below 2^53
        s = np.ldexp(rng.random((L, N)), rng.integers(-140, 5, (L, N))).astype(np.float32)
    elif kind == "halves":    # weights that end in exactly one half and round to even
        s = np.ldexp(rng.integers(1, 1 << 24, (L, N)).astype(np.float64), -33 - rng.integers(0, 26, (L, N))).astype(np.float32)
    else:
        s = rng.exponential(1.0, (L, N)).astype(np.float32)
    return s


@pytest.mark.parametrize("B,L,N,kind,tol", [
    (1, 3, 1, "wide", 0.0), (2, 2, 31, "ties", 0.0), (1, 4, 33, "halves", 1e-6), (1, 5, 1023, "exp", 1e-15),
    (1, 33, 1024, "ties", 1e-6), (2, 65, 1025, "wide", 1e-6), (1, 3, 2049, "halves", 1e-17), (1, 130, 700, "exp", 0.0),
    (1, 3, 64, "ties", 0.0), (2, 3, 255, "halves", 0.0), (1, 4, 256, "ties", 1e-6), (1, 4, 257, "ties", 1e-6),
    (1, 3, 768, "wide", 0.0), (2, 3, 769, "ties", 1e-9), (1, 2, 3072, "halves", 0.0),
    (1, 2, 4097, "ties", 0.0), (1, 2, 8193, "wide", 1e-9), (1, 3, 16384, "exp", 0.25), (1, 2, 16383, "halves", 2.0),
])
@pytest.mark.parametrize("ratio,max_iters", [(0.2, 2000), (0.7, 2000), (0.33, 3)])
def test_selection_bit_exact_at_edges(B, L, N, kind, tol, ratio, max_iters):
    from paper_2412_03409_b200.session import Session
    scores = np.stack([_scores(kind, L, N, 11 * b + N) for b in range(B)])
    budgets = [max(L, int(ratio * L * N)) + 5 * b for b in range(B)]
    s = Session(B, L, 2, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    s.search(torch.tensor(budgets), tol=tol, max_iters=max_iters, scores=torch.from_numpy(scores).cuda())
    for b, (order, cum, res) in enumerate(oracle_select(scores, budgets, tol, max_iters)):
        np.testing.assert_array_equal(s.order[b].cpu().numpy(), order)
        np.testing.assert_array_equal(s.cum[b].cpu().numpy().view(np.uint64), cum)
        np.testing.assert_array_equal(s.len[b].cpu().numpy(), res.len)
        assert s.p[b].item() == res.p and s.iters[b].item() == res.iters
    assert s.status.cpu().tolist() == [0] * B


def test_totals_out_of_range_are_reported():
    from paper_2412_03409_b200 import api
    from paper_2412_03409_b200.session import Session
    for values, code in [([2.0 ** 21] + [0.0] * 99, api.DEV_RANGE),            # one weight of 2^53
                         ([2.0 ** 15] * 64 + [0.0] * 36, api.DEV_RANGE),       # 64 of 2^47: a total of 2^53
                         ([2.0 ** 20] * 100, api.DEV_RANGE),                   # a sum that needs 59 bits
                         ([2.0 ** 15] * 63 + [0.0] * 37, api.DEV_OK),
                         ([-1.0] + [1.0] * 99, api.DEV_BAD_SCORE), ([float("inf")] + [1.0] * 99, api.DEV_BAD_SCORE),
                         ([float("nan")] * 100, api.DEV_BAD_SCORE)]:
        s = Session(1, 2, 2, 64, 100, torch.float32, np.ones(2), decode_cap=0, max_budget_rows=2)
        x = torch.ones(1, 2, 100, device="cuda")
        x[0, 1] = torch.tensor(values)
        s.search(50, scores=x)
        assert s.status.item() == code, values[:2]
        assert int(s.len.min()) >= 1 and int(s.len.max()) <= 100


def first_call(entry, N):
    """One selection of N tokens as the first call of its process, bit for bit against the oracle."""
    from paper_2412_03409_b200.session import Session
    L, budget = 2, N
    scores = np.stack([_scores("exp", L, N, N)])
    s = Session(1, L, 2, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    if entry == "search":
        s.search(budget, scores=torch.from_numpy(scores).cuda())
    else:
        s.apply_lengths(torch.tensor([N // 3, N // 5]), scores=torch.from_numpy(scores).cuda())
    (order, cum, res), = oracle_select(scores, [budget])
    np.testing.assert_array_equal(s.order[0].cpu().numpy(), order)
    np.testing.assert_array_equal(s.cum[0].cpu().numpy().view(np.uint64), cum)
    np.testing.assert_array_equal(s.len[0].cpu().numpy(), res.len if entry == "search" else [N // 3, N // 5])
    assert s.status.cpu().tolist() == [0]


# Around 48 KiB of shared memory (four and eight scores a thread); the limit that an earlier, longer call raised
# must not be what lets a launch through, so each length gets a process of its own.
FIRST_CALLS = [("search", 3456), ("apply", 3585), ("search", 4608), ("search", 4609), ("apply", 4609), ("search", 4736),
               ("search", 4864), ("apply", 4864), ("apply", 4865)]


def test_first_call_of_a_process():
    here = os.path.dirname(os.path.abspath(__file__))
    path = os.pathsep.join([here, os.path.dirname(here)])
    runs = [(c, subprocess.Popen([sys.executable, "-c", "import test_gpu_select_edges as t; t.first_call(%r, %d)" % c],
                                 cwd=os.path.dirname(here), env=dict(os.environ, PYTHONPATH=path),
                                 stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)) for c in FIRST_CALLS]
    failed = []
    for c, p in runs:
        out, _ = p.communicate(timeout=300)
        if p.returncode:
            failed.append((c, out[-400:]))
    assert not failed, failed

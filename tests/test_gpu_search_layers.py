"""The search where its warps' shares of a sample's layers change: one layer to a warp, two, four and eight kept in
registers, odd ones out of pairs, and layers beyond them; bisections to the tolerance, to the step limit and to neighbouring
numbers (past the rounds whose midpoints are exact sums).  Counts and p are compared exactly."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 31, 130])
@pytest.mark.parametrize("L", [1, 2, 32, 33, 63, 64, 65, 97, 128, 129, 255, 256, 257, 288, 289, 321])
def test_lengths_are_the_oracles(L, N):
    rng = np.random.default_rng(L * 1000 + N)
    scores = (rng.random((L, N)) ** rng.integers(1, 12, (L, 1)) * 4).astype(np.float32)
    scores[:, 0] += 1e-6  # (a layer without any weight is another test's)
    s = Session(1, L, 1, 64, N, torch.float32, np.ones(L), decode_cap=1)
    on_gpu = torch.from_numpy(scores[None]).cuda()
    for budget in sorted({L - 1, L, L * N // 3, L * N * 9 // 10, L * N - 1, L * N}):
        for tol, steps, slack, over in ((1e-6, 64, 0, 0), (0.0, 2000, 0, 0), (0.0, 7, 0, 0), (1e-3, 64, L // 8, L // 16)):
            s.search(budget, tol=tol, max_iters=steps, slack_rows=slack, slack_over_rows=over, scores=on_gpu)
            _, _, want = oracle.select_sample(scores, budget, tol, steps, slack, over)
            got = (int(s.status.item()), s.p.item(), s.iters.item())
            if budget < L:
                assert got[0] != 0 and want.status != 0
                continue
            assert got == (0, want.p, want.iters), (budget, tol, steps)
            np.testing.assert_array_equal(s.len[0].cpu().numpy(), want.len)

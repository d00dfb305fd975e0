"""The search evaluates five bisections at a time: it may end at any of them, for any reason (needs a B200)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N", [(1, 1), (3, 40), (31, 97), (40, 640), (129, 50), (300, 33), (5, 9000)])
@pytest.mark.parametrize("slack,over", [(0, 0), (7, 0), (40, 40)])
def test_every_last_step(L, N, slack, over):
    from paper_2412_03409_b200.session import Session
    scores = np.random.default_rng(L * N).exponential(1.0, (L, N)).astype(np.float32)
    scores[:, ::3] = 0.0
    budget = max(L, int(0.3 * L * N))
    s = Session(1, L, 1, 64, N, torch.float32, np.ones(L), decode_cap=0, max_budget_rows=L)
    on_gpu = torch.from_numpy(scores[None]).cuda()
    for tol, steps in [(0.0, list(range(13)) + [200]), (1e-3, [200]), (0.04, [200]), (1.0, [200])]:
        for max_iters in steps:
            s.search(budget, tol=tol, max_iters=max_iters, slack_rows=slack, slack_over_rows=over, scores=on_gpu)
            _, _, want = oracle.select_sample(scores, budget, tol, max_iters, slack, over)
            assert (s.p.item(), s.iters.item()) == (want.p, want.iters), (tol, max_iters)
            np.testing.assert_array_equal(s.len[0].cpu().numpy(), want.len)

"""fp32 prompts whose logits are kept for the column sums (2 to 8 tiles of 128 tokens; with heads of 64 16, with a CTA for
each) and the lengths around them (needs a B200).  Against 64 bits."""
import numpy as np
import pytest
import torch

from paper_2412_03409_b200 import api
from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu

# An fp32 logit is off by up to 2^-22 of the sum of its terms' magnitudes (here below 30): 7e-6; a probability as much of itself,
# and a score is a mean of sums of them.
TOL = 2e-5


def _exact(q, k, scale):
    x = torch.matmul(q.double(), k.double().transpose(-1, -2)) * torch.from_numpy(scale).double().cuda()[None, :, None, None, None]
    later = torch.ones(x.shape[-2:], dtype=torch.bool, device="cuda").triu(1)
    return torch.softmax(x.masked_fill_(later, -float("inf")), -1).masked_fill_(later, 0).sum(-2).mean(2)


@pytest.mark.parametrize("B,L,H,D,N", [
    (1, 1, 1, 64, 129), (1, 2, 3, 128, 129), (1, 1, 9, 64, 255), (2, 1, 8, 128, 256), (1, 3, 5, 64, 257), (1, 1, 2, 128, 1000),
    (1, 1, 2, 128, 1024), (1, 1, 2, 128, 1025), (1, 1, 1, 64, 1921), (1, 1, 1, 64, 2048), (1, 1, 1, 64, 2049),
    (1, 12, 16, 64, 150),      # more items than CTAs
    (3, 9, 17, 128, 130),
    (1, 3, 7, 64, 1024), (1, 1, 17, 64, 1025), (1, 1, 14, 64, 1280), (1, 1, 15, 64, 1280),   # ten tiles: 140 items, and 150 in two passes
])
@pytest.mark.parametrize("sign", [1, -1])
def test_scores(B, L, H, D, N, sign):
    g = torch.Generator(device="cuda").manual_seed(N * 3 + H)
    # heads and tokens in another order than the shape's
    q = torch.randn(B, L, N, H, D, device="cuda", generator=g).transpose(2, 3)
    k = (torch.randn(B, L, H, N, D + 4, device="cuda", generator=g) * 2)[..., :D]
    scale = sign * np.linspace(0.5, 1.5, L).astype(np.float32) / np.float32(np.sqrt(D))
    s = Session(B, L, H, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=L)
    s.scores.fill_(float("nan"))
    got = s.score(q, k).clone()
    ref = _exact(q, k, scale)
    assert ((got.double() - ref).abs() / ref.clamp(min=1e-3)).max().item() <= TOL
    s.ws_score.fill_(255)      # over a workspace of NaN words
    assert torch.equal(got, s.score(q, k))


# one tile: a cluster of a segment's heads takes the mean up to eight heads and 98 in all
@pytest.mark.parametrize("B,L,H,D,N", [(1, 1, 1, 128, 128), (1, 4, 4, 64, 128), (1, 3, 7, 64, 65), (2, 6, 8, 128, 127), (1, 7, 7, 128, 90),
                                       (1, 14, 7, 64, 100), (1, 33, 3, 64, 100), (1, 2, 9, 128, 100), (2, 8, 8, 64, 66)])
def test_one_tile(B, L, H, D, N):
    g = torch.Generator(device="cuda").manual_seed(N + L)
    q, k = (torch.randn(B, L, H, N, D, device="cuda", generator=g) for _ in range(2))
    q[0, L - 1, H - 1, N // 2, 3] = float("nan")
    scale = np.linspace(0.5, 1.5, L).astype(np.float32) / np.float32(np.sqrt(D))
    s = Session(B, L, H, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=L)
    got = [s.score(q, k).clone() for _ in range(3)]
    ref = _exact(q, k, scale)
    assert torch.equal(torch.isnan(got[0]), torch.isnan(ref)) and torch.equal(got[0].nan_to_num(7.0), got[2].nan_to_num(7.0))
    assert ((got[0].double() - ref).abs() / ref.clamp(min=1e-3)).nan_to_num(0.0).max().item() <= TOL


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 3.4e38])
def test_elements_that_have_no_split(D, bad):
    """What a NaN query or an infinite key does to the other keys is what the definition has, and no more."""
    N = 400
    g = torch.Generator(device="cuda").manual_seed(D)
    q, k = (torch.randn(1, 1, 2, N, D, device="cuda", generator=g) for _ in range(2))
    scale = np.full(1, D ** -0.5, np.float32)
    q[..., 0] = 2.0 ** -122 if bad == 3.4e38 else q[..., 0].abs() + 1
    (q if np.isnan(bad) else k)[0, 0, 1, 200, 0] = bad
    s = Session(1, 1, 2, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=1)
    got, ref = s.score(q, k)[0, 0].double(), _exact(q, k, scale)[0, 0]
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    ok = ~torch.isnan(ref)
    assert bool(ok.any()) or bad == float("inf")
    assert bool((((got - ref).abs() / ref.clamp(min=1e-3))[ok] <= TOL).all())


@pytest.mark.parametrize("D,N,longer", [(128, 512, 4096), (64, 1500, 2100), (128, 129, 1025)])
def test_workspace_of_a_longer_prompt(D, N, longer):
    """It holds less than keeping the logits takes, and serves all the same."""
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k = (torch.randn(1, 1, 2, N, D, device="cuda", generator=g) for _ in range(2))
    scale = np.full(1, 1 / np.sqrt(D), np.float32)
    s = Session(1, 1, 2, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=1)
    s.ws_score = api.alloc_workspace(api.make_shape(1, 1, 2, D, longer, torch.float32), api.WS_SCORE, "cuda")
    assert s.ws_score.numel() < api.alloc_workspace(s.shape, api.WS_SCORE, "cuda").numel()
    ref = _exact(q, k, scale)
    assert ((s.score(q, k).double() - ref).abs() / ref.clamp(min=1e-3)).max().item() <= TOL


@pytest.mark.parametrize("B,L,H,D,N", [(3, 71, 9, 64, 1000), (2, 40, 33, 128, 1024), (1, 3, 1800, 128, 1020), (1, 13, 900, 64, 300)])
def test_segments_in_turns(B, L, H, D, N):
    """More part sums than the workspace holds: as many segments at a time, no longer than the two passes' bound."""
    g = torch.Generator(device="cuda").manual_seed(N + H)
    q, k = (torch.randn(B, L, H, N, D, device="cuda", generator=g) for _ in range(2))
    scale = np.linspace(0.5, 1.5, L).astype(np.float32) / np.float32(np.sqrt(D))
    s = Session(B, L, H, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=L)
    tiles = (N + 127) // 128
    assert s.B * s.L * H * (tiles * (tiles + 1) // 2) * 2048 > 128 << 20      # (more than one turn)
    got = s.score(q, k).clone()
    for b, l in {(0, 0), (B // 2, L // 2), (B - 1, L - 1), (B - 1, 0)}:
        ref = torch.zeros(N, dtype=torch.float64, device="cuda")
        for h in range(H):
            ref += _exact(q[b:b + 1, l:l + 1, h:h + 1], k[b:b + 1, l:l + 1, h:h + 1], scale[l:l + 1])[0, 0]
        ref /= H
        assert ((got[b, l].double() - ref).abs() / ref.clamp(min=1e-3)).max().item() <= TOL
    # each segment by itself, in one turn: the same sums
    for b, l in {(0, L // 3), (B - 1, L - 1)}:
        one = Session(1, 1, H, D, N, torch.float32, scale[l:l + 1], decode_cap=0, max_budget_rows=1)
        assert torch.equal(one.score(q[b:b + 1, l:l + 1], k[b:b + 1, l:l + 1])[0, 0], got[b, l])


def test_with_a_log_sum_exp_the_least_will_do():
    """A call with the caller's log-sum-exp has no logits to keep, and a session none to make room for."""
    N = 600
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k = (torch.randn(1, 2, 3, N, 128, device="cuda", generator=g) for _ in range(2))
    scale = np.full(2, 128 ** -0.5, np.float32)
    s = Session(1, 2, 3, 128, N, torch.float32, scale, decode_cap=0, max_budget_rows=2)
    x = torch.matmul(q.double(), k.double().transpose(-1, -2)) * float(scale[0])
    later = torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1)
    lse = torch.logsumexp(x.masked_fill_(later, -float("inf")), -1).float()
    a = s.score(q, k, lse=lse).clone()
    assert s.ws_score is None and s.ws_score_lse.numel() == api.prefixkv_workspace_bytes(s.shape, api.WS_SCORE_LEAST)
    b = s.score(q, k)
    assert s.ws_score.numel() > s.ws_score_lse.numel()
    assert ((a - b).abs() / b.clamp(min=1e-3)).max().item() <= TOL

"""Scores of short bf16 prompts, both sums in one kernel, at the edges of its key tiles and query strips (needs a B200)."""
import numpy as np
import pytest
import torch

from helpers import check_scores

pytestmark = pytest.mark.gpu


def reference(q, k, scale):
    """The scores of every layer in 64 bits, and its largest logit."""
    B, L, _, N, _ = q.shape
    ref, top = np.empty((B, L, N)), np.zeros(L)
    mask = torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1)
    for b in range(B):
        for l in range(L):
            x = torch.matmul(q[b, l].double(), k[b, l].double().transpose(-1, -2)) * float(scale[l])
            top[l] = max(top[l], float(x.abs().max()))
            ref[b, l] = torch.softmax(x.masked_fill_(mask, -float("inf")), -1).sum(1).mean(0).cpu().numpy()
    return ref, top


# Up to five key tiles of 128 and ten strips of 64; more heads than SMs, and several for a CTA where tiles are few.
@pytest.mark.parametrize("L,H,N", [(40, 30, 1), (40, 30, 63), (20, 30, 65), (10, 31, 128), (10, 31, 129), (8, 40, 191), (10, 31, 192),
                                   (8, 20, 257), (8, 20, 320), (4, 40, 385), (4, 40, 511), (4, 39, 512), (4, 39, 513),
                                   (2, 64, 576), (4, 80, 577), (4, 80, 640), (1, 63, 640), (1, 64, 640)])
@pytest.mark.parametrize("D", [64, 128])
def test_scores_of_short_prompts(L, H, N, D):
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(N * 7 + D)
    q = torch.randn(1, L, N, H, D, device="cuda", generator=g).bfloat16().transpose(2, 3)
    k = (torch.randn(1, L, N, H, D, device="cuda", generator=g) * 2).bfloat16().transpose(2, 3)
    # Layers in turn: ordinary logits, of either sign; logits so large that their exponentials overflow, and so small
    # that they vanish, unless taken relative to the maximum.
    scale = np.resize(np.array([0.5, -0.5, 6.0, -6.0], np.float32), L) / np.float32(np.sqrt(D))
    k[:, 2::4, :, :, 0] = -300.0
    q[:, 2::4, ::2, :, 0] = 1.0     # even heads: every logit near -150 (D = 128); odd heads: of either sign
    ref, top = reference(q, k, scale)
    s = Session(1, L, H, D, N, torch.bfloat16, scale, decode_cap=0, max_budget_rows=L)
    s.scores.fill_(float("nan"))
    got = s.score(q, k).cpu().numpy()
    # A logit is a sum of D products rounded to 2^-24 of its partial sums, at most twice the largest logit, and
    # multiplied by the scale: some 4 * 2^-24 of that is the relative error of its exponential.
    for l in range(L):
        check_scores(got[0, l], ref[0, l], max(1e-5, 8 * top[l] * 2.0 ** -24))
    np.testing.assert_array_equal(got, s.score(q, k).cpu().numpy())


@pytest.mark.parametrize("N", [100, 500])
def test_one_head_out_of_range(N):
    """Heads that need the maximum among heads that do not, on the same SM: neither changes the others' scores."""
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k = (torch.randn(1, 700, 1, N, 64, device="cuda", generator=g).bfloat16() for _ in range(2))
    scale = np.full(700, 0.125, np.float32)
    s = Session(1, 700, 1, 64, N, torch.bfloat16, scale, decode_cap=0, max_budget_rows=700)
    plain = s.score(q, k).clone()
    big = [0, 1, 147, 148, 300, 699]
    scale[big] = 40.0
    s = Session(1, 700, 1, 64, N, torch.bfloat16, scale, decode_cap=0, max_budget_rows=700)
    got = s.score(q, k)
    rest = [l for l in range(700) if l not in big]
    assert torch.equal(got[0, rest], plain[0, rest])
    ref, top = reference(q[:, big], k[:, big], scale[big])
    check_scores(got[:, big].cpu().numpy(), ref, 8 * top.max() * 2.0 ** -24)


def test_a_wait_for_the_other_warp_that_runs_out():
    from paper_2412_03409_b200 import api
    status = torch.zeros(2, dtype=torch.int32, device="cuda")
    api.prefixkv_selftest_bounded_wait(3, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist() == [api.DEV_TIMEOUT, 0]


@pytest.mark.parametrize("N", [40, 64, 100, 128, 200, 256, 300, 450, 512, 640])
@pytest.mark.parametrize("where", ["quarter", "early queries", "late queries", "half", "low and masked", "one key"])
@pytest.mark.parametrize("size", [110.0, -110.0, 400.0, -400.0])
def test_ranges_that_differ_within_a_head(N, where, size):
    """Logits (log2) far from 0 for some of the keys or queries only: for one of the four warps that share a strip, for strips
    after the first, for one half of a strip, or beside keys that an infinite element masks."""
    from paper_2412_03409_b200.session import Session
    L, H, D = 10, 8, 64   # 80 heads: prompts of more than four tiles take this kernel too
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k = (torch.randn(1, L, H, N, D, device="cuda", generator=g) for _ in range(2))
    q[..., 0] = k[..., 0] = q[..., 1] = k[..., 1] = 0.0
    at = torch.arange(N, device="cuda")
    q[..., 0] = 1.0
    far = size / np.log2(np.e) * 8   # (a scale of 1 / 8 below)
    if where == "quarter":
        k[..., at % 128 // 32 == 1, 0] = far
    elif where == "early queries":
        q[..., at >= N // 3, 0] = 0.0
        k[..., 0] = far
    elif where == "late queries":
        q[..., at < N - 20, 0] = 0.0
        k[..., 0] = far
    elif where == "half":
        q[..., at % 64 < 32, 0] = 0.0
        k[..., 0] = far
    elif where == "low and masked":
        k[..., 0] = far
        q[..., 1] = q[..., 1].abs() + 1
        if N % 64 == 0:   # (no padding queries, whose zeros make NaN of an infinite element)
            k[..., N // 4:N // 2, 1] = -float("inf")
    else:
        k[..., N // 2, 0] = far
    q, k = q.bfloat16(), k.bfloat16()
    scale = np.full(L, 0.125, np.float32)
    x = torch.matmul(q.double(), k.double().transpose(-1, -2)) * 0.125
    x.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
    ref = torch.softmax(x, -1).sum(3).mean(2).cpu().numpy()
    s = Session(1, L, H, D, N, torch.bfloat16, scale, decode_cap=0, max_budget_rows=L)
    got = s.score(q, k).cpu().numpy()
    # (as above; logits of masked keys are none)
    check_scores(got, ref, max(1e-5, 8 * float(x[x.isfinite()].abs().max()) * 2.0 ** -24))
    np.testing.assert_array_equal(got, s.score(q, k).cpu().numpy())


@pytest.mark.parametrize("N", [60, 333])
def test_a_scale_of_zero(N):
    """Every query attends to its keys alike."""
    from paper_2412_03409_b200.session import Session
    q, k = (torch.randn(1, 2, 3, N, 64, device="cuda").bfloat16() for _ in range(2))
    s = Session(1, 2, 3, 64, N, torch.bfloat16, np.zeros(2, np.float32), decode_cap=0, max_budget_rows=2)
    want = np.cumsum((1.0 / np.arange(1, N + 1))[::-1])[::-1]
    for got in s.score(q, k)[0].cpu().numpy():
        check_scores(got, want, 1e-6)


@pytest.mark.parametrize("N", [300, 640])
def test_heads_out_of_range_are_not_done_twice(N):
    """Heads whose logits need the maximum from the start cost one walk more, not a second pass over everything."""
    from paper_2412_03409_b200.session import Session
    q, k = (torch.randn(1, 32, 32, N, 128, device="cuda").bfloat16() for _ in range(2))
    times = []
    for scale in (1.0, 40.0):
        s = Session(1, 32, 32, 128, N, torch.bfloat16, np.full(32, scale / 128 ** 0.5, np.float32), decode_cap=0, max_budget_rows=32)
        runs = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(10):
                s.score(q, k)
            b.record()
            torch.cuda.synchronize()
            runs.append(a.elapsed_time(b))
        times.append(sorted(runs[2:])[5])
    assert times[1] < 1.9 * times[0], times   # (1.4 measured; 2.5 with a first round that fails)


# Both sides of every line between this kernel and the two passes.
@pytest.mark.parametrize("heads,N,D", [(444, 100, 64), (445, 100, 64), (1036, 65, 128), (1037, 65, 128), (3, 384, 64), (3, 385, 64), (63, 450, 128), (64, 450, 128),
                                       (148, 600, 64), (149, 600, 64), (149, 599, 64), (166, 640, 128), (165, 640, 128)])
def test_at_the_lines_of_the_route(heads, N, D):
    from paper_2412_03409_b200.session import Session
    q, k = (torch.randn(1, heads, 1, N, D, device="cuda").bfloat16() for _ in range(2))
    scale = np.full(heads, D ** -0.5, np.float32)
    s = Session(1, heads, 1, D, N, torch.bfloat16, scale, decode_cap=0, max_budget_rows=heads)
    ref, _ = reference(q, k, scale)
    check_scores(s.score(q, k).cpu().numpy(), ref, 1e-5)

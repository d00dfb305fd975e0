"""Scores at the edges of the 128-token tiles, of both tensor-core kernels (needs a B200)."""
import numpy as np
import pytest
import torch

from helpers import check_scores, oracle_scores

pytestmark = pytest.mark.gpu

# A logit is a sum of 128 products of N(0, 1) x N(0, 2) numbers, scaled by D^-1/2: |logit| < 16 here, its
# fp32 rounding (and that of the normaliser) below 2^-23 * 16 = 2e-6, and exp doubles no relative error.
TOL = 1e-5


SHAPES = [(1, 1, 1, 64, 1), (1, 2, 3, 128, 127), (1, 2, 2, 64, 128), (1, 1, 2, 128, 129), (1, 2, 2, 64, 193),
          (1, 1, 2, 128, 257), (2, 1, 3, 64, 385), (1, 1, 2, 128, 1150),   # a set's turn comes round several times
          (1, 10, 20, 64, 65), (1, 5, 40, 128, 40),                        # one-tile items, more than SMs
          (1, 2, 3, 64, 63), (2, 2, 3, 64, 64),                            # fp32 with the caller's lse: FMA kernel
          (1, 13, 20, 64, 600)]                                            # items from the counters


@pytest.mark.parametrize("B,L,H,D,N", SHAPES)
@pytest.mark.parametrize("given_lse", [False, True])
@pytest.mark.parametrize("dtype,sign", [(torch.float32, 1), (torch.bfloat16, 1), (torch.bfloat16, -1)])
def test_scores_at_tile_edges(B, L, H, D, N, given_lse, dtype, sign):
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(N * 7 + D)
    # token-major storage seen through [B, L, H, N, D] strides
    q = torch.randn(B, L, N, H, D, device="cuda", generator=g).to(dtype).transpose(2, 3)
    k = (torch.randn(B, L, N, H, D, device="cuda", generator=g) * 2).to(dtype).transpose(2, 3)
    scale = np.full(L, sign * 0.5 / np.sqrt(D), np.float32)
    lse = None
    if given_lse:
        x = torch.matmul(q.double(), k.double().transpose(-1, -2)) * float(scale[0])
        x.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
        lse = torch.logsumexp(x, -1).float().contiguous()
    s = Session(B, L, H, D, N, dtype, scale, decode_cap=0, max_budget_rows=L)
    s.scores.fill_(float("nan"))
    got = s.score(q, k, lse=lse).cpu().numpy()
    segs = [(b, l) for b in range(B) for l in range(L)] if L < 13 else [(0, 0), (0, L - 1)]
    for (b, l), ref in oracle_scores(q, k, scale, segs=segs).items():
        check_scores(got[b, l], ref, TOL)
    np.testing.assert_array_equal(got, s.score(q, k, lse=lse).cpu().numpy())   # bitwise reproducible


@pytest.mark.parametrize("row", [3, 66, 130, 200])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_a_nan_is_not_lost(row, dtype):
    """A NaN in a query reaches every key that the query attends to, whichever unit computes its exponential."""
    from paper_2412_03409_b200.session import Session
    q = torch.randn(1, 1, 2, 300, 64, device="cuda").to(dtype)
    k = torch.randn(1, 1, 2, 300, 64, device="cuda").to(dtype)
    q[0, 0, 1, row, 5] = float("nan")
    s = Session(1, 1, 2, 64, 300, dtype, np.full(1, 0.125, np.float32), decode_cap=0, max_budget_rows=1)
    got = s.score(q, k).cpu().numpy()[0, 0]
    assert np.isnan(got[:row + 1]).all() and np.isfinite(got[row + 1:]).all()


def test_exponents_out_of_range():
    """A log-sum-exp far below (above) the logits makes infinite (zero) probabilities, never wrong finite ones."""
    from paper_2412_03409_b200.session import Session
    q = torch.zeros(1, 1, 1, 256, 64, device="cuda", dtype=torch.bfloat16)
    s = Session(1, 1, 1, 64, 256, torch.bfloat16, np.full(1, 0.125, np.float32), decode_cap=0, max_budget_rows=1)
    for value, want in [(-1000.0, np.inf), (1000.0, 0.0), (float("inf"), 0.0)]:
        got = s.score(q, q, lse=torch.full((1, 1, 1, 256), value, device="cuda")).cpu().numpy()
        assert (got == want).all()


@pytest.mark.parametrize("lo,hi", [(128, 192), (128, 256), (200, 300), (384, 448)])
@pytest.mark.parametrize("D", [64, 128])
def test_keys_masked_by_an_infinite_element(lo, hi, D):
    """Keys with logits of -infinity (an infinite element against queries of one sign there) have score 0 and leave the
    others' as they are without them, whole blocks of columns included."""
    from paper_2412_03409_b200.session import Session
    N = 512  # (no padding queries: zeros, whose logits against an infinite element are NaN)
    g = torch.Generator(device="cuda").manual_seed(lo + D)
    q = torch.randn(1, 1, 2, N, D, device="cuda", generator=g).bfloat16()
    k = torch.randn(1, 1, 2, N, D, device="cuda", generator=g).bfloat16()
    q[..., 0] = q[..., 0].abs() + 1
    k[..., lo:hi, 0] = -float("inf")
    s = Session(1, 1, 2, D, N, torch.bfloat16, np.full(1, D ** -0.5, np.float32), decode_cap=0, max_budget_rows=1)
    got = s.score(q, k)[0, 0].double().cpu().numpy()
    x = torch.matmul(q.double(), k.double().transpose(-1, -2))[0, 0] * float(np.float32(D ** -0.5))
    x.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
    ref = torch.softmax(x, -1).sum(1).mean(0).cpu().numpy()
    check_scores(got, ref, TOL)
    assert (got[lo:hi] == 0).all()


@pytest.mark.parametrize("N,lo,hi", [(512, 128, 256), (520, 200, 300), (777, 700, 770), (100, 1, 60), (128, 127, 128), (300, 0, 0)])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("given_lse", [False, True])
def test_fp32_infinite_and_huge_elements(N, lo, hi, D, given_lse):
    """As above in fp32, whose split cannot carry an infinite element, at every length; and an element next to the
    largest float."""
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(lo + D)
    q = torch.randn(1, 1, 2, N, D, device="cuda", generator=g)
    k = torch.randn(1, 1, 2, N, D, device="cuda", generator=g)
    q[..., 0] = q[..., 0].abs() + 1
    k[..., lo:hi, 0] = -float("inf")
    huge = N // 2 if hi == 0 else 0
    if huge:
        q[..., 0] = 2.0 ** -122
        k[..., huge, 0] = float(np.float32(3.4e38))   # above the largest bf16; a product of 64
    s = Session(1, 1, 2, D, N, torch.float32, np.full(1, D ** -0.5, np.float32), decode_cap=0, max_budget_rows=1)
    x = torch.matmul(q.double(), k.double().transpose(-1, -2))[0, 0] * float(np.float32(D ** -0.5))
    x.masked_fill_(torch.ones(N, N, dtype=torch.bool, device="cuda").triu(1), -float("inf"))
    lse = torch.logsumexp(x, -1).float()[None, None].contiguous() if given_lse else None
    got = s.score(q, k, lse=lse)[0, 0].double().cpu().numpy()
    check_scores(got, torch.softmax(x, -1).sum(1).mean(0).cpu().numpy(), TOL)
    assert (got[lo:hi] == 0).all()


@pytest.mark.parametrize("D", [64, 128])
def test_fp32_single_products(D):
    """Logits of one product each, of the last token with itself: dropped parts of the split are at most 2^-24 of the product,
    the last of the accumulations, which truncate, 2^-23, and those before it next to nothing."""
    from paper_2412_03409_b200.session import Session
    L, N = 4096, 1 if D == 128 else 65  # (64 tokens and fewer of D = 64 go to the FMA kernel)
    rng = np.random.default_rng(D)
    x, y = (np.float32(1) + rng.integers(0, 1 << 23, (2, L)) * np.float32(2.0 ** -23)).astype(np.float32)
    x[:2048] = y[:2048] = np.float32(1) + (0xfe80 + np.arange(2048) - 1024) * np.float32(2.0 ** -23)  # two large lower parts
    scale = (64 / (x.astype(np.float64) * y)).astype(np.float32)
    lse = (scale.astype(np.float64) * x * y).astype(np.float32)
    q, k = (torch.zeros(1, L, 1, N, D, device="cuda") for _ in range(2))
    place = torch.arange(L, device="cuda") % D
    q[0, torch.arange(L), 0, N - 1, place] = torch.from_numpy(x).cuda()
    k[0, torch.arange(L), 0, N - 1, place] = torch.from_numpy(y).cuda()
    given = torch.from_numpy(lse).cuda().view(1, L, 1, 1).expand(1, L, 1, N).contiguous()
    s = Session(1, L, 1, D, N, torch.float32, scale, decode_cap=0, max_budget_rows=L)
    got = s.score(q, k, lse=given)[0, :, N - 1].cpu().numpy().astype(np.float64)
    log2e = np.float32(np.log2(np.e))
    sc, l2 = (scale * log2e).astype(np.float64), (lse * log2e).astype(np.float64)   # rounded as the kernel rounds them
    exact = sc * (x.astype(np.float64) * y)
    error = (np.log2(got) + l2 - exact) / exact
    # (log2 of a score near 1 has the rounding of the score and of the exponential, 2^-22, over an exponent of 92)
    assert np.abs(error).max() <= 1.5 * 2.0 ** -23 + 2.0 ** -28

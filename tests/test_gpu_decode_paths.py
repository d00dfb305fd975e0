"""Decode calls that take each of the library's kernels, against the oracle on the cache as it stands
(needs a B200), and says which it is.  Few (segment, head) pairs: a cluster to each; from four pairs per SM (592) a CTA to each
or, where pairs are short or too long for one wave, the per-head kernel, the row-split kernel (more than 256 segments, more than 1024
rows, pruning) or, above 64 heads, the two-kernel path."""
import numpy as np
import pytest
import torch

import oracle
from helpers import CLUSTER, HEADS, PAIR, ROWS, SHARED, TWO, check_kernel, to_np32
from paper_2412_03409_b200 import workloads as wl

pytestmark = pytest.mark.gpu

# fp32: sums of a few thousand terms; bf16: outputs are averages of N(0, 1) values, |out| < 4, so one
# rounding to bf16 is at most 2^-9 * 4 = 8e-3
TOL = {torch.float32: 2e-5, torch.bfloat16: 8e-3}

CASES = [  # B, L, H, D, N, rows per layer, dtype, evict_distance, kernel
    (1, 2, 1, 64, 40, 1, torch.bfloat16, 0, CLUSTER),        # single cached row per layer
    (1, 1, 32, 128, 300, 33, torch.bfloat16, 0, CLUSTER),    # a row more than one round of a cluster's CTA
    (2, 3, 5, 64, 300, 131, torch.float32, 0, CLUSTER),
    (1, 1, 3, 128, 3000, 2900, torch.float32, 0, CLUSTER),   # eight CTAs of many rounds each
    (3, 1, 7, 64, 2500, 1111, torch.bfloat16, 0, CLUSTER),
    (1, 4, 80, 64, 200, 50, torch.bfloat16, 0, CLUSTER),     # above the row-split kernel's 64 heads
    (2, 2, 4, 128, 64, 16, torch.bfloat16, 3, CLUSTER),      # pruning: reused slots are skipped
    (1, 3, 9, 64, 90, 30, torch.float32, 2, CLUSTER),
    (1, 20, 32, 128, 200, 60, torch.bfloat16, 3, PAIR),      # 640 pairs with pruning
    (1, 20, 32, 64, 1100, 1050, torch.bfloat16, 0, PAIR),    # 640 pairs, long segments
    (1, 9, 72, 64, 100, 20, torch.bfloat16, 0, PAIR),        # 648 pairs, 72 heads
    (1, 9, 72, 64, 1300, 1200, torch.bfloat16, 0, PAIR),
    # short segments with pruning, heads of either size.  (Behind those of the row-split kernel: lanes per row, heads per warp, rows per
    # unit and block size.  Rows of up to 8.9 KB go in units of eight, up to 16.5 KB of four, up to 28.9 KB of two; many segments
    # leave less room for the ring.  test_what_goes_elsewhere has the other combinations.)
    (1, 38, 16, 128, 40, 12, torch.bfloat16, 3, PAIR),
    (1, 15, 40, 128, 40, 12, torch.bfloat16, 3, PAIR),
    (1, 10, 64, 128, 40, 12, torch.bfloat16, 3, PAIR),
    (4, 32, 64, 128, 24, 6, torch.bfloat16, 3, ROWS),        # 16, 4, 2, 17 warps
    (2, 19, 16, 64, 40, 12, torch.bfloat16, 3, PAIR),
    (2, 10, 32, 64, 40, 12, torch.bfloat16, 3, PAIR),
    (1, 15, 40, 64, 40, 12, torch.bfloat16, 3, PAIR),
    (1, 10, 64, 64, 40, 12, torch.bfloat16, 3, PAIR),
    (1, 38, 16, 128, 40, 12, torch.float32, 3, PAIR),
    (30, 32, 16, 128, 20, 4, torch.float32, 3, ROWS),        # 8, 1, 4
    (1, 20, 32, 128, 40, 12, torch.float32, 3, PAIR),
    (4, 32, 32, 128, 24, 6, torch.float32, 3, ROWS),         # 16, 2, 2
    (1, 15, 40, 128, 40, 12, torch.float32, 3, PAIR),
    (1, 11, 56, 128, 40, 12, torch.float32, 3, PAIR),
    (1, 38, 16, 64, 40, 12, torch.float32, 3, PAIR),
    (1, 20, 32, 64, 40, 12, torch.float32, 3, PAIR),
    (1, 15, 40, 64, 40, 12, torch.float32, 3, PAIR),
    (1, 10, 64, 64, 40, 12, torch.float32, 3, PAIR),
    (10, 32, 2, 128, 40, 9, torch.bfloat16, 0, PAIR),        # 320 segments
    (1, 1, 2, 128, 6600, 6500, torch.float32, 0, CLUSTER),   # two pairs of 6.7 MB each: split over all SMs
    (2, 12, 32, 128, 1100, 1040, torch.bfloat16, 0, ROWS),   # segments split over a few CTAs each
    (1, 24, 64, 128, 40, 12, torch.bfloat16, 3, ROWS),       # 1536 short pairs with pruning
    (9, 32, 16, 128, 40, 15, torch.bfloat16, 3, ROWS),       # 288 segments
    (40, 32, 16, 64, 24, 5, torch.bfloat16, 0, ROWS),        # 1280 segments: two launches, of 25 layers and of seven
    (1, 32, 48, 128, 100, 20, torch.bfloat16, 0, HEADS),     # 1536 short pairs
    (2, 16, 48, 64, 90, 40, torch.bfloat16, 0, HEADS),
    (1, 32, 48, 64, 100, 40, torch.float32, 0, HEADS),
    (1, 20, 40, 128, 500, 300, torch.float32, 0, HEADS),     # 800 pairs too long for one wave
    (1, 27, 32, 128, 600, 560, torch.bfloat16, 0, SHARED),
    (1, 27, 32, 64, 600, 560, torch.float32, 0, SHARED),
    (1, 9, 72, 128, 1300, 1200, torch.bfloat16, 0, TWO),     # 648 long pairs of 72 heads
    (9, 30, 72, 64, 24, 8, torch.bfloat16, 0, TWO),          # 270 segments of 72 heads
]
REPLAYED = [c for i, c in enumerate(CASES) if i in (4, 6, 8, 9) or (i >= 31 and c[0] < 40)]


def _ready(B, L, H, D, N, rows, dtype, d, T, seed=3, kernel=None):
    from paper_2412_03409_b200.session import Session
    g = torch.Generator(device="cuda").manual_seed(seed + N)
    scale = np.full(L, 1.0 / np.sqrt(D), np.float32)
    s = Session(B, L, H, D, N, dtype, scale, decode_cap=T, max_budget_rows=L * rows, evict_distance=d, poison=True)
    if kernel is not None:
        check_kernel(s, kernel)
    scores = np.stack([wl.synthetic_scores(L, N, seed + b) for b in range(B)])
    s.search(L * rows, scores=torch.from_numpy(scores).cuda())
    k, v = (torch.randn(B, L, H, N, D, device="cuda", generator=g).to(dtype) for _ in range(2))
    s.compact(k, v)
    tok = [[torch.randn(B, L, H, D, device="cuda", generator=g).to(dtype) for _ in range(3)] for _ in range(T)]
    return s, scale, tok


@pytest.mark.parametrize("B,L,H,D,N,rows,dtype,d,kernel", CASES)
def test_decode_steps_match_the_oracle(B, L, H, D, N, rows, dtype, d, kernel):
    T = 8 if d else 2
    s, scale, tok = _ready(B, L, H, D, N, rows, dtype, d, T, kernel=kernel)
    ring = {i: np.full(d + 1, -1, np.int32) for i in range(B * L)}
    len0 = s.cache.len.cpu().numpy()
    off = s.cache.row_offset.cpu().numpy()
    segs = range(B * L) if B * L * rows < 4000 else [0, B * L // 2, B * L - 1]
    for t in range(T):
        before = s.cache.len.cpu().numpy()
        rows_k, rows_v = to_np32(s.cache.k), to_np32(s.cache.v)
        q, kn, vn = tok[t]
        got = to_np32(s.decode(q, kn, vn))
        after = s.cache.len.cpu().numpy()
        new_k, new_v = to_np32(s.cache.k), to_np32(s.cache.v)
        for i in segs:
            b, l, n, o = i // L, i % L, int(before[i]), int(off[i])
            dst, n_after = n, n + 1
            if d:
                dst, _, n_after = oracle.decode_slot(int(len0[i]), N, t, n, d, ring[i])
            want_k, want_v = rows_k[o:o + n_after].copy(), rows_v[o:o + n_after].copy()
            want_k[dst], want_v[dst] = to_np32(kn[b, l]), to_np32(vn[b, l])
            assert after[i] == n_after
            np.testing.assert_array_equal(new_k[o:o + n_after], want_k)
            np.testing.assert_array_equal(new_v[o:o + n_after], want_v)
            ref = oracle.decode_attn(to_np32(q[b, l]), want_k, want_v, float(scale[l]))
            assert np.abs(got[b, l] - ref).max() <= TOL[dtype], (t, i)
    assert s.status.cpu().tolist() == [0] * B
    # nothing appended: the same query over the rows that are there; lengths stay
    if H <= 64:
        q = tok[0][0]
        n = s.cache.len.clone()
        got = to_np32(s.decode(q, None, None))
        assert torch.equal(n, s.cache.len)
        for i in segs:
            b, l, o = i // L, i % L, int(off[i])
            ref = oracle.decode_attn(to_np32(q[b, l]), new_k[o:o + int(n[i])], new_v[o:o + int(n[i])], float(scale[l]))
            assert np.abs(got[b, l] - ref).max() <= TOL[dtype]


@pytest.mark.parametrize("B,L,H,D,N,rows,dtype,d,kernel", REPLAYED)
@pytest.mark.parametrize("byte", [0x7f, 0xff])
def test_replay_and_stale_workspace(B, L, H, D, N, rows, dtype, d, kernel, byte):
    """A captured call replayed token after token, over a workspace that holds anything, gives bit for
    bit what separate calls give; a segment without rows is reported and zero."""
    T = 6
    a, _, tok = _ready(B, L, H, D, N, rows, dtype, d, T, kernel=kernel)
    b, _, _ = _ready(B, L, H, D, N, rows, dtype, d, T)
    warm, _, _ = _ready(B, L, H, D, N, rows, dtype, d, T)
    buf = [x.clone() for x in tok[0]]
    warm.decode(*buf)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.decode(*buf)
    b.ws_decode.fill_(byte)
    for t in range(T):
        for x, y in zip(buf, tok[t]):
            x.copy_(y)
        if t == T - 1:
            for s in (a, b):
                s.cache.len[B * L - 1] = 0
        graph.replay()
        ref = a.decode(*tok[t])
        torch.cuda.synchronize()
        assert torch.equal(b.out, ref), t
        assert torch.equal(a.cache.len, b.cache.len), t
    from paper_2412_03409_b200 import api
    assert a.status.cpu().tolist() == b.status.cpu().tolist() == [0] * (B - 1) + [api.DEV_CAPACITY]
    assert (a.out[B - 1, L - 1] == 0).all() and int(a.cache.len[B * L - 1]) == 0


@pytest.mark.parametrize("H,D,dtype", [(1, 64, torch.float32), (9, 128, torch.bfloat16), (72, 64, torch.bfloat16)])
@pytest.mark.parametrize("rows", [1, 3, 19, 70])
def test_a_nan_row_is_not_lost(H, D, dtype, rows):
    """A NaN in one head's key makes that head's output NaN, whichever warp gets the row and whatever else it gets."""
    s, _, tok = _ready(1, 1, H, D, 80, rows, dtype, 0, 1)
    q, kn, vn = tok[0]
    h, place, n = H // 2, int(s.cache.row_offset[0]), int(s.cache.len[0])
    clean = s.cache.k.clone()
    for row in range(n):
        s.cache.k.copy_(clean)
        s.cache.k[place + row, h, 3] = float("nan")
        s.cache.len.fill_(n)
        got = s.decode(q, kn, vn)[0, 0].cpu()
        assert torch.isnan(got[h]).all(), row
        assert torch.isfinite(got[torch.arange(H) != h]).all(), row


def test_a_wait_for_flags_that_runs_out():
    """Flags that come late leave nothing that a replay with the same token could mistake for its own."""
    from paper_2412_03409_b200 import api
    status = torch.zeros(2, dtype=torch.int32, device="cuda")
    api.prefixkv_selftest_bounded_wait(2, status)
    torch.cuda.synchronize()
    assert status.cpu().tolist() == [api.DEV_TIMEOUT, 0]


def test_refused_calls_stay_refused():
    """Pruning and attending without appending are for shapes within the row-split kernel's limits."""
    from paper_2412_03409_b200 import api
    s, _, tok = _ready(1, 1, 72, 64, 60, 20, torch.bfloat16, 2, 2)
    with pytest.raises(api.PrefixKVError):
        s.decode(*tok[0])
    s, _, tok = _ready(1, 1, 72, 64, 60, 20, torch.bfloat16, 0, 2)
    with pytest.raises(api.PrefixKVError):
        s.decode(tok[0][0], None, None)


@pytest.mark.parametrize("missing", ["q", "k_new", "layer_scale", "out", "dev_status", "ws"])
def test_a_missing_tensor_is_an_argument_error(missing):
    from paper_2412_03409_b200 import api
    s, _, tok = _ready(1, 1, 2, 64, 60, 20, torch.bfloat16, 0, 2)
    args = dict(zip(("q", "k_new", "v_new"), tok[0]), layer_scale=s.layer_scale, out=s.out, dev_status=s.status,
                ws=s.ws_decode)
    args[missing] = None
    with pytest.raises(api.PrefixKVError):
        api.prefixkv_decode_attn(s.shape, s.cache, **args)

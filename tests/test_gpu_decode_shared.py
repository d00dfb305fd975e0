"""Decode calls of long segments, whose tiles the per-head kernel shares out evenly over the CTAs (needs a B200): an item
may be begun by one CTA, gone on with by others and ended by another."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TILE = {(torch.bfloat16, 128): 32, (torch.bfloat16, 64): 64, (torch.float32, 128): 16, (torch.float32, 64): 32}
# as for the other kernels: sums of a few thousand terms; |out| < 4 rounded to bf16
TOL = {torch.float32: 2e-5, torch.bfloat16: 8e-3}


def ready(L, H, D, lens, dtype, T, seed=5):
    from paper_2412_03409_b200.session import Session
    N = max(lens)
    g = torch.Generator(device="cuda").manual_seed(seed)
    # (the mean capacity, 300 rows and more, is what sends the call to the shared form)
    s = Session(1, L, H, D, N, dtype, np.full(L, D ** -0.5, np.float32), decode_cap=T, max_budget_rows=max(sum(lens), 300 * L), poison=True)
    s.apply_lengths(torch.tensor(lens, dtype=torch.int32), scores=torch.rand(1, L, N, device="cuda", generator=g))
    k, v = (torch.randn(1, L, H, N, D, device="cuda", generator=g).to(dtype) for _ in range(2))
    s.compact(k, v)
    tok = [[torch.randn(1, L, H, D, device="cuda", generator=g).to(dtype) for _ in range(3)] for _ in range(T)]
    return s, tok


def reference(s, q, D):
    off, n = s.cache.row_offset.tolist(), s.cache.len.tolist()
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    for l in range(q.shape[1]):
        if n[l] < 1:
            continue
        k, v = (x[off[l]:off[l] + n[l]].double() for x in (s.cache.k, s.cache.v))   # [rows, H, D]
        p = torch.softmax(torch.einsum("hd,rhd->hr", q[0, l].double(), k) * float(np.float32(D ** -0.5)), -1)
        out[0, l] = torch.einsum("hr,rhd->hd", p, v)
    return out


def lengths(L, H, kind, tile):
    rng = np.random.default_rng(L * H)
    if kind == "even":
        return [300] * L
    if kind == "edges":      # whole tiles, a row more, a row less
        return [int(x) for x in rng.choice([1, tile - 1, tile, tile + 1, 11 * tile, 11 * tile + 1, 700], L)]
    long = 125 * tile        # items of 125 tiles, split over many CTAs or a few CTAs' own
    return [long if (l == L - 1 if kind == "long last" else l == 0) else 10 for l in range(L)]


@pytest.mark.parametrize("L,H,kind", [(37, 16, "even"), (75, 8, "edges"), (19, 32, "edges"), (40, 16, "long last"), (40, 16, "long first"),
                                      (250, 5, "edges"), (20, 40, "even")])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_shared_tiles(L, H, kind, D, dtype):
    T = 3
    a, tok = ready(L, H, D, lengths(L, H, kind, TILE[dtype, D]), dtype, T)
    b, _ = ready(L, H, D, lengths(L, H, kind, TILE[dtype, D]), dtype, T)
    refused = [L // 3, L - 2]    # segments that cannot take the step
    before = a.cache.len.clone()
    for s in (a, b):
        s.cache.len[refused] = 0
    buf = [x.clone() for x in tok[0]]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.decode(*buf)
    b.ws_decode.fill_(0xff)
    for t in range(T):
        for x, y in zip(buf, tok[t]):
            x.copy_(y)
        got = a.decode(*tok[t])
        graph.replay()
        torch.cuda.synchronize()
        want = before + t + 1
        want[refused] = 0
        assert torch.equal(a.cache.len, want)
        for l in (0, L - 1):     # the appended rows
            row = int(a.cache.row_offset[l]) + int(before[l]) + t
            assert torch.equal(a.cache.k[row], tok[t][1][0, l]) and torch.equal(a.cache.v[row], tok[t][2][0, l])
        ref = reference(a, tok[t][0], D)
        assert float((got.double() - ref).abs().max()) <= TOL[dtype], t
        assert torch.equal(got, b.out) and torch.equal(a.cache.len, b.cache.len), t   # (a captured call replayed: bit for bit)
    from paper_2412_03409_b200 import api
    assert a.status.tolist() == [api.DEV_CAPACITY]
    # nothing appended
    got = a.decode(tok[0][0], None, None)
    assert torch.equal(a.cache.len, want)
    assert float((got.double() - reference(a, tok[0][0], D)).abs().max()) <= TOL[dtype]

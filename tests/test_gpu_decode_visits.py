"""Decode calls pair by pair: the readers of a length are counted, and rows are asked for by a length read ahead
(needs a B200).  Outputs against attention in 64 bits over the rows as they stand."""
import numpy as np
import pytest
import torch

import test_gpu_decode_paths as paths
from helpers import CLUSTER, HEADS, PAIR, ROWS, SHARED, check_kernel
from paper_2412_03409_b200 import api
from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 2e-5, torch.bfloat16: 8e-3}  # one rounding to bf16 of |out| < 4


def _session(B, L, H, D, lens, dtype, T):
    s = Session(B, L, H, D, max(lens), dtype, np.full(L, 1.0 / np.sqrt(D), np.float32), decode_cap=T,
                max_budget_rows=int(np.ceil(sum(lens) / B)))
    cap = torch.tensor(lens, dtype=torch.int32, device="cuda") + T
    s.cache.cap.copy_(cap)
    s.cache.len.copy_(cap - T)
    s.cache.row_offset.copy_(torch.cat([cap.new_zeros(1), cap.cumsum(0)])[:s.cache.row_offset.numel()])
    g = torch.Generator(device="cuda").manual_seed(H * 131 + sum(lens))
    s.cache.k.copy_(torch.randn(s.cache.k.shape, device="cuda", generator=g).to(dtype))
    s.cache.v.copy_(torch.randn(s.cache.v.shape, device="cuda", generator=g).to(dtype))
    tok = [[torch.randn(B, L, H, D, device="cuda", generator=g).to(dtype) for _ in range(3)] for _ in range(T)]
    return s, tok


def _attend(s, q, i, n):
    """Segment i's output over its first n rows, 64 bits."""
    o, L = int(s.cache.row_offset[i]), q.shape[1]
    k, v = (x[o:o + n].double().reshape(n, q.shape[2], q.shape[3]) for x in (s.cache.k, s.cache.v))
    w = torch.einsum("hd,nhd->hn", q[i // L, i % L].double(), k) / np.sqrt(q.shape[3])
    return torch.einsum("hn,nhd->hd", torch.softmax(w, -1), v)


# readers of a length (heads x CTAs of a cluster) at and around powers of two; lengths around a CTA's and a round's rows
@pytest.mark.parametrize("B,L,H,D,lens,dtype", [
    (1, 1, 1, 64, [1], torch.bfloat16), (1, 1, 1, 128, [700], torch.float32), (1, 1, 2, 128, [255], torch.bfloat16),
    (1, 2, 31, 64, [32, 129], torch.bfloat16), (1, 1, 32, 128, [127], torch.bfloat16), (2, 1, 33, 64, [64, 33], torch.float32),
    (3, 1, 63, 64, [31, 257, 8], torch.bfloat16), (2, 2, 64, 128, [16, 17, 90, 5], torch.bfloat16), (1, 1, 80, 64, [300], torch.bfloat16),
    (8, 1, 40, 128, [410, 380, 409, 3, 411, 64, 128, 256], torch.bfloat16), (1, 1, 512, 64, [40], torch.bfloat16),
])
@pytest.mark.parametrize("layerwise", [False, True])
def test_tokens_back_to_back(B, L, H, D, lens, dtype, layerwise):
    """Every call but the first starts while the one in front may still be writing the lengths."""
    T = 5
    s, tok = _session(B, L, H, D, lens, dtype, T)
    check_kernel(s, CLUSTER)
    outs = [torch.empty_like(tok[0][0]) for _ in range(T)]
    torch.cuda.synchronize()
    for t in range(T):
        if layerwise:
            for l in range(L):
                s.decode(*tok[t], out=outs[t], layer_begin=l, layer_end=l + 1)
        else:
            s.decode(*tok[t], out=outs[t])
    torch.cuda.synchronize()
    assert s.cache.len.tolist() == [n + T for n in lens] and s.status.tolist() == [0] * B
    for i, n in enumerate(lens):
        o = int(s.cache.row_offset[i])
        for t in range(T):
            for mine, new in ((s.cache.k, tok[t][1]), (s.cache.v, tok[t][2])):
                assert torch.equal(mine[o + n + t].reshape(H, D), new[i // L, i % L])
            ref = _attend(s, tok[t][0], i, n + t + 1)
            assert (outs[t][i // L, i % L].double() - ref).abs().max().item() <= TOL[dtype], (i, t)


# a CTA to a pair: one wave of five, six and seven CTAs an SM (740, 888, 1036 pairs on a B200) and the next pair after
# each, and several waves (pairs of 96 rows and more, 112 with more than 256 segments); test_what_goes_elsewhere has the others
@pytest.mark.parametrize("B,L,H,D,rows,dtype", [
    (1, 37, 20, 128, 60, torch.bfloat16), (1, 13, 57, 64, 33, torch.bfloat16), (1, 24, 37, 64, 20, torch.float32), (1, 127, 7, 64, 50, torch.bfloat16),
    (2, 14, 37, 128, 30, torch.bfloat16), (1, 17, 61, 128, 230, torch.bfloat16), (1, 20, 74, 64, 300, torch.bfloat16), (2, 25, 32, 128, 140, torch.bfloat16),
    (1, 20, 80, 128, 100, torch.float32), (8, 33, 6, 128, 210, torch.bfloat16), (8, 33, 8, 64, 500, torch.bfloat16),
])
def test_a_cta_to_a_pair(B, L, H, D, rows, dtype):
    rng = np.random.default_rng(rows)
    lens = [int(x) for x in rng.integers(1, 2 * rows, B * L)]
    T = 3
    s, tok = _session(B, L, H, D, lens, dtype, T)
    check_kernel(s, PAIR)
    outs = [torch.empty_like(tok[0][0]) for _ in range(T)]
    torch.cuda.synchronize()
    for t in range(T):
        s.decode(*tok[t], out=outs[t])
    again = s.decode(tok[0][0], None, None) if H <= 64 else None
    torch.cuda.synchronize()
    assert s.cache.len.tolist() == [n + T for n in lens] and s.status.tolist() == [0] * B
    for i in sorted({0, 1, B * L // 2, B * L - 1}):
        n, o = lens[i], int(s.cache.row_offset[i])
        for t in range(T):
            assert torch.equal(s.cache.v[o + n + t].reshape(H, D), tok[t][2][i // L, i % L])
            ref = _attend(s, tok[t][0], i, n + t + 1)
            assert (outs[t][i // L, i % L].double() - ref).abs().max().item() <= TOL[dtype], (i, t)
        if again is not None:
            assert (again[i // L, i % L].double() - _attend(s, tok[0][0], i, n + T)).abs().max().item() <= TOL[dtype]


# (words whose lower bits would be a length, with bits set above them: anything but a length is refused)
@pytest.mark.parametrize("word", [0, -1, 2**31 - 1, -2**31, 0x7f7f7f7f, "full", "above", 30 + (1 << 20), 30 + (1 << 28), 5 + (3 << 28),
                                  5 + (3 << 26), 31 + (7 << 24), 31 + (100 << 24), 5 - 2**31, 30 - 2**31 + (1 << 26)])
@pytest.mark.parametrize("H", [1, 5, 64])
def test_a_segment_that_cannot_take_the_row_keeps_its_word(word, H):
    s, tok = _session(2, 1, H, 64, [40, 30], torch.bfloat16, 2)
    word = {"full": 32, "above": 33}.get(word, word)  # (of the second segment: 30 rows and two to come)
    s.cache.len[1] = word
    before = s.cache.k.clone()
    out = s.decode(*tok[0])
    torch.cuda.synchronize()
    assert s.status.tolist() == [0, api.DEV_CAPACITY]
    assert s.cache.len.tolist() == [41, word]
    assert (out[1] == 0).all()
    assert (out[0, 0].double() - _attend(s, tok[0][0], 0, 41)).abs().max().item() <= TOL[torch.bfloat16]
    o = int(s.cache.row_offset[1])
    assert torch.equal(s.cache.k[o:], before[o:])


@pytest.mark.parametrize("B,L,H,D,rows,dtype", [(1, 24, 16, 64, 90, torch.bfloat16), (1, 13, 57, 128, 33, torch.bfloat16), (3, 16, 8, 64, 31, torch.float32)])
def test_lengths_off_by_more_than_a_row_ahead_of_the_call(B, L, H, D, rows, dtype):
    """A CTA to a pair in one wave asks for a row more than the length read ahead has: right, a row short, and far off; to the last row of
    the cache."""
    T = 6
    lens = [rows + i % 3 for i in range(B * L)]
    s, tok = _session(B, L, H, D, lens, dtype, T)
    full = torch.tensor(lens, dtype=torch.int32, device="cuda")
    for t, back in enumerate((0, 0, 3, 0, 1, 0)):      # (the rows taken back are overwritten)
        if back:
            s.cache.len.sub_(back)
        n = [int(x) for x in (s.cache.len if t == 0 or back else last + 1).tolist()]
        last = torch.tensor(n, dtype=torch.int32, device="cuda")
        out = s.decode(*tok[t])
        if back == 0 and t % 2:
            continue                                   # (the next call right behind it)
        torch.cuda.synchronize()
        for i in (0, B * L // 2, B * L - 1):
            ref = _attend(s, tok[t][0], i, n[i] + 1)
            assert (out[i // L, i % L].double() - ref).abs().max().item() <= TOL[dtype], (t, i)
    assert s.cache.len.tolist() == [n + T - 4 for n in full.tolist()] and s.status.tolist() == [0] * B


@pytest.mark.parametrize("place", ["len", "row_offset"])
def test_a_plan_changed_just_before_the_call(place):
    """The rows that count are those of the plan after the kernel in front, whatever was there while it ran."""
    s, tok = _session(1, 2, 8, 64, [200, 90], torch.bfloat16, 4)
    for n in (200, 17, 131, 64):
        s.cache.len.copy_(torch.tensor([n, 90], dtype=torch.int32))
        if place == "row_offset":
            s.cache.row_offset[:2].copy_(torch.tensor([n % 3, 204 + n % 4]))
            s.cache.cap.copy_(torch.tensor([n + 1, 91], dtype=torch.int32))
        s.decode(*tok[0])      # changes the lengths while the next call is being set up
        out = s.decode(tok[1][0], None, None)
        torch.cuda.synchronize()
        for i, rows in enumerate((n + 1, 91)):
            ref = _attend(s, tok[1][0], i, rows)
            assert (out[0, i].double() - ref).abs().max().item() <= TOL[torch.bfloat16], (n, i)


# What the pair kernel leaves: more than 256 segments of few rows (row-split kernel, whose lanes, heads a warp, rows a unit and warps
# go by the row's bytes), pairs just too long for one wave (per-head kernel, tiles shared out where lengths differ), short ones of several waves.
@pytest.mark.parametrize("B,L,H,D,N,rows,dtype,d,kernel", [
    (9, 32, 16, 128, 40, 15, torch.bfloat16, 3, ROWS), (9, 32, 40, 128, 40, 15, torch.bfloat16, 3, ROWS), (9, 30, 64, 128, 24, 15, torch.bfloat16, 3, ROWS),
    (9, 32, 16, 64, 60, 30, torch.bfloat16, 3, ROWS), (9, 32, 32, 64, 60, 20, torch.bfloat16, 0, ROWS), (9, 32, 40, 64, 40, 15, torch.bfloat16, 3, ROWS),
    (9, 30, 64, 64, 40, 15, torch.bfloat16, 0, ROWS), (9, 32, 16, 128, 40, 12, torch.float32, 3, ROWS), (9, 32, 32, 128, 40, 12, torch.float32, 3, ROWS),
    (9, 30, 40, 128, 24, 8, torch.float32, 0, ROWS), (9, 32, 16, 64, 40, 12, torch.float32, 3, ROWS),
    (9, 32, 32, 64, 40, 12, torch.float32, 3, ROWS), (9, 30, 40, 64, 24, 9, torch.float32, 0, ROWS), (9, 30, 64, 64, 24, 9, torch.float32, 3, ROWS),
    (1, 32, 32, 128, 1500, 700, torch.bfloat16, 0, SHARED), (2, 18, 25, 128, 900, 660, torch.bfloat16, 0, SHARED), (2, 22, 30, 128, 800, 660, torch.bfloat16, 0, SHARED), (3, 32, 32, 64, 90, 40, torch.bfloat16, 0, HEADS),
    (2, 32, 32, 128, 90, 30, torch.float32, 0, HEADS),
])
def test_what_goes_elsewhere(B, L, H, D, N, rows, dtype, d, kernel):
    paths.test_decode_steps_match_the_oracle(B, L, H, D, N, rows, dtype, d, kernel)


@pytest.mark.parametrize("B,L,H,D,rows,dtype", [(1, 37, 16, 128, 60, torch.bfloat16), (1, 9, 8, 64, 500, torch.float32), (1, 16, 96, 128, 120, torch.bfloat16)])
def test_a_workspace_that_holds_anything(B, L, H, D, rows, dtype):
    """Counts are made anew over any words: over what another call's layout left, over all ones, and over the call's own."""
    T = 4
    lens = [rows + i % 5 for i in range(B * L)]
    a, tok = _session(B, L, H, D, lens, dtype, T)
    b, _ = _session(B, L, H, D, lens, dtype, T)
    for t in range(T):
        ref = a.decode(*tok[t]).clone()
        if t == 1:
            b.ws_decode.fill_(255)
        elif t == 2:        # a layer at a time: other places for the same segments
            b.cache.len.copy_(a.cache.len - 1)
            for l in range(L):
                b.decode(*tok[t], layer_begin=l, layer_end=l + 1)
            b.cache.len.copy_(a.cache.len - 1)
        got = b.decode(*tok[t])
        torch.cuda.synchronize()
        assert torch.equal(got, ref) and torch.equal(a.cache.len, b.cache.len), t
    assert a.cache.len.tolist() == [n + T for n in lens] and b.status.tolist() == [0] * B

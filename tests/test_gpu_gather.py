"""The compaction copy where its tiles of rows and groups of heads end: single heads, heads one below,
at and one above a group, a whole tile of rows and one more, several rounds of a CTA, and sources laid
out by head, by token and with a gap between rows.  Rows are moved, so every comparison is exact."""
import numpy as np
import pytest
import torch

from paper_2412_03409_b200 import api
from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu


def _source(layout, B, L, H, N, D, dtype, gen):
    if layout == "head":
        shape, order = (B, L, H, N, D), (0, 1, 2, 3, 4)
    elif layout == "token":
        shape, order = (B, L, N, H, D), (0, 1, 3, 2, 4)
    else:                                       # rows 16 bytes apart from their neighbours
        shape, order = (B, L, H, N, D + 16 // dtype.itemsize), (0, 1, 2, 3, 4)
    x = torch.randn(shape, generator=gen, device="cuda").to(dtype).permute(order)
    return x[..., :D]


@pytest.mark.parametrize("layout", ["head", "token", "gap"])
@pytest.mark.parametrize("dtype,D", [(torch.bfloat16, 64), (torch.bfloat16, 128), (torch.float32, 64),
                                     (torch.float32, 128)])
@pytest.mark.parametrize("B,L,H,N,keep", [
    (1, 1, 1, 1, 1.0), (2, 2, 7, 17, 0.5), (1, 3, 8, 16, 1.0), (2, 1, 9, 33, 1.0), (1, 2, 17, 129, 0.7),
    (1, 2, 40, 300, 0.2), (16, 64, 9, 210, 0.95)])
def test_rows_are_copied_exactly(B, L, H, N, keep, dtype, D, layout):
    if B * L * H * N * D * dtype.itemsize > 300 << 20:
        B //= 4 if dtype == torch.float32 else 2
    gen = torch.Generator(device="cuda").manual_seed(N * 100 + H)
    k, v = (_source(layout, B, L, H, N, D, dtype, gen) for _ in range(2))
    s = Session(B, L, H, D, N, dtype, torch.ones(L), decode_cap=3)
    s.cache.k.fill_(float("nan"))
    s.cache.v.fill_(float("nan"))
    scores = torch.rand((B, L, N), generator=gen, device="cuda")
    s.search(torch.full((B,), max(L, int(L * N * keep)), dtype=torch.int64), scores=scores)
    s.compact(k, v)
    torch.cuda.synchronize()
    assert s.status.cpu().tolist() == [0] * B
    lens, offs = s.cache.len.view(-1).tolist(), s.cache.row_offset.tolist()
    raw = torch.int16 if dtype == torch.bfloat16 else torch.int32
    for seg in range(B * L):
        b, l = divmod(seg, L)
        pos = s.order[b, l, :lens[seg]].sort().values.long()
        for src, dst in ((k, s.cache.k), (v, s.cache.v)):
            want = src[b, l][:, pos].transpose(0, 1).contiguous().view(raw)
            got = dst[offs[seg]:offs[seg + 1]]
            assert torch.equal(got[:lens[seg]].contiguous().view(raw), want), (seg, lens[seg])
            assert torch.isnan(got[lens[seg]:]).all()


def test_more_groups_of_heads_than_a_grid_holds():
    H, N, D = 8 * 65535 + 9, 3, 64
    shape = api.make_shape(1, 1, H, D, N, torch.bfloat16)
    gen = torch.Generator(device="cuda").manual_seed(3)
    k, v = (torch.randn((1, 1, H, N, D), generator=gen, device="cuda").bfloat16() for _ in range(2))
    cache = api.alloc_cache(shape, 2, 0, "cuda")
    order = torch.tensor([[[2, 0, 1]]], dtype=torch.int32, device="cuda")
    length = torch.tensor([[2]], dtype=torch.int32, device="cuda")
    kept = torch.empty((1, 1, N), dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.prefixkv_compact(shape, k, v, order, length, cache, status, None, kept=kept)
    torch.cuda.synchronize()
    assert status.tolist() == [0]
    for src, dst in ((k, cache.k), (v, cache.v)):
        assert torch.equal(dst[:2].view(2, H, D), src[0, 0][:, [0, 2]].transpose(0, 1))

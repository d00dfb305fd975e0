"""The compaction plan: lists, lengths and offsets at and around a word, a warp's words, a block's threads and the longest
prompt, with segments beyond the capacity and lengths out of range.  Compared exactly."""
import numpy as np
import pytest
import torch

from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("segments,N", [(1, 1), (3, 31), (3, 32), (2, 33), (40, 1023), (5, 1024), (5, 1025), (3, 1057), (2, 2048), (2, 2049),
                                        (1100, 40), (2, 16383), (2, 16384)])
@pytest.mark.parametrize("short", [False, True])
def test_plan(segments, N, short):
    rng = np.random.default_rng(N + segments)
    lens = rng.integers(1, N + 1, segments).astype(np.int32)
    lens[-1] = N
    bad = segments > 2
    if bad:
        lens[1] = N + 1                      # counted as none
    cap, used = 2, np.where(lens > N, 0, lens)
    total = int((used + cap).sum()) - (1 if short else 0)     # short: the last segment does not fit
    order = np.stack([rng.permutation(N) for _ in range(segments)]).astype(np.int32)
    s = Session(1, segments, 1, 64, N, torch.bfloat16, np.ones(segments), decode_cap=cap,
                max_budget_rows=total - cap * segments)
    s.order.copy_(torch.from_numpy(order[None]))
    s.len.copy_(torch.from_numpy(lens[None]))
    s.kept.fill_(-7)
    k = torch.randn(1, segments, 1, N, 64, device="cuda").bfloat16()
    s.compact(k, k)
    assert s.cache.total_cap_rows == total
    offs = np.concatenate([[0], np.cumsum(used + cap)])
    np.testing.assert_array_equal(s.cache.row_offset.cpu().numpy(), offs)
    fits = offs[1:] <= total
    assert fits.all() != short
    np.testing.assert_array_equal(s.cache.len.view(-1).cpu().numpy(), np.where(fits, used, 0))
    np.testing.assert_array_equal(s.cache.cap.view(-1).cpu().numpy(), np.where(fits, used + cap, 0))
    kept = s.kept[0].cpu().numpy()
    for i in range(segments):
        n = used[i] if fits[i] else 0
        np.testing.assert_array_equal(kept[i, :n], np.sort(order[i, :n]))
        assert (kept[i, n:] == -7).all()
    assert (s.status.item() != 0) == (bad or short)

"""The sort: runs merged, radix passes with any number of quads of warps, clusters of two and four.  Numbers of scores at and around
the runs' ends, the lines between the variants and shares that leave a cluster's last blocks without items, with many equal
scores and zeros.  Order and sums are compared exactly."""
import numpy as np
import pytest
import torch

from paper_2412_03409_b200.session import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["distinct", "few", "equal", "falling"])
@pytest.mark.parametrize("segments,N", [(1, n) for n in (1, 2, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 255, 256, 257, 384, 385, 640,
                                                         767, 768, 769, 1000, 1023, 1024, 1025, 1026, 1400, 2047, 2048, 2049, 3001,
                                                         4095, 4096, 4097)]
                         + [(33, 1030), (34, 1030), (34, 2049), (74, 1024), (75, 1024), (74, 2048), (74, 4096), (75, 2100), (148, 1000),
                            (149, 1000), (149, 768), (149, 769), (149, 1500), (149, 2817),
                            (75, 4500), (75, 6001), (34, 4097), (34, 6001), (74, 8192), (40, 9000), (75, 8193), (3, 16384), (40, 16384), (75, 16001)])
def test_order_and_sums(segments, N, kind):
    rng = np.random.default_rng(segments * 10000 + N)
    shape = (segments, N)
    scores = {"distinct": lambda: rng.random(shape), "few": lambda: rng.integers(0, 4, shape) / 8,
              "equal": lambda: np.full(shape, 0.25), "falling": lambda: np.broadcast_to(np.arange(N, 0, -1) / 64, shape)}[kind]()
    scores = np.ascontiguousarray(scores, np.float32)
    scores[:, 0] = 1.0  # (a layer has some weight)
    s = Session(1, segments, 1, 64, N, torch.float32, np.ones(segments), decode_cap=1)
    s.search(segments * N // 2 + segments, scores=torch.from_numpy(scores[None]).cuda())
    order, cum = s.order[0].cpu().numpy(), s.cum[0].cpu().numpy().view(np.uint64)
    assert s.status.item() == 0
    for i in range(segments):
        want = np.argsort(-scores[i], kind="stable")
        np.testing.assert_array_equal(order[i], want)
        weight = np.rint(scores[i][want].astype(np.float64) * 2.0**32).astype(np.uint64)
        np.testing.assert_array_equal(cum[i], np.cumsum(weight))

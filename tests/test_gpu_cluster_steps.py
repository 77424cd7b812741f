"""K-means iterations of two launches (few clusters): labels, cluster
hypervectors, accumulators and change counts against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle as orc
from _helpers import pack, unpack, words_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# clusters around the passes (8, 32), the end of the route (64); points around a
# block's 64 and the update's 16 parts of the runs; words of a part of a 16-word
# step and of a 32-word chunk; every point of a block in one cluster (K = 1);
# kept dims; one block an SM (9,728 points) and past it; past each line of the
# route (16,384 points, clusters x words, blocks x clusters x words, points x words)
@pytest.mark.parametrize("N,D,K,tp", [
    (1, 33, 1, (0.0, 1.0, 1)), (64, 128, 1, (0.0, 1.0, 1)), (65, 500, 8, (0.1, 0.8, 1)), (200, 513, 9, (0.0, 1.0, 3)),
    (1024, 1025, 26, (0.0, 1.0, 1)), (1025, 2100, 32, (0.0, 1.0, 2)), (1500, 4096, 33, (0.3, 1.0, 1)),
    (2500, 640, 64, (0.0, 1.0, 1)), (700, 640, 65, (0.0, 1.0, 1)), (9728, 1024, 3, (0.0, 1.0, 1)),
    (9729, 1030, 26, (0.0, 0.9, 1)), (16384, 96, 5, (0.0, 1.0, 1)), (16385, 96, 5, (0.0, 1.0, 1)),
    (9729, 4200, 2, (0.0, 1.0, 1)), (90, 40000, 9, (0.0, 1.0, 1)), (90, 40000, 10, (0.0, 1.0, 1)),
    (9700, 4096, 54, (0.0, 1.0, 1)), (9700, 4096, 53, (0.0, 1.0, 1)), (9700, 4096, 27, (0.0, 1.0, 1)),
    (9700, 4096, 26, (0.0, 1.0, 1)), (90, 40000, 8, (0.0, 1.0, 1)), (90, 40000, 7, (0.0, 1.0, 1)),
    (9728, 6100, 3, (0.0, 1.0, 1)), (9600, 6100, 3, (0.0, 1.0, 1))])
def test_iterations(N, D, K, tp):
    from paper_2606_26547_gb300 import hdc
    rng = np.random.default_rng(N + D + K)
    protos = rng.integers(0, 2, (K, D)).astype(np.uint8)
    bits = protos[rng.integers(0, K, N)] ^ (rng.random((N, D), dtype=np.float32) < 0.4).astype(np.uint8)
    init = bits[rng.integers(0, N, K)]       # equal initial clusters: ties, clusters without members
    H = torch.from_numpy(pack(bits, words_for(D)).view(np.int32)).cuda()
    first = torch.from_numpy(pack(init, words_for(D)).view(np.int32)).cuda()
    cfg = hdc.ApproxConfig(perf_start=tp[0], perf_end=tp[1], perf_stride=tp[2])
    lab, cls, acc, ch = hdc.cluster(H, D, first, 4, cfg)
    o_lab, o_cb, o_acc, o_ch = orc.kmeans(bits, init, 4, tp)
    assert np.array_equal(lab.cpu().numpy(), o_lab) and ch.cpu().numpy().tolist() == o_ch
    assert np.array_equal(acc.cpu().numpy(), o_acc)
    assert np.array_equal(unpack(cls.cpu().numpy().view(np.uint32), D), o_cb)

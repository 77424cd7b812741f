"""17 to 32 binary classes on the tensor cores: Hamming arg-min and the training
passes against the oracle, next to the routes on either side."""
import numpy as np
import pytest

import oracle as orc
from _helpers import pack, unpack

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# both ends of the route and one class past each; ragged tiles; part words; kept
# dims; rows past the route's 4,096 words
@pytest.mark.parametrize("C", [16, 17, 26, 32, 33])
@pytest.mark.parametrize("N,D,perf", [(1, 33, None), (129, 1000, (0.1, 0.9, 3)), (700, 4100, None), (300, 131073, None)])
def test_hamming(C, N, D, perf):
    from paper_2606_26547_gb300 import hdc
    rng = np.random.default_rng(C + N + D)
    q = rng.integers(0, 2, (N, D)).astype(np.uint8)
    c = rng.integers(0, 2, (C, D)).astype(np.uint8)
    c[C - 1] = c[1]
    q[0] = c[1]
    cfg = hdc.ApproxConfig(perf_start=perf[0], perf_end=perf[1], perf_stride=perf[2]) if perf else None
    dims = orc.kept_dims(D, *perf) if perf else orc.kept_dims(D)
    od = orc.hamming(orc.gather_cols(q, dims), orc.gather_cols(c, dims))
    Qt, Ct = T(pack(q).view(np.int32)), T(pack(c).view(np.int32))
    for use_ws in (True, False):
        labels, dd = hdc.hamming_argmin(Qt, Ct, D, cfg, dists=True, use_ws=use_ws)
        assert np.array_equal(dd.cpu().numpy(), od)
        assert np.array_equal(labels.cpu().numpy(), orc.argmin(od))


@pytest.mark.parametrize("C", [16, 17, 32, 33])
@pytest.mark.parametrize("N,D", [(300, 1000), (4001, 2100)])
def test_training(C, N, D):
    from paper_2606_26547_gb300 import hdc
    rng = np.random.default_rng(C + N)
    protos = rng.integers(0, 2, (C, D)).astype(np.uint8)
    y = rng.integers(0, C, N).astype(np.int32)
    bits = protos[y] ^ (rng.random((N, D), dtype=np.float32) < 0.47).astype(np.uint8)
    acc, cls, ups = hdc.train(T(pack(bits).view(np.int32)), T(y), D, C, 2)
    o_acc, o_ups = orc.train(bits, y, C, 2)
    assert np.array_equal(acc.cpu().numpy(), o_acc) and ups == o_ups
    assert np.array_equal(unpack(cls.cpu().numpy().view(np.uint32), D), orc.class_bits(o_acc))

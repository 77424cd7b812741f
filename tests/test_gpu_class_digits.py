"""b-bit class values as base-16 digit rows on the tensor cores: the cosine
classify of binary queries and the batched sweep, against the scores of the
definition in FP64 (integer dot products, one division), bit for bit."""
import numpy as np
import pytest

import oracle as orc
from _helpers import pack, unpack

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hdc():
    from paper_2606_26547_gb300 import hdc as m
    m.load()
    return m


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def classes(rng, C, D, scale):
    """Accumulators with an equal pair (a tie), a class of zeros (zero norm) and one constant class."""
    acc = np.rint(rng.standard_normal((C, D)) * scale).astype(np.int32)
    if C > 3:
        acc[C - 1] = acc[0]
        acc[2] = 0
    if C > 5:
        acc[4] = 3
    return acc


# P C around the padding of the class rows (16), one tile / two tiles a unit
# (128 rows) and the end of the route (256 rows); split dims; few and many rows
@pytest.mark.parametrize("bits,C", [(4, 1), (4, 16), (4, 17), (4, 129), (4, 256), (4, 257), (8, 5), (8, 64), (8, 65),
                                    (8, 128), (8, 129)])
@pytest.mark.parametrize("N,D", [(1, 300), (129, 2050), (5000, 1056)])
def test_cosine_scores(hdc, bits, C, N, D):
    rng = np.random.default_rng(bits * 1000 + C + N)
    F = 20
    X = rng.integers(-8, 8, (N, F)).astype(np.float32)
    Bt = rng.choice([-1.0, 1.0], (D, F)).astype(np.float32)
    acc = classes(rng, C, D, 40)
    cfg = hdc.ApproxConfig(enc="fp8", class_bits=bits, perf_start=0.02, perf_end=0.97, perf_stride=2)
    m = hdc.Model(T(Bt), cfg, acc=T(acc))
    labels, scores = hdc.classify(T(X), m, sims=True)
    only = hdc.classify(T(X), m)
    dims = orc.kept_dims(D, 0.02, 0.97, 2)
    q = unpack(hdc.encode(T(X), m).cpu().numpy().view(np.uint32), dims.size)
    v = orc.class_quantise(acc, bits)[:, dims].astype(np.int64)
    dot = (1 - 2 * q.astype(np.int64)) @ v.T
    nrm = np.sqrt((v * v).sum(1).astype(np.float64))
    ref = np.where(nrm == 0, 0.0, dot / np.where(nrm == 0, 1.0, nrm))
    assert np.array_equal(scores.cpu().numpy(), ref)
    assert np.array_equal(labels.cpu().numpy(), ref.argmax(1))
    assert torch.equal(labels, only)


# 26 classes x 4 entries x (1 + 1 + 2) digit rows: two passes; 8 digit rows a
# class (unquantised); 33 of those: the popcount route; large accumulators (the
# 64-bit class division)
@pytest.mark.parametrize("C,widths,scale", [(6, (1, 4, 8), 30), (26, (1, 4, 8), 30), (6, (0,), 2000), (32, (0, 8), 30),
                                            (33, (0,), 30), (10, (8, 4), 2e7)])
@pytest.mark.parametrize("N,D", [(1, 96), (300, 1056), (9000, 2100)])
def test_sweep_labels(hdc, C, widths, scale, N, D):
    rng = np.random.default_rng(C + N)
    entries = [(0.0, 1.0, 1), (0.1, 0.9, 2), (0.03, 1.0, 8), (0.0, 0.5, 32)]
    acc = classes(rng, C, D, scale)
    h = rng.integers(0, 2, (N, D)).astype(np.uint8)
    y = rng.integers(0, C, N).astype(np.int32)
    sw = hdc.Sweep(D, C, [e[2] for e in entries], widths, N, torch.device("cuda"), words_per_chunk=4, keep_labels=True,
                   starts=[e[0] for e in entries], ends=[e[1] for e in entries])
    correct = sw(T(pack(h).view(np.int32)), T(y), T(acc)).cpu().numpy()
    s = 1 - 2 * h.astype(np.int64)
    for j, b in enumerate(widths):
        full = acc.astype(np.int64) if b == 0 else np.where(acc < 0, -1, 1) if b == 1 else orc.class_quantise(acc, b)
        for i, e in enumerate(entries):
            dims = orc.kept_dims(D, *e)
            v = full[:, dims].astype(np.int64)
            dot = s[:, dims] @ v.T
            nrm = np.sqrt((v * v).sum(1).astype(np.float64))
            ref = (-dot).argmin(1) if b == 1 else np.where(nrm == 0, 0.0, dot / np.where(nrm == 0, 1.0, nrm)).argmax(1)
            assert np.array_equal(sw.labels[j, i].cpu().numpy(), ref), (b, e)
            assert correct[j, i] == int((ref == y).sum())

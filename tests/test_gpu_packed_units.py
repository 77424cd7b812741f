"""The tensor-core Hamming arg-min of packed rows where its work units change:
one or two 128-row tiles a unit, the dims of a unit split over a cluster of
CTAs, partial query chunks (1,024 dims) and 256-dim tiles, one or two distance
accumulators, with and without the class workspace."""
import numpy as np
import pytest

import oracle as orc
from _helpers import pack

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hdc():
    from paper_2606_26547_gb300 import hdc as m
    m.load()
    return m


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("N,D", [(1, 1024), (128, 1025), (129, 2047), (257, 8200), (1000, 3000), (9000, 1280),
                                 (19456, 520), (19457, 1100), (40000, 300)])
@pytest.mark.parametrize("C", [33, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("perf", [None, (0.03, 0.91, 3)])
def test_hamming_units(hdc, N, D, C, perf):
    rng = np.random.default_rng(N * 3 + D + C)
    W = hdc.words(D)
    q = rng.integers(0, 2 ** 32, (N, W), dtype=np.uint32)
    q[:, D // 32:] = 0                       # pad bits zero: whole words of random dims, the partial word all +1
    c = rng.integers(0, 2, (C, D)).astype(np.uint8)
    c[:, D // 32 * 32:] = 0
    c[C - 1] = c[0]                          # a tie across the class range
    rows = np.unique(np.r_[0, N - 1, rng.integers(0, N, 250)])
    qb = np.unpackbits(q[rows].view(np.uint8), axis=1, bitorder="little")[:, :D]
    dims = orc.kept_dims(D, *perf) if perf else orc.kept_dims(D)
    od = orc.hamming(orc.gather_cols(qb, dims), orc.gather_cols(c, dims))
    cfg = hdc.ApproxConfig(perf_start=perf[0], perf_end=perf[1], perf_stride=perf[2]) if perf else None
    for use_ws in (True, False):
        labels, dd = hdc.hamming_argmin(T(q.view(np.int32)), T(pack(c).view(np.int32)), D, cfg, dists=True,
                                        use_ws=use_ws)
        assert hdc.stream_status() == 0
        assert np.array_equal(dd.cpu().numpy()[rows].astype(np.int64), od)
        assert np.array_equal(labels.cpu().numpy()[rows], orc.argmin(od))
        # every row: its label is the lowest class of its smallest distance
        assert torch.equal(labels.long(), dd.argmin(1))


def unpack_pm1(words, D):
    bits = (words[:, :, None] >> torch.arange(32, device=words.device, dtype=torch.int32)) & 1
    return 1.0 - 2.0 * bits.reshape(words.shape[0], -1)[:, :D].float()


@pytest.mark.parametrize("N,D,C", [(30000, 4096, 256), (80000, 8192, 100), (80000, 4096, 97), (80000, 4096, 40)])
def test_hamming_units_every_row(hdc, N, D, C):
    """Several units a CTA while the distances are written: every distance of
    every row equals the +-1 product (sums of at most D ones: exact in FP32)."""
    g = torch.Generator(device="cuda").manual_seed(C)
    W = hdc.words(D)
    q, c = (torch.randint(-2 ** 31, 2 ** 31 - 1, (n, W), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
            for n in (N, C))
    k = unpack_pm1(c, D)
    ref = torch.cat([(D - unpack_pm1(q[r:r + 10000], D) @ k.t()) / 2 for r in range(0, N, 10000)]).to(torch.int32)
    for use_ws in (True, False, True, False):
        labels, dd = hdc.hamming_argmin(q, c, D, dists=True, use_ws=use_ws)
        assert torch.equal(dd, ref)
        assert torch.equal(labels.long(), ref.argmin(1))

"""Level-ID encoding of many queries (a query a thread, popcounts over feature
words) against the kernel of small batches, bit for bit, and the oracle."""
import numpy as np
import pytest

import oracle as orc
from _helpers import unpack

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SMALL = 1000     # rows of a call that stays on the other kernel, up to 19 slices of 1,024 dims


@pytest.fixture(scope="module")
def hdc():
    from paper_2606_26547_gb300 import hdc as m
    m.load()
    orc.build()
    return m


def make(hdc, F, D, L, ends, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    bit = lambda *shape: torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.uint8)
    lo = bit(D)
    hi = {"random": bit(D), "equal": lo, "opposite": 1 - lo}[ends]
    flip = torch.randint(1, L, (D,), generator=g, device="cuda", dtype=torch.int32)
    return (bit(F, D), lo, hi, flip), g


def check(hdc, m, X, unaligned=False):
    N = X.shape[0]
    if unaligned:
        out = torch.empty(N * m.W + 1, dtype=torch.int32, device="cuda")[1:].view(N, m.W)
    else:
        out = torch.empty((N, m.W), dtype=torch.int32, device="cuda")
    out.fill_(-1)
    hdc.levelid_encode(X, m, out=out)
    for r in list(range(0, N, SMALL))[-8:]:
        assert torch.equal(out[r:r + SMALL], hdc.levelid_encode(X[r:r + SMALL].contiguous(), m))
    for r in range(0, min(N, 4 * SMALL), SMALL):
        assert torch.equal(out[r:r + SMALL], hdc.levelid_encode(X[r:r + SMALL].contiguous(), m))
    return out


# feature words around the kernels' 8, 12, 16, 20 and 25 (256 .. 800 features), the
# route's lines in features with few and many levels; levels 2, 128 and past the planes (129);
# words of a part of a slice and several slices; level end points that agree
# everywhere, nowhere (past 600 dims of a slice they stay on the other kernel below 740 features); a ragged last warp and block; result rows off 16 bytes
@pytest.mark.parametrize("F,D,L,N,ends", [
    (192, 1024, 2, 30001, "random"), (193, 1024, 2, 30001, "random"), (225, 33, 3, 30000, "random"),
    (256, 1024, 32, 30011, "random"), (272, 1000, 5, 30011, "random"),
    (271, 1000, 5, 30011, "random"), (447, 1000, 33, 30011, "random"), (448, 1000, 33, 30011, "random"), (384, 1024, 16, 30005, "opposite"),
    (385, 1000, 32, 30005, "random"), (512, 1100, 100, 15005, "opposite"), (513, 1024, 128, 30300, "random"),
    (617, 1056, 128, 15100, "random"), (640, 1024, 127, 30300, "opposite"), (641, 2050, 64, 10001, "random"),
    (800, 1024, 128, 30033, "opposite"), (801, 1024, 128, 30033, "random"), (200, 1024, 129, 30033, "random"),
    (200, 1024, 20, 30033, "equal"), (617, 5000, 128, 6100, "random"), (200, 200000, 16, 160, "random"),
    (513, 600, 128, 30300, "opposite"), (513, 601, 128, 30300, "opposite"), (739, 1024, 8, 30300, "opposite"),
    (740, 1024, 8, 30300, "opposite"),
    (617, 1024, 128, 80000, "random")])
def test_many(hdc, F, D, L, N, ends):
    hvs, g = make(hdc, F, D, L, ends, F + D)
    m = hdc.LevelIdModel(*hvs, L, -2.0, 2.5)
    X = torch.randn((N, F), generator=g, device="cuda") * 1.5
    X[3, 0], X[5, F - 1], X[7, F // 2] = float("nan"), float("inf"), -float("inf")
    X[9] = 2.5
    if D < 6000:
        out = check(hdc, m, X, unaligned=F % 2 == 1)
        rows = np.r_[0:12, N - 5:N]
    else:
        out = torch.empty((N, m.W), dtype=torch.int32, device="cuda")
        hdc.levelid_encode(X, m, out=out)
        for r in (0, 60, N - 50):
            assert torch.equal(out[r:r + 50], hdc.levelid_encode(X[r:r + 50].contiguous(), m))
        rows = np.r_[0:12]
    ids, lo, hi, flip = (t.cpu().numpy() for t in hvs)
    pick = torch.as_tensor(rows, device="cuda")
    ref, _ = orc.levelid_encode(X[pick].cpu().numpy(), ids, lo, hi, flip, L, -2.0, 2.5, np.arange(D))
    assert np.array_equal(unpack(out[pick].cpu().numpy().view(np.uint32), D), ref)


# few queries: one and four a warp and the rows' kernel past them; features around
# the 16-row groups and the counter's planes (1,024); part words, several slices
@pytest.mark.parametrize("F,D,L,N", [(1, 33, 2, 1), (15, 100, 5, 8), (16, 1024, 7, 9), (35, 1030, 130, 300),
                                     (20, 100, 5, 1216), (20, 100, 5, 1217), (21, 130, 5, 4864), (20, 100, 5, 4865),
                                     (617, 1024, 128, 11), (1030, 200, 20, 3), (1030, 200, 20, 1300), (1500, 70, 60, 5)])
def test_few(hdc, F, D, L, N):
    hvs, g = make(hdc, F, D, L, "random", N + F)
    m = hdc.LevelIdModel(*hvs, L, -2.0, 2.5)
    X = torch.randn((N, F), generator=g, device="cuda") * 1.5
    X[0, 0], X[N - 1, F - 1], X[N // 2, F // 2] = float("nan"), float("inf"), -float("inf")
    out = hdc.levelid_encode(X, m)
    ids, lo, hi, flip = (t.cpu().numpy() for t in hvs)
    ref, _ = orc.levelid_encode(X.cpu().numpy(), ids, lo, hi, flip, L, -2.0, 2.5, np.arange(D))
    assert np.array_equal(unpack(out.cpu().numpy().view(np.uint32), D), ref)


def test_level_rows_that_switch_twice(hdc):
    """A level table of the caller's own: the slice with such a dim takes the other kernel."""
    F, D, L, N = 250, 3000, 16, 10100
    hvs, g = make(hdc, F, D, L, "random", 5)
    m = hdc.LevelIdModel(*hvs, L, -2.0, 2.5)
    X = torch.randn((N, F), generator=g, device="cuda")
    before = hdc.levelid_encode(X, m)
    W, off = m.W, (F * m.W * 4 + 255) // 256 * 256
    level = m.buf[off:off + L * W * 4].view(torch.int32).view(L, W)
    level[4, 40] ^= -1                                 # level 4 of the dims 1,280 .. 1,311
    out = check(hdc, m, X)
    assert torch.equal(out[:, :32], before[:, :32]) and not torch.equal(out[:, 40], before[:, 40])

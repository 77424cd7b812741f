"""Level-ID encoding of few queries around its load steps (256 features one query
a warp, 128 four a warp), partial last warps among them, against the oracle."""
import numpy as np
import pytest

import oracle as orc
from _helpers import unpack

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("F", [31, 33, 127, 128, 129, 225, 255, 256, 257, 385, 511, 513])
@pytest.mark.parametrize("N", [1, 10, 1217, 1219])     # one query a warp, then four
def test_against_oracle(F, N):
    from paper_2606_26547_gb300 import hdc
    orc.build()
    D, L = 100, 9
    g = torch.Generator(device="cuda").manual_seed(F + N)
    bit = lambda *shape: torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.uint8)
    hvs = bit(F, D), bit(D), bit(D), torch.randint(1, L, (D,), generator=g, device="cuda", dtype=torch.int32)
    m = hdc.LevelIdModel(*hvs, L, -2.0, 2.5)
    X = torch.randn((N, F), generator=g, device="cuda") * 1.5
    X[0, 0], X[N - 1, F - 1], X[N // 2, F // 2] = float("nan"), float("inf"), -float("inf")
    out = torch.full((N, m.W), -1, dtype=torch.int32, device="cuda")
    hdc.levelid_encode(X, m, out=out)
    ids, lo, hi, flip = (t.cpu().numpy() for t in hvs)
    ref, _ = orc.levelid_encode(X.cpu().numpy(), ids, lo, hi, flip, L, -2.0, 2.5, np.arange(D))
    assert np.array_equal(unpack(out.cpu().numpy().view(np.uint32), D), ref)

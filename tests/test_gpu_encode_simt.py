"""The FP32 encoder's tiles: 256- and 128-dim blocks, ragged rows, dims and K
slabs, aligned and unaligned query rows, against an exact integer product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hdc():
    from paper_2606_26547_gb300 import hdc as m
    m.load()
    return m


# 19 x 8 blocks of 256 dims fill 152 SMs once (the wide tile); a few blocks (the narrow one)
@pytest.mark.parametrize("N,D", [(2431, 2047), (2432, 2048), (2305, 1801), (1, 257), (129, 300), (700, 4100)])
@pytest.mark.parametrize("F", [1, 15, 16, 17, 20, 33])
def test_encode_fp32_exact(hdc, N, D, F):
    g = torch.Generator(device="cuda").manual_seed(N + F)
    X = torch.randint(-8, 8, (N, F), generator=g, device="cuda").float()
    Bt = torch.randint(-8, 8, (D, F), generator=g, device="cuda").float()
    H, S = hdc.encode(X, hdc.Model(Bt, hdc.ApproxConfig(enc="fp32")), scores=True)
    ref = (X.double() @ Bt.double().t())
    assert torch.equal(S.double(), ref)
    bits = (H[:, :, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    bits = bits.reshape(N, -1)
    assert torch.equal(bits[:, :D].bool(), ref < 0) and not bits[:, D:].any()
    # rows that start off a 16-byte boundary
    buf = torch.empty(N * F + 1, device="cuda")
    Xo = buf[1:].view(N, F).copy_(X)
    assert torch.equal(hdc.encode(Xo, hdc.Model(Bt, hdc.ApproxConfig(enc="fp32"))), H)

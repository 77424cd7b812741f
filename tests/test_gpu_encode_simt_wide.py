"""The FP32 encoder around the least features of its 256-dim tile, against an
exact integer product."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 19 x 8 blocks of 256 dims fill 152 SMs once; ragged rows, dims and K slabs
@pytest.mark.parametrize("N,D", [(2431, 2047), (2432, 2048), (2305, 1801), (129, 300)])
@pytest.mark.parametrize("F", [255, 256, 257, 260, 271, 272, 273])
def test_exact(N, D, F):
    from paper_2606_26547_gb300 import hdc
    g = torch.Generator(device="cuda").manual_seed(N + F)
    X = torch.randint(-8, 8, (N, F), generator=g, device="cuda").float()
    Bt = torch.randint(-8, 8, (D, F), generator=g, device="cuda").float()
    m = hdc.Model(Bt, hdc.ApproxConfig(enc="fp32"))
    H, S = hdc.encode(X, m, scores=True)
    ref = X.double() @ Bt.double().t()
    assert torch.equal(S.double(), ref)
    bits = (H[:, :, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    bits = bits.reshape(N, -1)
    assert torch.equal(bits[:, :D].bool(), ref < 0) and not bits[:, D:].any()
    buf = torch.empty(N * F + 1, device="cuda")   # rows that start off a 16-byte boundary
    assert torch.equal(hdc.encode(buf[1:].view(N, F).copy_(X), m), H)

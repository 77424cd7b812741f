"""Encodes whose query tiles split into dim ranges over the SMs: the packed words
and projections of a batch equal those of its rows in other batches, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# one dim tile, ragged ones, many; batches of one tile, some, about the SMs' number,
# one past it, several waves
@pytest.mark.parametrize("enc", ["bf16", "fp8"])
@pytest.mark.parametrize("F,D", [(100, 200), (617, 1000), (784, 5130)])
def test_batches_agree(F, D, enc):
    from paper_2606_26547_gb300 import hdc
    g = torch.Generator(device="cuda").manual_seed(F + D)
    Bt = (torch.randint(0, 2, (D, F), generator=g, device="cuda") * 2 - 1).float()
    X = torch.randn((47000, F), generator=g, device="cuda")
    m = hdc.Model(Bt, hdc.ApproxConfig(enc=enc))
    whole = hdc.encode(X, m)
    for n in (1, 128, 129, 1000, 9728, 19400, 19457, 30000):
        assert torch.equal(hdc.encode(X[:n].contiguous(), m), whole[:n])
    H, S = hdc.encode(X[:300].contiguous(), m, scores=True)
    H1, S1 = hdc.encode(X[299:300].contiguous(), m, scores=True)
    assert torch.equal(H, whole[:300]) and torch.equal(S[299:], S1) and torch.equal(H[299:], H1)

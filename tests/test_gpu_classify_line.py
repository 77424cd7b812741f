"""Small batches of 33..112 classes on both sides of the line between the fused
kernel and the encode + packed Hamming, against exact integer projections."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# nine and ten dim tiles of four E4M3 stages (one BF16 stage: two and more), with
# one query tile and with half as many as SMs
@pytest.mark.parametrize("enc,F", [("fp8", 512), ("bf16", 512), ("fp8", 100)])
@pytest.mark.parametrize("D", [900, 1728, 1729, 4000, 7500])
@pytest.mark.parametrize("N", [1, 129, 4000, 9728])
def test_exact(enc, F, D, N):
    from paper_2606_26547_gb300 import hdc
    C = 50
    g = torch.Generator(device="cuda").manual_seed(F + D)
    Bt = (torch.randint(0, 2, (D, F), generator=g, device="cuda") * 2 - 1).float()
    acc = torch.randint(-9, 10, (C, D), generator=g, device="cuda", dtype=torch.int32)
    acc[C - 1] = acc[1]          # a tie across the class range
    X = torch.randint(-8, 9, (N, F), generator=g, device="cuda").float()
    s = torch.where(X @ Bt.t() < 0, -1.0, 1.0)
    ref = ((D - s @ torch.where(acc < 0, -1.0, 1.0).t()) / 2).to(torch.int32)
    m = hdc.Model(Bt, hdc.ApproxConfig(enc=enc), acc=acc)
    labels, dists = hdc.classify(X, m, sims=True)
    assert torch.equal(dists, ref) and torch.equal(labels.long(), ref.argmin(1))
    assert torch.equal(hdc.classify(X, m), labels)

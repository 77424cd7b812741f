"""Small batches of 33..112 binary classes (encode split over the SMs, then the packed
Hamming) against the fused kernel of large ones: labels and distances bit for bit."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# both ends of the classes; stages around the route's 24 (784 features: 7 an E4M3 tile
# of 192 dims); rows of one tile, some, the route's last and the first past it
@pytest.mark.parametrize("enc", ["bf16", "fp8"])
@pytest.mark.parametrize("C,D", [(33, 570), (33, 1000), (112, 2050), (64, 2050)])
def test_small_batches_equal_large(C, D, enc):
    from paper_2606_26547_gb300 import hdc
    g = torch.Generator(device="cuda").manual_seed(C + D)
    F = 784
    Bt = (torch.randint(0, 2, (D, F), generator=g, device="cuda") * 2 - 1).float()
    acc = torch.randint(-9, 10, (C, D), generator=g, device="cuda", dtype=torch.int32)
    acc[C - 1] = acc[1]
    X = torch.randn((20500, F), generator=g, device="cuda")
    m = hdc.Model(Bt, hdc.ApproxConfig(enc=enc), acc=acc)
    labels, dists = hdc.classify(X, m, sims=True)
    for n in (1, 128, 129, 3000, 9728, 9729):
        lab, dd = hdc.classify(X[:n].contiguous(), m, sims=True)
        assert torch.equal(lab, labels[:n]) and torch.equal(dd, dists[:n])
        assert torch.equal(hdc.classify(X[:n].contiguous(), m), labels[:n])

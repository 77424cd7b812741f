"""Forms of the packed Hamming arg-min that the sizes choose between: one or two
row tiles a unit, a unit's dims over one to eight CTAs (few chunks of 1,024 dims,
uneven and even shares, batches at the limits of what is resident together)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def pm1(words, D):
    bits = (words[:, :, None] >> torch.arange(32, device=words.device, dtype=torch.int32)) & 1
    return 1.0 - 2.0 * bits.reshape(words.shape[0], -1)[:, :D].float()


@pytest.mark.parametrize("D", [1024, 2049, 4000, 8200, 20000, 60000, 131072])
@pytest.mark.parametrize("N", [100, 1792, 1793, 3000, 3585])
@pytest.mark.parametrize("C", [33, 64, 128, 129, 256])
def test_distances(N, D, C):
    from paper_2606_26547_gb300 import hdc
    g = torch.Generator(device="cuda").manual_seed(N + D + C)
    W = hdc.words(D)
    q, c = (torch.randint(-2 ** 31, 2 ** 31 - 1, (n, W), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
            for n in (N, C))
    for t in (q, c):
        t[:, D // 32:] = 0           # whole words of random dims, the rest +1
    k = pm1(c, D)
    ref = torch.cat([(D - pm1(q[r:r + 500], D) @ k.t()) / 2 for r in range(0, N, 500)]).to(torch.int32)   # exact below 2^24
    for use_ws in (True, False):
        labels, dd = hdc.hamming_argmin(q, c, D, dists=True, use_ws=use_ws)
        assert torch.equal(dd, ref) and torch.equal(labels.long(), ref.argmin(1))
        assert torch.equal(hdc.hamming_argmin(q, c, D, use_ws=use_ws), labels)


# distances of few rows and of class groups of one or two leave as single words
@pytest.mark.parametrize("N", [1, 31, 33, 64, 65])
@pytest.mark.parametrize("C", [33, 34, 35, 65, 67, 161, 255])
def test_distances_of_few_rows(N, C):
    test_distances(N, 1000, C)

"""17 to 32 binary classes on both sides of the line between the popcount and the
packed tensor-core kernel: distances against the +-1 product, a retraining epoch
against one of the same rows in a larger call's route."""
import numpy as np
import pytest

import oracle as orc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def rows(n, D, seed):
    from paper_2606_26547_gb300 import hdc
    g = torch.Generator(device="cuda").manual_seed(seed)
    h = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, hdc.words(D)), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    h[:, D // 32:] = 0      # whole words of random dims, the rest +1
    return h


def pm1(words, D, keep):
    bits = (words[:, :, None] >> torch.arange(32, device=words.device, dtype=torch.int32)) & 1
    return (1.0 - 2.0 * bits.reshape(words.shape[0], -1)[:, :D].float()) * keep


# 64 and 68 words; 260,000 words of rows and more; the narrowest rows
@pytest.mark.parametrize("N,D", [(1, 2048), (1, 2049), (300, 2049), (4062, 2048), (4063, 2048), (4063, 2040), (65000, 100),
                                 (65001, 100), (16250, 500), (16251, 500)])
@pytest.mark.parametrize("C", [17, 32])
@pytest.mark.parametrize("perf", [None, (0.1, 0.9, 3)])
def test_hamming(N, D, C, perf):
    from paper_2606_26547_gb300 import hdc
    q, c = rows(N, D, N + D), rows(C, D, C)
    c[C - 1] = c[1]          # a tie across the class range
    keep = torch.ones(D, device="cuda")
    cfg = None
    if perf:
        keep.zero_()
        keep[torch.from_numpy(np.asarray(orc.kept_dims(D, *perf), dtype=np.int64)).cuda()] = 1.0
        cfg = hdc.ApproxConfig(perf_start=perf[0], perf_end=perf[1], perf_stride=perf[2])
    ref = ((keep.sum() - pm1(q, D, keep) @ pm1(c, D, 1.0).t()) / 2).to(torch.int32)
    labels, dd = hdc.hamming_argmin(q, c, D, cfg, dists=True)
    assert torch.equal(dd, ref) and torch.equal(labels.long(), ref.argmin(1))
    assert torch.equal(hdc.hamming_argmin(q, c, D, cfg), labels)


# 32 and 36 words with the classes in scratch; both sides of 260,000 words
@pytest.mark.parametrize("N,D", [(500, 1024), (500, 1025), (8125, 1024), (8126, 1024)])
@pytest.mark.parametrize("C", [17, 32])
def test_epoch(N, D, C):
    from paper_2606_26547_gb300 import hdc
    H = rows(N, D, N + C)
    y = torch.arange(N, device="cuda", dtype=torch.int32) % C
    cls, acc = rows(C, D, 5), torch.zeros((C, D), dtype=torch.int32, device="cuda")
    pred = hdc.hamming_argmin(H, cls, D)
    wrong = (pred != y).float()
    s = pm1(H, D, 1.0) * wrong[:, None]
    ref = torch.zeros((C, D), device="cuda").index_add_(0, y.long(), s).index_add_(0, pred.long(), s, alpha=-1)
    ups = torch.zeros(1, dtype=torch.int32, device="cuda")
    hdc.train_epoch(H, y, D, C, 1, acc, cls, n_updates=ups)
    assert int(ups) == int(wrong.sum()) and torch.equal(acc, ref.to(torch.int32))

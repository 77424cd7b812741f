"""More rows than one launch of the packed tensor-core kernel takes (row
coordinates of 32 bits): every row is a class's or zero, the marked ones around
the first launch's last row and at both ends."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, LAST, D = 2 ** 31 + 300, 0x7fffff00, 128
MARKS = [0, 7, LAST - 2, LAST - 1, LAST, LAST + 1, 2 ** 31 - 1, 2 ** 31, N - 1]


@pytest.fixture(scope="module")
def rows():
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB")
    yield torch.zeros((N, 4), dtype=torch.int32, device="cuda")
    torch.cuda.empty_cache()


def mark(rows, cls):
    """Rows MARKS become class rows; their classes."""
    want = [3 * i % cls.shape[0] for i in range(len(MARKS))]
    for r, c in zip(MARKS, want):
        rows[r] = cls[c]
    return want


def class_rows(C):
    g = torch.Generator(device="cuda").manual_seed(C)
    return torch.randint(-2 ** 31, 2 ** 31 - 1, (C, 4), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)


@pytest.mark.parametrize("C,use_ws", [(20, False), (40, False), (40, True), (200, True)])
def test_hamming(rows, C, use_ws):
    from paper_2606_26547_gb300 import hdc
    cls = class_rows(C)
    want = mark(rows, cls)
    zero = int(hdc.hamming_argmin(torch.zeros((1, 4), dtype=torch.int32, device="cuda"), cls, D)[0])
    labels = hdc.hamming_argmin(rows, cls, D, use_ws=use_ws)
    assert labels[MARKS].tolist() == want
    labels[MARKS] = zero
    assert bool((labels == zero).all()) and hdc.stream_status() == 0


def test_sweep(rows):
    from paper_2606_26547_gb300 import hdc
    C = 9
    cls = class_rows(C)
    want = mark(rows, cls)
    bits = (cls[:, :, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    acc = (1 - 2 * bits.reshape(C, D)).to(torch.int32) * 5
    zero = int(hdc.hamming_argmin(torch.zeros((1, 4), dtype=torch.int32, device="cuda"), cls, D)[0])
    y = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    y[MARKS] = torch.tensor(want, dtype=torch.int32, device="cuda")
    sw = hdc.Sweep(D, C, [1], [1, 4], N, torch.device("cuda"), keep_labels=True)   # +-5 alike: both widths give the sign's order
    assert sw(rows, y, acc).tolist() == [[len(MARKS)], [len(MARKS)]]
    for k in range(2):
        labels = sw.labels[k, 0]
        assert labels[MARKS].tolist() == want
        labels[MARKS] = zero
        assert bool((labels == zero).all())
    assert hdc.stream_status() == 0


def test_cosine():
    from paper_2606_26547_gb300 import hdc
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB")
    g = torch.Generator(device="cuda").manual_seed(1)
    Bt = (torch.randint(0, 2, (D, 1), generator=g, device="cuda") * 2 - 1).float()
    acc = torch.randint(-60, 61, (7, D), generator=g, device="cuda", dtype=torch.int32)
    m = hdc.Model(Bt, hdc.ApproxConfig(enc="fp32", class_bits=4), acc=acc)
    plus, minus = hdc.classify(torch.tensor([[1.0], [-1.0]], device="cuda"), m).tolist()
    assert plus != minus
    X = torch.ones((N, 1), device="cuda")
    X[MARKS] = -1.0
    labels = hdc.classify(X, m)
    assert labels[MARKS].tolist() == [minus] * len(MARKS)
    labels[MARKS] = plus
    assert bool((labels == plus).all()) and hdc.stream_status() == 0

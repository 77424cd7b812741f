"""Calls whose kernels start while their predecessor ends (programmatic
launches), each followed at once by a reader of what it wrote: captured in a
graph, and on two streams from two host threads at a time, against the same
calls alone on one stream, which the oracle's tests cover."""
import threading

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def rows(n, D, g):
    from paper_2606_26547_gb300 import hdc
    h = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, hdc.words(D)), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    h[:, D // 32:] = 0      # whole words of random dims, the rest +1
    return h


def training(C):
    """Bundling, two epochs, and the arg-min of their class rows without and with a workspace."""
    from paper_2606_26547_gb300 import hdc
    N, D = 5000, 2080

    def make(g):
        H, y = rows(N, D, g), torch.randint(0, C, (N,), generator=g, device="cuda", dtype=torch.int32)
        acc, cls = torch.zeros((C, D), dtype=torch.int32, device="cuda"), torch.zeros((C, hdc.words(D)), dtype=torch.int32, device="cuda")
        ups = torch.zeros(2, dtype=torch.int32, device="cuda")

        def call():
            hdc.train_epoch(H, y, D, C, 0, acc, cls)
            out = []
            for e in range(2):
                hdc.train_epoch(H, y, D, C, 1, acc, cls, n_updates=ups[e:e + 1])
                out += hdc.hamming_argmin(H, cls, D, dists=True, use_ws=False)
            out += hdc.hamming_argmin(H, cls, D, dists=True)
            return out + [acc, cls, ups]
        return call
    return make


def clustering(N, K):
    from paper_2606_26547_gb300 import hdc

    def make(g):
        H = rows(N, 1056, g)
        return lambda: list(hdc.cluster(H, 1056, H[:K].clone(), 3))
    return make


def classify(N, C, enc, bits, float_query=False):
    from paper_2606_26547_gb300 import hdc
    F, D = 128, 2050

    def make(g):
        Bt = (torch.randint(0, 2, (D, F), generator=g, device="cuda") * 2 - 1).float()
        acc = torch.randint(-60, 61, (C, D), generator=g, device="cuda", dtype=torch.int32)
        m = hdc.Model(Bt, hdc.ApproxConfig(enc=enc, class_bits=bits, float_query=float_query), acc=acc)
        X = torch.randn((N, F), generator=g, device="cuda")
        return lambda: [hdc.classify(X, m), *hdc.classify(X, m, sims=True)]
    return make


def sweep(N, C):
    from paper_2606_26547_gb300 import hdc
    D = 2080

    def make(g):
        H, y = rows(N, D, g), torch.randint(0, C, (N,), generator=g, device="cuda", dtype=torch.int32)
        acc = torch.randint(-60, 61, (C, D), generator=g, device="cuda", dtype=torch.int32)
        sw = hdc.Sweep(D, C, [1, 2, 8], [1, 4, 8], N, torch.device("cuda"), keep_labels=True)
        return lambda: [sw(H, y, acc), sw.labels]
    return make


def levelid(N, L):
    from paper_2606_26547_gb300 import hdc
    F, D = 500, 1056

    def make(g):
        bit = lambda *s: torch.randint(0, 2, s, generator=g, device="cuda", dtype=torch.uint8)
        m = hdc.LevelIdModel(bit(F, D), bit(D), bit(D), torch.randint(1, L, (D,), generator=g, device="cuda", dtype=torch.int32),
                             L, -2.0, 2.0)
        X = torch.randn((N, F), generator=g, device="cuda")

        def call():
            H = hdc.levelid_encode(X, m)
            return [H, hdc.hamming_argmin(H, H[:20].clone(), D)]
        return call
    return make


CALLS = {
    "train_10": lambda: training(10), "train_26": lambda: training(26), "train_100": lambda: training(100),
    "train_400": lambda: training(400), "cluster_few": lambda: clustering(3000, 26), "cluster_many": lambda: clustering(20000, 40),
    "binary_fp8": lambda: classify(700, 10, "fp8", 1), "binary_100": lambda: classify(700, 100, "bf16", 1),
    "binary_200": lambda: classify(700, 200, "fp8", 1), "cosine_8": lambda: classify(5000, 26, "fp8", 8),
    "float_4": lambda: classify(5000, 26, "bf16", 4, True), "sweep": lambda: sweep(3000, 26),
    "levelid_few": lambda: levelid(9, 100), "levelid_many": lambda: levelid(20000, 100),
}


@pytest.mark.parametrize("name", CALLS)
def test_captured(name):
    from paper_2606_26547_gb300 import hdc
    call = CALLS[name]()(torch.Generator(device="cuda").manual_seed(3))
    ref = [t.clone() for t in call()]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call()
    for _ in range(3):
        for t in out:
            t.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        assert hdc.stream_status() == 0
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


@pytest.mark.parametrize("first,second", [("train_10", "train_26"), ("train_100", "binary_100"), ("cluster_few", "sweep"),
                                          ("cosine_8", "binary_200"), ("float_4", "cluster_many"), ("binary_fp8", "levelid_many"),
                                          ("train_400", "levelid_few")])
def test_two_streams(first, second):
    from paper_2606_26547_gb300 import hdc
    calls = [CALLS[n]()(torch.Generator(device="cuda").manual_seed(k)) for k, n in enumerate((first, second))]
    refs = [[t.clone() for t in c()] for c in calls]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(10):
                    out = calls[k]()
                    if not all(torch.equal(a, b) for a, b in zip(out, refs[k])):
                        bad.append((k, "differs"))
                s.synchronize()
        except Exception as e:   # a failed call must not pass for a finished thread
            bad.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad and hdc.stream_status() == 0

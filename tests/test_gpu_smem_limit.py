"""Two host threads in one kernel with different shared-memory sizes: a call must
not lower the limit under the other's launches (a launch past it is refused)."""
import threading

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def rows(n, W, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-2 ** 31, 2 ** 31 - 1, (n, W), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)


def cluster(D, iters):          # 61 and 157 KB
    from paper_2606_26547_gb300 import hdc
    H = rows(64, hdc.words(D), D)
    return lambda: hdc.cluster(H, hdc.words(D) * 32, H[:3].clone(), iters)


def hamming(C):                 # one 128-row tile a unit: class rings of different sizes
    from paper_2606_26547_gb300 import hdc
    Q, K = rows(64, 64, 1), rows(C, 64, C)
    return lambda: hdc.hamming_argmin(Q, K, 2048)


def encode(F):                  # the quantiser's row slots
    from paper_2606_26547_gb300 import hdc
    m = hdc.Model(torch.ones((64, F), device="cuda"), hdc.ApproxConfig(enc="bf16"))
    X = torch.ones((9, F), device="cuda")
    return lambda: hdc.encode(X, m)


def classify(C, float_query=False):
    from paper_2606_26547_gb300 import hdc
    cfg = hdc.ApproxConfig(enc="bf16", class_bits=4 if float_query else 1, float_query=float_query)
    acc = torch.ones((C, 64), dtype=torch.int32, device="cuda")
    m = hdc.Model(torch.ones((64, 64), device="cuda"), cfg, acc=acc)
    X = torch.ones((300, 64), device="cuda")
    return lambda: hdc.classify(X, m)


def cosine(C):                  # past the digit rows' 256: the popcount form
    from paper_2606_26547_gb300 import hdc
    acc = torch.ones((C, 640), dtype=torch.int32, device="cuda")
    m = hdc.Model(torch.ones((640, 64), device="cuda"), hdc.ApproxConfig(enc="bf16", class_bits=8), acc=acc)
    X = torch.ones((300, 64), device="cuda")
    return lambda: hdc.classify(X, m)


def levelid(F, N):
    from paper_2606_26547_gb300 import hdc
    z = torch.zeros(64, dtype=torch.uint8, device="cuda")
    m = hdc.LevelIdModel(torch.zeros((F, 64), dtype=torch.uint8, device="cuda"), z, z, torch.ones(64, dtype=torch.int32, device="cuda"),
                         4, -1.0, 1.0)
    X = torch.zeros((N, F), device="cuda")
    return lambda: hdc.levelid_encode(X, m)


def sweep(C):                   # over 256 digit rows a configuration: the popcount form
    from paper_2606_26547_gb300 import hdc
    H, y = rows(100, 4, 1), torch.zeros(100, dtype=torch.int32, device="cuda")
    acc = torch.ones((C, 128), dtype=torch.int32, device="cuda")
    sw = hdc.Sweep(128, C, [1], [0], 100, torch.device("cuda"), 64, 4)
    return lambda: sw(H, y, acc)


PAIRS = {
    "cluster": lambda: (cluster(16000, 300), cluster(6000, 1)), "hamming": lambda: (hamming(256), hamming(144)),
    "quantiser": lambda: (encode(1500), encode(800)), "quantiser_span": lambda: (encode(1501), encode(801)),
    "binary": lambda: (classify(112), classify(40)), "float": lambda: (classify(128, True), classify(36, True)),
    "cosine": lambda: (cosine(250), cosine(140)), "levelid": lambda: (levelid(1400, 5000), levelid(1100, 5000)),
    "levelid_few": lambda: (levelid(1400, 3), levelid(1100, 3)), "sweep": lambda: (sweep(200), sweep(110)),
}


@pytest.mark.parametrize("name", PAIRS)
def test_two_threads(name):
    calls, bad, done = PAIRS[name](), [], threading.Event()
    for c in calls:
        c()
    torch.cuda.synchronize()

    def work(k):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                n = 0
                while not bad and (n < (40 if name == "cluster" else 3000) if k == 0 else not done.is_set()):
                    calls[k]()
                    n += 1
                s.synchronize()
        except Exception as e:
            bad.append(repr(e))
        finally:
            done.set()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad

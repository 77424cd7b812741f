"""Timed cases of the library: the calls that its users' programs make, over the range of sizes.

Every case is one pass through the public binding (paper_2606_26547_gb300.hdc) on device tensors, with what
a program keeps between calls (the prepared model, workspaces, output buffers) made beforehand.  Sizes are those of
the repository's workloads (synth.WORKLOADS), of its serving mix and of the paper's applications.  Kinds:

  classify  FP32 queries -> nearest class with the distances or scores (hdc.classify)
  encode    FP32 rows -> packed hypervectors (hdc.encode)
  train     bundling and retraining epochs over packed samples (hdc.train_epoch)
  hamming   Hamming arg-min of packed hypervectors (hdc.hamming_argmin)
  sweep     class width x perforation configurations of one trained model (hdc.Sweep)
  cluster   K-means over packed hypervectors (hdc.cluster)
  levelid   FP32 rows -> packed hypervectors by the Level-ID encoder (hdc.levelid_encode)

Queries and training rows are Gaussian mixtures (centroids N(0, 1), within-class deviation `sigma`), base
hypermatrices N(0, 1); packed samples are random prototypes with every bit flipped with probability `flip`.
"""
import math

import torch

from paper_2606_26547_gb300 import hdc

# kept configuration fields of a classify / encode / hamming case, with their defaults
_CONFIG = {"enc": "fp32", "start": 0.0, "end": 1.0, "stride": 1, "bits": 1, "float_query": False}
_TRAIN_ROWS = 40   # training rows per class behind a classify case's class accumulators


def listed():
    return [
        # serving, the smallest request: one row against a resident 10-class model
        {"name": "serve_one", "kind": "classify", "F": 784, "D": 8192, "C": 10, "N": 1, "sigma": 0.6, "enc": "bf16"},
        # serving, one batch of queued requests (rows of 561 floats: no 16-byte alignment), ragged
        {"name": "serve_batch", "kind": "classify", "F": 561, "D": 4096, "C": 6, "N": 2357, "sigma": 8.3,
         "enc": "bf16"},
        # the approximated classifier at full load: E4M3, every second dimension, binary classes
        {"name": "bulk_binary", "kind": "classify", "F": 784, "D": 10000, "C": 10, "N": 1048576, "sigma": 0.6,
         "enc": "fp8", "stride": 2},
        # many classes
        {"name": "many_classes", "kind": "classify", "F": 1024, "D": 16384, "C": 100, "N": 131149, "sigma": 0.6,
         "enc": "fp8", "stride": 2},
        # 8-bit class hypervectors with the cosine score: the widest class width of the tuner's space
        {"name": "cosine_8bit", "kind": "classify", "F": 617, "D": 2048, "C": 26, "N": 100003, "sigma": 5.2,
         "enc": "fp8", "bits": 8},
        # float query hypervectors: the paper's unapproximated similarity
        {"name": "float_query", "kind": "classify", "F": 784, "D": 10000, "C": 10, "N": 262144, "sigma": 0.6,
         "enc": "fp8", "stride": 2, "bits": 8, "float_query": True},
        # the plain exact form: a training set encoded in FP32 at the full dimensionality
        {"name": "encode_exact", "kind": "encode", "F": 561, "D": 10000, "N": 10000, "sigma": 8.3, "enc": "fp32"},
        # bundling and two retraining epochs
        {"name": "train", "kind": "train", "N": 60000, "D": 10000, "C": 10, "epochs": 2, "flip": 0.48},
        # nearest of 100 packed class hypervectors
        {"name": "hamming_100", "kind": "hamming", "N": 100000, "D": 16384, "C": 100, "flip": 0.4},
        # one round of the tuner: 4 strides x 3 class widths of one model on the validation set
        {"name": "sweep", "kind": "sweep", "N": 10000, "D": 10000, "C": 6, "flip": 0.45, "strides": "1,2,4,8",
         "starts": "0,0,0,0", "ends": "1,1,1,1", "widths": "1,4,8"},
        # HD-Clustering, 20 iterations
        {"name": "cluster", "kind": "cluster", "N": 7797, "D": 1024, "C": 26, "epochs": 20, "flip": 0.44},
        # Level-ID encoding
        {"name": "levelid", "kind": "levelid", "F": 617, "D": 1024, "N": 262144, "L": 128, "sigma": 1.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _perforation(rng):
    """Most configurations keep every dim or every 2nd, 4th, 8th; some cut the ends."""
    c = {"stride": rng.choice((1, 1, 2, 2, 4, 8, 3))}
    if rng.random() < 0.3:
        c["start"] = rng.choice((0.0, 0.05, 0.1, 0.36))
        c["end"] = rng.choice((0.5, 0.84, 0.92, 0.97))
    return c


def draw(rng):
    kind = rng.choice(("classify",) * 6 + ("encode", "train", "train", "hamming", "hamming", "sweep", "cluster",
                                           "levelid"))
    if kind == "classify":
        c = {"kind": kind, "F": rng.choice((561, 617, 784, 1024, rng.randint(64, 1024))), "D": _log(rng, 1024, 16384),
             "C": rng.choice((6, 10, 26, 100, _log(rng, 2, 256))), "N": _log(rng, 1, 1 << 20),
             "sigma": rng.choice((0.6, 5.2, 8.3)), "enc": rng.choice(("bf16", "fp8", "fp8")), **_perforation(rng)}
        c["bits"] = rng.choice((1, 1, 1, 4, 8))
        c["float_query"] = c["bits"] > 1 and rng.random() < 0.5
        most = 4.0e12 if c["bits"] == 1 else 2.0e12   # operations, under the largest listed case's
        if c["bits"] > 1 and not c["float_query"]:
            c["C"] = min(c["C"], 26)
            most = min(most, 2.0e11)
        c["N"] = max(1, min(c["N"], int(most / (2.0 * c["F"] * c["D"]))))
        return c
    if kind == "encode":
        c = {"kind": kind, "F": rng.choice((561, 617, 784, rng.randint(64, 1024))), "D": _log(rng, 1024, 10000),
             "N": _log(rng, 1, 60000), "sigma": rng.choice((0.6, 5.2, 8.3)),
             "enc": rng.choice(("fp32", "bf16", "fp8")), **_perforation(rng)}
        most = 1.1e11 if c["enc"] == "fp32" else 1.0e12
        c["N"] = max(1, min(c["N"], int(most / (2.0 * c["F"] * c["D"]))))
        return c
    if kind == "train":
        return {"kind": kind, "N": _log(rng, 500, 100000), "D": _log(rng, 1024, 16384),
                "C": rng.choice((6, 10, 26, 100, rng.randint(2, 128))), "epochs": rng.randint(0, 3),
                "flip": rng.choice((0.4, 0.48))}
    if kind == "hamming":
        return {"kind": kind, "N": _log(rng, 1, 200000), "D": _log(rng, 1024, 16384),
                "C": rng.choice((6, 10, 26, 100, _log(rng, 2, 256))), "flip": 0.4, **_perforation(rng)}
    if kind == "sweep":
        n = rng.randint(1, 4)
        cut = rng.random() < 0.5
        return {"kind": kind, "N": _log(rng, 500, 10000), "D": _log(rng, 1024, 10000), "C": rng.choice((6, 10, 26)),
                "flip": 0.45, "strides": ",".join(str(rng.choice((1, 2, 4, 8))) for _ in range(n)),
                "starts": ",".join(str(rng.randint(0, 30) / 100 if cut else 0) for _ in range(n)),
                "ends": ",".join(str(rng.randint(50, 100) / 100 if cut else 1) for _ in range(n)),
                "widths": rng.choice(("1,4,8", "1,4,8", "4,8", "1", "8"))}
    if kind == "cluster":
        return {"kind": kind, "N": _log(rng, 500, 8000), "D": _log(rng, 512, 4096), "C": rng.randint(4, 64),
                "epochs": rng.randint(3, 20), "flip": 0.44}
    F, D = rng.choice((561, 617, rng.randint(32, 784))), _log(rng, 512, 10000)
    most = 262144.0 * 617 * 1024
    return {"kind": kind, "F": F, "D": D, "N": max(1, min(_log(rng, 1, 262144), int(most / (F * D)))),
            "L": rng.choice((16, 32, 64, 128)), "sigma": 1.0}


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + stream)


def _mixture(n, F, C, sigma, seed, stream):
    """n rows of the C-class mixture of `seed` (labels n mod C), FP32."""
    mu = torch.randn((C, F), generator=_gen(seed, 0), device="cuda")
    y = torch.arange(n, device="cuda") % C
    x = torch.randn((n, F), generator=_gen(seed, stream), device="cuda")
    x.mul_(sigma)
    for r in range(0, n, 1 << 16):   # the centroids added in slices: no second N x F array
        x[r:r + (1 << 16)] += mu[y[r:r + (1 << 16)]]
    return x, y


def _base(D, F, seed):
    return torch.randn((D, F), generator=_gen(seed, 1), device="cuda")


def _class_sums(Bt, C, sigma, seed):
    """Class accumulators C x D (int32): the bundled signs of _TRAIN_ROWS training rows of every class."""
    x, y = _mixture(C * _TRAIN_ROWS, Bt.shape[1], C, sigma, seed, 2)
    h = torch.where(x @ Bt.t() < 0, -1.0, 1.0)
    acc = torch.zeros((C, Bt.shape[0]), device="cuda")
    return acc.index_add_(0, y, h).to(torch.int32)


def _pack(bits, W):
    """Rows of booleans -> W int32 words a row, zero past the last dim."""
    n, D = bits.shape
    pad = torch.zeros((n, W * 32), dtype=torch.bool, device=bits.device)
    pad[:, :D] = bits
    shifts = torch.arange(32, device=bits.device, dtype=torch.int64)
    return (pad.view(n, W, 32).to(torch.int64) << shifts).sum(-1).to(torch.int32)


def _samples(n, D, C, flip, seed):
    """Packed samples around C random prototypes, their labels (int32) and the prototypes (packed)."""
    W = (D + 127) // 128 * 4
    protos = torch.rand((C, D), generator=_gen(seed, 3), device="cuda") < 0.5
    y = torch.randint(0, C, (n,), generator=_gen(seed, 4), device="cuda")
    g = _gen(seed, 5)
    H = torch.empty((n, W), dtype=torch.int32, device="cuda")
    step = max(1, (1 << 27) // D)
    for r in range(0, n, step):
        k = min(step, n - r)
        H[r:r + k] = _pack(protos[y[r:r + k]] ^ (torch.rand((k, D), generator=g, device="cuda") < flip), W)
    return H, y.to(torch.int32), _pack(protos, W)


def _config(case):
    c = {k: case.get(k, v) for k, v in _CONFIG.items()}
    return hdc.ApproxConfig(enc=c["enc"], perf_start=c["start"], perf_end=c["end"], perf_stride=c["stride"],
                            class_bits=c["bits"], float_query=c["float_query"])


def _numbers(text, kind):
    return [kind(v) for v in text.split(",")]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("classify", "encode"):
        Bt = _base(case["D"], case["F"], seed)
        C = case.get("C", 10)
        s["X"], _ = _mixture(case["N"], case["F"], C, case["sigma"], seed, 6)
        acc = _class_sums(Bt, C, case["sigma"], seed) if kind == "classify" else None
        s["model"] = hdc.Model(Bt, _config(case), acc=acc)
        s["ws"] = s["model"].workspace(case["N"])
        if kind == "classify":
            s["labels"] = torch.empty(case["N"], dtype=torch.int32, device="cuda")
        else:
            s["out"] = torch.empty((case["N"], s["model"].W), dtype=torch.int32, device="cuda")
    elif kind == "levelid":
        F, D, L = case["F"], case["D"], case["L"]
        g = _gen(seed, 7)
        bit = lambda *shape: torch.randint(0, 2, shape, generator=g, device="cuda", dtype=torch.uint8)
        flip = torch.randint(1, L, (D,), generator=g, device="cuda", dtype=torch.int32)
        s["model"] = hdc.LevelIdModel(bit(F, D), bit(D), bit(D), flip, L, -3.0, 3.0)
        s["X"] = torch.randn((case["N"], F), generator=g, device="cuda")
        s["out"] = torch.empty((case["N"], s["model"].W), dtype=torch.int32, device="cuda")
    else:
        N, D, C = case["N"], case["D"], case["C"]
        s["D"], s["C"] = D, C
        s["H"], s["y"], s["cls"] = _samples(N, D, C, case["flip"], seed)
        if kind == "train":
            s["acc"] = torch.empty((C, D), dtype=torch.int32, device="cuda")
            s["updates"] = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(case["epochs"])]
            s["ws"] = hdc.train_workspace(N, D, C, s["H"].device)
        elif kind == "hamming":
            s["config"] = _config(case)
            s["ws"] = hdc.hamming_workspace(C, D, s["H"].device)
        elif kind == "sweep":
            s["acc"] = torch.empty((C, D), dtype=torch.int32, device="cuda")
            hdc.train_epoch(s["H"], s["y"], D, C, 0, s["acc"], s["cls"])
            s["sweep"] = hdc.Sweep(D, C, _numbers(case["strides"], int), _numbers(case["widths"], int), N,
                                   s["H"].device, keep_labels=True, ends=_numbers(case["ends"], float),
                                   starts=_numbers(case["starts"], float))
        else:
            s["iters"] = case["epochs"]
            pick = torch.randperm(N, generator=_gen(seed, 8), device="cuda")[:C]
            s["init"] = s["H"][pick].contiguous()
    return s


def run(s):
    kind = s["kind"]
    if kind == "classify":
        return hdc.classify(s["X"], s["model"], sims=True, ws=s["ws"], labels=s["labels"])
    if kind == "encode":
        return hdc.encode(s["X"], s["model"], ws=s["ws"], out=s["out"])
    if kind == "levelid":
        return hdc.levelid_encode(s["X"], s["model"], out=s["out"])
    if kind == "train":
        hdc.train_epoch(s["H"], s["y"], s["D"], s["C"], 0, s["acc"], s["cls"], ws=s["ws"])
        for nu in s["updates"]:
            hdc.train_epoch(s["H"], s["y"], s["D"], s["C"], 1, s["acc"], s["cls"], n_updates=nu, ws=s["ws"])
        return s["acc"], s["cls"], s["updates"]
    if kind == "hamming":
        return hdc.hamming_argmin(s["H"], s["cls"], s["D"], s["config"], dists=True, ws=s["ws"])
    if kind == "sweep":
        return s["sweep"](s["H"], s["y"], s["acc"]), s["sweep"].labels
    return hdc.cluster(s["H"], s["D"], s["init"], s["iters"])


# ------------------------------------------------------------- what a pass needs

def _kept(case):
    s0 = math.floor(case.get("start", 0.0) * case["D"])
    e0 = math.floor(case.get("end", 1.0) * case["D"])
    return max(1, -(-(e0 - s0) // case.get("stride", 1)))


def work(case):
    """Bytes (inputs and outputs once) and operations (a multiply-add or a counted bit is two) of one pass."""
    kind, N, D = case["kind"], case["N"], case["D"]
    C, row = case.get("C", 0), (case["D"] + 127) // 128 * 16   # bytes of a packed row
    if kind == "levelid":
        return {"bytes": 4 * N * case["F"] + N * row + (case["F"] + case["L"]) * row, "flops": 2 * N * case["F"] * D}
    if kind in ("classify", "encode"):
        F, K = case["F"], _kept(case)
        es = {"fp32": 4, "bf16": 2, "fp8": 1}[case["enc"]]
        out = 4 * N + (8 if case.get("bits", 1) > 1 else 4) * N * C if kind == "classify" else N * ((K + 127) // 128 * 16)
        return {"bytes": 4 * N * F + es * K * F + C * K * case.get("bits", 1) // 8 + out,
                "flops": 2 * N * K * F + 2 * N * K * C}
    if kind == "train":   # every epoch predicts, and counts the updated rows (at least the bundling counts every row)
        e = case["epochs"]
        return {"bytes": (1 + e) * (N * row + 4 * N) + (1 + e) * C * (4 * D + row), "flops": 2 * N * D * (1 + e * C)}
    if kind == "hamming":
        return {"bytes": N * row + C * row + 4 * N * (1 + C), "flops": 2 * N * _kept(case) * C}
    if kind == "sweep":
        n = len(_numbers(case["strides"], int)) * len(_numbers(case["widths"], int))
        return {"bytes": N * row + 4 * C * D + 4 * N * (1 + n), "flops": 2 * N * D * C * len(_numbers(case["widths"], int))}
    e = case["epochs"]
    return {"bytes": N * row + 4 * N + C * (4 * D + row), "flops": 2 * N * D * (e * (C + 1) + C)}


# ------------------------------------------------------------- 64-bit values

def _class_values(acc, bits):
    """b-bit class values: per class, round(acc * Q / max|acc|), halves away from zero."""
    a = acc.to(torch.int64)
    if bits == 1:
        return torch.where(a < 0, -1, 1).double()
    Q = 2 ** (bits - 1) - 1
    M = a.abs().amax(1, keepdim=True).clamp_min(1)
    return (a.sign() * torch.div(2 * a.abs() * Q + M, 2 * M, rounding_mode="floor")).double()


def _operand(x, enc):
    """Rows in FP64 as the encoding's element type holds them: BF16, or E4M3 under a power-of-two scale per row (the
    smallest with the row's largest magnitude at most 448)."""
    if enc == "bf16":
        return x.to(torch.bfloat16).double()
    if enc == "fp8":
        m, e = torch.frexp(x.abs().amax(1, keepdim=True).double() / 448.0)
        k = torch.where(m == 0, 0, torch.where(m == 0.5, e - 1, e)).double()
        return (x.double() * torch.exp2(-k)).float().to(torch.float8_e4m3fn).double() * torch.exp2(k)
    return x.double()


def exact(case, seed):
    """The cosine scores of a classify case, its operands those of the element type; None for whole numbers."""
    if case["kind"] != "classify" or case.get("bits", 1) == 1:
        return None
    N, F, K = case["N"], case["F"], _kept(case)
    if 2.0 * N * F * K > 4.0e12:
        return None
    Bt = _base(case["D"], F, seed)
    s0 = math.floor(case.get("start", 0.0) * case["D"])
    e0 = math.floor(case.get("end", 1.0) * case["D"])
    keep = slice(s0, e0, case.get("stride", 1))
    X, _ = _mixture(N, F, case["C"], case["sigma"], seed, 6)
    v = _class_values(_class_sums(Bt, case["C"], case["sigma"], seed), case["bits"])[:, keep]
    vn = v.norm(dim=1)
    B = _operand(Bt[keep], case["enc"]).t().contiguous()
    out = torch.empty((N, case["C"]), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // K)
    for r in range(0, N, step):
        q = _operand(X[r:r + step], case["enc"]) @ B
        if case.get("float_query"):
            n = q.norm(dim=1, keepdim=True) * vn
        else:
            q = torch.where(q < 0, -1.0, 1.0).double()
            n = vn.expand(q.shape[0], -1)
        out[r:r + step] = torch.where(n == 0, 0.0, (q @ v.t()) / n)
    return None, out

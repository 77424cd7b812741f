"""The sweep autotuner where the launch shape is not read (no GPU)."""
import ctypes

import pytest

from paper_2606_26547_gb300 import autotune, build, hdc


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()


# both sides of the digit rows (256 a configuration) and of the words (4,096)
@pytest.mark.parametrize("D,C,bits", [(1000, 256, (1, 4)), (1000, 257, (1, 4)), (1000, 128, (1, 8)), (1000, 129, (1, 8)),
                                      (1000, 32, (0, 4)), (1000, 33, (0, 4)), (131072, 26, (1, 4, 8)), (131073, 26, (1, 4, 8))])
def test_route_is_the_librarys(D, C, bits):
    """The workspace holds digit rows and one array of sums, or bit planes and two."""
    up = lambda n: (n + 255) // 256 * 256
    strides, W = (1, 2, 4), hdc.words(D)
    n = ctypes.c_size_t()
    spec = hdc.sweep_spec(strides, bits)
    assert hdc.load().hdc_sweep_workspace_bytes(D, C, ctypes.byref(spec), ctypes.byref(n)) == 0
    rows = sum({0: 8, 8: 2}.get(b, 1) * C * len(strides) for b in bits)
    planes = sum({0: 32}.get(b, b) for b in bits)
    sums = up(len(bits) * len(strides) * C * 8)
    digits, popcounts = up(rows * ((W + 7) // 8) * 256), up(planes * C * W * 4) + sums
    assert n.value == sums + (digits if autotune.tensor_core_sweep(D, C, bits) else popcounts)


def test_nothing_is_timed(monkeypatch):
    calls = []

    class Sweep:
        def __init__(self, *a):
            self.shape = a[-2:]

        def __call__(self, H, y, acc):
            calls.append(self.shape)
            if len(calls) < 3:
                raise hdc.HdcError("hdc_sweep_eval", 2)

    def fail(*a, **k):
        raise AssertionError("timed or cached")

    class H:
        shape, device = (100, 32), "cpu"

    monkeypatch.setattr(hdc, "Sweep", Sweep)
    for name in ("Event", "synchronize"):
        monkeypatch.setattr(autotune.torch.cuda, name, fail)
    for name in ("_load", "_store"):
        monkeypatch.setattr(autotune, name, fail)
    assert autotune.tune_sweep(H, None, None, 1000, 26, (1, 2), (1, 4, 8)) == autotune.CANDIDATES[2]
    assert calls == list(autotune.CANDIDATES[:3])

"""Kernels that start while the one before them in the stream still runs wait for
it (early_wait, grid_wait); what it wrote is then visible to ordinary loads, not
to non-coherent ones, whose data must not change while the kernel runs."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_26547_gb300", "csrc")


def bodies():
    """(file, name, body) of every function that holds one of the waits."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\([^;{]*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end]
            if re.search(r"\b(early_wait|grid_wait)\s*\(", body):
                yield os.path.basename(path), m.group(1), body


def test_kernels_found():
    names = {n for _, n, _ in bodies()}
    assert {"hist_kernel", "scan_kernel", "scatter_kernel", "count_kernel", "reduce_kernel", "assign_count_kernel",
            "update_kernel", "tc_encode_kernel", "tc_hamming_packed_kernel", "tc_cosine_kernel"} <= names


@pytest.mark.parametrize("what", [r"__ldg\b", r"\bld\.global(\.\w+)*\.nc\b"])
def test_no_non_coherent_loads(what):
    found = [(f, n) for f, n, body in bodies() if re.search(what, body)]
    assert not found

"""Register spills of the two-pixel trace kernels, all numbers of nodes per row, from
the compiler (no GPU).

A few words spilled cost nothing that shows; the guarded rows, which spilled more, had
lost to the one-pixel form in small launches.  Rows of 7 nodes are allowed twice as
much: with the registers for it they were measured slower.
"""
import os
import re
import subprocess

import pytest

from paper_1505_07674_gb300 import _build as B


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    try:
        exe = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    obj = os.path.join(tmp_path_factory.mktemp("k"), "k.o")
    r = subprocess.run([exe, *B.ARCH, *B.NVCC_FLAGS, "-Xptxas", "-v", "-c",
                        os.path.join(B.CSRC, "lensed_kernels.cu"), "-o", obj], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out, cur = {}, None
    for line in r.stderr.splitlines():
        m = re.search(r"(?:Compiling entry function|Function properties for) '?(\S+?)'?(?: for|$)", line)
        if m:
            cur = m.group(1)
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m and cur:
            out[cur] = int(m.group(1)) + int(m.group(2))
    return out


# <mode, nodes, exact, queue>: FP32 (MIXED's first pass too), and MIXED_FF with a
# second pass; <0, 4, false, false> are the guarded rows beyond 8 nodes
TWO_PIXEL = ([f"Li0ELi{g}ELb1ELb0E" for g in range(1, 9)] + ["Li0ELi4ELb0ELb0E"] +
             [f"Li3ELi{g}ELb1ELb1E" for g in range(1, 9)])


@pytest.mark.parametrize("form", ["k_trace_rowsI", "k_trace_rows_pqI"])
@pytest.mark.parametrize("args", TWO_PIXEL)
def test_two_pixel_kernels_spill_at_most_a_few_words(report, form, args):
    found = {k: v for k, v in report.items() if form + args in k}
    assert len(found) == 1, sorted(report)[:5]
    assert max(found.values()) <= (64 if "Li7E" in args else 32), found

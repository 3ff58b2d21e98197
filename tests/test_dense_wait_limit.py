"""The poll limit of the dense sampling's cluster barrier against the work that one CTA may do between two
barriers while the others wait (host only: the limit is compiled from the library's header).

Work by the FP64 rate of one SM (two multiply-adds a clock, 1.9 GHz): four multiply-adds for each of the n^2
entries and each column of a triangular solve, and 64 x 64 / 2 complex ones a row of a panel in global memory,
whose 1024 column passes cross L2 at 100 GB/s.  A poll takes at least 1 us (3.8 measured).  The limit must allow
four times the work."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CASES = [(64, 1), (1600, 2), (3200, 1), (10000, 1), (20000, 4), (50000, 1), (130000, 32), (180000, 1)]


@pytest.fixture(scope="module")
def limits(tmp_path_factory):
    from paper_1510_07522_gb300 import _build
    d = tmp_path_factory.mktemp("wait")
    src, exe = d / "limit.cu", d / "limit"
    src.write_text('#include <cstdio>\n#include "dense_lu.cuh"\nint main() {\n' + "".join(
        f'    std::printf("%llu\\n", rsrr::dense_wait_polls({n}, {c}));\n' for n, c in CASES) + "}\n")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-I" + os.path.join(ROOT, "include"),
                    "-I" + _build.CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    return dict(zip(CASES, map(int, out)))


@pytest.mark.parametrize("n,cols", CASES)
def test_limit_covers_the_work(limits, n, cols):
    clock = 1.9e9
    solve = n * n * cols * 4 / 2 / clock
    panel = n * (64 * 64 / 2 * 4 / 2 / clock + 1024 * 2 * 16 / 100e9)
    assert limits[n, cols] * 1e-6 >= 4 * max(solve, panel)
    assert limits[n, cols] >= 1 << 21

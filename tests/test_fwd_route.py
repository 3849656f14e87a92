"""The size rules that choose a forward kernel (csrc/fwd_route.h), compiled on the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _eval(tmp_path, exprs):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "route.cpp", tmp_path / "route"
    src.write_text('#include <cstdio>\n#include "fwd_route.h"\nusing namespace pinn;\nint main() {\n' +
                   "".join(f'  printf("%d\\n", (int)({e}));\n' for e in exprs) + "}\n")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2604_15645_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True, timeout=300)
    return [bool(int(x)) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]


def test_pairs_only_where_they_are_faster(tmp_path):
    """(width, K, points, low half on value rows only) measured with both kernels."""
    cases = [  # slower in pairs
             (512, 128, 20000, False, False), (512, 256, 200000, False, False), (512, 64, 200000, True, False),
             (768, 128, 60000, False, False), (1024, 256, 200000, True, False),
             (512, 512, 2000, False, False), (512, 512, 6000, False, False), (1024, 1024, 6000, False, False),
             (256, 512, 6000, False, False), (256, 128, 40000, True, False),
             (1024, 1024, 60000, True, False), (512, 2048, 200000, True, False),
             (384, 512, 200000, False, False), (264, 264, 200000, False, False),   # odd numbers of m-tiles
             # faster in pairs
             (512, 384, 20000, False, True), (512, 512, 20000, False, True), (512, 512, 200000, True, True),
             (768, 768, 60000, False, True), (1024, 1024, 200000, False, True), (256, 512, 60000, False, True)]
    exprs = [f"fwd_in_pairs({(w + 127) // 128}, {(n + 63) // 64}, {k}, {str(v).lower()}, 152)" for w, k, n, v, _ in cases]
    exprs += ["fwd_in_pairs(4, 1 << 30, 512, false, 152)", "fwd_in_pairs(4, 100000, 512, false, 1)"]
    assert _eval(tmp_path, exprs) == [c[4] for c in cases] + [True, False]


def test_one_kernel_needs_more_than_one_layer(tmp_path):
    assert _eval(tmp_path, [f"fwd_in_one_kernel({n})" for n in (0, 1, 2, 3, 16)]) == [False, False, True, True, True]

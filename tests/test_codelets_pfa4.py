"""The pruned 20- and 28-point codelets (Good-Thomas 4 x 5 and 4 x 7) built for the host and
checked against numpy's FFT: zero upper half of the inputs, lower half of the outputs kept,
both signs, in double and in float (the tolerances of test_codelets.py)."""
import os
import subprocess

import numpy as np
import pytest

from paper_2405_01522_gb300 import build as pkg_build
from test_codelets import CSRC, PROGRAM, _dft, _inputs

MAIN = r"""
int main() {
  half<20, -1, double>(); half<20, 1, double>(); half<28, -1, double>(); half<28, 1, double>();
  half<20, -1, float>(); half<20, 1, float>(); half<28, -1, float>(); half<28, 1, float>();
}
"""


@pytest.mark.parametrize("size,tol", [(8, 1e-13), (4, 3e-6)])
def test_pruned_four_by_q(tmp_path, size, tol):
    src, exe = str(tmp_path / "c.cu"), str(tmp_path / "c")
    with open(src, "w") as f:
        f.write(PROGRAM[:PROGRAM.index("template <typename R> void all()")] + MAIN)
    r = subprocess.run([pkg_build.NVCC, "-O2", "-std=c++17", "-I", CSRC, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    seen = 0
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines():
        tag, n, s, sz, *vals = line.split()
        n, s = int(n), int(s)
        if int(sz) != size:
            continue
        z = np.array(vals, dtype=float).reshape(-1, 2)
        x = _inputs(n)
        if tag == "halfin":
            x[n // 2:] = 0
        ref = _dft(x, s)[: len(z)]
        assert np.max(np.abs(z[:, 0] + 1j * z[:, 1] - ref)) <= tol * np.max(np.abs(ref)), (tag, n, s)
        seen += 1
    assert seen == 8

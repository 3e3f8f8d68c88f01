"""Block fixed-point arithmetic of the float64 FFT lines, run on the host (nvcc compiles the same
functions for it): conversions at every exponent."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2412_17445_gb300", "csrc")


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    """name -> remaining columns of the lines that the host program prints."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("fx") / "fixed_lines")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "native", "fixed_lines.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = {}
    for line in r.stdout.splitlines():
        name, *cols = line.split()
        out.setdefault(name, []).append(cols)
    return out


@pytest.mark.parametrize("name", ["integers_to_float64", "float64_to_integers"])
def test_conversions(report, name):
    """Correct rounding: no differing value, from subnormal results to the largest binade."""
    (n, bad), = report[name]
    assert int(n) > 100000 and int(bad) == 0

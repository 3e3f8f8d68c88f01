"""Block fixed-point arithmetic of the float64 FFT lines, run on the host (nvcc compiles the same
functions for it): conversions at every exponent, and whole lines of every length and plan."""
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


def test_compiled_plans(report):
    (n, bad), = report["plans"]
    assert int(bad) == 0


def test_lines(report):
    """RMS error of a transformed line over the RMS of the result.  A component is rounded to float64
    once (0.6e-16 of itself); a stage rounds to units of 2^-59 of the line's largest component times
    the shifts so far, which the sum of magnitudes, at most sqrt(N) times the norm, keeps within
    2^-2.5 sqrt(N) of it: 2e-17 of the RMS at N = 4096, and the up to 8 stages add in the square with the
    rotations' like share: below 2.5e-16 for every line.  An overflow, which the constant, alternating and
    single-frequency lines at the largest mantissa are made for (moduli of 2^62.5 of 2^63), is an
    error of order one."""
    rows = report["line"]
    lengths = {int(r[0]) for r in rows}
    assert {2, 3, 48, 729, 768, 1024, 3072, 4096} <= lengths and {r[3] for r in rows} >= {"constant", "wave", "peak"}
    worst = max(rows, key=lambda r: float(r[4]))
    assert float(worst[4]) < 2.5e-16, worst

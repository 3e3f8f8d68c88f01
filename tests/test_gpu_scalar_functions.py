"""recip_nr, rsqrt_nr and round_to<float> of the float64 kernels, over all exponents and at extreme
mantissas, against correctly rounded values."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    """(x, recip, rsqrt, float32 rounding, taken by rsqrt)"""
    from paper_2412_17445_gb300 import build
    d = tmp_path_factory.mktemp("scalar")
    exe = str(d / "scalar_functions")
    inc = [os.path.join(os.path.dirname(HERE), "include"), build.CSRC]
    r = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I", inc[0], "-I", inc[1],
                       os.path.join(HERE, "native", "scalar_functions.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    rng = np.random.default_rng(1)
    top = (1 << 52) - 1
    ex = np.repeat(np.arange(2048, dtype=np.uint64), 400)
    man = rng.integers(0, 1 << 52, ex.size, dtype=np.uint64)
    edge = np.array([0, 1, 2, top, top - 1, 1 << 51, (1 << 51) - 1, (1 << 51) + 1, 1 << 29, (1 << 29) - 1, (1 << 28),
                     (1 << 28) + 1, (1 << 28) - 1, top - (1 << 28), top - (1 << 28) + 1, 3 << 28, (3 << 28) + 1],
                    dtype=np.uint64)
    man = man.reshape(2048, 400)
    man[:, :edge.size] = edge
    man[:, edge.size:100] = (man[:, edge.size:100] >> np.uint64(28)) << np.uint64(28)  # float32 ties
    bits = (ex << np.uint64(52)) | man.reshape(-1)
    bits[1::2] |= np.uint64(1 << 63) * (rng.random(bits[1::2].size) < 0.5).astype(np.uint64)
    x = np.concatenate([bits.view(np.float64), [0.0, -0.0, np.inf, -np.inf, np.nan]])
    x.tofile(d / "in")
    r = subprocess.run([exe, str(d / "in"), str(d / "out")], capture_output=True, text=True)
    assert r.returncode == 0
    out = np.fromfile(d / "out").reshape(-1, 4)
    return x, out[:, 0], out[:, 1], out[:, 2], out[:, 3] > 0


def _steps(a, b):
    """Distance in representable numbers (same sign)."""
    return np.abs(a.view(np.int64) - b.view(np.int64))


def test_recip(values):
    """The seed is good to 2^-21, the correction leaves its cube, 2^-63, and the last operation rounds once:
    within one step of the rounded quotient, and the library's result where the seed declines."""
    x, got, *_ = values
    want = 1.0 / x
    ok = np.isfinite(want) & (want != 0)
    assert np.array_equal(np.signbit(got[ok]), np.signbit(want[ok]))
    assert np.max(_steps(got[ok], want[ok])) <= 1
    e = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(2047)
    lib = (e < 2) | (e > 2043)
    assert np.array_equal(got[lib], want[lib], equal_nan=True)


def test_rsqrt(values):
    """As recip; x r rounds once more, half of which reaches the result: one unit in the last place of the
    exact value, two steps across a power of two.  Takes the positive numbers of exponents 2 to 2043."""
    x, _, got, _, ok = values
    e = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(2047)
    assert np.array_equal(ok, ~np.signbit(x) & (e >= 2) & (e <= 2043))
    assert not np.any(got[~ok])
    # 1 / sqrt by float64 and one correction with the residual in two parts, exact to 2^-60
    xs = x[ok]
    m, k = np.frexp(xs)
    odd = k % 2 != 0
    m = np.where(odd, 2 * m, m)
    k = np.where(odd, k - 1, k) // 2
    r = 1.0 / np.sqrt(m)
    from fractions import Fraction
    pick = np.random.default_rng(2).choice(xs.size, 20000, replace=False)
    g = np.ldexp(got[ok], k)  # scaled to 1 / sqrt(m), exact
    assert np.max(np.abs(g - r) / r) < 4e-16
    for i in pick:
        v = Fraction(float(g[i]))
        ulp = Fraction(float(np.spacing(g[i])))
        mm = Fraction(float(m[i]))
        assert (v - ulp) ** 2 * mm <= 1 <= (v + ulp) ** 2 * mm, xs[i]


def test_round_to_float32(values):
    """Bit for bit the conversion to float32, NaN to NaN."""
    x, _, _, got, _ = values
    with np.errstate(all="ignore"):
        want = x.astype(np.float32).astype(np.float64)
    assert np.array_equal(got, want, equal_nan=True)
    assert np.array_equal(np.signbit(got[~np.isnan(x)]), np.signbit(want[~np.isnan(x)]))

"""Float64 FFT lines in block fixed point: accuracy against the oracle at the edges of the plans,
and what a shared exponent per line must keep (powers of two, zeros, non-finite values)."""
import numpy as np
import pytest

from oracle import solver
from paper_2412_17445_gb300 import binding as B
from paper_2412_17445_gb300 import microstructure as ms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2412_17445_gb300 import build
    build.build()
    B.lib()


# line lengths of one to seven stages, compiled and runtime plans; one line a block to several
# warps a line; column groups of one to sixteen lines
SHAPES = [(2, 2), (3, 2), (4, 1024), (1024, 6), (729, 8), (8, 2187), (512, 48), (81, 64), (6, 4, 3), (128, 9, 48)]


def _setup(shape, seed):
    inp = ms.random_rve(shape, seed, notch=False)
    eps, E, phi, H = ms.random_state(inp, seed + 1)
    g = B.RVE(inp)
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.linearize(B.RVE_CTRL_STRAIN, E)
    return inp, g, (eps, E, phi, H)


def _apply(g, x, xE):
    import torch
    xd = torch.tensor(x, dtype=torch.float64, device="cuda")
    e = torch.tensor([xE], dtype=torch.float64, device="cuda")
    y, yE = torch.zeros_like(xd), torch.zeros_like(e)
    g.apply_device(xd.data_ptr(), e.data_ptr(), y.data_ptr(), yE.data_ptr())
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["noise", "peak", "rows"])
def test_apply_accuracy(shape, kind):
    """Strain rows of an apply against the oracle.  Each transform pass is off by a few roundings
    of its lines' norms; two transforms of at most 22 stages a side: 100 roundings (2.2e-14) of the
    largest value for noise, times sqrt(n) at most for a field whose norm one voxel holds."""
    inp, g, (eps, E, phi, H) = _setup(shape, 11)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((g.m, g.n))
    if kind == "peak":       # one voxel holds the norm: lines that are never shifted
        x *= 1e-9
        x[:, g.n // 2] = 1.0
    elif kind == "rows":     # rows of very different magnitude: one exponent a line
        x *= np.repeat(10.0 ** (-12.0 * rng.random(g.n // shape[-1])), shape[-1])
    pb = solver.problem_from_input(inp)
    lin = solver.Linearization(pb, eps, E, phi, H)
    Jo = solver.jacobian_apply(lin, (B.tensor_from_mandel(x, shape), np.zeros(shape), 0.0), solver.STRAIN)
    Je, _, _ = g.apply(x, np.zeros(g.n), 0.0)
    ref = B.mandel_from_tensor(Jo[0])
    assert np.sqrt(np.mean((Je - ref) ** 2)) < 2.2e-14 * np.max(np.abs(ref))
    g.close()


@pytest.mark.parametrize("shape", [(48, 64), (27, 81), (16, 12, 6)])
def test_shared_exponent(shape):
    """An apply commutes with powers of two bit for bit, keeps zeros, and a NaN or an infinity in
    one voxel reaches every strain value."""
    _, g, _ = _setup(shape, 21)
    rng = np.random.default_rng(6)
    x = rng.standard_normal((g.m + 1) * g.n)
    y = _apply(g, x, 0.25)
    for k in (-300, 300):
        assert np.array_equal(_apply(g, np.ldexp(x, k), np.ldexp(0.25, k)), np.ldexp(y, k))
    assert not np.any(_apply(g, np.zeros_like(x), 0.0))
    for bad in (np.nan, np.inf):
        z = x.copy()
        z[g.n // 3] = bad
        assert np.all(np.isnan(_apply(g, z, 0.25)[:g.m * g.n]))
    g.close()


@pytest.mark.parametrize("shape", [(48, 64), (27, 81), (16, 12, 6)])
def test_subnormal_results(shape):
    """Operands far below the normal range (2^-1040) give the scaled result of the operands at unit
    magnitude, off by the subnormal roundings alone: about three units of 2^-1074 an entry after
    the projection, which carries the factor 1 / n, times sqrt(n) through the two inverse transforms
    of the RMS (the roundings before the projection and in the last pass are smaller by sqrt(n))."""
    _, g, _ = _setup(shape, 21)
    rng = np.random.default_rng(7)
    k = 1040
    small = np.ldexp(rng.standard_normal((g.m + 1) * g.n), -k)  # rounded to the subnormal grid
    want = _apply(g, np.ldexp(small, k), 0.25)
    got = np.ldexp(_apply(g, small, np.ldexp(0.25, -k)), k)
    err = np.sqrt(np.mean((got - want).reshape(g.m + 1, -1) ** 2, axis=1))
    assert np.all(err <= 4.0 * np.sqrt(g.n) * 2.0 ** (k - 1074)), err
    g.close()


# (row pairs, columns) a block: groups of 2, 4 and 16 columns with and without a partial last group, several
# row pairs with a partial last block; lines of 128 (one warp a group) and 144 elements (two)
TILED = [((48, 36), (3, 4)), ((27, 64), (4, 16)), ((144, 54), (2, 2)), ((128, 144), (5, 4)), ((16, 12, 18), (3, 4)),
         ((9, 64, 48), (4, 16)), ((8, 27, 16), (2, 2))]


@pytest.mark.parametrize("shape,tiles", TILED)
@pytest.mark.parametrize("kind", ["noise", "wave"])
def test_apply_accuracy_of_tiles(shape, tiles, kind, monkeypatch):
    """Strain rows of an apply against the oracle: a dozen roundings of the pointwise tensor products and
    five conversions of the lines here, two transforms of up to 13 stages a side at half a rounding in the
    oracle, all adding in the square: below 12 roundings (1.3e-15) of the RMS of the stress that is
    projected, at most the largest 3 lam + 2 mu times the strain's."""
    monkeypatch.setenv("RVE_TILES", "%d,%d" % tiles)
    inp, g, (eps, E, phi, H) = _setup(shape, 11)
    g.autotune()
    rng = np.random.default_rng(5)
    if kind == "noise":
        x = rng.standard_normal((g.m, g.n))
    else:  # one frequency, the rows of a pair alike
        i = np.indices(shape)
        t = sum((3 + a) * i[a] / shape[a] for a in range(len(shape)))
        x = np.cos(2 * np.pi * t).reshape(1, -1) * rng.standard_normal((g.m, 1))
    pb = solver.problem_from_input(inp)
    lin = solver.Linearization(pb, eps, E, phi, H)
    Jo = solver.jacobian_apply(lin, (B.tensor_from_mandel(x, shape), np.zeros(shape), 0.0), solver.STRAIN)
    Je, _, _ = g.apply(x, np.zeros(g.n), 0.0)
    ref = B.mandel_from_tensor(Jo[0])
    stiff = np.max(inp.E / (1 - 2 * inp.nu))
    assert np.sqrt(np.mean((Je - ref) ** 2)) < 1.3e-15 * stiff * np.sqrt(np.mean(x ** 2))
    g.close()

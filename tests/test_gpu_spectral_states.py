"""Spectral split of the constitutive update at strain states that are hard for an eigen-solver:
the residual and the tangent against the oracle."""
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


def _states(kind, shape, d):
    rng = np.random.default_rng(4)
    a = rng.standard_normal(shape + (d, d))
    a = 0.5 * (a + np.swapaxes(a, -1, -2))
    eye = np.eye(d)
    p = 0.5 + rng.random(shape + (1, 1))
    if kind == "near_degenerate":    # equal eigenvalues but for 1e-9, away from zero
        return p * eye + 1e-9 * a
    if kind == "round_off":          # equal eigenvalues but for round-off
        return -p * eye + 1e-15 * a
    if kind == "diagonal":
        return a * eye
    if kind == "rank_one":
        v = rng.standard_normal(shape + (d,))
        return v[..., :, None] * v[..., None, :] + 0.1 * eye
    if kind == "small":              # far below unit magnitude, entries over ten decades
        return 1e-30 * (a * eye + 10.0 ** (-10 * rng.random(shape + (1, 1))) * a)
    return np.zeros_like(a)


@pytest.mark.parametrize("shape", [(12, 16), (6, 8, 4)])
@pytest.mark.parametrize("kind", ["near_degenerate", "round_off", "diagonal", "rank_one", "small", "zero"])
def test_residual_and_tangent(shape, kind):
    """1e-11 of the operand scale, as for random states."""
    d = len(shape)
    inp = ms.random_rve(shape, 7)
    _, _, phi, H = ms.random_state(inp, 8)
    eps = _states(kind, shape, d)
    E = 0.0
    pb = solver.problem_from_input(inp)
    lin = solver.Linearization(pb, eps, E, phi, H)
    F1o, F2o, _ = solver.residual(lin, solver.STRAIN, E)
    g = B.RVE(inp)
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.linearize(B.RVE_CTRL_STRAIN, E)
    F1, F2, _ = g.residual()
    assert np.max(np.abs(F1 - B.mandel_from_tensor(F1o))) <= 1e-11 * np.max(np.abs(lin.sigma))
    assert np.max(np.abs(F2 - F2o.reshape(-1))) <= 1e-11 * np.max(np.abs(F2o))
    de, dp, dE = ms.random_direction(inp, 9)
    Jo = solver.jacobian_apply(lin, (de, dp, dE), solver.STRAIN)
    Je, Jp, _ = g.apply(B.mandel_from_tensor(de), dp, dE)
    assert np.max(np.abs(Je - B.mandel_from_tensor(Jo[0]))) < 1e-11 * np.max(np.abs(Jo[0]))
    assert np.max(np.abs(Jp - Jo[1].reshape(-1))) < 1e-11 * np.max(np.abs(Jo[1]))
    g.close()


@pytest.mark.parametrize("k", [1010, 1040])
def test_residual_of_tiny_strains(k):
    """The stress is positively homogeneous in the strain: strains at 2^-k, their eigenvectors included,
    give the residual of the same strains at unit magnitude.  1e-11 of the stress scale as above;
    near and below 2^-1022 also the subnormal roundings, in units u = 2^-1074: about 2 u a strain
    entry and as much again in the eigenvalues, times the stiffness, and four u an entry, times sqrt(n),
    through the transforms of the RMS."""
    shape = (6, 8, 4)
    inp = ms.random_rve(shape, 7)
    _, _, phi, H = ms.random_state(inp, 8)
    a = np.random.default_rng(4).standard_normal(shape + (3, 3))
    small = np.ldexp(B.mandel_from_tensor(a + np.swapaxes(a, -1, -2)), -k)
    stiff = np.max(inp.E * (1 - inp.nu) / ((1 + inp.nu) * (1 - 2 * inp.nu)))
    g = B.RVE(inp)
    F = []
    for eps in (np.ldexp(small, k), small):
        g.set_state(eps, phi, H, 0.0)
        g.linearize(B.RVE_CTRL_STRAIN, 0.0)
        F.append(g.residual()[0])
    scale = stiff * np.max(np.abs(np.ldexp(small, k)))
    err = np.sqrt(np.mean((np.ldexp(F[1], k) - F[0]) ** 2))
    assert err <= 1e-11 * scale + 4 * (np.sqrt(g.n) + 2 * stiff + 2) * 2.0 ** (k - 1074)
    g.close()

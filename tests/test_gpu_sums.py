"""Reduction of the per-block partials (exact integer accumulation): the constraint row's sum of an
operator apply, where cancelling, tiny, huge and non-finite values all pass through it."""
import math

import numpy as np
import pytest

from paper_2412_17445_gb300 import binding as B
from paper_2412_17445_gb300 import microstructure as ms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2412_17445_gb300 import build
    build.build()
    B.lib()


def _yE(g, torch, x):
    xd = torch.tensor(x, dtype=torch.float64, device="cuda")
    xE = torch.zeros(1, dtype=torch.float64, device="cuda")
    y, yE = torch.empty_like(xd), torch.zeros_like(xE)
    g.apply_device(xd.data_ptr(), xE.data_ptr(), y.data_ptr(), yE.data_ptr())
    torch.cuda.synchronize()
    return float(yE)


# 1, 32, 36, 256, 288 and 1024 partials: a lane's batch is 8 values, a warp's 256
@pytest.mark.parametrize("shape", [(2, 48), (64, 48), (72, 27), (512, 16), (576, 8), (2048, 8)])
def test_constraint_sum(shape, monkeypatch):
    """yE = sum w dphi of a float64 apply.  With dphi non-zero in one voxel of one row pair per
    block, a partial is that product alone, so the sum over blocks is compared with math.fsum of
    the products: one rounding, 2^-52 relative to the result, cancellation included."""
    import torch
    monkeypatch.setenv("RVE_TILES", "1,1")  # one row pair per block
    inp = ms.random_rve(shape, seed=5, notch=False)
    eps, E, phi, H = ms.random_state(inp, 7)
    g = B.RVE(inp)
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.autotune()
    g.linearize(B.RVE_CTRL_CRACK, 1.0)
    ny, nx = shape
    rng = np.random.default_rng(3)
    n = ny * nx
    vox = [r * nx + int(rng.integers(nx)) for r in range(0, ny, 2)]
    w = np.empty(len(vox))
    for i, v in enumerate(vox):  # w at the voxels: one unit entry at a time (a single partial)
        if i < 40 or i % 61 == 0:
            x = np.zeros(4 * n)
            x[3 * n + v] = 1.0
            w[i] = _yE(g, torch, x)
        else:
            w[i] = np.nan
    use = [i for i in range(len(vox)) if np.isfinite(w[i])]
    for scale in (1.0, 1e-300, 1e250):
        x = np.zeros(4 * n)
        d = rng.standard_normal(len(use)) * 10.0 ** rng.uniform(-12, 12, len(use)) * scale
        if len(use) > 2:  # cancel the largest products to rounding
            k = np.argsort(np.abs(d * w[use]))[::-1]
            d[k[1]] = -d[k[0]] * w[use][k[0]] / w[use][k[1]]
        for i, di in zip(use, d):
            x[3 * n + vox[i]] = di
        got = _yE(g, torch, x)
        want = math.fsum(w[i] * di for i, di in zip(use, d))
        assert abs(got - want) <= 2.0 ** -52 * abs(want), (got, want)
    for bad in (np.inf, -np.inf, np.nan):
        x = np.zeros(4 * n)
        x[3 * n + vox[use[-1]]] = bad
        got = _yE(g, torch, x)
        assert not np.isfinite(got)
    g.close()



# partials of one batch (36), of two (288) and of four (1024)
@pytest.mark.parametrize("shape", [(72, 27), (576, 8), (2048, 8)])
def test_constraint_sum_below_a_cancelled_pair(shape, monkeypatch):
    """Two partials that cancel exactly, in the first batch or a later one, and survivors 2^40 to 2^1500
    below them: the sum is that of the survivors, to one rounding (math.fsum of the products),
    also where those cancel in turn down to a last one."""
    import torch
    monkeypatch.setenv("RVE_TILES", "1,1")  # one row pair per block
    inp = ms.random_rve(shape, seed=5, notch=False)
    eps, E, phi, H = ms.random_state(inp, 7)
    g = B.RVE(inp)
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.autotune()
    g.linearize(B.RVE_CTRL_CRACK, 1.0)
    ny, nx = shape
    n, nb = ny * nx, ny // 2
    rng = np.random.default_rng(3)
    blocks = [0, 1, 5, nb // 2, nb // 2 + 1, nb - 7, nb - 2, nb - 1]
    vox = [2 * r * nx + int(rng.integers(nx)) for r in blocks]
    w = []
    for v in vox:  # w at the voxels: one unit entry at a time (a single partial)
        x = np.zeros(4 * n)
        x[3 * n + v] = 1.0
        w.append(_yE(g, torch, x))

    def check(d):
        x = np.zeros(4 * n)
        for v, di in zip(vox, d):
            x[3 * n + v] = di
        want = math.fsum(wi * di for wi, di in zip(w, d))
        got = _yE(g, torch, x)
        assert abs(got - want) <= 2.0 ** -52 * abs(want), (d, got, want)

    for down in (40, 60, 80, 107, 130, 400, 1500):
        for i, j in ((0, 1), (0, 7), (6, 7), (3, 5)):
            rest = [k for k in range(8) if k not in (i, j)]
            d = np.zeros(8)
            d[i], d[j] = np.ldexp(w[j], down // 2), -np.ldexp(w[i], down // 2)  # equal products
            d[rest] = np.ldexp(rng.standard_normal(6), -(down - down // 2))
            check(d)
            a, b = rest[0], rest[1]  # a second pair cancels: one survivor far below it
            d[rest] = 0.0
            d[a], d[b] = np.ldexp(w[b], -down // 4), -np.ldexp(w[a], -down // 4)
            d[rest[2]] = np.ldexp(1.0, -(down - down // 2))
            check(d)
            d[rest[2]] = 0.0
            check(d)
    g.close()

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


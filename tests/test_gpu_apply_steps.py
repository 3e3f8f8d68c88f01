"""Float32 passes at the lengths where their steps change: two radix-3 stages in one step (odd and even
counts of them), column passes read into and written from registers with one, two and three steps,
and the E slot that one more block forms."""
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


def _rve(shape, seed, precision=B.RVE_MIXED, control=B.RVE_CTRL_CRACK):
    inp = ms.random_rve(shape, seed)
    st = ms.random_state(inp, seed + 1)
    g = B.RVE(inp, precision=precision)
    eps, E, phi, H = st
    g.set_state(B.mandel_from_tensor(eps), phi, H, E)
    g.linearize(control, 1.0)
    return inp, st, g


@pytest.mark.parametrize("shape", [(9, 3), (27, 81), (243, 4), (6, 729), (768, 18), (18, 768), (1024, 512), (192, 3, 4),
                                   (4, 192, 6), (3, 4, 192), (48, 64, 12), (96, 128, 2), (128, 48, 18)])
def test_mixed_apply(shape):
    """1e-5 of the largest value, the tolerance of the float32 apply."""
    inp, (eps, E, phi, H), g = _rve(shape, 31)
    pb = solver.problem_from_input(inp)
    lin = solver.Linearization(pb, eps, E, phi, H)
    de, dp, dE = ms.random_direction(inp, 33)
    Jo = solver.jacobian_apply(lin, (de, dp, dE), solver.CRACK)
    Je, Jp, JE = g.apply(B.mandel_from_tensor(de), dp, dE)
    assert np.max(np.abs(Je - B.mandel_from_tensor(Jo[0]))) < 1e-5 * np.max(np.abs(Jo[0]))
    assert np.max(np.abs(Jp - Jo[1].reshape(-1))) < 1e-5 * np.max(np.abs(Jo[1]))
    assert abs(JE - Jo[2]) < 1e-5 * max(abs(Jo[2]), 1.0)
    g.close()


@pytest.mark.parametrize("shape", [(64, 48), (27, 9), (512, 512), (6, 8, 4)])
@pytest.mark.parametrize("precision", [B.RVE_MIXED, B.RVE_FP64])
def test_e_slot_of_a_mixed_group(shape, precision):
    """A group with both controls gives each member's own result bit for bit."""
    import torch
    gs = [_rve(shape, 41 + k, precision, c)[2] for k, c in enumerate([B.RVE_CTRL_CRACK, B.RVE_CTRL_STRAIN,
                                                                      B.RVE_CTRL_CRACK])]
    dt = torch.float32 if precision == B.RVE_MIXED else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(5)
    xs = [torch.randn((g.m + 1) * g.n, generator=gen, dtype=dt, device="cuda") for g in gs]
    es = [torch.randn(1, generator=gen, dtype=torch.float64, device="cuda") for _ in gs]
    ref = []
    for g, x, e in zip(gs, xs, es):
        y, yE = torch.zeros_like(x), torch.zeros_like(e)
        g.apply_device(x.data_ptr(), e.data_ptr(), y.data_ptr(), yE.data_ptr())
        torch.cuda.synchronize()
        ref.append((y, yE))
    ys, yEs = [torch.zeros_like(x) for x in xs], [torch.zeros_like(e) for e in es]
    B.apply_device_batch(gs, *[[t.data_ptr() for t in ts] for ts in (xs, es, ys, yEs)])
    torch.cuda.synchronize()
    for (y, yE), yb, yEb in zip(ref, ys, yEs):
        assert torch.equal(y, yb) and torch.equal(yE, yEb)
    assert torch.equal(yEs[1], es[1])  # strain control: the E slot itself
    for g in gs:
        g.close()


def test_few_large_column_blocks_spread_over_the_gpu():
    """Twice the columns at twice the length of a row are twice the work: an apply of half of them, whose
    129 column blocks of 73 KB leave SMs idle, takes well below the time of the whole (0.55 of it;
    0.84 when blocks of the next pass settle on whichever SM has room first)."""
    import torch
    times = []
    for shape in ((2048, 256), (2048, 512)):
        _, _, g = _rve(shape, 51)
        x = torch.randn((g.m + 1) * g.n, dtype=torch.float32, device="cuda")
        e = torch.ones(1, dtype=torch.float64, device="cuda")
        y, yE = torch.zeros_like(x), torch.zeros_like(e)
        g.set_stream(torch.cuda.current_stream().cuda_stream)
        best = []
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(20):
                g.apply_device(x.data_ptr(), e.data_ptr(), y.data_ptr(), yE.data_ptr())
            t1.record()
            torch.cuda.synchronize()
            best.append(t0.elapsed_time(t1))
        times.append(min(best[1:]))
        g.close()
    assert times[0] < 0.7 * times[1], times


def test_tuned_increment_of_768_points():
    """The two-row-pair, 512-thread passes of 768 points in the modes of a solve: a tuned MIXED increment
    against the float64 handle's, to the 1e-5 that MIXED is held to."""
    inp = ms.fibre_composite(n=768, ny=256, radius=12.0, fraction=0.4, notch_len=32, seed=3)
    steps = []
    for precision in (B.RVE_MIXED, B.RVE_FP64):
        g = B.RVE(inp, precision=precision, newton_tol=1e-8, krylov_tol=1e-2)
        g.startup()
        steps.append(g.crack_increment(1.0))
        g.close()
    m, d = steps
    assert m["fallbacks"] == 0
    assert abs(m["E"] - d["E"]) <= 1e-5 * abs(d["E"]) and abs(m["gamma"] - d["gamma"]) <= 1e-5 * abs(d["gamma"])
    assert np.max(np.abs(np.subtract(m["sigma"], d["sigma"]))) <= 1e-5 * np.max(np.abs(d["sigma"]))


@pytest.mark.parametrize("shape", [(256, 768), (18, 768), (6, 8, 4)])
def test_constraint_row_terms(shape):
    """The constraint row of a tuned MIXED apply against its terms: each a product of two float32 numbers, a
    dozen of them and the lanes of a warp summed in float32, ten roundings (6e-7) of the terms' magnitudes."""
    inp, (eps, E, phi, H), g = _rve(shape, 61)
    g.autotune()
    lin = solver.Linearization(solver.problem_from_input(inp), eps, E, phi, H)
    de, dp, dE = ms.random_direction(inp, 63)
    _, _, JE = g.apply(B.mandel_from_tensor(de), dp, dE)
    terms = lin.w * dp
    assert abs(JE - np.sum(terms)) <= 6e-7 * np.sum(np.abs(terms))
    g.close()

"""Timed cases of the public entry points: what a user of the library has it do.

A case is one of three calls, each through `paper_2412_17445_gb300.binding`:

  apply      the scaled Newton operator y = S J x on device buffers (`RVE.apply_device`, or
             `apply_device_batch` for several RVEs of one shape), the call that a Krylov solver
             repeats hundreds of times per crack increment;
  newton     a new linearisation at the committed state followed by one operator apply
             (`RVE.linearize`, `RVE.apply_device`), the work at the head of a Newton iteration;
  increment  one crack-length increment of each RVE from a given committed state
             (`RVE.set_state`, `RVE.crack_increment` or `batch_crack_increment`, `RVE.field`).

Grids are nz x ny x nx with nz = 1 for plane strain; extents are 2^a 3^b.  Microstructures are
fibre composites, porous solids and notched panels as in the benchmark; the linearisation point
is a notch's phase-field profile under uniaxial load with fluctuating strain and history.
"""
import math

import numpy as np
import torch

from paper_2412_17445_gb300 import binding as B
from paper_2412_17445_gb300 import microstructure as ms

SMOOTH = sorted(2 ** a * 3 ** b for a in range(11) for b in range(7) if 2 ** a * 3 ** b <= 1024)


def _case(kind, nz, ny, nx, precision, count=1, split="spectral", gamma="rotated", control="crack"):
    return {"kind": kind, "nz": nz, "ny": ny, "nx": nx, "precision": precision, "count": count, "split": split,
            "gamma": gamma, "control": control}


def listed():
    out = []

    def add(name, *args, **kw):
        out.append(dict(_case(*args, **kw), name=name))

    # one apply of the small float64 panel: launches and latency
    add("apply_panel64_f64", "apply", 1, 64, 64, "f64")
    # one RVE of the benchmarked 512^2 composite, alone on the GPU
    add("apply_512_mixed", "apply", 1, 512, 512, "mixed")
    # four of them in one launch per pass, the grouping of a batch of increments
    add("apply_4x512_mixed", "apply", 1, 512, 512, "mixed", count=4)
    # the float64 solver on the same grid
    add("apply_512_f64", "apply", 1, 512, 512, "f64")
    # an odd-sided grid (no Nyquist column, a half-empty last row pair), isotropic degradation
    add("apply_243x729_mixed", "apply", 1, 243, 729, "mixed", split="none", gamma="continuous", control="strain")
    # the 128^3 porous solid
    add("apply_128cube_mixed", "apply", 128, 128, 128, "mixed")
    # the largest served grid
    add("apply_192cube_mixed", "apply", 192, 192, 192, "mixed")
    # a group of small uneven 3D RVEs, as in the ragged batch
    add("apply_4x96x64x48_mixed", "apply", 96, 64, 48, "mixed", count=4)
    # head of a Newton iteration, 2D and 3D
    add("newton_512_mixed", "newton", 1, 512, 512, "mixed")
    add("newton_96cube_mixed", "newton", 96, 96, 96, "mixed")
    # the float64 single-RVE crack run of the small panel: one increment
    add("increment_panel64_f64", "increment", 1, 64, 64, "f64")
    # the batched crack run: four 512^2 composites, one increment each
    add("increment_4x512_mixed", "increment", 1, 512, 512, "mixed", count=4)
    return out


def _side(rng, lo, hi):
    """A 2^a 3^b extent, its logarithm uniform over [lo, hi]."""
    want = math.log(lo) + rng.random() * math.log(hi / lo)
    return min((s for s in SMOOTH if lo <= s <= hi), key=lambda s: abs(math.log(s) - want))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "newton"])
    if rng.random() < 0.08:
        # a crack increment of one small 2D RVE
        side = rng.choice([48, 64, 96, 128])
        return _case("increment", 1, side, side, rng.choice(["mixed", "f64"]))
    precision = "mixed" if rng.random() < 0.75 else "f64"
    split = "spectral" if rng.random() < 0.8 else "none"
    gamma = "rotated" if rng.random() < 0.85 else "continuous"
    control = "crack" if rng.random() < 0.8 else "strain"
    if rng.random() < 0.55:
        nz, ny, nx = 1, _side(rng, 48, 1024), _side(rng, 48, 1024)
    else:
        nz, ny, nx = _side(rng, 16, 192), _side(rng, 16, 192), _side(rng, 16, 192)
    if rng.random() < 0.5:  # the usual grids: square, cubic, or sides that a user picks from
        if nz == 1:
            ny, nx = (rng.choice([128, 192, 256, 384, 512, 768, 1024]) for _ in range(2))
        else:
            nz, ny, nx = (rng.choice([32, 48, 64, 96, 128]) for _ in range(3))
    count = 1
    if kind == "apply" and nz * ny * nx <= 1 << 19 and rng.random() < 0.5:
        count = rng.randint(2, 6)
    return _case(kind, nz, ny, nx, precision, count, split, gamma, control)


# ---- inputs -----------------------------------------------------------------------------

def _shape(case):
    return (case["ny"], case["nx"]) if case["nz"] == 1 else (case["nz"], case["ny"], case["nx"])


def _input(case, seed):
    """The microstructure of one RVE."""
    shape = _shape(case)
    rng = np.random.default_rng(seed)
    if case["kind"] == "increment" and case["count"] == 1:
        n = shape[0]
        return ms.homogeneous_panel(n, notch_len=n // 4 + int(rng.integers(-2, 3)), nu=float(rng.uniform(0.25, 0.35)),
                                    Gc=float(rng.uniform(0.8e-3, 1.2e-3)))
    if len(shape) == 2:
        r = 12.0 if min(shape) >= 128 else 3.0
        inp = ms.fibre_composite(n=shape[1], ny=shape[0], radius=r, fraction=0.4 if min(shape) >= 128 else 0.2,
                                 notch_len=min(32, shape[1] // 4), seed=seed)
    else:
        inp = ms.porous_solid(shape=shape, radius=min(8.0, max(3.0, min(shape) / 8.0)), porosity=0.1,
                              notch_radius=min(10.0, min(shape) / 5.0), seed=seed, E_pore=1e-3)
    return inp


def _state(inp, seed):
    """A linearisation point: (eps_tilde Mandel (m, n), phi (n,), H (n,), E), float64 on the GPU."""
    shape = tuple(inp.shape)
    d = len(shape)
    m = 3 if d == 2 else 6
    n = int(np.prod(shape))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    f64 = dict(dtype=torch.float64, device="cuda")
    E = 4e-3 * (1.0 + 0.5 * float(torch.rand((), generator=g, **f64)))
    eps = 0.3 * E * torch.randn((m, n), generator=g, **f64)
    notch = torch.from_numpy(np.ascontiguousarray(inp.notch)).cuda()
    idx = torch.nonzero(notch.reshape(shape), as_tuple=False).double()
    # distance to the notch's plane segment, for the profile exp(-|x| / ell) around it
    ax = [torch.arange(s, **f64) for s in shape]
    lo, hi = idx.min(0).values, idx.max(0).values
    dist2 = torch.zeros(shape, **f64)
    for a in range(d):
        c = torch.clamp(lo[a] - ax[a], min=0.0) + torch.clamp(ax[a] - hi[a], min=0.0)
        dist2 += (c * c).reshape([-1 if b == a else 1 for b in range(d)])
    phi = 0.95 * torch.exp(-torch.sqrt(dist2) / float(inp.ell)).reshape(-1)
    phi = phi + 0.02 * torch.rand(n, generator=g, **f64)
    phi = torch.where(notch.reshape(-1) > 0, torch.ones_like(phi), phi)
    H = 0.5 * E * E * torch.rand(n, generator=g, **f64) * (torch.rand(n, generator=g, **f64) < 0.5)
    return eps, phi, H, E


def _x(seed, c, n, dtype):
    """A Krylov direction: c channels of n values and the E slot, the phase field growing on average."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    x = torch.randn(c * n, generator=g, dtype=torch.float32, device="cuda").to(dtype)
    x[(c - 1) * n:] += 0.5
    xE = torch.randn(1, generator=g, dtype=torch.float64, device="cuda")
    return x, xE


def _sub(seed, k):
    return int(seed) * 1009 + 13 * k + 1


def _rve(case, inp, **kw):
    return B.RVE(inp, precision=B.RVE_MIXED if case["precision"] == "mixed" else B.RVE_FP64,
                 split=B.RVE_SPLIT_SPECTRAL if case["split"] == "spectral" else B.RVE_SPLIT_NONE,
                 gamma_op=B.RVE_GAMMA_ROTATED if case["gamma"] == "rotated" else B.RVE_GAMMA_CONTINUOUS, **kw)


def prepare(case, seed):
    st = {"case": case, "rves": []}
    if case["kind"] == "increment":
        # the committed states of a running crack: start-up of each RVE
        inps = [_input(case, _sub(seed, k)) for k in range(case["count"])]
        # mixed runs at the benchmark's Newton tolerance, float64 runs at the default one
        tol = {"newton_tol": 1e-8} if case["precision"] == "mixed" else {}
        st["rves"] = [_rve(case, inp, **tol) for inp in inps]
        st["states"] = []
        for g in st["rves"]:
            su = g.startup()
            st["states"].append((g.field(B.RVE_FIELD_EPS_T), g.field(B.RVE_FIELD_PHI), g.field(B.RVE_FIELD_H), su["E"],
                                 su["tau"]))
        return st
    ctrl = B.RVE_CTRL_CRACK if case["control"] == "crack" else B.RVE_CTRL_STRAIN
    dt = torch.float32 if case["precision"] == "mixed" else torch.float64
    bufs = []
    yE = torch.zeros(case["count"], dtype=torch.float64, device="cuda")
    for k in range(case["count"]):
        inp = _input(case, _sub(seed, k))
        g = _rve(case, inp)
        eps, phi, H, E = _state(inp, _sub(seed, k))
        g.set_state(eps.cpu().numpy(), phi.cpu().numpy(), H.cpu().numpy(), E)
        g.linearize(ctrl, 1.0)
        g.autotune()
        x, xE = _x(_sub(seed, k), g.m + 1, g.n, dt)
        bufs.append((x, xE, torch.zeros_like(x), yE[k:k + 1]))
        st["rves"].append(g)
    st["ctrl"] = ctrl
    st["yE"] = yE
    st["bufs"] = bufs
    st["ptrs"] = [[b[i].data_ptr() for b in bufs] for i in range(4)]
    return st


def run(st):
    case, rves = st["case"], st["rves"]
    if case["kind"] == "increment":
        for g, s in zip(rves, st["states"]):
            g.set_state(*s)
        if len(rves) == 1:
            steps = [rves[0].crack_increment(1.0)]
        else:
            steps, status = B.batch_crack_increment(rves, [1.0] * len(rves))
            if any(status):
                raise RuntimeError(f"increment failed: {status}")
        # a mixed run holds its increments to the Newton tolerance, well within 32 bits
        dt = np.float32 if case["precision"] == "mixed" else np.float64
        return [{"phi": g.field(B.RVE_FIELD_PHI).astype(dt), "E": dt(r["E"]), "sigma": np.array(r["sigma"], dt),
                 "gamma": dt(r["gamma"])} for g, r in zip(rves, steps)]
    if case["kind"] == "newton":
        rves[0].linearize(st["ctrl"], 1.0)
    if len(rves) == 1:
        rves[0].apply_device(*(p[0] for p in st["ptrs"]))
    else:
        B.apply_device_batch(rves, *st["ptrs"])
    # the E slots in the precision of the vectors that they belong to
    return {"y": [b[2] for b in st["bufs"]], "yE": st["yE"].to(st["bufs"][0][0].dtype)}


def work(case):
    """Compulsory bytes and operations of one pass.  An apply reads the vector (c channels), the
    tangent channels of the linearisation and writes the result; its operations are the forward
    and inverse real FFTs of c channels and the pointwise tangent products.  A linearisation
    reads strain, phase field, history (float64) and material and writes stress, history,
    residual, right-hand side and tangent.  An increment counts 600 applies, about what the
    benchmarked composite needs, with the Krylov vectors of two applies per iteration read and
    written once."""
    d = 2 if case["nz"] == 1 else 3
    m = 3 if d == 2 else 6
    c = m + 1
    n = case["nz"] * case["ny"] * case["nx"]
    tan = m * (m + 1) // 2 + m + 5
    p = 4 if case["precision"] == "mixed" else 8
    apply_bytes = p * (2 * c + tan) * n
    apply_flops = n * (2 * c * 2.5 * math.log2(n) + 2 * m * m + 10 * m)
    if case["kind"] == "apply":
        b, f = apply_bytes, apply_flops
    elif case["kind"] == "newton":
        b = apply_bytes + (8 * (m + 2) + 1 + 8 * (m + 1) + 8 * c + p * c + p * tan) * n
        f = apply_flops + n * (2 * c * 2.5 * math.log2(n) + 40 * m * m)
    else:
        b = 600 * (apply_bytes + 4 * p * c * n)
        f = 600 * (apply_flops + 6 * c * n)
    return {"bytes": case["count"] * b, "flops": case["count"] * f}


# ---- the same results in 64 bits, plain torch ------------------------------------------

def _tensor(mv, d):
    """(m, n) Mandel -> (n, d, d)."""
    n = mv.shape[1]
    t = torch.empty((n, d, d), dtype=torch.float64, device=mv.device)
    r = 1.0 / math.sqrt(2.0)
    for a in range(d):
        t[:, a, a] = mv[a]
    pairs = [(0, 1)] if d == 2 else [(1, 2), (0, 2), (0, 1)]
    for k, (a, b) in enumerate(pairs):
        t[:, a, b] = t[:, b, a] = r * mv[d + k]
    return t


def _mandel(t):
    d = t.shape[-1]
    pairs = [(0, 1)] if d == 2 else [(1, 2), (0, 2), (0, 1)]
    return torch.stack([t[:, a, a] for a in range(d)] + [math.sqrt(2.0) * t[:, a, b] for a, b in pairs])


def _eigh(e):
    """Eigenvalues (n, d) and eigenvectors (columns of (n, d, d)) by cyclic Jacobi rotations."""
    n, d = e.shape[0], e.shape[-1]
    A = [[e[:, i, j].clone() for j in range(d)] for i in range(d)]
    Q = [[torch.full((n,), float(i == j), dtype=torch.float64, device=e.device) for j in range(d)] for i in range(d)]
    for _ in range(8 if d == 3 else 1):
        for p in range(d):
            for q in range(p + 1, d):
                flat = A[p][q] == 0
                theta = (A[q][q] - A[p][p]) / torch.where(flat, torch.ones_like(A[p][q]), 2 * A[p][q])
                t = torch.where(theta >= 0, 1.0, -1.0) / (theta.abs() + torch.sqrt(theta * theta + 1))
                t = torch.where(flat, torch.zeros_like(t), t)
                c = 1 / torch.sqrt(t * t + 1)
                s = t * c
                for r in range(d):
                    A[r][p], A[r][q] = c * A[r][p] - s * A[r][q], s * A[r][p] + c * A[r][q]
                for r in range(d):
                    A[p][r], A[q][r] = c * A[p][r] - s * A[q][r], s * A[p][r] + c * A[q][r]
                for r in range(d):
                    Q[r][p], Q[r][q] = c * Q[r][p] - s * Q[r][q], s * Q[r][p] + c * Q[r][q]
    return torch.stack([A[i][i] for i in range(d)], 1), torch.stack([torch.stack(row, 1) for row in Q], 1)


def _freqs(shape, gamma):
    """Per axis (x, y[, z]) the direction symbols and |xi|^2, each shaped to broadcast on the grid."""
    d = len(shape)
    sn, cs, x2 = [], [], []
    for a in range(d):
        N = shape[d - 1 - a]
        k = torch.arange(N, dtype=torch.float64, device="cuda")
        k = torch.where(2 * k < N, k, k - N)
        xi = 2.0 * math.pi * k / N
        nyq = 2 * k == -N
        if gamma == "rotated":
            s, c = torch.sin(xi / 2), torch.where(nyq, torch.zeros_like(xi), torch.cos(xi / 2))
        else:
            s, c = torch.where(nyq, torch.zeros_like(xi), xi), torch.ones_like(xi)
        view = [1] * d
        view[d - 1 - a] = N
        sn.append(s.reshape(view))
        cs.append(c.reshape(view))
        x2.append((xi * xi).reshape(view))
    return sn, cs, x2


def _project(t, shape, gamma):
    """F^-1[ Gamma : F[t] ] of a field of symmetric tensors (n, d, d)."""
    d = len(shape)
    sn, cs, _ = _freqs(shape, gamma)
    nvec = []
    for a in range(d):
        v = sn[a]
        for b in range(d):
            if b != a:
                v = v * cs[b]
        nvec.append(v.expand(shape))
    nn = sum(v * v for v in nvec)
    inv = torch.where(nn > 0, 1.0 / torch.sqrt(torch.where(nn > 0, nn, torch.ones_like(nn))), torch.zeros_like(nn))
    nvec = [v * inv for v in nvec]
    hat = {}
    for a in range(d):
        for b in range(a, d):
            hat[a, b] = hat[b, a] = torch.fft.fftn(t[:, a, b].reshape(shape))
    v = [sum(hat[a, b] * nvec[b] for b in range(d)) for a in range(d)]
    s = sum(v[a] * nvec[a] for a in range(d))
    out = torch.empty_like(t)
    for a in range(d):
        for b in range(a, d):
            q = v[a] * nvec[b] + nvec[a] * v[b] - s * nvec[a] * nvec[b]
            out[:, a, b] = out[:, b, a] = torch.fft.ifftn(q).real.reshape(-1)
    return out


def _laplace(u, shape, x2):
    return torch.fft.ifftn(torch.fft.fftn(u.reshape(shape)) * sum(x2)).real.reshape(-1)


def _exact_one(case, seed):
    shape = _shape(case)
    d = len(shape)
    m = 3 if d == 2 else 6
    inp = _input(case, seed)
    eps, phi, H0, E = _state(inp, seed)
    n = phi.numel()
    x, xE = _x(seed, m + 1, n, torch.float32 if case["precision"] == "mixed" else torch.float64)
    x = x.double().reshape(m + 1, n)
    xE = float(xE)
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()  # noqa: E731
    ph = torch.from_numpy(np.ascontiguousarray(inp.phase).reshape(-1)).long().cuda()
    Em, nu, Gct = cuda(inp.E), cuda(inp.nu), cuda(inp.Gc)
    lam_t, mu_t = Em * nu / ((1 + nu) * (1 - 2 * nu)), Em / (2 * (1 + nu))
    lam, mu, Gc = lam_t[ph], mu_t[ph], Gct[ph]
    s1 = 1.0 / float((lam_t + 2 * mu_t).max())
    ell = float(inp.ell)
    notch = torch.from_numpy(np.ascontiguousarray(inp.notch).reshape(-1)).cuda() > 0
    f = torch.from_numpy(np.asarray(inp.f, dtype=np.float64)).cuda()
    eye = torch.eye(d, dtype=torch.float64, device="cuda")
    e = _tensor(eps, d) + f * E
    g = (1 - phi) ** 2
    gp = -2 * (1 - phi)
    tr = torch.einsum("nii->n", e)
    de = _tensor(x[:m], d) + f * xE
    trd = torch.einsum("nii->n", de)
    if case["split"] == "spectral":
        z, Q = _eigh(e)
        zp = torch.clamp(z, min=0.0)
        trp = torch.clamp(tr, min=0.0)
        psi = 0.5 * lam * trp ** 2 + mu * (zp ** 2).sum(1)
        ep = torch.einsum("nik,nk,njk->nij", Q, zp, Q)
        drive = 2 * mu[:, None, None] * ep + (lam * trp)[:, None, None] * eye
        dz = z[:, :, None] - z[:, None, :]
        tie = dz.abs() <= 1e-12 * z.abs().max(1).values[:, None, None]
        mean = 0.5 * (z[:, :, None] + z[:, None, :])
        L = torch.where(tie, (mean > 0).double(), (zp[:, :, None] - zp[:, None, :]) / torch.where(tie, torch.ones_like(dz), dz))
        dp = torch.einsum("nip,npq,njq->nij", Q, L * torch.einsum("nip,nij,njq->npq", Q, de, Q), Q)
        hp = (tr > 0).double()
        vol = g * lam * hp + lam * (1 - hp)
        dsig = 2 * (g * mu)[:, None, None] * dp + 2 * mu[:, None, None] * (de - dp) + (vol * trd)[:, None, None] * eye
    else:
        psi = 0.5 * lam * tr ** 2 + mu * (e * e).sum((1, 2))
        drive = 2 * mu[:, None, None] * e + (lam * tr)[:, None, None] * eye
        dsig = g[:, None, None] * (2 * mu[:, None, None] * de + (lam * trd)[:, None, None] * eye)
    Hc = torch.maximum(psi, H0)
    chi = (psi >= H0).double()
    Lbar = 0.0
    _, _, x2 = _freqs(shape, case["gamma"])
    for q in x2:
        Lbar += float(q.mean())
    free = (~notch).double()
    dphi = x[m] * free
    t = s1 * (dsig + (free * gp * dphi)[:, None, None] * drive)
    y = torch.empty((m + 1, n), dtype=torch.float64, device="cuda")
    y[:m] = _mandel(_project(t, shape, case["gamma"]))
    s2 = 1.0 / (Gc / ell + 2 * Hc + Gc * ell * Lbar)
    coup = (drive * de).sum((1, 2))
    y[m] = free * s2 * (chi * gp * coup + (Gc / ell + 2 * Hc) * dphi + Gc * ell * _laplace(dphi, shape, x2)) + notch * x[m]
    if case["control"] == "crack":
        w = free * (phi / ell + ell * _laplace(phi, shape, x2))
        yE = (w * dphi).sum().reshape(1)
    else:
        yE = torch.tensor([xE], dtype=torch.float64, device="cuda")
    return {"y": y.reshape(-1), "yE": yE}


def exact(case, seed):
    """What run() returns, in 64 bits; an increment has no plain closed evaluation."""
    if case["kind"] == "increment":
        return None
    one = [_exact_one(case, _sub(seed, k)) for k in range(case["count"])]
    return {"y": [o["y"] for o in one], "yE": torch.cat([o["yE"] for o in one])}

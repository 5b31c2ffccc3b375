"""Measured workloads of the folded-spectrum library, through its public Python entry points.

Every case is a call that a program using the library makes: the H application on
device blocks (both precisions; stored and generated projectors), the eigensolves,
the folded linear solve, ChebFD, k-interpolation, the dense eigensolver and the
training step of the learned preconditioner.  Inputs are Gaussian-well boxes with
Gaussian s/p projectors on jittered simple-cubic sites, made from the seed alone.
Units are Hartree atomic units.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1907_06821_gb300 as fs

SPACING = 0.5556          # bohr per grid point of the boxes without a cell of their own
DEV = "cuda"


# ---------------------------------------------------------------- cases
def listed():
    return [
        # one small box: every kernel of an H application is shorter than its launch
        dict(name="apply_c64_tiny", kind="apply", c64=True, n0=16, n1=16, n2=32, L0=10.0, L1=10.0, L2=20.0, ecut=5.0,
             kpt=0.0, natom=8, nproj=4, lattice=5.0, bands=8),
        # the block H application of the wire's solver, the call most of a mixed solve is made of
        dict(name="apply_c64_wire", kind="apply", c64=True, n0=72, n1=72, n2=144, L0=40.0, L1=40.0, L2=80.0, ecut=10.0,
             kpt=0.0, natom=256, nproj=8, lattice=5.0, bands=272),
        # the long wire: 1.3 million plane waves, projectors formed where they are used
        dict(name="apply_c64_longwire", kind="apply", c64=True, n0=108, n1=108, n2=432, L0=60.0, L1=60.0, L2=240.0,
             ecut=10.0, kpt=0.0, natom=990, nproj=8, lattice=6.0, bands=96),
        # FP64 H application at the wire's size: FP64 checks, ChebFD and linear solves are made of it
        dict(name="apply_f64_wire", kind="apply", c64=False, n0=72, n1=72, n2=144, L0=40.0, L1=40.0, L2=80.0,
             ecut=10.0, kpt=0.0, natom=256, nproj=8, lattice=5.0, bands=16),
        # a whole plain FP64 solve of the smallest box: many small steps, launches and latency
        dict(name="solve_f64_tiny", kind="solve", c64=False, n0=16, n1=16, n2=32, L0=10.0, L1=10.0, L2=20.0, ecut=5.0,
             natom=8, nproj=4, lattice=5.0, eref=0.0, states=8),
        # fragments of uneven grids solved together in mixed precision
        dict(name="batch_c64_fragments", kind="batch", grids="24x24x24,32x32x32,24x24x48,30x30x30",
             states="12,32,24,20", atoms="8,27,16,20", ecut=7.5, threads=4),
        # a whole mixed-precision solve in the interior of the medium box's spectrum
        dict(name="solve_c64_medium", kind="solve", c64=True, n0=48, n1=48, n2=96, L0=24.0, L1=24.0, L2=48.0,
             ecut=10.0, natom=64, nproj=8, lattice=5.0, eref=0.05, states=32),
        # the Rayleigh-Ritz problem of the wire's block (three blocks of 272 bands)
        dict(name="eigh_wire", kind="eigh", n=816, m=272, general=True),
        # interpolation between two k-points on the medium box's sphere
        dict(name="kinterp_medium", kind="kinterp", n0=48, n1=48, n2=96, L0=24.0, L1=24.0, L2=48.0, ecut=10.0,
             b1=128, b2=136, alpha=0.35),
        # a bounded number of PCG steps for four wave packets in the medium box
        dict(name="linear_medium", kind="linear", n0=48, n1=48, n2=96, L0=24.0, L1=24.0, L2=48.0, ecut=10.0, natom=64,
             nproj=8, lattice=5.0, eref=0.05, nrhs=4, steps=12),
        # one filter step of ChebFD on a fragment
        dict(name="chebfd_fragment", kind="chebfd", n0=32, n1=32, n2=32, ecut=7.5, natom=27, nproj=4, lattice=5.0,
             degree=60, nvec=64),
        # one full-batch training step of the learned preconditioner on a recorded solve's rows
        dict(name="learned_grad", kind="learned", rows=153312),
    ]


GRID = (16, 18, 20, 24, 30, 32, 36, 40, 45, 48, 54, 60, 64, 72)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, most):
    n = [rng.choice(GRID[:11]) for _ in range(2)] + [rng.choice(GRID)]
    while n[0] * n[1] * n[2] > most:
        n[n.index(max(n))] = rng.choice(GRID[:8])
    return n


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "apply", "solve", "eigh", "kinterp", "linear", "chebfd", "learned"))
    if kind == "apply":
        c64 = rng.random() < 0.5
        n = _draw_grid(rng, 54 * 54 * 72)
        ecut = round(rng.uniform(3.0, 10.0), 2)
        natom = _log(rng, 1, 128)
        nproj = rng.choice((0, 1, 4, 8))
        work = max(1, natom * nproj) * _npw_estimate(n, [SPACING * v for v in n], ecut)
        bands = max(1, min(_log(rng, 1, 272), int((4e10 if c64 else 3e9) / work)))
        return dict(kind="apply", c64=c64, n0=n[0], n1=n[1], n2=n[2], ecut=ecut, kpt=round(rng.uniform(-0.1, 0.1), 3),
                    natom=natom, nproj=nproj, lattice=round(rng.uniform(3.0, 6.0), 2), bands=bands)
    if kind == "solve":
        n = [rng.choice((16, 18, 20, 24)), rng.choice((16, 18, 20, 24)), rng.choice((24, 30, 32))]
        return dict(kind="solve", c64=rng.random() < 0.5, n0=n[0], n1=n[1], n2=n[2],
                    ecut=round(rng.uniform(3.0, 5.0), 2), natom=rng.choice((8, 12, 18)), nproj=4, lattice=4.0,
                    eref=-1.0, states=rng.randint(4, 20))
    if kind == "eigh":
        n = _log(rng, 4, 816)
        return dict(kind="eigh", n=n, m=max(1, rng.randint(n // 4, n // 2)), general=rng.random() < 0.5)
    if kind == "kinterp":
        n = _draw_grid(rng, 36 * 36 * 72)
        b1 = _log(rng, 3, 128)
        return dict(kind="kinterp", n0=n[0], n1=n[1], n2=n[2], ecut=round(rng.uniform(5.0, 10.0), 2), b1=b1,
                    b2=b1 + rng.randint(0, 12), alpha=round(rng.uniform(0.05, 0.95), 3))
    if kind == "linear":
        n = _draw_grid(rng, 40 * 40 * 48)
        return dict(kind="linear", n0=n[0], n1=n[1], n2=n[2], ecut=round(rng.uniform(4.0, 10.0), 2),
                    natom=_log(rng, 2, 48), nproj=4, lattice=4.5, eref=round(rng.uniform(-0.2, 0.3), 3),
                    nrhs=rng.randint(1, 7), steps=rng.randint(3, 12))
    if kind == "chebfd":
        n = [rng.choice((18, 20, 24, 30))] * 2 + [rng.choice((24, 30, 32, 36))]
        return dict(kind="chebfd", n0=n[0], n1=n[1], n2=n[2], ecut=round(rng.uniform(4.0, 7.5), 2),
                    natom=rng.randint(4, 20), nproj=4, lattice=4.5, degree=rng.randint(20, 60),
                    nvec=rng.randint(6, max(6, int(n[0] * n[1] * n[2] * SPACING ** 3 / 90.0))))
    return dict(kind="learned", rows=_log(rng, 40, 150000))


# ---------------------------------------------------------------- inputs
def _grid(c):
    return [c["n0"], c["n1"], c["n2"]]


def _cell(c):
    return [float(c.get("L%d" % d, SPACING * c["n%d" % d])) for d in range(3)]


def _npw_estimate(n, L, ecut):
    return max(1.0, L[0] * L[1] * L[2] * (2.0 * ecut) ** 1.5 / (6.0 * math.pi ** 2))


def _box(n, L, ecut, kpt, natom, nproj, lattice, seed):
    """Positions, depths, V(r) and projectors of a box of jittered simple-cubic sites."""
    rng = np.random.default_rng(seed)
    L = np.asarray(L, dtype=np.float64)
    # as many sites along z as the cell is longer than wide
    nx = max(1, int(round((natom * L[0] * L[1] / L[2] ** 2) ** (1.0 / 3.0))))
    nz = -(-natom // (nx * nx))
    cand = np.array([[i, j, l] for l in range(nz) for i in range(nx) for j in range(nx)], dtype=np.float64)[:natom]
    a = np.minimum(lattice, L / np.array([nx, nx, nz]))
    sites = L / 2 + (cand - (np.array([nx, nx, nz]) - 1) / 2.0) * a
    pos = np.mod(sites + rng.normal(0.0, 0.1, size=sites.shape), L)
    U = rng.uniform(1.0, 3.0, size=natom)
    ax = []
    for d in range(3):  # periodic Gaussians along each axis
        x = np.arange(n[d]) * (L[d] / n[d])
        images = range(-2, 3) if L[d] > 8.0 else range(-4, 5)
        ax.append(sum(np.exp(-0.5 * (x[None, :] - pos[:, d:d + 1] - t * L[d]) ** 2) for t in images))
    v = -np.einsum("axy,az->xyz", (U[:, None] * ax[0])[:, :, None] * ax[1][:, None, :], ax[2], optimize=True)
    widths = {0: [], 1: [1.0], 4: [1.0], 8: [0.8, 1.2]}[nproj]
    proj = []
    for w in widths:
        proj += [(0, 0, w)] + ([(1, d, w) for d in range(3)] if nproj >= 4 else [])
    D = np.zeros((natom, nproj, nproj))
    for p in range(nproj):
        D[:, p, p] = rng.uniform(0.1, 0.5, size=natom)
    k = np.array([kpt, -0.5 * kpt, 0.3 * kpt])
    return dict(L=L, n=tuple(n), ecut=ecut, k=k, vloc=v, pos=pos, proj=proj, D=D, U=U)


def _case_box(c, seed):
    return _box(_grid(c), _cell(c), c["ecut"], c.get("kpt", 0.0), c["natom"], c["nproj"], c["lattice"], seed)


def _context(b, **kw):
    return fs.Context(b["L"], b["n"], b["ecut"], b["k"], b["vloc"], pos=b["pos"], proj=b["proj"], D=b["D"], **kw)


def _randn(gen, *shape, dtype=torch.complex128):
    return torch.randn(*shape, dtype=dtype, device=DEV, generator=gen)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _kin(b):
    """(q [npw][3], |q|^2 / 2, Miller indices) of the sphere, in the library's order."""
    bb = 2.0 * np.pi / b["L"]
    qmax = math.sqrt(2.0 * b["ecut"])
    h = [int(math.floor((qmax + abs(b["k"][d])) / bb[d])) + 1 for d in range(3)]
    g = np.stack(np.meshgrid(*[np.arange(-h[d], h[d] + 1) for d in range(3)], indexing="ij"), -1).reshape(-1, 3)
    q = b["k"][None, :] + g * bb[None, :]
    kin = 0.5 * ((q[:, 0] * q[:, 0] + q[:, 1] * q[:, 1]) + q[:, 2] * q[:, 2])
    keep = kin <= b["ecut"]
    return q[keep], kin[keep], g[keep]


def _bands(kin, gen, nb):
    """Random bands with the decay of plane-wave states, unit norm."""
    x = _randn(gen, nb, kin.shape[0]) / (1.0 + kin)[None, :]
    return x / torch.linalg.vector_norm(x, dim=1, keepdim=True)


def _packets(b, nrhs, seed):
    """Unit-norm Gaussian wave packets along z (analytic Fourier coefficients)."""
    q, _, _ = _kin(b)
    q = torch.as_tensor(q, device=DEV)
    rng = np.random.default_rng(seed + 77)
    out = []
    for _ in range(nrhs):
        r0 = rng.uniform(0.2, 0.8, size=3) * b["L"]
        env = torch.exp(-2.0 * (q[:, 0] ** 2 + q[:, 1] ** 2) - 4.5 * (q[:, 2] - 0.8) ** 2)
        w = torch.polar(env, -(q[:, 0] * r0[0] + q[:, 1] * r0[1] + (q[:, 2] - 0.8) * r0[2]))
        out.append(w / torch.linalg.vector_norm(w))
    return torch.stack(out)


def _hermitian(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return (a + a.conj().T) / (2.0 * math.sqrt(n))


def _eigh_inputs(c, seed):
    rng = np.random.default_rng(seed)
    n = c["n"]
    A = np.asfortranarray(_hermitian(rng, n))
    B = np.asfortranarray(np.eye(n) + 0.3 * _hermitian(rng, n)) if c["general"] else None
    u = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    return A, B, u


def _kinterp_inputs(c, npw, seed):
    """Orthonormal blocks of two near k-points and their eigenvalues."""
    g = _gen(seed)
    rng = np.random.default_rng(seed)
    P2 = torch.linalg.qr(_randn(g, npw, c["b2"]))[0].T.contiguous()
    mix = torch.eye(c["b1"], c["b2"], dtype=torch.complex128, device=DEV) + 0.2 * _randn(g, c["b1"], c["b2"]) / math.sqrt(c["b2"])
    P1 = mix @ P2 + 0.3 * _randn(g, c["b1"], npw) / math.sqrt(npw)
    P1 = torch.linalg.qr(P1.T)[0].T.contiguous()
    e1, e2 = np.sort(rng.uniform(-0.3, 0.4, c["b1"])), np.sort(rng.uniform(-0.3, 0.4, c["b2"]))
    return P1, e1, P2, e2, _randn(g, npw)


def _learned_inputs(c, seed):
    rng = np.random.default_rng(seed)
    n = c["rows"]
    F = np.stack([(np.arange(n) % 32 + 0.5) / 32, rng.normal(-0.5, 1.0, n), rng.uniform(-1, 1, n),
                  rng.uniform(-0.6, -0.1, n)], axis=1).astype(np.float32)
    zt = np.clip(rng.normal(0.0, 0.7, n), -2.3, 2.3).astype(np.float32)
    wt = (rng.random(n) ** 2 / 16).astype(np.float32)
    parts = []
    for i, (a, b) in enumerate(((4, 128), (128, 128), (128, 128), (128, 1))):
        lim = 1.0 / math.sqrt(a)
        parts += [rng.uniform(-lim, lim, a * b), rng.uniform(-lim, lim, b)]
    return F, zt, wt, np.concatenate(parts).astype(np.float32)


def _batch_boxes(c, seed):
    boxes = []
    for i, (g, s, a) in enumerate(zip(c["grids"].split(","), c["states"].split(","), c["atoms"].split(","))):
        n = [int(v) for v in g.split("x")]
        b = _box(n, [SPACING * v for v in n], c["ecut"], 0.0, int(a), 4, 4.0, 1000 * seed + i)
        b["e_ref"] = -0.5 * float(np.mean(b["U"]))
        boxes.append((b, int(s)))
    return boxes


def _guard(states):
    return max(4, states // 16)


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(case=c)
    if kind == "apply":
        b = _case_box(c, seed)
        s["ctx"] = _context(b, precision=fs.FS_MIXED if c["c64"] else fs.FS_FP64)
        kin = torch.as_tensor(_kin(b)[1], device=DEV)
        g = _gen(seed)
        dt = torch.complex64 if c["c64"] else torch.complex128
        s["psi"] = torch.empty(c["bands"], s["ctx"].npw, dtype=dt, device=DEV)
        for i in range(0, c["bands"], 16):
            s["psi"][i:i + 16] = _bands(kin, g, min(16, c["bands"] - i)).to(dt)
        s["out"] = torch.empty_like(s["psi"])
    elif kind == "solve":
        b = _case_box(c, seed)
        s["ctx"] = _context(b, precision=fs.FS_MIXED if c["c64"] else fs.FS_FP64, maxit=3000)
        torch.cuda.synchronize()
        x0 = _randn(_gen(seed), c["states"] + _guard(c["states"]), s["ctx"].npw)
        torch.cuda.synchronize()
        s["ctx"].set_initial_states(x0, damp=True)
    elif kind == "batch":
        boxes = _batch_boxes(c, seed)
        s["ctx"] = [_context(b, precision=fs.FS_MIXED, maxit=3000) for b, _ in boxes]
        for i, (ctx, (b, n)) in enumerate(zip(s["ctx"], boxes)):
            x0 = _randn(_gen(seed + i), n + _guard(n), ctx.npw)
            torch.cuda.synchronize()
            ctx.set_initial_states(x0, damp=True)
        s["e"], s["n"] = [b["e_ref"] for b, _ in boxes], [n for _, n in boxes]
        s["batch"] = fs.Batch(s["ctx"], nthreads=c["threads"])
    elif kind == "eigh":
        s["ctx"] = _context(_box([16, 16, 16], [10.0, 10.0, 10.0], 3.0, 0.0, 1, 0, 5.0, seed))
        s["A"], s["B"], s["u"] = _eigh_inputs(c, seed)
    elif kind == "kinterp":
        s["ctx"] = _context(_box(_grid(c), _cell(c), c["ecut"], 0.0, 1, 0, 5.0, seed))
        s["in"] = _kinterp_inputs(c, s["ctx"].npw, seed)
    elif kind == "linear":
        b = _case_box(c, seed)
        s["ctx"] = _context(b)
        s["w"] = _packets(b, c["nrhs"], seed)
    elif kind == "chebfd":
        b = _case_box(c, seed)
        s["ctx"] = _context(b)
        s["bounds"] = (float(b["vloc"].min()) - 0.1, c["ecut"] + 3.0)
        s["seed"] = seed % (1 << 31)
    else:
        s["ctx"] = _context(_box([16, 16, 16], [10.0, 10.0, 10.0], 3.0, 0.0, 1, 0, 5.0, seed))
        F, zt, wt, w = _learned_inputs(c, seed)
        s["ctx"].precond_weights(w)
        s["in"] = [torch.as_tensor(v, device=DEV) for v in (F, zt, wt)]
    torch.cuda.synchronize()
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "apply":
        return s["ctx"].apply_H(s["psi"], out=s["out"], shift=0.05)
    if kind == "solve":
        return np.sort(s["ctx"].solve(c["eref"], c["states"], tol=1e-6)["eps"])
    if kind == "batch":
        r = s["batch"].solve(s["e"], s["n"], tol=1e-6)
        return [np.sort(x["eps"]) for x in r] + [int(x["nconv"]) for x in r]
    if kind == "eigh":
        w, Z = s["ctx"].dense_eigh(s["A"], m=c["m"], B=s["B"])
        p = np.conj(s["u"]) @ Z
        return w, Z * (np.conj(p) / np.abs(p))[None, :]
    if kind == "kinterp":
        P1, e1, P2, e2, u = s["in"]
        e, psi = s["ctx"].kinterp(c["alpha"], e1, P1, e2, P2)
        p = psi @ u.conj()   # the phase of every band against one fixed vector
        psi *= (p.conj() / p.abs())[:, None]
        return e, psi
    if kind == "linear":
        psi, _ = s["ctx"].linear_solve(s["w"], c["eref"], tol=1e-12, maxit=c["steps"], allow_unconverged=True)
        return psi
    if kind == "chebfd":
        lo, hi = s["bounds"]
        r = s["ctx"].chebfd(-0.5, 1.0, lo, hi, c["degree"], c["nvec"], 1, seed=s["seed"])
        return r["eps"]
    return s["ctx"].precond_loss_grad(*s["in"])


# ---------------------------------------------------------------- what a pass cannot do without
def _apply_work(n, L, ecut, nptot, bands, size):
    npw, grid = _npw_estimate(n, L, ecut), float(n[0] * n[1] * n[2])
    return (2.0 * bands * npw * size + grid * size / 2,
            bands * (10.0 * grid * math.log2(grid) + 16.0 * nptot * npw))


def _solve_work(n, L, ecut, nptot, states, size, its):
    """its block iterations: two H applications, Gram products and rotations of three blocks."""
    npw, m = _npw_estimate(n, L, ecut), states + _guard(states)
    by, fl = _apply_work(n, L, ecut, nptot, 2 * m, size)
    return its * (by + 8.0 * m * npw * size), its * (fl + 8.0 * npw * m * m * 15.0 + 100.0 * (3.0 * m) ** 3)


def work(case):
    c, kind = case, case["kind"]
    if kind == "apply":
        by, fl = _apply_work(_grid(c), _cell(c), c["ecut"], c["natom"] * c["nproj"], c["bands"], 8 if c["c64"] else 16)
    elif kind == "solve":
        by, fl = _solve_work(_grid(c), _cell(c), c["ecut"], c["natom"] * c["nproj"], c["states"],
                             8 if c["c64"] else 16, 60)
    elif kind == "batch":
        by = fl = 0.0
        for g, s, a in zip(c["grids"].split(","), c["states"].split(","), c["atoms"].split(",")):
            n = [int(v) for v in g.split("x")]
            x, y = _solve_work(n, [SPACING * v for v in n], c["ecut"], 4 * int(a), int(s), 8, 60)
            by, fl = by + x, fl + y
    elif kind == "eigh":
        n, m = float(c["n"]), float(c["m"])
        by = 16.0 * (n * n * (2 if c["general"] else 1) + n * m)
        fl = 16.0 / 3.0 * n ** 3 + 8.0 * n * n * m + (32.0 / 3.0 * n ** 3 if c["general"] else 0.0)
    elif kind == "kinterp":
        npw = _npw_estimate(_grid(c), _cell(c), c["ecut"])
        by = 16.0 * npw * (2 * c["b1"] + c["b2"])
        fl = 8.0 * npw * c["b1"] * (2.0 * c["b2"] + c["b1"])
    elif kind == "linear":
        by, fl = _apply_work(_grid(c), _cell(c), c["ecut"], c["natom"] * c["nproj"], c["nrhs"], 16)
        by, fl = by * 2 * c["steps"], fl * 2 * c["steps"]
    elif kind == "chebfd":
        by, fl = _apply_work(_grid(c), _cell(c), c["ecut"], c["natom"] * c["nproj"], c["nvec"], 16)
        by, fl = by * c["degree"], fl * c["degree"]
    else:
        by, fl = 24.0 * c["rows"] + 8.0 * 33793, 6.0 * 33280.0 * c["rows"]
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------------------- 64-bit values
class _Ham:
    """H on the sphere in plain FP64 torch: FFT local part and a projector table."""

    def __init__(self, b):
        q, kin, g = _kin(b)
        self.n = b["n"]
        self.kin = torch.as_tensor(kin, device=DEV)
        n = self.n
        self.at = torch.as_tensor(((g[:, 0] % n[0]) * n[1] + g[:, 1] % n[1]) * n[2] + g[:, 2] % n[2], device=DEV)
        self.v = torch.as_tensor(b["vloc"], device=DEV)
        self.D = torch.as_tensor(b["D"], device=DEV, dtype=torch.float64)
        self.q = torch.as_tensor(q, device=DEV)
        self.b, self.npw = b, len(kin)
        self.omega = float(np.prod(b["L"]))

    def beta(self, a):
        """Projector rows of atom a, [nproj][npw]."""
        ph = -(self.q @ torch.as_tensor(self.b["pos"][a], device=DEV))
        rows = []
        for l, ax, w in self.b["proj"]:
            r = (math.pi * w * w) ** -0.75 * (2.0 * math.pi * w * w) ** 1.5 / math.sqrt(self.omega) * torch.exp(-w * w * self.kin_free())
            rows.append(torch.polar(r, ph) if l == 0 else
                        torch.polar(math.sqrt(2.0) * w * r * torch.ones_like(ph), ph) * (-1j * self.q[:, ax]))
        return torch.stack(rows)

    def kin_free(self):
        return 0.5 * (self.q * self.q).sum(1)

    def apply(self, x, shift=0.0):
        out = torch.empty_like(x)
        ng = self.n[0] * self.n[1] * self.n[2]
        for i in range(0, x.shape[0], 16):
            xb = x[i:i + 16]
            f = torch.zeros(xb.shape[0], ng, dtype=torch.complex128, device=DEV)
            f[:, self.at] = xb
            f = f.view(-1, *self.n)
            f = torch.fft.fftn(torch.fft.ifftn(f, dim=(1, 2, 3)) * self.v, dim=(1, 2, 3)).reshape(xb.shape[0], ng)
            out[i:i + 16] = f[:, self.at] + (self.kin - shift) * xb
        if self.b["proj"]:
            step = max(1, int(5e8 // (self.npw * 16 * len(self.b["proj"]))))
            for a0 in range(0, len(self.b["pos"]), step):
                a1 = min(a0 + step, len(self.b["pos"]))
                be = torch.stack([self.beta(a) for a in range(a0, a1)])         # [atom][proj][npw]
                p = torch.einsum("apg,bg->bap", be.conj(), x)
                qd = torch.einsum("aij,baj->bai", self.D[a0:a1].to(torch.complex128), p)
                out += torch.einsum("bap,apg->bg", qd, be)
        return out

    def dense(self):
        return self.apply(torch.eye(self.npw, dtype=torch.complex128, device=DEV)).T


def _nearest(b, e_ref, states):
    """The eigenvalues nearest e_ref, ascending (None for a sphere too large for brute force)."""
    h = _Ham(b)
    if h.npw > 2400:
        return None
    w = np.linalg.eigvalsh(h.dense().cpu().numpy())
    return np.sort(w[np.argsort(np.abs(w - e_ref), kind="stable")[:states]])


def _exact_linear(b, w, e, steps, dE=0.5):
    """Polak-Ribiere PCG on (H - e)^2 psi = (H - e) w, all right-hand sides together."""
    h = _Ham(b)
    m = 1.0 / ((h.kin - e) ** 2 + dE * dE)
    dot = lambda x, y: (x.conj() * y).sum(1).real  # noqa: E731
    psi = torch.zeros_like(w)
    r = h.apply(w, e)
    z = m * r
    p, zr = z.clone(), dot(z, r)
    for it in range(steps):
        ap = h.apply(h.apply(p, e), e)
        a = (zr / dot(p, ap))[:, None]
        psi = psi + a * p
        old, r = r, r - a * ap
        z = m * r
        beta = torch.clamp((dot(z, r) - dot(z, old)) / zr, min=0.0)
        zr = dot(z, r)
        p = z + beta[:, None] * p
    return psi


def _exact_learned(F, zt, wt, theta):
    """Loss and gradient: weights rounded to BF16 in the forward pass, master weights in the backward pass."""
    def bf(x):
        return torch.as_tensor(x).to(torch.bfloat16).double()
    F, zt, wt = (torch.as_tensor(v).double() for v in (F, zt, wt))
    W, o = [], 0
    for a, b in ((4, 128), (128, 128), (128, 128), (128, 1)):
        W.append((theta[o:o + a * b].reshape(b, a), torch.as_tensor(theta[o + a * b:o + a * b + b]).double()))
        o += a * b + b
    h = [F]
    for i, (w, bias) in enumerate(W):
        pre = h[-1] @ bf(w).T + bias
        h.append(torch.tanh(pre) if i < 3 else pre)
    r = h[4][:, 0] - zt
    sw = wt.sum()
    loss = float((wt * r * r).sum() / sw)
    g, grads = (2.0 * wt * r / sw)[:, None], []
    for i in (3, 2, 1, 0):
        grads.append((g.T @ h[i], g.sum(0)))
        if i:
            g = (g @ torch.as_tensor(W[i][0]).double()) * (1.0 - h[i] ** 2)
    return loss, np.concatenate([np.concatenate([x.numpy().ravel(), y.numpy()]) for x, y in reversed(grads)])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "apply":
        if c["natom"] * c["nproj"] > 4000:
            return None
        b = _case_box(c, seed)
        h = _Ham(b)
        g = _gen(seed)
        dt = torch.complex64 if c["c64"] else torch.complex128
        psi = torch.cat([_bands(h.kin, g, min(16, c["bands"] - i)).to(dt) for i in range(0, c["bands"], 16)])
        return h.apply(psi.to(torch.complex128), 0.05)
    if kind == "solve":
        return _nearest(_case_box(c, seed), c["eref"], c["states"])
    if kind == "batch":
        return [_nearest(b, b["e_ref"], n) for b, n in _batch_boxes(c, seed)] + [None] * len(c["states"].split(","))
    if kind == "eigh":
        A, B, u = _eigh_inputs(c, seed)
        if B is None:
            w, Z = np.linalg.eigh(A)
        else:
            li = np.linalg.inv(np.linalg.cholesky(B))
            w, Z = np.linalg.eigh(li @ A @ li.conj().T)
            Z = li.conj().T @ Z
        Z = Z[:, :c["m"]]
        p = np.conj(u) @ Z
        return w[:c["m"]], Z * (np.conj(p) / np.abs(p))[None, :]
    if kind == "kinterp":
        b = _box(_grid(c), _cell(c), c["ecut"], 0.0, 1, 0, 5.0, seed)
        P1, e1, P2, e2, u = _kinterp_inputs(c, len(_kin(b)[1]), seed)
        S = (P1 @ P2.conj().T).cpu()          # S_il = <psi_l(k2)|psi_i(k1)>
        U = torch.linalg.solve_triangular(torch.linalg.cholesky(S @ S.conj().T), S, upper=False)
        al = c["alpha"]
        H = (1 - al) * (U.conj() * torch.as_tensor(e2)) @ U.T + al * torch.diag(torch.as_tensor(e1)).to(S.dtype)
        w, C = torch.linalg.eigh(H)
        C, U = C.to(DEV), U.to(DEV)
        psi = al * C.T @ P1 + (1 - al) * (C.T @ U) @ P2
        p = psi @ u.conj()
        return w, psi * (p.conj() / p.abs())[:, None]
    if kind == "linear":
        b = _case_box(c, seed)
        return _exact_linear(b, _packets(b, c["nrhs"], seed), c["eref"], c["steps"])
    if kind == "chebfd":
        return None   # the start vectors are the library's own
    return _exact_learned(*_learned_inputs(c, seed))

"""Performance cases: the calls a real-space orbital-free DFT program makes through the C ABI.

Every case names its kind, its grid (points per axis; the spacing is that of the aluminium
cells, 7.6 bohr / 32 points) and its options.  Inputs are what the calls meet in a run: charges
of Gaussian ions with smooth electron densities, density-like fields, right-hand sides of the
kernel map, all made on the GPU from a seed.

Kinds:
  laplacian    one Laplacian sweep of a field, FP32 or FP64, finite-difference order 2, 6 or 12
  poisson      one Poisson solve, plain FP64 or mixed precision, from a zero guess
  kernel       the complex shifted systems of the WT kernel for one right-hand side, mixed
  lr_map       the whole kernel map V[u] (potential and energy) of the WT functional, mixed
  ions         nuclear charge, self energy and Hellmann-Feynman forces of a cell
  batched      Poisson solves of several uneven cells in one call, mixed
  network      one application of the learned preconditioner to a residual
  ground       a whole WT ground state and its forces, mixed, converged tightly
"""
import math

import numpy as np
import torch

from paper_1412_8250_gb300 import binding as B, functionals as Fn, workloads as W

H = W.A_LATTICE / 32.0          # grid spacing, bohr
ELECTRON_WIDTH = 1.9            # width (bohr) of the Gaussians the test electron densities sum
POISSON_TOL = 1e-11             # relative residual: the long waves of a large cell amplify what is left
WT_ALPHA = (5.0 + math.sqrt(5.0)) / 6.0
WT_BETA = (5.0 - math.sqrt(5.0)) / 6.0


def listed():
    return [
        # the stencil rate a user quotes: single precision, the largest grid (3999 atoms)
        dict(name="laplacian_f32_320", kind="laplacian", n1=320, n2=320, n3=320, order=12, dtype="f32"),
        # the same operator in double precision on the 108-atom grid: one small, short call
        dict(name="laplacian_f64_96", kind="laplacian", n1=96, n2=96, n3=96, order=12, dtype="f64"),
        # the 4-atom unit cell's electrostatics: the smallest solve, all launch latency
        dict(name="poisson_32", kind="poisson", n1=32, n2=32, n3=32, order=12, form="mixed"),
        # the 108-atom cell's electrostatics, the solve a ground state repeats most
        dict(name="poisson_96", kind="poisson", n1=96, n2=96, n3=96, order=12, form="mixed"),
        # the 3999-atom cell's electrostatics: the largest solve
        dict(name="poisson_320", kind="poisson", n1=320, n2=320, n3=320, order=12, form="mixed"),
        # plain double-precision CG on a ragged grid that no multigrid coarsens, order 6
        dict(name="poisson_f64_ragged", kind="poisson", n1=45, n2=50, n3=54, order=6, form="f64"),
        # the two shifted systems of one density power at 864 atoms
        dict(name="kernel_192", kind="kernel", n1=192, n2=192, n3=192, order=12),
        # one outer iteration's kernel map on the 108-atom cell
        dict(name="lr_map_96", kind="lr_map", n1=96, n2=96, n3=96, order=12),
        # the ion terms of one geometry of the 108-atom cell
        dict(name="ions_108", kind="ions", r1=3, r2=3, r3=3, points=32),
        # several independent cells at once, 2 to 4 unit cells per axis
        dict(name="batched_12", kind="batched", cells=12, reps_seed=3),
        # the learned preconditioner on the 864-atom grid
        dict(name="network_192", kind="network", n1=192, n2=192, n3=192),
        # the whole calculation: 108 atoms, ground state and forces
        dict(name="ground_108", kind="ground", r1=3, r2=3, r3=3, points=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, most, multiple=1):
    """Three extents, log-uniform in [lo, hi], no more than `most` points in all."""
    while True:
        n = [max(multiple, multiple * int(round(_log_int(rng, lo, hi) / multiple))) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return dict(n1=n[0], n2=n[1], n3=n[2])


def draw(rng):
    kind = rng.choice(["laplacian", "laplacian", "poisson", "poisson", "poisson", "kernel", "lr_map",
                       "ions", "batched", "network", "ground"])
    if kind == "laplacian":
        return dict(kind=kind, **_grid(rng, 16, 400, 320 ** 3), order=rng.choice([2, 6, 12, 12]),
                    dtype=rng.choice(["f32", "f64"]))
    if kind == "poisson":
        form = rng.choice(["mixed", "mixed", "mixed", "f64"])
        if form == "f64":
            g = _grid(rng, 12, 80, 64 ** 3)
        elif rng.random() < 0.25:        # ragged: plain CG passes
            g = _grid(rng, 12, 80, 64 ** 3)
        else:                            # extents a multigrid hierarchy takes
            g = _grid(rng, 24, 360, 320 ** 3, multiple=8)
        return dict(kind=kind, **g, order=rng.choice([6, 12, 12, 12]), form=form)
    if kind in ("kernel", "lr_map"):
        most = 192 ** 3 if kind == "kernel" else 128 ** 3
        if rng.random() < 0.2:
            g = _grid(rng, 16, 64, 48 ** 3)
        else:
            g = _grid(rng, 24, 224, most, multiple=8)
        return dict(kind=kind, **g, order=12)
    if kind == "ions":
        return dict(kind=kind, r1=rng.randint(1, 4), r2=rng.randint(1, 4), r3=rng.randint(1, 4),
                    points=rng.choice([20, 24, 27, 32]))
    if kind == "batched":
        return dict(kind=kind, cells=_log_int(rng, 2, 32), reps_seed=rng.randint(4, 1 << 20))
    if kind == "network":
        return dict(kind=kind, **_grid(rng, 16, 256, 192 ** 3))
    r = rng.choice([(1, 1, 1), (1, 1, 2), (1, 2, 2), (2, 2, 2), (2, 2, 3), (1, 3, 3)])
    return dict(kind="ground", r1=r[0], r2=r[1], r3=r[2], points=rng.choice([24, 32]))


# ------------------------------------------------------------------------------- inputs
class _Grids:
    """Grid handles, given back with the state that holds them."""

    def __init__(self):
        self.handles = []

    def new(self, n, L, half_order):
        h = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
        self.handles.append(h)
        return h

    def __del__(self):
        torch.cuda.synchronize()
        for h in self.handles:
            B.of_grid_destroy(h)


def _n(case):
    return case["n1"], case["n2"], case["n3"]


def _lengths(n):
    return tuple(H * k for k in n)


def _atoms(n, seed):
    """Ions at the aluminium density (four per 32^3 points), on a jittered regular lattice."""
    rng = np.random.default_rng(seed)
    k = [max(1, int(round(x / 32.0 * 4.0 ** (1.0 / 3.0)))) for x in n]
    i = np.stack(np.meshgrid(*[np.arange(m) for m in k], indexing="ij"), -1).reshape(-1, 3)
    return (i + 0.5 + rng.uniform(-0.2, 0.2, i.shape)) / np.array(k) * np.array(_lengths(n))


def _gaussians(n, R, sigma, amplitude):
    """sum over the ions and their periodic images of amplitude * unit Gaussians, shape (n3, n2, n1)."""
    L = _lengths(n)
    R = torch.as_tensor(R, dtype=torch.float64, device="cuda")
    axes = []
    for a in range(3):
        x = torch.arange(n[a], dtype=torch.float64, device="cuda") * H
        d = x[None, :] - R[:, a, None]
        f = torch.zeros_like(d)
        reach = int(math.ceil(8.0 * sigma / L[a])) + 1
        for m in range(-reach, reach + 1):
            f += torch.exp(-((d + m * L[a]) ** 2) / (2.0 * sigma * sigma))
        axes.append(f)
    fx, fy, fz = axes
    fx = fx * (amplitude * (2.0 * math.pi * sigma * sigma) ** -1.5)
    out = torch.empty((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    step = max(1, int(2 ** 26 // max(1, R.shape[0] * n[1])))
    for z in range(0, n[2], step):
        yz = torch.einsum("jz,jy->zyj", fz[:, z:z + step], fy)
        out[z:z + step] = torch.matmul(yz, fx)
    return out


def _electrons(n, seed):
    """A positive electron density at the valence of aluminium."""
    return _gaussians(n, _atoms(n, seed), ELECTRON_WIDTH, W.Z_ION) + 1e-3


def _charge(n, seed):
    """Electrons minus ions: the right-hand side of the electrostatic problem."""
    R = _atoms(n, seed)
    return (_gaussians(n, R, ELECTRON_WIDTH, W.Z_ION) - _gaussians(n, R, W.SIGMA_LR, W.Z_ION))


def _weights(half_order):
    w = [-sum(1.0 / (q * q) for q in range(1, half_order + 1)) / (H * H)]
    for p in range(1, half_order + 1):
        c = math.factorial(half_order) ** 2 / (math.factorial(half_order - p) * math.factorial(half_order + p))
        w.append((2.0 if p % 2 else -2.0) * c / (H * H * p * p))
    return w


def _laplacian(f, half_order):
    """The periodic central-difference Laplacian in plain torch, in the field's precision."""
    w = _weights(half_order)
    out = (6.0 * w[0]) * f
    for p in range(1, half_order + 1):
        for a in range(3):
            out += w[p] * (torch.roll(f, p, a) + torch.roll(f, -p, a))
    return out


def _symbol(n, half_order):
    """Eigenvalues of -L_h on the plane waves of the half-spectrum transform, (n3, n2, n1 // 2 + 1)."""
    w = _weights(half_order)

    def axis(m, count):
        t = 2.0 * math.pi * torch.arange(count, dtype=torch.float64, device="cuda") / m
        s = torch.zeros_like(t)
        for p in range(1, half_order + 1):
            s += 4.0 * w[p] * torch.sin(0.5 * p * t) ** 2
        return s

    # the weights sum to zero, so that -L_h e^{ikx} = sum_p 2 w_p (1 - cos(p k h)) e^{ikx}
    return (axis(n[2], n[2])[:, None, None] + axis(n[1], n[1])[None, :, None]
            + axis(n[0], n[0] // 2 + 1)[None, None, :])


def _kf2(case):
    n = _n(case)
    volume = math.prod(_lengths(n))
    return Fn.kf2(W.Z_ION * _atoms(n, 0).shape[0], volume)


def _opts(form, tol=1e-10):
    o = B.of_default_solve_opts()            # relative residual 1e-10, the default
    o.tol = tol
    o.precision = B.OF_F64 if form == "f64" else B.OF_F32
    return o


def _cell(case, seed, displacement=0.1):
    return W.fcc_supercell((case["r1"], case["r2"], case["r3"]), points_per_cell=case["points"],
                           displacement=displacement, seed=seed, sigma=W.SIGMA_LR, rc=W.R_CUT_LR)


def _batch_sizes(case):
    rng = np.random.default_rng(case["reps_seed"])
    return [tuple(int(32 * r) for r in rng.integers(2, 5, size=3)) for _ in range(case["cells"])]


def _smooth(n, seed):
    """A smooth field of a few long waves (a potential)."""
    g = np.random.default_rng(seed)
    axes = [torch.arange(k, dtype=torch.float64, device="cuda") * (2.0 * math.pi / k) for k in n]
    out = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    for _ in range(6):
        k, ph, a = g.integers(-3, 4, size=3), g.uniform(0, 2 * math.pi), g.uniform(0.05, 0.25)
        out += a * torch.cos(float(k[2]) * axes[2][:, None, None] + float(k[1]) * axes[1][None, :, None]
                             + float(k[0]) * axes[0][None, None, :] + ph)
    return out


def _field32(n, seed):
    """A Krylov residual: a density's curvature with the rough part an iteration leaves."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = _charge(n, seed)
    r = r / r.square().mean().sqrt()
    r += 0.5 * torch.randn(r.shape, dtype=torch.float64, device="cuda", generator=gen)
    return (r - r.mean()).to(torch.float32)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, grids=_Grids())
    if kind == "laplacian":
        n = _n(case)
        u = torch.sqrt(_electrons(n, seed))
        s["x"] = u.to(torch.float32) if case["dtype"] == "f32" else u
        s["y"] = torch.empty_like(s["x"])
        s["h"] = s["grids"].new(n, _lengths(n), case["order"] // 2)
    elif kind == "poisson":
        n = _n(case)
        s["rho"] = _charge(n, seed)
        s["phi"] = torch.zeros_like(s["rho"])
        s["h"] = s["grids"].new(n, _lengths(n), case["order"] // 2)
        s["opts"] = _opts(case["form"], POISSON_TOL)
    elif kind == "kernel":
        n = _n(case)
        s["f"] = _laplacian(_electrons(n, seed) ** WT_ALPHA, case["order"] // 2) * (-1.0 / _kf2(case))
        s["W"] = torch.zeros((len(Fn.P00),) + tuple(s["f"].shape), dtype=torch.complex128, device="cuda")
        s["h"] = s["grids"].new(n, _lengths(n), case["order"] // 2)
        s["kf2"], s["opts"] = _kf2(case), _opts("mixed")
    elif kind == "lr_map":
        n = _n(case)
        s["u"] = torch.sqrt(_electrons(n, seed))
        s["v"] = torch.empty_like(s["u"])
        s["h"] = s["grids"].new(n, _lengths(n), case["order"] // 2)
        s["kf2"], s["fn"], s["opts"] = _kf2(case), Fn.wt(), _opts("mixed")
    elif kind == "ions":
        c = _cell(case, seed)
        s["sys"] = B.make_system(c.R, c.Z, c.sigma, c.rc)
        s["phi"] = _smooth(c.n, seed)
        s["b"] = torch.empty_like(s["phi"])
        s["h"] = s["grids"].new(c.n, c.L, 6)
    elif kind == "batched":
        sizes = _batch_sizes(case)
        s["rho"] = [_charge(n, seed + 1000 * k) for k, n in enumerate(sizes)]
        s["phi"] = [torch.zeros_like(r) for r in s["rho"]]
        s["h"] = [s["grids"].new(n, _lengths(n), 6) for n in sizes]
        s["opts"] = _opts("mixed", POISSON_TOL)
    elif kind == "network":
        n = _n(case)
        s["r"] = _field32(n, seed)
        s["z"] = torch.empty_like(s["r"])
        s["h"] = s["grids"].new(n, _lengths(n), 6)
        s["net"] = _Network(W.initial_network(seed=seed, scale=1.0))
    elif kind == "ground":
        c = _cell(case, seed, displacement=0.4)      # a hot snapshot: forces well above their error
        s["sys"], s["fn"] = B.make_system(c.R, c.Z, c.sigma, c.rc), Fn.wt()
        s["u"] = torch.ones(c.shape, dtype=torch.float64, device="cuda")
        s["phi"] = torch.zeros_like(s["u"])
        s["h"] = s["grids"].new(c.n, c.L, 6)
        s["opts"] = _ground_opts()
    else:
        raise ValueError(kind)
    return s


class _Network:
    """A learned-preconditioner handle, given back with the state that holds it."""

    def __init__(self, params):
        self.handle = B.of_precond_create(params)

    def __del__(self):
        torch.cuda.synchronize()
        B.of_precond_destroy(self.handle)


def _ground_opts():
    """The mixed form with the preconditioned NLCG, converged as far as a mesh-convergence study
    wants it (forces to about 1e-11)."""
    o = B.of_default_scf_opts()
    o.precision = B.OF_F32
    o.anderson_m, o.anderson_zeta = 3, 1.0
    o.nlcg_precond_shift, o.nlcg_precond_low = 1.5, 0.01
    o.nlcg_tol, o.fp_tol, o.nlcg_tol_rel = 2e-11, 1e-11, 3e-2
    o.poisson.tol = o.kernel.tol = 1e-11
    o.poisson.inner_tol = 3e-4
    return o


# --------------------------------------------------------------------------------- calls
def run(s):
    kind = s["case"]["kind"]
    if kind == "laplacian":
        B.of_laplacian_apply(s["h"], B.OF_F32 if s["case"]["dtype"] == "f32" else B.OF_F64, s["x"], s["y"])
        return s["y"]
    if kind == "poisson":
        s["phi"].zero_()
        B.of_poisson_solve(s["h"], s["rho"], s["phi"], s["opts"])
        return s["phi"]
    if kind == "kernel":
        s["W"].zero_()
        B.of_kernel_solve(s["h"], s["f"], Fn.P00, Fn.Q00, s["kf2"], s["W"], s["opts"])
        return s["W"]
    if kind == "lr_map":
        t, _ = B.of_lr_potential(s["h"], s["fn"], s["kf2"], s["u"], s["v"], None, s["opts"])
        return dict(v=s["v"], t=np.float64(t))
    if kind == "ions":
        e = B.of_pseudocharge(s["h"], s["sys"], s["b"])
        f = B.of_forces(s["h"], s["sys"], None, s["phi"])
        return dict(b=s["b"], e_self=np.float64(e), forces=f)
    if kind == "batched":
        for p in s["phi"]:
            p.zero_()
        B.of_poisson_solve_batched(s["h"], s["rho"], s["phi"], s["opts"])
        return s["phi"]
    if kind == "network":
        B.of_precond_apply(s["h"], s["net"].handle, s["r"], s["z"])
        return s["z"]
    s["u"].fill_(1.0)
    res = B.of_scf_ground_state(s["h"], s["sys"], s["fn"], s["opts"], s["u"], s["phi"])
    f = B.of_forces(s["h"], s["sys"], s["u"], s["phi"])
    return dict(u=s["u"], phi=s["phi"], forces=f,
                energies=np.array([res.energy, res.e_tf, res.e_vw, res.e_lr, res.e_xc, res.e_es]))


# ---------------------------------------------------------------------------------- work
def work(case):
    """Bytes: each input field read once and each output field written once.  Operations: what
    one application of the case's operator to its fields takes, a solve counted as one."""
    kind = case["kind"]
    if kind in ("ions", "ground"):
        points = case["r1"] * case["r2"] * case["r3"] * case["points"] ** 3
        atoms = 4 * case["r1"] * case["r2"] * case["r3"]
        ball = 4.0 / 3.0 * math.pi * (W.R_CUT_LR * case["points"] / W.A_LATTICE) ** 3
        if kind == "ions":       # read phi, write b; a charge and a force term per ion and point in reach
            return dict(bytes=16.0 * points, flops=40.0 * atoms * ball)
        return dict(bytes=32.0 * points, flops=80.0 * points + 40.0 * atoms * ball)
    if kind == "batched":
        points = sum(math.prod(n) for n in _batch_sizes(case))
        return dict(bytes=16.0 * points, flops=74.0 * points)
    points = math.prod(_n(case))
    taps = 2.0 * (3.0 * case.get("order", 2) + 1.0)
    if kind == "laplacian":
        return dict(bytes=(8.0 if case["dtype"] == "f32" else 16.0) * points, flops=taps * points)
    if kind == "poisson":
        return dict(bytes=16.0 * points, flops=taps * points)
    if kind == "kernel":         # one real right-hand side, two complex solutions
        return dict(bytes=40.0 * points, flops=4.0 * taps * points)
    if kind == "lr_map":         # u in, V out; four complex systems between them
        return dict(bytes=16.0 * points, flops=10.0 * taps * points)
    return dict(bytes=8.0 * points, flops=2.0 * 27.0 * (16 + 256 + 16) * points)


# --------------------------------------------------------------------------------- exact
def _poisson_exact(rho, half_order):
    n = rho.shape[::-1]
    lam = _symbol(n, half_order)
    lam[0, 0, 0] = 1.0
    k = torch.fft.rfftn(rho) * (4.0 * math.pi)
    k[0, 0, 0] = 0.0
    return torch.fft.irfftn(k / lam, s=rho.shape)


def _shifted_exact(f, P, Q, kf2, half_order):
    """(-(1/kf2) L_h + Q)^{-1} P f of a real f: the real and imaginary parts are real filters."""
    g = 1.0 / (_symbol(f.shape[::-1], half_order) / kf2 + Q) * P
    k = torch.fft.rfftn(f)
    return torch.complex(torch.fft.irfftn(k * g.real, s=f.shape), torch.fft.irfftn(k * g.imag, s=f.shape))


def _ions_exact(case, seed):
    c = _cell(case, seed)
    L, n = np.array(c.L), c.n
    h = [L[a] / n[a] for a in range(3)]
    dV = h[0] * h[1] * h[2]
    phi = _smooth(n, seed)
    s, rc = c.sigma, c.rc
    norm = (2.0 * math.pi * s * s) ** -1.5
    b = torch.zeros_like(phi)
    e_self, F = 0.0, np.zeros_like(c.R)
    for J in range(c.n_atoms):
        idx, dist = [], []
        for a in range(3):
            lo, hi = math.ceil((c.R[J, a] - rc) / h[a]), math.floor((c.R[J, a] + rc) / h[a])
            i = torch.arange(lo, hi + 1, device="cuda")
            idx.append(torch.remainder(i, n[a]))
            dist.append(i.to(torch.float64) * h[a] - c.R[J, a])
        dx, dy, dz = dist[0][None, None, :], dist[1][None, :, None], dist[2][:, None, None]
        r2 = dx * dx + dy * dy + dz * dz
        r = torch.sqrt(r2)
        bj = torch.where(r2 <= rc * rc, -c.Z[J] * norm * torch.exp(-r2 / (2.0 * s * s)), 0.0)
        v = torch.where(r < 1e-12, -c.Z[J] * math.sqrt(2.0 / math.pi) / s,
                        -c.Z[J] * torch.erf(r / (math.sqrt(2.0) * s)) / torch.clamp(r, min=1e-12))
        at = (idx[2][:, None, None], idx[1][None, :, None], idx[0][None, None, :])
        b.index_put_(at, bj, accumulate=True)
        e_self -= 0.5 * dV * float((bj * v).sum())
        w = -bj / (s * s) * (phi[at] - v) * dV
        F[J] = [float((w * x).sum()) for x in (dx, dy, dz)]
    # the overlap correction of point reference charges
    cut = 14.0 * s
    reps = [int(math.ceil(cut / x)) + 1 for x in L]
    T = np.stack(np.meshgrid(*[np.arange(-m, m + 1) for m in reps], indexing="ij"), -1).reshape(-1, 3) * L
    R, T = torch.as_tensor(c.R, device="cuda"), torch.as_tensor(T, device="cuda")
    Z = torch.as_tensor(c.Z, device="cuda")
    for I in range(c.n_atoms):
        d = R[I] - R[:, None, :] - T[None, :, :]
        r = d.square().sum(-1).sqrt()
        use = (r <= cut) & (r > 1e-9)
        r = torch.where(use, r, 1.0)
        ec = torch.special.erfc(r / (2.0 * s))
        gp = -torch.exp(-r * r / (4.0 * s * s)) / (s * math.sqrt(math.pi) * r) - ec / (r * r)
        w = torch.where(use, -Z[I] * Z[:, None] * gp / r, 0.0)
        F[I] += (w[..., None] * d).sum((0, 1)).cpu().numpy()
    return dict(b=b, e_self=np.float64(e_self), forces=F)


def _network_exact(case, seed):
    """The network's formula on its parameters and its input, every value in 64 bits."""
    r = _field32(_n(case), seed).to(torch.float64)
    p = torch.as_tensor(W.initial_network(seed=seed, scale=1.0), device="cuda").to(torch.float64)
    C, T = 16, 27
    w1, p = p[:C * T].view(C, 1, T), p[C * T:]
    b1, p = p[:C], p[C:]
    w2, p = p[:C * C * T].view(C, C, T), p[C * C * T:]
    b2, p = p[:C], p[C:]
    w3, b3 = p[:C * T].view(1, C, T), p[C * T:]

    def conv(a, w, bias):
        out = bias.view(-1, 1, 1, 1).expand((w.shape[0],) + a.shape[1:]).clone()
        for t in range(T):
            at = torch.roll(a, (1 - t // 9, 1 - t // 3 % 3, 1 - t % 3), (1, 2, 3))
            out += torch.einsum("oc,czyx->ozyx", w[:, :, t], at)
        return out

    s = r.square().mean().sqrt()
    a = torch.nn.functional.gelu(conv((r / s)[None], w1, b1))
    a = torch.nn.functional.gelu(conv(a, w2, b2))
    return (conv(a, w3, b3) * s)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "laplacian":
        u = torch.sqrt(_electrons(_n(case), seed))
        u = u.to(torch.float32).to(torch.float64) if case["dtype"] == "f32" else u
        return _laplacian(u, case["order"] // 2)
    if kind == "poisson":
        return _poisson_exact(_charge(_n(case), seed), case["order"] // 2)
    if kind == "kernel":
        f = _laplacian(_electrons(_n(case), seed) ** WT_ALPHA, case["order"] // 2) * (-1.0 / _kf2(case))
        return torch.stack([_shifted_exact(f, P, Q, _kf2(case), case["order"] // 2)
                            for P, Q in zip(Fn.P00, Fn.Q00)])
    if kind == "lr_map":
        N, kf2 = case["order"] // 2, _kf2(case)
        rho = _electrons(_n(case), seed)
        pots = []
        for e in (WT_ALPHA, WT_BETA):
            f = _laplacian(rho ** e, N) * (-1.0 / kf2)
            pots.append(sum(2.0 * _shifted_exact(f, P, Q, kf2, N).real for P, Q in zip(Fn.P00, Fn.Q00)))
        Va, Vb = pots
        cf = 0.3 * (3.0 * math.pi ** 2) ** (2.0 / 3.0)
        v = cf * (WT_ALPHA * rho ** (WT_ALPHA - 1.0) * Vb + WT_BETA * rho ** (WT_BETA - 1.0) * Va)
        t = 0.5 * cf * float((rho ** WT_ALPHA * Vb + rho ** WT_BETA * Va).sum()) * H ** 3
        return dict(v=v, t=np.float64(t))
    if kind == "ions":
        return _ions_exact(case, seed)
    if kind == "batched":
        return [_poisson_exact(_charge(n, seed + 1000 * k), 6) for k, n in enumerate(_batch_sizes(case))]
    if kind == "network":
        return _network_exact(case, seed)
    return None

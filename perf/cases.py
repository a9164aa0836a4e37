"""Performance cases of the coarse-grid projection library: what a flow solver has it do, through its public calls.

Every case is one kind of work on one mesh size.  The meshes are the O-grid
around a cylinder of ``inputs.ogrid``, the velocities ``inputs.velocity``; the
previous time step's solutions (initial guesses, network inputs) come from a
direct solver in this file, so that the inputs do not depend on the library.

Kinds
  pressure  one pressure-correction step: right-hand side, Poisson solve from the previous step's
            solution, prolongation, pressure gradient, velocity update
  potential one potential step: right-hand side, Poisson solve, prolongation, gradient and Lorentz force
  solve     one Poisson solve from the previous step's solution (FP64 or mixed precision)
  batch     many uneven independent systems in one batched mixed-precision solve
  maps      the mapping and field calls of one step with the solution in hand
  spmv      the product with the coarse stiffness matrix alone
  guess     one prediction of the learned initial guess
  train     one minibatch's gradient of the learned initial guess

``exact`` gives the same outputs in 64 bits: the operators assembled with
numpy, the Poisson systems solved directly by a Fourier transform over the
angle and one tridiagonal system per mode.
"""
from __future__ import annotations

import collections
import math

import numpy as np
import torch

from paper_2003_00082_gb300 import cgp, inputs

DEV = "cuda"
RHO_OVER_DT = 1.0 / inputs.DT
STUART = 1.0


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one potential step of a small case (a parameter study, a unit of an ensemble): the solver's latency
        dict(name="potential-64x32", kind="potential", n_theta=64, n_r=32, levels=1, tol=1e-10),
        # the benchmark's size and launch: the pressure correction of a 525,312-node flow, warm started
        dict(name="pressure-512x256-tuned", kind="pressure", n_theta=512, n_r=256, levels=1, tol=1e-10, tuned=True),
        # a mesh of no round size, solved as a program does that tunes nothing
        dict(name="solve-321x163-fp64", kind="solve", n_theta=321, n_r=163, levels=1, tol=1e-10, mixed=False,
             far_field=False),
        # the far-field Dirichlet variant on a mid-size ragged mesh
        dict(name="solve-129x67-far-field", kind="solve", n_theta=129, n_r=67, levels=1, tol=1e-10, mixed=False,
             far_field=True),
        # mixed precision on the small mesh's noisy sequence
        dict(name="solve-64x32-mixed", kind="solve", n_theta=64, n_r=32, levels=1, tol=1e-10, mixed=True,
             far_field=False),
        # mixed precision at the benchmark's size, in the launch its autotuner picks
        dict(name="solve-512x256-mixed-tuned", kind="solve", n_theta=512, n_r=256, levels=1, tol=1e-10, mixed=True,
             far_field=False, tuned=True),
        # uneven independent systems (several meshes at once), in the launch the batch autotuner picks
        dict(name="batch-16-uneven", kind="batch", count=16, pick=7, tol=1e-10, tuned=True),
        # the streaming kernels of one step at the benchmark's size
        dict(name="maps-512x256", kind="maps", n_theta=512, n_r=256, levels=1),
        # the same fine size from a coarser mesh: three prolongation levels
        dict(name="maps-128x64-k3", kind="maps", n_theta=128, n_r=64, levels=3),
        # the product alone on a matrix larger than the L2 cache
        dict(name="spmv-2048x1024-fp64", kind="spmv", n_theta=2048, n_r=1024, levels=1, single=False, stencil=False),
        # the learned initial guess at the size it is trained on: one prediction per time step
        dict(name="guess-64x32", kind="guess", n_theta=64, n_r=32),
        # and one minibatch of its training
        dict(name="train-64x32-b16", kind="train", n_theta=64, n_r=32, batch=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """An O-grid size: n_theta over its logarithm, n_r about half of it, odd ones as likely as even ones."""
    nt = _log_int(rng, lo, hi)
    return dict(n_theta=nt, n_r=max(4, int(round(nt * rng.uniform(0.4, 0.5)))))


def _tunes(rng, size):
    """Whether the program keeps the large launch shape: half of those with a mesh for it."""
    return rng.random() < 0.5 and size["n_theta"] >= 192


def draw(rng):
    kind = rng.choice(["pressure", "potential", "solve", "solve", "solve", "batch", "maps", "spmv", "guess", "train"])
    if kind == "pressure":
        size = _grid(rng, 64, 400)
        return dict(kind=kind, levels=rng.choice([1, 1, 2]), tol=1e-10, tuned=_tunes(rng, size), **size)
    if kind == "potential":
        # the Lorentz force is the small difference of two large terms far from the cylinder: sizes
        # where 64 bits leave its rounding below what outputs are compared to
        return dict(kind=kind, levels=rng.choice([1, 2]), tol=1e-10, **_grid(rng, 24, 72))
    if kind == "solve":
        size = _grid(rng, 24, 480)
        return dict(kind=kind, levels=1, tol=rng.choice([1e-10, 1e-11]), mixed=rng.random() < 0.5,
                    far_field=rng.random() < 0.3, tuned=_tunes(rng, size), **size)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 16), pick=rng.randint(8, 1000), tol=1e-10, tuned=rng.random() < 0.5)
    if kind == "maps":
        levels = rng.choice([1, 2, 3])
        return dict(kind=kind, levels=levels, **_grid(rng, 24, 512 >> (levels - 1)))
    if kind == "spmv":
        return dict(kind=kind, levels=1, single=rng.random() < 0.5, stencil=rng.random() < 0.3, **_grid(rng, 128, 2048))
    if kind == "guess":
        return dict(kind=kind, **_grid(rng, 24, 128))
    return dict(kind=kind, batch=rng.randint(1, 16), **_grid(rng, 24, 64))


def _batch_sizes(case):
    """Mesh sizes of a batch: 64, 128, 256 and 512 angles as in the batched workload, a third of them off by a few."""
    rng = np.random.default_rng(case["pick"])
    nt = rng.choice([64, 128, 256, 512], size=case["count"], p=[0.35, 0.3, 0.2, 0.15])
    nt = nt - np.where(rng.random(case["count"]) < 0.33, rng.integers(1, 12, size=case["count"]), 0)
    return [(int(k), int(k) // 2) for k in nt]


# ---------------------------------------------------------------------------
# geometry, operators and the direct solver (numpy only)
# ---------------------------------------------------------------------------
_geo = collections.OrderedDict()


def _refine(xy, tri):
    """One uniform 4-way split: midpoints numbered by sorted edge, children as the library orders them."""
    n = xy.shape[0]
    t = tri.astype(np.int64)
    ends = np.stack([t, np.roll(t, -1, axis=1)], axis=2)                # sides ab, bc, ca
    key = ends.min(axis=2) * n + ends.max(axis=2)
    uniq, inv = np.unique(key.ravel(), return_inverse=True)
    mid = n + inv.reshape(-1, 3)
    edges = np.stack([uniq // n, uniq % n], axis=1)
    fine = np.concatenate([xy, 0.5 * (xy[edges[:, 0]] + xy[edges[:, 1]])])
    a, b, c = t.T
    ab, bc, ca = mid.T
    kids = np.stack([a, ab, ca, ab, b, bc, ca, bc, c, ab, bc, ca], axis=1).reshape(-1, 3)
    return fine, kids, edges


class _Geometry:
    """An O-grid, its splits, its P1 operators as triplets and the factors of the direct solver."""

    def __init__(self, nt, nr, levels):
        self.nt, self.nr = nt, nr
        self.xy, self.tri = inputs.ogrid(nt, nr)
        self.n = self.xy.shape[0]
        self.levels = []
        xy, tri = self.xy, self.tri
        for _ in range(levels):
            xy, tri, edges = _refine(xy, tri)
            self.levels.append(edges)
        self.xy_f, self.tri_f = xy, tri
        self._ops = None

    @property
    def ops(self):
        """(rows, cols, K, Gx, Gy) triplets: K = int grad.grad, G_ij = int psi_j d psi_i."""
        if self._ops is None:
            area, gx, gy = _gradients(self.xy, self.tri)
            t = self.tri.astype(np.int64)
            rows = np.repeat(t, 3, axis=1).ravel()
            cols = np.tile(t, (1, 3)).ravel()
            K = (area[:, None, None] * (gx[:, :, None] * gx[:, None, :] + gy[:, :, None] * gy[:, None, :])).ravel()
            Gx = np.repeat(area[:, None] / 3.0 * gx, 3, axis=1).ravel()
            Gy = np.repeat(area[:, None] / 3.0 * gy, 3, axis=1).ravel()
            self._ops = rows, cols, K, Gx, Gy
        return self._ops

    def mul(self, vals, x):
        rows, cols = self.ops[:2]
        return np.bincount(rows, weights=vals * x[cols], minlength=self.n)

    def rhs(self, Fx, Fy):
        rows, cols, _, Gx, Gy = self.ops
        return np.bincount(rows, weights=Gx * Fx[cols] + Gy * Fy[cols], minlength=self.n)

    def poisson(self, b, far_field=False):
        """K x = b by a Fourier transform over the angle; mean zero, or zero on the outer ring."""
        nt, nj = self.nt, self.nr + 1
        rows, cols, K = self.ops[:3]
        # K does not change along the angle: the entries of the rows at angle 0 give every mode's tridiagonal system
        at = rows % nt == 0
        r, c, k = rows[at] // nt, cols[at], K[at]
        m = np.arange(nt // 2 + 1)
        step = c % nt
        sym = k[:, None] * np.exp(2j * np.pi * np.outer(np.where(step > 1, -1, step), m) / nt)
        dj = c // nt - r
        diag, up = np.zeros((nj, m.size), complex), np.zeros((nj, m.size), complex)
        np.add.at(diag, r[dj == 0], sym[dj == 0])
        np.add.at(up, r[dj == 1], sym[dj == 1])
        if far_field:
            diag[-1], up[-2] = 1.0, 0.0
        else:
            diag[0, 0], up[0, 0] = 1.0, 0.0                              # the constant: pinned, projected afterwards
        low = np.conj(up)
        fac, inv = np.empty_like(diag), np.empty_like(diag)
        inv[0] = 1.0 / diag[0]
        for j in range(1, nj):
            fac[j] = low[j - 1] * inv[j - 1]
            inv[j] = 1.0 / (diag[j] - fac[j] * up[j - 1])

        def project(v):
            if far_field:
                v = v.copy()
                v[-nt:] = 0.0
                return v
            return v - v.mean()

        def direct(v):
            f = np.fft.rfft(v.reshape(nj, nt), axis=1)
            if not far_field:
                f[0, 0] = 0.0
            for j in range(1, nj):
                f[j] -= fac[j] * f[j - 1]
            f[-1] *= inv[-1]
            for j in range(nj - 2, -1, -1):
                f[j] = (f[j] - up[j] * f[j + 1]) * inv[j]
            return project(np.fft.irfft(f, n=nt, axis=1).ravel())

        b = project(b)
        x = direct(b)
        for _ in range(2):
            x = project(x + direct(project(b - self.mul(K, x))))
        return x

    def prolong(self, x):
        for edges in self.levels:
            x = np.concatenate([x, 0.5 * (x[edges[:, 0]] + x[edges[:, 1]])])
        return x


def _gradients(xy, tri):
    p = xy[tri]
    x, y = p[:, :, 0], p[:, :, 1]
    area2 = (x[:, 1] - x[:, 0]) * (y[:, 2] - y[:, 0]) - (x[:, 2] - x[:, 0]) * (y[:, 1] - y[:, 0])
    gx = (np.roll(y, -1, axis=1) - np.roll(y, -2, axis=1)) / area2[:, None]
    gy = (np.roll(x, -2, axis=1) - np.roll(x, -1, axis=1)) / area2[:, None]
    return 0.5 * area2, gx, gy


def _geometry(nt, nr, levels=1):
    key = (nt, nr, levels)
    if key not in _geo:
        while len(_geo) >= 20:
            _geo.popitem(last=False)
        _geo[key] = _Geometry(nt, nr, levels)
    _geo.move_to_end(key)
    return _geo[key]


def _velocity(g, step, seed):
    return inputs.velocity(g.xy_f, step, seed, vortices=True, noise_std=1e-3)


def _b_field(seed):
    """B_o k-hat and a unit in-plane part at a seeded angle."""
    return inputs.magnetic_field(angle=float(np.random.default_rng(seed).uniform(0.0, 2.0 * np.pi)))


def _source(g, u, v, B, pressure):
    n = g.n
    return (RHO_OVER_DT * u[:n], RHO_OVER_DT * v[:n]) if pressure else (B[2] * v[:n], -B[2] * u[:n])


def _fields(g, x_f, u, v, B, sigma):
    """Gradient and Lorentz force per fine triangle, x components of all triangles first."""
    _, gx, gy = _gradients(g.xy_f, g.tri_f)
    f = x_f[g.tri_f]
    dx, dy = (gx * f).sum(axis=1), (gy * f).sum(axis=1)
    um, vm = u[g.tri_f].mean(axis=1), v[g.tri_f].mean(axis=1)
    jx, jy, jz = sigma * (-dx + vm * B[2]), sigma * (-dy - um * B[2]), sigma * (um * B[1] - vm * B[0])
    return np.concatenate([dx, dy]), np.concatenate([jy * B[2] - jz * B[1], jz * B[0] - jx * B[2]])


def _corrected(g, p_f, u, v):
    """u - (dt / rho) grad p with the gradient brought to the nodes by the lumped mass."""
    area, gx, gy = _gradients(g.xy_f, g.tri_f)
    f = p_f[g.tri_f]
    t = g.tri_f.ravel()
    mass = np.bincount(t, weights=np.repeat(area, 3))
    out = []
    for w, q in ((u, gx), (v, gy)):
        grad = np.bincount(t, weights=np.repeat(area * (q * f).sum(axis=1), 3)) / mass
        out.append(w - grad / RHO_OVER_DT)
    return out


# ---------------------------------------------------------------------------
# meshes kept by the program, as a time-stepping program keeps them
# ---------------------------------------------------------------------------
_kept = collections.OrderedDict()


def _keep(key, make, most=14):
    if key not in _kept:
        while len(_kept) >= most:
            _kept.popitem(last=False)
        _kept[key] = make()
    _kept.move_to_end(key)
    return _kept[key]


def _mesh(case, instance=0):
    key = (case["kind"], case["n_theta"], case["n_r"], case.get("levels", 1), bool(case.get("mixed")),
           bool(case.get("far_field")), bool(case.get("tuned")), bool(case.get("single")), bool(case.get("stencil")),
           instance)

    def make():
        xy, tri = inputs.ogrid(case["n_theta"], case["n_r"])
        m = cgp.Mesh(xy, tri, case.get("levels", 1))
        if case.get("tuned") or case.get("stencil"):
            cgp.cgp_mesh_set_ogrid(m.handle, case["n_theta"], case["n_r"])
        if case.get("far_field"):
            cgp.cgp_set_far_field(m.handle, 1)
        if case["kind"] == "spmv":
            cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SPMV_FP32 if case["single"] else cgp.CGP_TUNE_SPMV_FP64,
                               0, 0, 0, 1 if case["stencil"] else 0)
        elif case.get("tuned") and case["kind"] != "batch":
            # the shapes cgp_autotune finds at the benchmark's size and a program keeps: one 512-thread block
            # per SM with tagged reductions, in FP64 on O-grid tiles
            mixed = case.get("mixed")
            cgp.cgp_set_tuning(m.handle, cgp.CGP_TUNE_SOLVE_MIXED if mixed else cgp.CGP_TUNE_SOLVE_FP64,
                               512, 1, 152, 8 if mixed else 40)
        return m

    return _keep(key, make)


def _batch_meshes(case):
    key = ("batch", case["count"], case["pick"])

    def make():
        return [cgp.Mesh(*inputs.ogrid(nt, nr)) for nt, nr in _batch_sizes(case)]

    return _keep(key, make)


# ---------------------------------------------------------------------------
# inputs (host arrays, from the seed alone)
# ---------------------------------------------------------------------------
def _step_inputs(case, seed):
    g = _geometry(case["n_theta"], case["n_r"], case.get("levels", 1))
    step = 2 + seed % 150
    B = _b_field(seed)
    pressure = case["kind"] == "pressure"
    u, v = _velocity(g, step, seed)
    up, vp = _velocity(g, step - 1, seed)
    before = g.poisson(g.rhs(*_source(g, up, vp, B, pressure)), case.get("far_field", False))
    return g, B, u, v, before


def _network_inputs(case, seed, count):
    """`count` successive samples (b(t), phi(t-1), phi(t-2), phi(t)) and He-normal weights with a small decoder
    (outputs of order one, as the increments that the network predicts)."""
    g = _geometry(case["n_theta"], case["n_r"])
    first = seed % 100
    b, phi = [], []
    for t in range(first, first + count + 2):
        u, v = _velocity(g, t, seed)
        b.append(g.rhs(*_source(g, u, v, (0.0, 0.0, 1.0), False)))
        phi.append(g.poisson(b[-1]))
    b, phi = np.stack(b), np.stack(phi)
    rng = np.random.default_rng(seed)
    params = []
    for rows, cols in _layers():
        params.append(rng.standard_normal(rows * cols) * math.sqrt(2.0 / cols) * (1.0 if rows > 1 else 1.0 / 64.0))
        params.append(np.zeros(rows))
    return g, b[2:], phi[1:-1], phi[:-2], phi[2:], np.concatenate(params).astype(np.float32)


def _layers():
    """(rows, columns) of the network's dense layers, each followed by its bias."""
    return [(64, 5)] + [(64, 131), (64, 128)] * 3 + [(1, 64)]


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


def _new(n, dtype=torch.float64):
    return torch.empty(n, dtype=dtype, device=DEV)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        meshes = _batch_meshes(case)
        bs, x0 = [], []
        for k, (nt, nr) in enumerate(_batch_sizes(case)):
            g, _, b, before = _batch_instance(nt, nr, seed, k)
            bs.append(_d(b))
            x0.append(_d(before))
        xs = [torch.empty_like(x) for x in x0]
        batch = cgp.Batch(meshes, bs, xs, tol=case["tol"], precision=cgp.CGP_MIXED, use_x0=True)
        if case["tuned"]:
            batch.set_tuning(512, 1, 1, 104)   # waves of 2048 rows a block, tagged reductions
        return dict(kind=kind, batch=batch, x0=x0, xs=xs)
    if kind in ("guess", "train"):
        g, b, p1, p2, pt, params = _network_inputs(case, seed, case.get("batch", 1))
        m = _mesh(case)
        net = cgp.GNN(m, case.get("batch", 1), params)
        return dict(kind=kind, net=net, mesh=m, b=_d(b), p1=_d(p1), p2=_d(p2), pt=_d(pt), x0=_new(m.n_c),
                    batch=case.get("batch", 1))
    m = _mesh(case)
    if kind == "spmv":
        dtype = torch.float32 if case["single"] else torch.float64
        return dict(kind=kind, mesh=m, precision=cgp.CGP_FP32 if case["single"] else cgp.CGP_FP64,
                    x=_d(_spmv_input(m.n_c, seed)).to(dtype), y=_new(m.n_c, dtype))
    g, B, u, v, before = _step_inputs(case, seed)
    s = dict(kind=kind, mesh=m, B=B, u=_d(u), v=_d(v), x0=_d(before), x=_new(m.n_c), tol=case.get("tol"))
    if kind == "solve":
        s.update(b=_d(g.rhs(*_source(g, u, v, B, False))), precision=cgp.CGP_MIXED if case["mixed"] else cgp.CGP_FP64)
        return s
    s.update(b=_new(m.n_c), x_f=_new(m.n_f), grad=_new(2 * m.t_f))
    if kind in ("potential", "maps"):
        s.update(force=_new(2 * m.t_f))
    if kind in ("pressure", "maps"):
        s.update(u1=_new(m.n_f), v1=_new(m.n_f))
    if kind == "maps":
        s.update(b2=_new(m.n_c), uc=_new(m.n_c), vc=_new(m.n_c))
    return s


def _batch_instance(nt, nr, seed, k):
    g = _geometry(nt, nr)
    own = (seed * 1000 + k) % (1 << 31)
    B = _b_field(own)
    step = 2 + own % 150
    before = g.poisson(g.rhs(*_source(g, *_coarse_velocity(g, step - 1, own), B, False)))
    return g, B, g.rhs(*_source(g, *_coarse_velocity(g, step, own), B, False)), before


def _coarse_velocity(g, step, seed):
    return inputs.velocity(g.xy, step, seed, vortices=True, noise_std=1e-3)


def _spmv_input(n, seed):
    return np.random.default_rng(seed).standard_normal(n)


def run(s):
    kind = s["kind"]
    if kind == "batch":
        for x, x0 in zip(s["xs"], s["x0"]):
            x.copy_(x0)
        cgp.cgp_batch_solve(s["batch"])
        return s["xs"]
    if kind == "guess":
        cgp.cgp_gnn_predict(s["net"], s["b"], s["p1"], s["p2"], s["x0"])
        return s["x0"]
    if kind == "train":
        return cgp.cgp_gnn_gradients(s["net"], s["batch"], s["b"], s["p1"], s["p2"], s["pt"])
    h = s["mesh"].handle
    if kind == "spmv":
        cgp.cgp_spmv(h, s["precision"], s["x"], s["y"])
        return s["y"]
    if kind == "solve":
        s["x"].copy_(s["x0"])
        cgp.cgp_poisson_solve_async(h, s["b"], s["x"], tol=s["tol"], precision=s["precision"], use_x0=True)
        return s["x"]
    if kind == "maps":
        cgp.cgp_restrict(h, cgp.CGP_RHS_POTENTIAL, s["B"], RHO_OVER_DT, s["u"], s["v"], s["b"], s["uc"], s["vc"])
        cgp.cgp_restrict(h, cgp.CGP_RHS_PRESSURE, s["B"], RHO_OVER_DT, s["u"], s["v"], s["b2"])
        cgp.cgp_prolong(h, s["x0"], s["x_f"])
        cgp.cgp_lorentz(h, s["x_f"], s["u"], s["v"], s["B"], STUART, s["grad"], s["force"])
        cgp.cgp_velocity_correct(h, s["x_f"], s["u"], s["v"], 1.0 / RHO_OVER_DT, s["u1"], s["v1"])
        return [s[k] for k in ("uc", "vc", "b", "b2", "x_f", "grad", "force", "u1", "v1")]
    s["x"].copy_(s["x0"])
    pressure = kind == "pressure"
    cgp.cgp_restrict(h, cgp.CGP_RHS_PRESSURE if pressure else cgp.CGP_RHS_POTENTIAL, s["B"], RHO_OVER_DT, s["u"],
                     s["v"], s["b"])
    cgp.cgp_poisson_solve_async(h, s["b"], s["x"], tol=s["tol"], use_x0=True)
    cgp.cgp_prolong(h, s["x"], s["x_f"])
    if pressure:
        cgp.cgp_lorentz(h, s["x_f"], None, None, s["B"], STUART, s["grad"], None)
        cgp.cgp_velocity_correct(h, s["x_f"], s["u"], s["v"], 1.0 / RHO_OVER_DT, s["u1"], s["v1"])
        return [s[k] for k in ("b", "x_f", "grad", "u1", "v1")]
    cgp.cgp_lorentz(h, s["x_f"], s["u"], s["v"], s["B"], STUART, s["grad"], s["force"])
    return [s[k] for k in ("b", "x_f", "grad", "force")]


# ---------------------------------------------------------------------------
# work and the exact answer
# ---------------------------------------------------------------------------
def _solve_work(nt, nr, tol):
    """A Poisson solve: the system, b and x0 in, x out, and the flops of plain CG (2 nnz + 13 n an iteration).

    The iterations of Jacobi-PCG from the previous step's solution grow with the angles and the digits
    asked for: about 0.26 n_theta per digit.
    """
    z = inputs.ogrid_sizes(nt, nr)
    n, nnz = z["n_c"], z["nnz"]
    its = 0.26 * nt * -math.log10(tol)
    return 12 * nnz + 4 * n + 32 * n, its * (2 * nnz + 13 * n)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_solve_work(nt, nr, case["tol"]) for nt, nr in _batch_sizes(case)]
        return dict(bytes=sum(b for b, _ in each), flops=sum(f for _, f in each))
    z = inputs.ogrid_sizes(case["n_theta"], case["n_r"])
    n, nnz, t_f, n_f, e = z["n_c"], z["nnz"], z["t_c"], z["n_c"], 0
    for _ in range(case.get("levels", 1)):
        new = n_f + t_f                      # edges of an annulus: nodes + triangles
        e, n_f, t_f = e + new, n_f + new, 4 * t_f
    if kind == "spmv":
        s = 4 if case["single"] else 8
        index = 0 if case["stencil"] else 4 * nnz + 4 * n
        return dict(bytes=s * nnz + index + 2 * s * n, flops=2 * nnz)
    if kind in ("guess", "train"):
        batch, edges = case.get("batch", 1), nnz - n
        flops = batch * 3 * (2 * n * 64 * 128 * 2 + 4 * edges * 64)
        weights = 4 * sum(r * c + r for r, c in _layers())
        if kind == "guess":
            return dict(bytes=weights + 32 * n + 4 * edges, flops=flops)
        return dict(bytes=2 * weights + batch * 36 * n + 4 * edges, flops=3 * flops)
    if kind == "solve":
        b, f = _solve_work(case["n_theta"], case["n_r"], case["tol"])
        return dict(bytes=b, flops=f)
    rhs = 20 * nnz + 16 * n + 12 * n                     # Gx, Gy and pattern, velocity, b
    prolong = 8 * n + 8 * n_f + 8 * e
    grad = 8 * n_f + 16 * n_f + 12 * t_f // 4 * 2 + 16 * t_f   # x_f, coordinates, indices, gradient
    correct = 8 * n_f * 5 + 16 * n_f + 24 * t_f          # p, u, v in and out, coordinates, incidence
    if kind == "maps":
        return dict(bytes=rhs * 2 + 16 * n + prolong + grad + 16 * n_f + 16 * t_f + correct,
                    flops=8 * nnz + 2 * e + 40 * t_f + 60 * t_f)
    b, f = _solve_work(case["n_theta"], case["n_r"], case["tol"])
    if kind == "pressure":
        return dict(bytes=b + rhs + prolong + grad + correct, flops=f + 4 * nnz + 2 * e + 75 * t_f)
    return dict(bytes=b + rhs + prolong + grad + 16 * n_f + 16 * t_f, flops=f + 4 * nnz + 2 * e + 40 * t_f)


def _network(g, params, b, p1, p2):
    """The network in 64 bits: (raw outputs, output scale), differentiable in `params`."""
    rows, cols, K = g.ops[:3]
    nz = np.unique(rows * g.n + cols)
    dst, src = nz // g.n, nz % g.n
    off = dst != src
    dst, src = dst[off], src[off]
    d = g.xy[src] - g.xy[dst]
    length = np.sqrt((d * d).sum(axis=1))
    e = torch.as_tensor(np.concatenate([d, length[:, None]], axis=1) / length.mean())
    dst, src = torch.as_tensor(dst), torch.as_tensor(src)
    r = b - g.mul(K, p1)
    scale = [max(float(np.sqrt(np.mean(w * w))), 1e-30) for w in (r, p1 - p2, b)]
    f = torch.as_tensor(np.stack([r / scale[0], (p1 - p2) / scale[1], b / scale[2], g.xy[:, 0] / 15.0,
                                  g.xy[:, 1] / 15.0], axis=1))
    W, at = [], 0
    for rows_, cols_ in _layers():
        W.append((params[at:at + rows_ * cols_].reshape(rows_, cols_),
                  params[at + rows_ * cols_:at + rows_ * cols_ + rows_]))
        at += rows_ * cols_ + rows_
    h = torch.relu(f @ W[0][0].T + W[0][1])
    for l in range(3):
        (Wm, bm), (Wu, bu) = W[1 + 2 * l], W[2 + 2 * l]
        msg = torch.relu((h @ Wm[:, :64].T)[dst] + (h @ Wm[:, 64:128].T)[src] + e @ Wm[:, 128:].T + bm)
        a = torch.zeros_like(h).index_add(0, dst, msg)
        h = h + torch.relu(h @ Wu[:, :64].T + a @ Wu[:, 64:].T + bu)
    return (h @ W[-1][0].T)[:, 0] + W[-1][1], scale[1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, (nt, nr) in enumerate(_batch_sizes(case)):
            g, _, b, _ = _batch_instance(nt, nr, seed, k)
            out.append(g.poisson(b))
        return out
    if kind in ("guess", "train"):
        g, b, p1, p2, pt, params = _network_inputs(case, seed, case.get("batch", 1))
        p = torch.tensor(params, dtype=torch.float64, requires_grad=kind == "train")
        if kind == "guess":
            out, s_d = _network(g, p, b[0], p1[0], p2[0])
            return p1[0] + s_d * out.numpy()
        outs, loss = [], 0.0
        for k in range(case["batch"]):
            out, s_d = _network(g, p, b[k], p1[k], p2[k])
            loss = loss + ((out - torch.as_tensor((pt[k] - p1[k]) / s_d)) ** 2).sum() / (case["batch"] * g.n)
            outs.append(out.detach())
        loss.backward()
        return p.grad.numpy(), torch.stack(outs).numpy(), float(loss.detach())
    if kind == "spmv":
        g = _geometry(case["n_theta"], case["n_r"])
        x = _spmv_input(g.n, seed)
        return g.mul(g.ops[2], x.astype(np.float32).astype(np.float64) if case["single"] else x)
    g, B, u, v, before = _step_inputs(case, seed)
    b = g.rhs(*_source(g, u, v, B, kind == "pressure"))
    if kind == "solve":
        return g.poisson(b, case.get("far_field", False))
    if kind == "maps":
        x_f = g.prolong(before)
        grad, force = _fields(g, x_f, u, v, B, STUART)
        u1, v1 = _corrected(g, x_f, u, v)
        return [u[:g.n], v[:g.n], b, g.rhs(*_source(g, u, v, B, True)), x_f, grad, force, u1, v1]
    x_f = g.prolong(g.poisson(b))
    grad, force = _fields(g, x_f, u, v, B, STUART)
    if kind == "pressure":
        u1, v1 = _corrected(g, x_f, u, v)
        return [b, x_f, grad, u1, v1]
    return [b, x_f, grad, force]

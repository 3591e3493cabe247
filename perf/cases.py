"""Performance cases of the library: what a user's program has it do, at the sizes in use.

Every case is one call (or one call pair) of the public Python API on device tensors:

  step     one adaptive SDC step of a monodomain model on a structured grid or a shell
  emi      one step of a cell-by-cell model, Jacobi or two-level preconditioner
  batch    one step of many stacked 2D instances
  adjoint  one taped step and its discrete adjoint
  solve    one stand-alone node solve

States are a travelling front (the profile of a 1D cable integrated here by explicit
Euler, placed by the seed), so that the active sets are those of a simulation under way.
`exact` restates the step in plain torch, element by element, with node solves to 1e-13.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import workloads as W
from paper_2311_07206_gb300 import Batch, Context, default_options
from paper_2311_07206_gb300 import binding as api
from workloads import emi as WE
from workloads import meshes as WM

AP = dict(ga=8.0, gs=8.0, a=0.15, eps=0.002, mu1=0.2, mu2=0.3, cw=1.0)
ALPHA = 0.1          # the library's default drop tolerance is ALPHA TOL
RHO = 0.05           # contraction rate given to the energy-norm stop


# ---- the cases ---------------------------------------------------------------------

def _step(name, nx, ny, nz, h, M, dt, sweeps, tol, phase="front", energy=False, shell=0.0):
    return dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, h=h, M=M, dt=dt, sweeps=sweeps,
                tol=tol, phase=phase, energy=energy, shell=shell)


def listed():
    return [
        # the smallest monodomain run: 4,225 dofs in 2D, every launch and wait counts
        _step("square_65", 65, 65, 1, 0.3125, 3, 0.1, 4, 1e-4),
        # higher order with a large step and the energy-norm stop on a mid-size slab
        _step("slab_58k_order6", 101, 36, 16, 0.2, 6, 0.2, 12, 1e-5, energy=True),
        # the headline slab while the corner is stimulated: the active sets shrink quickly
        _step("slab_442k_stimulus", 201, 71, 31, 0.1, 4, 0.05, 5, 1e-5, phase="stimulus"),
        # the headline slab with a front crossing it: most of a simulation's steps
        _step("slab_442k_front", 201, 71, 31, 0.1, 4, 0.05, 5, 1e-5),
        # above what the node solves hold on chip, and odd in every direction
        _step("slab_813k", 247, 89, 37, 0.1, 4, 0.05, 5, 1e-5, phase="stimulus"),
        # unstructured rows: randomly numbered tissue with fibre tensors, renumbered inside
        _step("shell_89k", 0, 0, 0, 0.175, 3, 0.05, 5, 1e-4, shell=0.175),
        # cell-by-cell in 2D, small and ill-conditioned: thousands of CG iterations
        dict(name="branched_8k", kind="emi", geometry="branched", h=5.0, cx=0, cy=0, cz=0,
             M=3, dt=0.02, sweeps=4, tol=1e-4, two_level=False, box=0),
        # cell-by-cell bricks with Jacobi alone
        dict(name="bricks_53k", kind="emi", geometry="bricks", h=2.0, cx=2, cy=1, cz=1,
             M=3, dt=0.02, sweeps=4, tol=1e-5, two_level=False, box=0),
        # cell-by-cell bricks with the two-level preconditioner, dofs numbered by block
        dict(name="bricks_131k_two_level", kind="emi", geometry="bricks", h=2.0, cx=2, cy=2, cz=2,
             M=3, dt=0.02, sweeps=4, tol=1e-5, two_level=True, box=4),
        # instances of uneven size advanced by the same launches
        dict(name="batch_32", kind="batch", count=32, nmin=64, nmax=256, sizes=3, M=3, dt=0.1,
             sweeps=4, tol=1e-4),
        # a step and its reverse pass, as a checkpointed gradient runs them
        dict(name="adjoint_58k", kind="adjoint", nx=101, ny=36, nz=16, h=0.2, M=3, dt=0.05,
             sweeps=4, tol=1e-5),
        # one node system solved on its own
        dict(name="solve_21k", kind="solve", nx=61, ny=23, nz=15, h=0.1, noalloc=False,
             c=0.0125),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step2d", "step3d", "step3d", "step3d", "shell", "emi", "batch",
                       "adjoint", "solve"])
    M = rng.choice([2, 3, 4, 4, 6])
    sweeps = rng.choice([3, 4, 5])
    tol = rng.choice([1e-4, 1e-5])
    if kind == "step2d":
        n = round(_log(rng, 48, 640))
        c = _step("", n, max(33, n + rng.randint(-9, 9)), 1, 0.3125, min(M, 4), 0.1, sweeps, 1e-4)
    elif kind == "step3d":
        n = _log(rng, 8e3, 8e5)
        s = (n / (201 * 71 * 31)) ** (1 / 3)
        c = _step("", max(9, round(201 * s) + rng.randint(-3, 3)),
                  max(7, round(71 * s) + rng.randint(-2, 2)), max(5, round(31 * s)),
                  0.1, M, 0.05, sweeps, tol, phase=rng.choice(["front", "stimulus"]),
                  energy=rng.random() < 0.25)
    elif kind == "shell":
        h = _log(rng, 0.17, 0.35)
        c = _step("", 0, 0, 0, h, 3, 0.05, sweeps, 1e-4, shell=h)
    elif kind == "emi":
        two = rng.random() < 0.5
        cx, cy, cz = rng.choice([(1, 1, 1), (2, 1, 1), (1, 2, 1), (2, 2, 1)])
        if rng.random() < 0.3:
            c = dict(kind="emi", geometry="branched", h=rng.choice([5.0, 10.0]), cx=0, cy=0, cz=0,
                     M=3, dt=0.02, sweeps=sweeps, tol=1e-4, two_level=False, box=0)
        else:
            c = dict(kind="emi", geometry="bricks", h=2.0, cx=cx, cy=cy, cz=cz, M=3, dt=0.02,
                     sweeps=min(sweeps, 4), tol=1e-5, two_level=two,
                     box=rng.choice([2, 4]) if two else 0)
    elif kind == "batch":
        c = dict(kind="batch", count=rng.randint(5, 32), nmin=48, nmax=round(_log(rng, 96, 256)),
                 sizes=rng.randint(0, 999), M=min(M, 4), dt=0.1, sweeps=sweeps, tol=1e-4)
    elif kind == "adjoint":
        n = _log(rng, 8e3, 6e4)
        s = (n / (101 * 36 * 16)) ** (1 / 3)
        c = dict(kind="adjoint", nx=round(101 * s), ny=round(36 * s), nz=max(5, round(16 * s)),
                 h=0.2, M=min(M, 4), dt=0.05, sweeps=min(sweeps, 4), tol=1e-5)
    else:
        n = _log(rng, 3e3, 6e4)
        s = (n / (61 * 23 * 15)) ** (1 / 3)
        c = dict(kind="solve", nx=round(61 * s), ny=round(23 * s), nz=max(5, round(15 * s)),
                 h=0.1, noalloc=rng.random() < 0.5, c=0.0125)
    c.pop("name", None)
    return c


# ---- inputs ------------------------------------------------------------------------

@functools.lru_cache(maxsize=1)
def _cable():
    """Profile (xi, v, w) of the front travelling along a cable with D = 1, xi = 0 where
    v = 1/2, positive ahead of it."""
    h, dt, n = 0.05, 0.001, 700
    x = np.arange(n) * h
    v, w = np.where(x < 3.0, 1.0, 0.0), np.zeros(n)
    while True:
        lap = np.empty(n)
        lap[1:-1] = v[2:] - 2.0 * v[1:-1] + v[:-2]
        lap[0], lap[-1] = 2.0 * (v[1] - v[0]), 2.0 * (v[-2] - v[-1])
        dv = lap / h ** 2 - AP["ga"] * v * (v - AP["a"]) * (v - 1.0) - v * w
        dw = (AP["eps"] + AP["mu1"] * w / (v + AP["mu2"])) * (
            -w - AP["gs"] * v * (v - AP["a"] - 1.0))
        v, w = v + dt * dv, w + dt * dw
        if v[500] > 0.5:
            break
    k = int(np.nonzero(v > 0.5)[0][-1])
    front = x[k] + h * (v[k] - 0.5) / (v[k] - v[k + 1])
    return x - front, v, w


def _front(xi):
    x, v, w = _cable()
    return np.interp(xi, x, v), np.interp(xi, x, w)


@functools.lru_cache(maxsize=3)
def _mesh(nx, ny, nz, h, shell):
    if shell:
        return WM.ventricle_shell(shell, W.SEED_BASE + 5)
    return WM.kuhn3d(nx, ny, nz, h) if nz > 1 else WM.grid2d(nx, ny, h)


def _mono(case):
    """Mesh, conductivity tensor and stimulated nodes of a monodomain case."""
    mesh = _mesh(case["nx"], case["ny"], case["nz"], case["h"], case.get("shell", 0.0))
    if case.get("shell"):
        sigma = np.eye(3)
    else:
        sigma = np.diag([1.0, 0.25, 0.25]) if mesh.dim == 3 else np.eye(3)
    stim = np.zeros(0, np.int32)
    if case.get("phase") == "stimulus":
        stim = np.nonzero((mesh.xyz <= 1.5 + 1e-12).all(axis=1))[0].astype(np.int32)
    return mesh, sigma, stim


def _mono_state(case, mesh, seed):
    rng = np.random.default_rng(seed)
    if case.get("phase") == "stimulus":
        # early wave around the stimulated corner, slower across the fibres
        d = np.sqrt(mesh.xyz[:, 0] ** 2 + 4.0 * mesh.xyz[:, 1] ** 2 + 4.0 * mesh.xyz[:, 2] ** 2)
        return _front(d - rng.uniform(1.6, 3.0))
    if case.get("shell"):
        z = mesh.xyz[:, 2] - mesh.xyz[:, 2].min()
        return _front((z - rng.uniform(3.0, 6.0)) / math.sqrt(0.5))
    x = mesh.xyz[:, 0]
    return _front(x - rng.uniform(0.3, 0.7) * x.max())


@functools.lru_cache(maxsize=2)
def _emi(geometry, h, cx, cy, cz, box):
    if geometry == "branched":
        wl, blocks = WE.emi_branched_2d(h=h, sweeps=4), None
    else:
        wl, blocks = WE.emi_bricks(cells=(cx, cy, cz), h=h), None
    if box:
        order, blocks = WE.block_major(wl, WE.coarse_blocks(wl, split=(2 * box, box, box)))
        wl = WE.renumber(wl, order)
    return wl, blocks


def _emi_case(case):
    return _emi(case["geometry"], case["h"], case["cx"], case["cy"], case["cz"], case["box"])


def _emi_state(wl, seed):
    rng = np.random.default_rng(seed)
    cell = int(rng.integers(1, int(wl.labels.max()) + 1))
    return np.where(wl.labels == cell, rng.uniform(0.8, 1.0), 0.0), np.zeros(wl.n_pairs)


@functools.lru_cache(maxsize=2)
def _instances(count, nmin, nmax, sizes):
    return tuple(W.batch_instances(count, 1000 + sizes, nmin=nmin, nmax=nmax))


def _batch_state(wls, seed):
    rng = np.random.default_rng(seed)
    vs, ws = [], []
    for wl in wls:
        cx, cy = wl.mesh.xyz.max(axis=0) * rng.uniform(0.2, 0.8, size=2)
        d = np.hypot(wl.mesh.xyz[:, 0] - cx, wl.mesh.xyz[:, 1] - cy)
        v, w = _front((d - rng.uniform(1.0, 8.0)) / math.sqrt(wl.meta["D"]))
        vs.append(v)
        ws.append(w)
    return np.concatenate(vs), np.concatenate(ws)


def _adjoint_inputs(case, seed):
    mesh = _mesh(case["nx"], case["ny"], case["nz"], case["h"], 0.0)
    rng = np.random.default_rng(seed)
    v, w = _front(mesh.xyz[:, 0] - rng.uniform(0.3, 0.7) * mesh.xyz[:, 0].max())
    scale = 1.0 + 0.1 * rng.standard_normal(mesh.n_nodes)
    lam = np.zeros(mesh.n_nodes)
    lam[rng.choice(mesh.n_nodes, size=256)] = rng.standard_normal(256)
    return mesh, v, w, scale, lam, 0.1 * rng.standard_normal(mesh.n_nodes)


def _solve_inputs(case, seed):
    mesh = _mesh(case["nx"], case["ny"], case["nz"], case["h"], 0.0)
    rng = np.random.default_rng(seed)
    v, w = _front(mesh.xyz[:, 0] - rng.uniform(0.3, 0.7) * mesh.xyz[:, 0].max())
    J = AP["ga"] * (3.0 * v * v - 2.0 * (1.0 + AP["a"]) * v + AP["a"]) + w
    return mesh, J, rng.standard_normal(mesh.n_nodes) * np.exp(-4.0 * (v - 0.5) ** 2)


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _options(case):
    kw = {}
    if case.get("energy"):
        kw = dict(energy_stop=1, sdc_rho=RHO)
    if case.get("shell"):
        kw["reorder"] = 1
    if case["kind"] == "emi":
        kw["w_frozen"] = 1 if case["geometry"] == "branched" else 0
        kw["cg_maxit"] = 20000
    return default_options(**kw)


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    kind = case["kind"]
    if kind == "step":
        mesh, sigma, stim = _mono(case)
        ctx = Context(mesh.dim, mesh.xyz, mesh.elems, sigma=sigma, elem_sigma=mesh.elem_sigma,
                      ionic=AP, M=case["M"], options=_options(case), stream=stream)
        if stim.size:
            ctx.set_stimulus(stim, 2.0, 0.0, 1.0)
        v, w = _mono_state(case, mesh, seed)
    elif kind == "emi":
        wl, blocks = _emi_case(case)
        emi = dict(pair_k=wl.pair_k, pair_l=wl.pair_l, pair_area=wl.pair_area,
                   pair_kind=wl.pair_kind, robin=wl.robin, Cm=wl.Cm, g_gap=wl.g_gap)
        ctx = Context(wl.mesh.dim, wl.mesh.xyz, wl.mesh.elems, sigma=np.eye(3),
                      elem_sigma=wl.mesh.elem_sigma, ionic=AP, M=case["M"],
                      options=_options(case), stream=stream, emi=emi)
        if case["two_level"]:
            ctx.set_coarse_blocks(blocks)
        v, w = _emi_state(wl, seed)
    elif kind == "batch":
        wls = [_with_order(wl, case["M"]) for wl in
               _instances(case["count"], case["nmin"], case["nmax"], case["sizes"])]
        ctx = Batch(wls, stream=stream)
        v, w = _batch_state(wls, seed)
    elif kind == "adjoint":
        mesh, v, w, scale, lam_v, lam_w = _adjoint_inputs(case, seed)
        ctx = Context(mesh.dim, mesh.xyz, mesh.elems, sigma=np.diag([1.0, 0.25, 0.25]),
                      dof_scale=scale, ionic=AP, M=case["M"], stream=stream)
        z = _dev(np.zeros(mesh.n_nodes))
        return dict(case=case, ctx=ctx, v0=_dev(v), w0=_dev(w), v=z.clone(), w=z.clone(),
                    tape=ctx.new_tape(case["sweeps"], z.device), lam_v=_dev(lam_v),
                    lam_w=_dev(lam_w), lam_v0=z.clone(), lam_w0=z.clone(), grad_scale=z.clone())
    else:
        mesh, J, b = _solve_inputs(case, seed)
        ell = _ell(mesh)
        dev = {k: torch.tensor(a, device="cuda") for k, a in ell.items() if k not in ("ld", "width")}
        return dict(case=case, n=mesh.n_nodes, ld=ell["ld"], width=ell["width"], J=_dev(J),
                    b=_dev(b) * dev["mass"], x=_dev(np.zeros(mesh.n_nodes)), stream=stream, **dev)
    v0, w0 = _dev(v), _dev(w)
    return dict(case=case, ctx=ctx, v0=v0, w0=w0, v=v0.clone(), w=w0.clone())


def _with_order(wl, M):
    import copy
    wl = copy.copy(wl)
    wl.M, wl.ionic = M, AP
    return wl


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        f = api.pcg_solve_noalloc if case["noalloc"] else api.pcg_solve
        f(state["n"], state["val"], state["col"], state["len"], state["ld"], state["width"],
          state["diag"], state["mass"], state["J"], case["c"], state["b"], state["x"],
          stream=state["stream"])
        return {"x": state["x"]}
    v, w, ctx = state["v"], state["w"], state["ctx"]
    v.copy_(state["v0"])
    w.copy_(state["w0"])
    if case["kind"] == "adjoint":
        ctx.step_taped(v, w, 2.0, case["dt"], case["sweeps"], case["tol"], state["tape"])
        state["grad_scale"].zero_()
        grad_ionic = np.zeros(3)
        ctx.adjoint(state["tape"], state["v0"], state["w0"], case["dt"], state["lam_v"],
                    state["lam_w"], state["lam_v0"], state["lam_w0"],
                    grad_scale=state["grad_scale"], grad_ionic=grad_ionic)
        return {"v": v, "w": w, "lam_v0": state["lam_v0"], "lam_w0": state["lam_w0"],
                "grad_scale": state["grad_scale"], "grad_ionic": grad_ionic}
    t = 0.5 if case.get("phase") == "stimulus" else 2.0
    ctx.step(v, w, t, case["dt"], case["sweeps"], case["tol"])
    return {"v": v, "w": w}


# ---- work --------------------------------------------------------------------------

def _size(case):
    """(dofs, stored entries per row, gating variables, CG iterations of a first-sweep solve)."""
    if case["kind"] == "emi":
        wl, blocks = _emi_case(case)
        return wl.n, (5.0 if wl.mesh.dim == 2 else 7.5), wl.n_pairs, (
            300 if case["two_level"] else 1000)
    if case["kind"] == "batch":
        wls = _instances(case["count"], case["nmin"], case["nmax"], case["sizes"])
        n = sum(wl.n for wl in wls)
        return n, 5.0, n, 15
    if case.get("shell"):
        n = _mesh(0, 0, 0, case["h"], case["shell"]).n_nodes
        return n, 13.5, n, 20
    n = case["nx"] * case["ny"] * case["nz"]
    return n, (7.0 if case["nz"] > 1 else 5.0), n, 20


def work(case):
    """The matrix and the state read once and the new state written once; the floating
    operations of one sweep over all dofs (textbook CG: z + 8 multiply-adds per row and
    iteration), the least that a step takes."""
    n, z, nw, its = _size(case)
    matrix = n * (12.0 * z + 8.0)
    if case["kind"] == "solve":
        return {"bytes": matrix + 24.0 * n, "flops": 2.0 * its * n * (z + 8.0)}
    passes = 2 if case["kind"] == "adjoint" else 1
    return {"bytes": passes * matrix + passes * 16.0 * (n + nw),
            "flops": passes * 2.0 * case["M"] * its * n * (z + 8.0)}


# ---- the same results in plain torch -----------------------------------------------

def _radau(M):
    """Radau-IIA nodes, cumulative quadrature Q and the LU-trick matrix Qhat."""
    P = np.polynomial.legendre.Legendre
    poly = P.basis(M) - P.basis(M - 1)                 # zeros: interior nodes and 1
    tau = np.sort((poly.roots().real + 1.0) / 2.0)
    tau[-1] = 1.0
    for _ in range(3):                                 # polish the interior nodes
        x = 2.0 * tau[:-1] - 1.0
        tau[:-1] -= 0.5 * poly(x) / poly.deriv()(x)
    p = np.arange(M)
    V = tau[None, :] ** p[:, None]
    Q = np.linalg.solve(V, (tau[None, :] ** (p[:, None] + 1)) / (p[:, None] + 1)).T
    U = Q.T.copy()
    for c in range(M):
        for r in range(c + 1, M):
            U[r] -= U[r, c] / U[c, c] * U[c]
    return Q, np.triu(U).T


class _Stiffness:
    """P1 stiffness matrix applied element by element (differentiable in the node scale)."""

    def __init__(self, mesh, sigma, dev):
        self.n = mesh.n_nodes
        el = torch.tensor(mesh.elems.astype(np.int64), device=dev)
        x = torch.tensor(mesh.xyz, device=dev)[el]
        d, nv = mesh.dim, mesh.dim + 1
        E = (x[:, 1:] - x[:, :1]).transpose(1, 2)      # columns: edges from vertex 0
        G = torch.linalg.inv(E)                        # rows: gradients of vertices 1..d
        G = torch.cat([-G.sum(1, keepdim=True), G], 1)
        vol = torch.linalg.det(E).abs() / math.factorial(d)
        S = torch.tensor(np.asarray(sigma, dtype=np.float64), device=dev)
        S = (S.expand(len(el), 3, 3) if S.dim() == 2 else S)[:, :d, :d]
        self.Ke = vol[:, None, None] * (G @ S @ G.transpose(1, 2))
        self.el, self.nv = el, nv
        self.mass = torch.zeros(self.n, dtype=torch.float64, device=dev).index_add_(
            0, el.reshape(-1), (vol / nv).repeat_interleave(nv))
        self.scale = None

    def __call__(self, x):
        y = torch.einsum("eab,eb->ea", self.Ke, x[self.el])
        if self.scale is not None:
            y = y * self.scale[self.el].mean(1, keepdim=True)
        return torch.zeros_like(x).index_add(0, self.el.reshape(-1), y.reshape(-1))

    def diag(self):
        y = torch.diagonal(self.Ke, dim1=1, dim2=2)
        if self.scale is not None:
            y = y * self.scale.detach()[self.el].mean(1, keepdim=True)
        return torch.zeros(self.n, dtype=torch.float64, device=self.el.device).index_add_(
            0, self.el.reshape(-1), y.reshape(-1))


def _cg(A, d, b, rtol=1e-13, maxit=30000):
    x, r = torch.zeros_like(b), b.clone()
    z = r / d
    p, rz = z.clone(), torch.dot(r, z)
    lim = rtol * rtol * rz
    for k in range(maxit):
        if k % 8 == 0 and not bool(rz > lim):
            break
        q = A(p)
        al = torch.where(rz > 0, rz / torch.dot(p, q), torch.zeros_like(rz))
        x, r = x + al * p, r - al * q
        z = r / d
        new = torch.dot(r, z)
        p, rz = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * p, new
    return x


class _Inverse(torch.autograd.Function):
    """A^-1 b for a symmetric A held fixed."""

    @staticmethod
    def forward(ctx, b, A, d):
        ctx.A, ctx.d = A, d
        return _cg(A, d, b)

    @staticmethod
    def backward(ctx, g):
        return _cg(ctx.A, ctx.d, g.contiguous()), None, None


def _solve(A, d, b):
    """A^-1 b, differentiable in b and in what A holds: x0 + A^-1 (b - A x0)."""
    with torch.no_grad():
        x0 = _cg(A, d, b)
    if not torch.is_grad_enabled():
        return x0

    def fixed(p):
        with torch.no_grad():
            return A(p)
    return x0 + _Inverse.apply(b - A(x0), fixed, d)


def _sdc_step(K, kdiag, area, Cm, gap, g_gap, gather, scatter, scatter_abs, touched, stim, v0, w0,
              ion, M, dt, sweeps, tol, energy=False, frozen=False):
    """One adaptive SDC step.  Ionic currents and gating live on sites: the nodes of a
    monodomain model (gather and scatter are the identity), the membrane pairs of a
    cell-by-cell one (gather: potential difference, scatter: its transpose)."""
    ga, gs, a, eps, mu1, mu2, cw = (ion[k] for k in ("ga", "gs", "a", "eps", "mu1", "mu2", "cw"))
    Q, Qh = _radau(M)
    live = ~gap
    V, Wn = [v0] * M, [w0] * M
    mask = torch.ones_like(v0, dtype=torch.bool)
    for _ in range(sweeps):
        if not bool(mask.any()):
            break
        on = mask.to(torch.float64)
        f, J = [], []
        for j in range(M):
            v = gather(V[j])
            I = torch.where(live, ga * v * (v - a) * (v - 1.0) + v * Wn[j], g_gap * v)
            J.append(torch.where(live, ga * (3.0 * v * v - 2.0 * (1.0 + a) * v + a) + Wn[j],
                                 g_gap * torch.ones_like(v)))
            f.append(-K(V[j]) - scatter(area * (I - stim)))
        b = [on * (scatter(area * Cm * gather(v0 - V[m])) + dt * sum(Q[m, j] * f[j]
                                                                     for j in range(M)))
             for m in range(M)]
        dv, E = [], 0.0
        for m in range(M):
            c = dt * Qh[m, m]

            def A(x, Jm=J[m], c=c, on=on):
                return on * (scatter(area * (Cm + c * Jm) * gather(on * x)) + c * K(on * x)
                             ) + (1.0 - on) * x
            d = (on * (scatter_abs(area * (Cm + c * J[m])) + c * kdiag) + (1.0 - on)).detach()
            x = _solve(A, d, b[m])
            E = E + torch.dot(x, A(x)).detach()
            g = on * (K(x) + scatter(area * J[m] * gather(x)))
            for k in range(m + 1, M):
                b[k] = b[k] - dt * Qh[k, m] * g
            dv.append(x)
        V = [V[m] + dv[m] for m in range(M)]
        if not frozen:
            R, dR = [], []
            for m in range(M):
                v = gather(V[m])
                G, H = -Wn[m] - gs * v * (v - a - 1.0), eps + mu1 * Wn[m] / (v + mu2)
                R.append(cw * H * G)
                dR.append(cw * (mu1 / (v + mu2) * G - H))
            e, act = [], touched(mask) & live
            for m in range(M):
                s = w0 + dt * sum(Q[m, j] * R[j] for j in range(M)) - Wn[m]
                s = s + dt * sum(Qh[m, j] * dR[j] * e[j] for j in range(m))
                e.append(torch.where(act, s / (1.0 - dt * Qh[m, m] * dR[m]), torch.zeros_like(s)))
            Wn = [Wn[m] + e[m] for m in range(M)]
        if energy and float(E) <= ((1.0 - RHO) / RHO * tol) ** 2:
            break
        mask = mask & (torch.stack(dv).detach().abs().amax(0) >= ALPHA * tol)
    return V[-1], Wn[-1]


def _mono_exact(mesh, sigma, stim, v, w, case, dev, scale=None, ion=None):
    K = _Stiffness(mesh, mesh.elem_sigma if mesh.elem_sigma is not None else sigma, dev)
    K.scale = scale
    amp = torch.zeros(K.n, dtype=torch.float64, device=dev)
    if stim.size:
        amp[torch.tensor(stim.astype(np.int64), device=dev)] = 2.0
    same = lambda x: x
    return _sdc_step(K, K.diag(), K.mass, 1.0, torch.zeros(K.n, dtype=torch.bool, device=dev), 0.0,
                     same, same, same, same, amp, v, w, ion or AP, case["M"], case["dt"],
                     case["sweeps"], case["tol"], energy=bool(case.get("energy")))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=dev)
    kind = case["kind"]
    if kind == "solve":
        mesh, J, b = _solve_inputs(case, seed)
        K = _Stiffness(mesh, np.diag([1.0, 0.25, 0.25]), dev)
        s, c = K.mass * (1.0 + case["c"] * t(J)), case["c"]
        with torch.no_grad():
            return {"x": _cg(lambda x: s * x + c * K(x), s + c * K.diag(), t(b) * K.mass)}
    if kind == "adjoint":
        mesh, v, w, scale, lam_v, lam_w = _adjoint_inputs(case, seed)
        v, w, scale = (t(x).requires_grad_() for x in (v, w, scale))
        ion = dict(AP)
        for k in ("ga", "gs", "a"):
            ion[k] = torch.tensor(AP[k], dtype=torch.float64, device=dev, requires_grad=True)
        v1, w1 = _mono_exact(mesh, np.diag([1.0, 0.25, 0.25]), np.zeros(0, np.int32), v, w, case,
                             dev, scale, ion)
        g = torch.autograd.grad(torch.dot(t(lam_v), v1) + torch.dot(t(lam_w), w1),
                                [v, w, scale, ion["ga"], ion["gs"], ion["a"]])
        return {"v": v1.detach(), "w": w1.detach(), "lam_v0": g[0], "lam_w0": g[1],
                "grad_scale": g[2], "grad_ionic": torch.stack(g[3:])}
    with torch.no_grad():
        if kind == "step":
            mesh, sigma, stim = _mono(case)
            v, w = _mono_state(case, mesh, seed)
            v, w = _mono_exact(mesh, sigma, stim, t(v), t(w), case, dev)
            return {"v": v, "w": w}
        if kind == "batch":
            wls = _instances(case["count"], case["nmin"], case["nmax"], case["sizes"])
            v, w = _batch_state(wls, seed)
            vs, ws, at = [], [], 0
            for wl in wls:
                v1, w1 = _mono_exact(wl.mesh, wl.sigma, np.zeros(0, np.int32),
                                     t(v[at:at + wl.n]), t(w[at:at + wl.n]), case, dev)
                vs.append(v1)
                ws.append(w1)
                at += wl.n
            return {"v": torch.cat(vs), "w": torch.cat(ws)}
        wl, _ = _emi_case(case)
        u, w = _emi_state(wl, seed)
        K = _Stiffness(wl.mesh, wl.mesh.elem_sigma, dev)
        robin = t(wl.robin)
        pk, pl = (torch.tensor(x.astype(np.int64), device=dev) for x in (wl.pair_k, wl.pair_l))
        gather = lambda x: x[pk] - x[pl]
        scatter = lambda y: torch.zeros(K.n, dtype=torch.float64, device=dev).index_add_(
            0, pk, y).index_add_(0, pl, -y)
        scatter_abs = lambda y: torch.zeros(K.n, dtype=torch.float64, device=dev).index_add_(
            0, pk, y).index_add_(0, pl, y)
        u, w = _sdc_step(lambda x: K(x) + robin * x, K.diag() + robin, t(wl.pair_area), wl.Cm,
                         torch.tensor(wl.pair_kind == 1, device=dev), wl.g_gap, gather, scatter,
                         scatter_abs, lambda on: on[pk] | on[pl],
                         torch.zeros(wl.n_pairs, dtype=torch.float64, device=dev), t(u), t(w), AP,
                         case["M"], case["dt"], case["sweeps"], case["tol"],
                         frozen=case["geometry"] == "branched")
        return {"v": u, "w": w}


def _ell(mesh):
    """Stiffness matrix of the mesh (fibres along x) as the node solve takes it: diagonal,
    column-major off-diagonal slots, lumped mass."""
    K = _Stiffness(mesh, np.diag([1.0, 0.25, 0.25]), "cpu")
    n, nv = K.n, K.nv
    el, Ke = K.el.numpy(), K.Ke.numpy()
    key = (el[:, :, None] * np.int64(n) + el[:, None, :]).reshape(-1)
    key, inv = np.unique(key, return_inverse=True)
    val = np.bincount(inv.reshape(-1), weights=Ke.reshape(-1))
    row, col = key // n, key % n
    diag = np.zeros(n)
    diag[row[row == col]] = val[row == col]
    keep = (row != col) & (np.abs(val) > 1e-12 * np.sqrt(diag[row] * diag[col]))
    row, col, val = row[keep], col[keep], val[keep]
    length = np.bincount(row, minlength=n)
    slot = np.arange(row.size) - np.concatenate([[0], np.cumsum(length)[:-1]])[row]
    ld, width = (n + 31) // 32 * 32, int(length.max())
    ev, ec = np.zeros((width, ld)), np.zeros((width, ld), dtype=np.int32)
    ev[slot, row], ec[slot, row] = val, col
    return dict(val=ev, col=ec, len=length.astype(np.int32), diag=diag, mass=K.mass.numpy(),
                ld=ld, width=width)

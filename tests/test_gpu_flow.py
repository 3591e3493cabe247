"""The node-solve kernels that keep every vector on chip (cg_flow.cuh) against the oracle at
the edges of their launch rule: chunks of 32 rows, CTAs of 128 rows, one or more rows per
thread, x in shared or global memory, two or three buffers for r and w; and solves whose
gamma leaves the window of the fixed-point sums in one iteration, downwards and upwards.

Tolerance: that of the parity tests, 1e-10 relative in the max norm and CG counts to one
(both sides stop at rtol = 1e-10).
"""

import numpy as np
import pytest

import oracle
import workloads as W
from workloads.configs import AP_BENCH, Workload
from workloads.meshes import grid2d

pytestmark = pytest.mark.gpu

RTOL = 1e-10


@pytest.fixture(scope="module")
def torch_dev():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_07206_gb300 import build as b
    b.build()
    return torch, torch.device("cuda:0")


def _workload(nx, ny, h, dt, M=2, sweeps=2, tol=0.0, v=None):
    mesh = grid2d(nx, ny, h)
    rng = np.random.default_rng(nx * 1000 + ny)
    v0 = rng.uniform(0.0, 1.0, mesh.n_nodes) if v is None else v(rng, mesh.n_nodes)
    return Workload("grid", mesh, np.diag([1.0, 0.5, 1.0]), dict(AP_BENCH), M=M, dt=dt,
                    sweeps=sweeps, tol=tol, steps=1, v0=v0, w0=np.zeros(mesh.n_nodes))


def _check(wl, torch, dev, **opts):
    from paper_2311_07206_gb300 import Context, default_options
    ctx = Context.from_workload(wl, options=default_options(cg_maxit=20000, **opts),
                                stream=torch.cuda.current_stream(dev).cuda_stream)
    v = torch.tensor(wl.v0, dtype=torch.float64, device=dev)
    w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    st = ctx.step(v, w, 0.0, wl.dt, wl.sweeps, wl.tol)
    ctx.close()
    r = oracle.System.from_mesh(wl.mesh, wl.sigma).step(wl.ionic, wl.M, wl.v0, wl.w0, wl.dt,
                                                        wl.sweeps, wl.tol, cg_maxit=20000)
    assert r["status"] == 0
    for a, b in ((v, r["v"]), (w, r["w"])):
        assert np.abs(a.cpu().numpy() - b).max() <= RTOL * max(1.0, np.abs(b).max())
    for k in range(wl.sweeps):
        for m in range(wl.M):
            a, b = st.cg_iters[k][m], r["stats"].cg_iters[k * 8 + m]
            # ill-conditioned solves: counts differ by rounding, within 10 %
            assert abs(a - b) <= max(1, b // 10), (k, m, a, b)
    return st


@pytest.mark.parametrize("pipelined", [0, 1])
@pytest.mark.parametrize("nx,ny,blocks", [
    (2, 2, 0), (4, 8, 0), (3, 11, 0), (8, 16, 0), (3, 43, 0),    # one chunk, one CTA, and one more
    (139, 140, 0),                                               # 152 CTAs of 128 rows, and more
    (28, 32, 1), (23, 39, 1),                                    # one row per thread, then more
    (61, 63, 1), (64, 65, 1),                                    # x on chip, then in global memory
    (64, 90, 1), (67, 86, 1),                                    # three buffers, then two
])
def test_edges_of_the_launch_rule(torch_dev, nx, ny, blocks, pipelined):
    torch, dev = torch_dev
    _check(_workload(nx, ny, 0.3, 0.1), torch, dev, cg_pipelined=pipelined, cg_max_blocks=blocks)


@pytest.mark.parametrize("pipelined", [0, 1])
def test_gamma_falls_below_the_window(torch_dev, pipelined):
    """c K / m ~ 1e-5: gamma falls by about 1e-10 (2^-33) per iteration."""
    torch, dev = torch_dev
    st = _check(_workload(40, 37, 0.3, 1e-6), torch, dev, cg_pipelined=pipelined)
    assert st.cg_iters[0][0] <= 4


def test_gamma_rises_above_the_window(torch_dev):
    """The right-hand side is the lowest mode with a trace of high modes: the first step of
    CG, exact for the low mode, lifts the others by (lambda_high / lambda_low)^2 > 2^10."""
    torch, dev = torch_dev
    wl = _workload(40, 37, 2e-3, 0.1, sweeps=1,
                   v=lambda rng, n: 0.5 + 1e-8 * rng.standard_normal(n))
    # gamma_1 / gamma_0 of the same CG on the host: the case does what it says
    S = oracle.System.from_mesh(wl.mesh, wl.sigma)
    K, m = S.dense()
    c = wl.dt * oracle.collocation(wl.M)[2][0, 0]
    v = wl.v0
    J = 8.0 * (3.0 * v * v - 2.0 * 1.15 * v + 0.15)
    f = -K @ v - m * 8.0 * v * (v - 0.15) * (v - 1.0)
    b = wl.dt * oracle.collocation(wl.M)[1][0].sum() * f
    A = np.diag(m * (1.0 + c * J)) + c * K
    d = np.diag(A)
    r1 = b - (b @ (b / d)) / ((b / d) @ A @ (b / d)) * (A @ (b / d))
    assert (r1 @ (r1 / d)) / (b @ (b / d)) > 2.0 ** 11
    _check(wl, torch, dev, cg_pipelined=0)


@pytest.mark.parametrize("blocks", [0, 1, 3])
def test_two_level_edges(torch_dev, blocks):
    """Cell-by-cell bricks of 4,176 dofs in 72 blocks: on many CTAs (pieces of one warp and
    less), on one CTA (two buffers, x in global memory, rows many times the threads) and on
    three (pieces across CTAs).  Counts to 5 %, as the two-level parity tests have them."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import Context, default_options
    from workloads.emi import coarse_blocks, emi_bricks
    wl = emi_bricks(cells=(2, 1, 1), cell_um=(24.0, 14.0, 10.0), h=2.0, margin=2, sweeps=2)
    lab = coarse_blocks(wl, split=(6, 2, 2), min_dofs=300)
    assert (wl.n, lab.max() + 1) == (4176, 72)
    ctx = Context.from_emi(wl, options=default_options(cg_max_blocks=blocks),
                           stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx.set_coarse_blocks(lab)
    u = torch.tensor(wl.u0, dtype=torch.float64, device=dev)
    w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    st = ctx.step(u, w, 0.0, wl.dt, wl.sweeps, wl.tol)
    ctx.close()
    r = oracle.System.from_mesh(wl.mesh).step_emi(wl, wl.u0, wl.w0, coarse=lab)
    assert r["status"] == 0
    for a, b in ((u, r["u"]), (w, r["w"])):
        assert np.abs(a.cpu().numpy() - b).max() <= RTOL * max(1.0, np.abs(b).max())
    for k in range(wl.sweeps):
        for m in range(wl.M):
            a, b = st.cg_iters[k][m], r["stats"].cg_iters[k * 8 + m]
            assert abs(a - b) <= max(2, b // 20), (k, m, a, b)


def test_launch_ids_wrap(torch_dev):
    """A context numbers its solves with 12 bits and clears the published words when the
    number wraps: 4,500 solves of the same step give the same bits every time (the sums are
    exact, so nothing depends on the order of the CTAs)."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import Context, default_options
    wl = _workload(20, 17, 0.3, 0.1, M=3, sweeps=1)      # 340 rows: four CTAs
    ctx = Context.from_workload(wl, options=default_options(),
                                stream=torch.cuda.current_stream(dev).cuda_stream)
    v0 = torch.tensor(wl.v0, dtype=torch.float64, device=dev)
    w0 = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    first = None
    for k in range(1500):
        v, w = v0.clone(), w0.clone()
        ctx.step(v, w, 0.0, wl.dt, wl.sweeps, wl.tol)
        if first is None:
            first = (v, w)
        elif k % 50 == 0 or 1360 < k < 1370:            # 1,365 steps: the wrap
            assert torch.equal(v, first[0]) and torch.equal(w, first[1]), k
    ctx.close()


@pytest.mark.parametrize("nx,ny", [(365, 356), (365, 357)])   # 129,940 rows and 130,305
def test_stand_alone_solves_on_both_sides_of_the_arrangements(torch_dev, nx, ny):
    """sdc_pcg_solve in the pipelined and in the classical kernel: a five-point matrix with
    mass 1 and c K of condition about 10.  The recurrence residual is at 1e-10; the true one
    differs by rounding, below 30 iterations x cond x 2^-52 ~ 1e-13: bound 1.01e-10."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import binding
    n = nx * ny
    ld = (n + 31) // 32 * 32
    i = np.arange(n)
    x_, y_ = i % nx, i // nx
    val, col = np.zeros((4, ld)), np.zeros((4, ld), dtype=np.int32)
    ln = np.zeros(n, dtype=np.int32)
    kd = np.zeros(n)
    for ok, off in ((x_ > 0, -1), (x_ < nx - 1, 1), (y_ > 0, -nx), (y_ < ny - 1, nx)):
        r = i[ok]
        val[ln[r], r], col[ln[r], r] = -1.0, r + off
        ln[r] += 1
        kd[r] += 1.0
    rng = np.random.default_rng(n)
    mass, J, c = np.ones(n), rng.uniform(0.0, 0.2, n), 1.0
    b = rng.standard_normal(n)
    t = lambda a: torch.tensor(a, device=dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    it, rr = binding.pcg_solve(n, t(val), t(col), t(ln), ld, 4, t(kd), t(mass), t(J), c, t(b), x,
                               rtol=1e-10, maxit=1000,
                               stream=torch.cuda.current_stream(dev).cuda_stream)
    assert 5 < it < 60 and rr <= 1e-10
    xh = x.cpu().numpy()
    d = mass * (1.0 + c * J) + c * kd
    Ax = d * xh
    for k in range(4):
        m = ln > k
        Ax[m] += c * val[k, :n][m] * xh[col[k, :n][m]]
    r = b - Ax
    assert np.sqrt((r * r / d).sum() / (b * b / d).sum()) <= 1.01e-10


@pytest.mark.parametrize("nx,ny", [(512, 256), (331, 396)])   # 1,024 blocks of 128 rows, and 1,025
def test_selection_on_both_sides_of_its_launch_rule(torch_dev, nx, ny):
    """A front over a third of the grid: the rows far from it leave the set after a sweep.  The
    sizes of the sets are the oracle's."""
    torch, dev = torch_dev
    wl = _workload(nx, ny, 0.3, 0.05, sweeps=3, tol=1e-4,
                   v=lambda rng, n: (np.arange(n) < n // 3).astype(float))
    st = _check(wl, torch, dev)
    r = oracle.System.from_mesh(wl.mesh, wl.sigma).step(wl.ionic, wl.M, wl.v0, wl.w0, wl.dt,
                                                        wl.sweeps, wl.tol, cg_maxit=20000)
    n = list(st.n_active)[:wl.sweeps]
    assert n == list(r["stats"].n_active)[:wl.sweeps]
    assert 0 < n[1] < n[0]

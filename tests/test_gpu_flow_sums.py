"""The sums of the on-chip node solves where the partial sums of more than 131,072 threads are
close to each other (spatially uniform states, slow trends), and at the top of the FP64 range.

Tolerance: that of the parity tests, 1e-10 relative in the max norm (both sides stop at
rtol = 1e-10).  A spatially uniform state stays uniform (K 1 = 0), so its step is that of a
small mesh.
"""

import numpy as np
import pytest

import oracle
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


def _workload(nx, ny, v0):
    mesh = grid2d(nx, ny, 0.3)
    return Workload("grid", mesh, np.diag([1.0, 0.5, 1.0]), dict(AP_BENCH), M=2, dt=0.1, sweeps=2,
                    tol=0.0, steps=1, v0=v0(mesh), w0=np.zeros(mesh.n_nodes))


def _context(wl, torch, dev, **opts):
    from paper_2311_07206_gb300 import Context, default_options
    return Context.from_workload(wl, options=default_options(**opts),
                                 stream=torch.cuda.current_stream(dev).cuda_stream)


def _step(ctx, wl, v0, torch, dev):
    v = torch.tensor(v0, dtype=torch.float64, device=dev)
    w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    ctx.step(v, w, 0.0, wl.dt, wl.sweeps, wl.tol)
    return v.cpu().numpy(), w.cpu().numpy()


@pytest.mark.parametrize("pipelined", [0, 1])
@pytest.mark.parametrize("nx,ny", [(456, 342), (666, 665)])   # 155,952 and 442,890 rows
def test_uniform_states(torch_dev, nx, ny, pipelined):
    torch, dev = torch_dev
    wl = _workload(nx, ny, lambda m: np.full(m.n_nodes, 0.5))
    small = _workload(3, 3, lambda m: np.full(m.n_nodes, 0.5))
    S = oracle.System.from_mesh(small.mesh, small.sigma)
    ctx = _context(wl, torch, dev, cg_pipelined=pipelined)
    for amp in np.exp(np.linspace(np.log(0.2), np.log(0.9), 12)):
        v, w = _step(ctx, wl, np.full(wl.n, amp), torch, dev)
        r = S.step(small.ionic, small.M, np.full(9, amp), np.zeros(9), small.dt, small.sweeps, 0.0)
        assert r["status"] == 0
        assert np.abs(v - r["v"][4]).max() <= RTOL and np.abs(w - r["w"][4]).max() <= RTOL
    ctx.close()


@pytest.mark.parametrize("pipelined", [0, 1])
def test_linear_trend(torch_dev, pipelined):
    torch, dev = torch_dev
    wl = _workload(456, 342, lambda m: 0.4 + 0.02 * m.xyz[:, 0] / m.xyz[:, 0].max())
    S = oracle.System.from_mesh(wl.mesh, wl.sigma)
    ctx = _context(wl, torch, dev, cg_pipelined=pipelined)
    for amp in (1.0, 1.2, 1.5):
        v, w = _step(ctx, wl, amp * wl.v0, torch, dev)
        r = S.step(wl.ionic, wl.M, amp * wl.v0, wl.w0, wl.dt, wl.sweeps, 0.0)
        assert r["status"] == 0
        assert np.abs(v - r["v"]).max() <= RTOL and np.abs(w - r["w"]).max() <= RTOL
    ctx.close()


def _diagonal_solve(n, b, torch, dev):
    """sdc_pcg_solve with the identity: x = b after one iteration."""
    from paper_2311_07206_gb300 import binding
    t = lambda a: torch.tensor(a, device=dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    it, rr = binding.pcg_solve(n, t(np.zeros(n)), t(np.zeros(n, np.int32)),
                               t(np.zeros(n, np.int32)), n, 1, t(np.zeros(n)), t(np.ones(n)),
                               t(np.zeros(n)), 1.0, t(b), x, rtol=1e-10, maxit=50,
                               stream=torch.cuda.current_stream(dev).cuda_stream)
    return it, x.cpu().numpy()


@pytest.mark.parametrize("n", [131_072, 155_648, 442_401])
def test_equal_right_hand_sides(torch_dev, n):
    torch, dev = torch_dev
    for amp in np.exp(np.linspace(0.0, np.log(2.0), 12)):
        it, x = _diagonal_solve(n, np.full(n, amp), torch, dev)
        assert it == 1 and np.abs(x - amp).max() <= RTOL


@pytest.mark.parametrize("n", [5, 4_000, 200_000])
def test_top_of_the_range(torch_dev, n):
    """b'b of 2^1022.5 and 2^1023.5 is solved as any other; above 2^1024 the solve ends as not
    finite."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import SdcError
    from paper_2311_07206_gb300 import binding as B
    for e in (1000.0, 1022.5, 1023.5):
        b = np.full(n, 2.0 ** (e / 2.0) / np.sqrt(n))
        it, x = _diagonal_solve(n, b, torch, dev)
        assert it == 1 and np.abs(x / b - 1.0).max() <= RTOL
    for e in (1024.5, 1030.0):
        with pytest.raises(SdcError) as err:
            _diagonal_solve(n, np.full(n, 2.0 ** (e / 2.0) / np.sqrt(n)), torch, dev)
        assert err.value.status == B.SDC_E_NONFINITE


@pytest.mark.parametrize("blocks", [0, 1])
@pytest.mark.parametrize("pipelined", [0, 1])
def test_waits_that_run_out(torch_dev, pipelined, blocks):
    """Budgets from one cycle to more than an exchange takes, so that barrier, words and sums run
    out of time here and there: a step either reports SDC_E_TIMEOUT or gives the full result, on
    the same context, whatever the steps before it did."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import SdcError
    from paper_2311_07206_gb300 import binding as B
    wl = _workload(41, 37, lambda m: 0.5 + 0.3 * np.sin(m.xyz[:, 0]))
    r = oracle.System.from_mesh(wl.mesh, wl.sigma).step(wl.ionic, wl.M, wl.v0, wl.w0, wl.dt,
                                                        wl.sweeps, 0.0)
    assert r["status"] == 0
    done = timeouts = 0
    for budget in (1, 300, 1_000, 2_000, 4_000, 10_000, 4_000_000_000):
        ctx = _context(wl, torch, dev, cg_pipelined=pipelined, cg_max_blocks=blocks,
                       spin_budget=budget)
        for _ in range(6):
            try:
                v, w = _step(ctx, wl, wl.v0, torch, dev)
            except SdcError as e:
                assert e.status == B.SDC_E_TIMEOUT and budget < 4_000_000_000
                timeouts += 1
                continue
            done += 1
            assert np.abs(v - r["v"]).max() <= RTOL and np.abs(w - r["w"]).max() <= RTOL
        ctx.close()
    assert done >= 6 and (timeouts >= 1 or blocks == 1)


@pytest.mark.parametrize("pipelined", [-1, 0, 1])
def test_a_high_iteration_limit_changes_nothing(torch_dev, pipelined):
    """cg_maxit of 1,000,000 and above: the same kernels, the same bits."""
    torch, dev = torch_dev
    wl = _workload(67, 61, lambda m: 0.5 + 0.3 * np.sin(m.xyz[:, 0]))
    out = []
    for maxit in (10_000, 1_000_000, 2**31 - 1):
        ctx = _context(wl, torch, dev, cg_pipelined=pipelined, cg_maxit=maxit)
        out.append(_step(ctx, wl, wl.v0, torch, dev))
        ctx.close()
    for v, w in out[1:]:
        assert np.array_equal(v, out[0][0]) and np.array_equal(w, out[0][1])


def test_more_iterations_than_a_tag_counts(torch_dev):
    """A chain of 1,000 links over thirteen decades does not converge in a million iterations;
    the words' tags wrap at 2^20 on the way, and the solve ends at its limit, with no wait run
    out."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import SdcError
    from paper_2311_07206_gb300 import binding as B
    n, ld = 1_000, 1_024
    rng = np.random.default_rng(1)
    k = np.exp(30.0 * rng.uniform(0.0, 1.0, n - 1))
    val, col, ln = np.zeros((2, ld)), np.zeros((2, ld), np.int32), np.zeros(n, np.int32)
    for i in range(n):
        for j in (i - 1, i + 1):
            if 0 <= j < n:
                val[ln[i], i], col[ln[i], i] = -k[min(i, j)], j
                ln[i] += 1
    kd = np.concatenate([k, [0.0]]) + np.concatenate([[0.0], k])
    t = lambda a: torch.tensor(a, device=dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    with pytest.raises(SdcError) as e:
        B.pcg_solve(n, t(val), t(col), t(ln), ld, 2, t(kd), t(np.full(n, 1e-6)), t(np.zeros(n)),
                    1.0, t(rng.uniform(-0.5, 0.5, n)), x, rtol=1e-14, maxit=1_060_000,
                    stream=torch.cuda.current_stream(dev).cuda_stream)
    assert e.value.status == B.SDC_E_CG_NOCONV


def test_a_row_longer_than_65535(torch_dev):
    """An arrow matrix whose first row has 65,699 off-diagonals (52 GB of slots, nearly all
    unused), against its Schur complement."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import binding
    n = 65_700
    ld, width = (n + 31) // 32 * 32, n - 1
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info(dev)[0] < 80e9:
        pytest.skip("not enough device memory")
    rng = np.random.default_rng(7)
    a = -rng.uniform(0.5, 1.5, n - 1)
    kd = np.concatenate([[-a.sum()], -a])
    b = rng.standard_normal(n)
    t = lambda q: torch.tensor(q, device=dev)
    val = torch.zeros((width, ld), dtype=torch.float64, device=dev)
    col = torch.zeros((width, ld), dtype=torch.int32, device=dev)
    val[:, 0], col[:, 0] = t(a), t(np.arange(1, n, dtype=np.int32))
    val[0, 1:n] = t(a)
    ln = np.ones(n, np.int32)
    ln[0] = n - 1
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    c = 0.5
    binding.pcg_solve(n, val, col, t(ln), ld, width, t(kd), t(np.ones(n)), t(np.zeros(n)), c, t(b),
                      x, rtol=1e-12, maxit=500, stream=torch.cuda.current_stream(dev).cuda_stream)
    d = 1.0 + c * kd
    x0 = (b[0] - (c * a * b[1:] / d[1:]).sum()) / (d[0] - (c * c * a * a / d[1:]).sum())
    want = np.concatenate([[x0], (b[1:] - c * a * x0) / d[1:]])
    assert np.abs(x.cpu().numpy() - want).max() <= RTOL * np.abs(want).max()
    del val, col
    torch.cuda.empty_cache()


def test_no_room_for_the_on_chip_workspace(torch_dev):
    """A tridiagonal matrix declared 65,000 slots wide: scaled values of every slot would take
    364 GB; the solve runs in the kernels that keep none."""
    torch, dev = torch_dev
    linalg = pytest.importorskip("scipy.linalg")
    from paper_2311_07206_gb300 import binding
    n, width = 700_000, 65_000
    ld = (n + 31) // 32 * 32
    val, col = np.zeros((2, ld)), np.zeros((2, ld), np.int32)
    i = np.arange(n)
    val[:, :n] = -1.0
    col[0, :n] = np.where(i > 0, i - 1, 1)
    col[1, :n] = np.minimum(i + 1, n - 1)
    ln = np.full(n, 2, np.int32)
    ln[0] = ln[-1] = 1
    kd = np.full(n, 2.0)
    kd[0] = kd[-1] = 1.0
    b = np.random.default_rng(8).standard_normal(n)
    t = lambda a: torch.tensor(a, device=dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    it, rr = binding.pcg_solve(n, t(val), t(col), t(ln), ld, width, t(kd), t(np.ones(n)),
                               t(np.zeros(n)), 1.0, t(b), x, rtol=1e-12, maxit=500,
                               stream=torch.cuda.current_stream(dev).cuda_stream)
    ab = np.zeros((3, n))
    ab[0, 1:], ab[1], ab[2, :-1] = -1.0, 1.0 + kd, -1.0
    want = linalg.solve_banded((1, 1), ab, b)
    assert rr <= 1e-12 and np.abs(x.cpu().numpy() - want).max() <= RTOL * np.abs(want).max()


def _grid_ell(nx, ny):
    n = nx * ny
    ld = (n + 31) // 32 * 32
    i = np.arange(n)
    val, col = np.zeros((4, ld)), np.zeros((4, ld), np.int32)
    ln, kd = np.zeros(n, np.int32), np.zeros(n)
    for ok, off in ((i % nx > 0, -1), (i % nx < nx - 1, 1), (i >= nx, -nx), (i < n - nx, nx)):
        r = i[ok]
        val[ln[r], r], col[ln[r], r] = -1.0, r + off
        ln[r] += 1
        kd[r] += 1.0
    return n, ld, val, col, ln, kd


@pytest.mark.parametrize("case", ["rise", "fall"])
def test_repeated_sums_in_the_pipelined_arrangement(torch_dev, case):
    """One to four iterations of a stand-alone solve (pipelined at this size) against the same
    iterates of plain CG.  Rise: the lowest mode with a trace of others, gamma grows by 2^11
    in the first iteration.  Fall: an almost diagonal matrix, 2^-30 an iteration."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import SdcError
    from paper_2311_07206_gb300 import binding as B
    n, ld, val, col, ln, kd = _grid_ell(61, 53)
    rng = np.random.default_rng(9)
    c, mass = (1.0, np.full(n, 1e-4)) if case == "rise" else (1e-5, np.ones(n))
    d = mass + c * kd

    def A(x):
        y = d * x
        for k in range(4):
            m = ln > k
            y[m] += c * val[k, :n][m] * x[col[k, :n][m]]
        return y
    b = d * (1.0 + 5e-3 * rng.standard_normal(n)) if case == "rise" else rng.standard_normal(n)
    t = lambda a: torch.tensor(a, device=dev)
    x, r = np.zeros(n), b.copy()
    p, g, ratio = np.zeros(n), 1.0, []
    for it in range(1, 5):
        g1 = r @ (r / d)
        p = r / d + (g1 / g if it > 1 else 0.0) * p
        q = A(p)
        a = g1 / (p @ q)
        x, r, g = x + a * p, r - a * q, g1
        ratio.append((r @ (r / d)) / g)
        dx = torch.zeros(n, dtype=torch.float64, device=dev)
        with pytest.raises(SdcError) as e:
            B.pcg_solve(n, t(val), t(col), t(ln), ld, 4, t(kd), t(mass), t(np.zeros(n)), c, t(b),
                        dx, rtol=1e-150, maxit=it, stream=torch.cuda.current_stream(dev).cuda_stream)
        assert e.value.status == B.SDC_E_CG_NOCONV
        assert np.abs(dx.cpu().numpy() - x).max() <= RTOL * np.abs(x).max(), it
    assert ratio[0] > 2.0**11 if case == "rise" else max(ratio[:2]) < 2.0**-25


def test_repeated_sums_in_the_two_level_solves(torch_dev):
    """Every dof a block of its own: the coarse matrix is the operator, and gamma falls by
    2^4 and more an iteration."""
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import Context, default_options
    from workloads.emi import emi_tiny
    wl = emi_tiny("two_cells")
    lab = np.arange(wl.n, dtype=np.int32)
    r = oracle.System.from_mesh(wl.mesh).step_emi(wl, wl.u0, wl.w0, coarse=lab)
    assert r["status"] == 0
    for blocks in (0, 1, 3):
        ctx = Context.from_emi(wl, options=default_options(cg_max_blocks=blocks),
                               stream=torch.cuda.current_stream(dev).cuda_stream)
        ctx.set_coarse_blocks(lab)
        u = torch.tensor(wl.u0, dtype=torch.float64, device=dev)
        w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
        st = ctx.step(u, w, 0.0, wl.dt, wl.sweeps, wl.tol)
        ctx.close()
        for a, b in ((u, r["u"]), (w, r["w"])):
            assert np.abs(a.cpu().numpy() - b).max() <= RTOL * max(1.0, np.abs(b).max())
        for m in range(wl.M):
            assert st.cg_iters[0][m] <= 20 and abs(st.cg_iters[0][m] - r["stats"].cg_iters[m]) <= 2

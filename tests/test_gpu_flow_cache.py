"""The launch rule of the node solves on large irregular meshes: on both sides of its limits (what
an iteration reads again against the L2 cache, numberings whose columns are scattered) a step and
a stand-alone solve agree with the kernels with every vector in global memory, and with the
same problem in its other numbering.

Tolerance: that of the parity tests, 1e-10 relative in the max norm (all sides stop at rtol = 1e-10).
"""

import numpy as np
import pytest

from workloads.configs import AP_BENCH, Workload
from workloads.meshes import Mesh, kuhn3d

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


def _mesh(nx, scattered):
    """A cube, thirteen off-diagonals a row with the full tensor below; scattered: numbered at
    random.  Returns the mesh and the new number of each of its nodes."""
    m = kuhn3d(nx, nx, nx, 0.2)
    perm = np.arange(m.n_nodes)
    if scattered:
        perm = np.random.default_rng(nx).permutation(m.n_nodes)
        xyz = np.empty_like(m.xyz)
        xyz[perm] = m.xyz
        m = Mesh(3, xyz, perm[m.elems].astype(np.int32))
    return m, perm


def _workload(nx, scattered):
    m, perm = _mesh(nx, scattered)
    f = np.array([0.6, 0.64, 0.48])
    r = np.linalg.norm(m.xyz, axis=1)
    return Workload("cube", m, 0.25 * np.eye(3) + 0.75 * np.outer(f, f), dict(AP_BENCH), M=2,
                    dt=0.05, sweeps=2, tol=1e-6, steps=1, v0=np.clip(1.5 - r / 3.0, 0.0, 1.0),
                    w0=np.zeros(m.n_nodes)), perm


def _step(wl, torch, dev, **opts):
    from paper_2311_07206_gb300 import Context, default_options
    ctx = Context.from_workload(wl, options=default_options(**opts),
                                stream=torch.cuda.current_stream(dev).cuda_stream)
    v = torch.tensor(wl.v0, dtype=torch.float64, device=dev)
    w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    st = ctx.step(v, w, 0.0, wl.dt, wl.sweeps, wl.tol)
    m = ctx.matrix()
    ctx.close()
    return v.cpu().numpy(), w.cpu().numpy(), st, m


@pytest.mark.parametrize("nx,scattered", [
    (60, False), (60, True),     # 216,000 rows: on chip; scattered, in the pipelined arrangement
    (74, True), (76, True),      # 405,224 and 438,976: on either side of the limit
    (76, False), (80, False),    # the same in order, and 512,000
])
def test_steps_on_both_sides(torch_dev, nx, scattered):
    torch, dev = torch_dev
    wl, _ = _workload(nx, scattered)
    v, w, st, _ = _step(wl, torch, dev)
    assert 0 < st.n_active[1] < wl.n
    for opts in ({"cg_variant": 1}, {"cg_pipelined": 1}, {"cg_variant": 2}):
        a, b, s, _ = _step(wl, torch, dev, **opts)
        assert np.abs(v - a).max() <= RTOL and np.abs(w - b).max() <= RTOL
        assert list(s.n_active) == list(st.n_active)
        for k in range(wl.sweeps):
            for m in range(wl.M):
                assert abs(s.cg_iters[k][m] - st.cg_iters[k][m]) <= 1


@pytest.mark.parametrize("nx", [78, 80])     # 474,552 and 512,000 rows: the rule asks from 500k on
def test_stand_alone_solves_in_both_numberings(torch_dev, nx):
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import binding
    x = []
    for scattered in (False, True):
        wl, perm = _workload(nx, scattered)
        _, _, _, (rp, ci, val, mass) = _step(wl, torch, dev)
        n = wl.n
        rows = np.repeat(np.arange(n), np.diff(rp))
        off = ci != rows
        kd = np.zeros(n)
        kd[rows[~off]] = val[~off]
        r, c, a = rows[off], ci[off], val[off]
        ln = np.bincount(r, minlength=n).astype(np.int32)
        slot = np.arange(len(r)) - (np.cumsum(ln) - ln)[r]
        ld, width = (n + 31) // 32 * 32, int(ln.max())
        ev, ec = np.zeros((width, ld)), np.zeros((width, ld), np.int32)
        ev[slot, r], ec[slot, r] = a, c
        b = np.empty(n)
        b[perm] = np.random.default_rng(2).standard_normal(n) * mass[perm]
        t = lambda q: torch.tensor(q, device=dev)
        out = torch.zeros(n, dtype=torch.float64, device=dev)
        it, rr = binding.pcg_solve(n, t(ev), t(ec), t(ln), ld, width, t(kd), t(mass),
                                   t(np.full(n, 0.5)), 0.05, t(b), out, rtol=1e-12, maxit=500,
                                   stream=torch.cuda.current_stream(dev).cuda_stream)
        assert 5 < it < 200 and rr <= 1e-12
        x.append(out.cpu().numpy()[perm])
    assert np.abs(x[0] - x[1]).max() <= RTOL * np.abs(x[0]).max()

"""The autotuner times no value that leaves every launch as it is: where all node solves run in the
scaled form on chip, the block sizes and row limits of the other kernels keep their settings."""

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_dev():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_07206_gb300 import build as b
    b.build()
    return torch, torch.device("cuda:0")


@pytest.mark.parametrize("variant,scaled", [(0, 1), (1, 1), (0, 0)])
def test_only_launches_that_differ_are_timed(torch_dev, variant, scaled):
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import Context, default_options
    wl = W.w0_square()
    o = default_options(cg_variant=variant, cg_scaled=scaled)
    ctx = Context.from_workload(wl, options=o, stream=torch.cuda.current_stream(dev).cuda_stream)
    v = torch.tensor(wl.v0, dtype=torch.float64, device=dev)
    w = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    rep = ctx.autotune(v, w, 0.0, wl.dt, wl.sweeps, wl.tol, trial_steps=2)
    ctx.close()
    if variant == 0 and scaled == 1:
        if rep["cg_scaled"] == 1:
            # the start, cg_pipelined, cg_scaled, rows per block
            assert rep["trials"] == 1 + 2 + 2 + 4
            assert rep["smem_block"] == o.cg_smem_block_size
            assert rep["general_block"] == o.cg_block_size
            assert rep["cluster_rows"] == o.cg_cluster_rows and rep["big_rows"] == 300000
    else:
        assert rep["trials"] > 1 + 2 + 2 + 4

"""An adjoint call that finds too little device memory reports it, and the next one, with the
memory there, starts over: its results are those of a context that never met the shortage."""

import numpy as np
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


def test_adjoint_after_a_shortage(torch_dev):
    torch, dev = torch_dev
    from paper_2311_07206_gb300 import Context, SdcError, default_options
    from paper_2311_07206_gb300 import binding as B
    wl = W.w0_square(n=513)      # eight vectors of 6.3 MB
    v0 = torch.tensor(wl.v0, dtype=torch.float64, device=dev)
    w0 = torch.tensor(wl.w0, dtype=torch.float64, device=dev)
    lam = torch.ones_like(v0)
    out = []
    for short in (True, False):
        ctx = Context.from_workload(wl, options=default_options(),
                                    stream=torch.cuda.current_stream(dev).cuda_stream)
        tape = ctx.new_tape(2, dev)
        v, w = v0.clone(), w0.clone()
        ctx.step_taped(v, w, 0.0, wl.dt, 2, wl.tol, tape)
        g = [torch.zeros_like(v0) for _ in range(3)]
        run = lambda: ctx.adjoint(tape, v0, w0, wl.dt, lam, lam, g[0], g[1], grad_scale=g[2])
        if short:
            torch.cuda.synchronize(dev)
            torch.cuda.empty_cache()
            fill, chunk = [], torch.cuda.mem_get_info(dev)[0]
            while chunk >= 1 << 21:      # all but about 24 MB, in as many pieces as it takes
                chunk = min(chunk, torch.cuda.mem_get_info(dev)[0] - (24 << 20))
                try:
                    if chunk >= 1 << 21:
                        fill.append(torch.empty(chunk, dtype=torch.uint8, device=dev))
                except torch.cuda.OutOfMemoryError:
                    chunk //= 2
            with pytest.raises(SdcError) as e:
                run()
            assert e.value.status == B.SDC_E_NOMEM
            del fill
            torch.cuda.empty_cache()
        run()
        torch.cuda.synchronize(dev)
        out.append([x.cpu().numpy() for x in g])
        ctx.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)

"""recip and quot (csrc/device_common.cuh), which take the place of the FP64 division in the node
solves' scalars, the update and the adjoint, against the exact quotient: random operands of both
signs, the neighbourhood of the binades' edges, and both sides of the limits beyond which they
divide.

Bound: 0.5 ulp for the last rounding and 2^-4 for the cut of the series (see the comment at the
functions), 0.5625 ulp, checked as 0.57 with the error from an exact residual.
"""

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

KERNEL = r"""
#include "device_common.cuh"
namespace {
__global__ void k(int n, const double* a, const double* b, double* q, double* rq, double* r,
                  double* rr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = sdc::quot(a[i], b[i]);
    rq[i] = fma(-q[i], b[i], a[i]);
    r[i] = sdc::recip(b[i]);
    rr[i] = fma(-r[i], b[i], 1.0);
}
}
extern "C" int run(int n, const double* a, const double* b, double* q, double* rq, double* r,
                   double* rr) {
    k<<<(n + 255) / 256, 256>>>(n, a, b, q, rq, r, rr);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_07206_gb300 import build as b
    d = tmp_path_factory.mktemp("quotient")
    (d / "k.cu").write_text(KERNEL)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", str(d / "k.so"),
                    str(d / "k.cu")], check=True)
    lib = C.CDLL(str(d / "k.so"))

    def call(a, b_):
        x = [torch.tensor(v, dtype=torch.float64, device="cuda:0") for v in (a, b_)]
        o = [torch.empty_like(x[0]) for _ in range(4)]
        torch.cuda.synchronize()
        assert lib.run(len(a), *[C.c_void_p(t.data_ptr()) for t in x + o]) == 0
        return [t.cpu().numpy() for t in o]
    return call


def _significands(rng, n):
    """Random ones, and a third at the edges of the binade."""
    s = 1.0 + rng.integers(0, 1 << 52, n) * 2.0 ** -52
    k = rng.integers(0, 64, n) * 2.0 ** -52
    edge = rng.integers(0, 6, n)
    return np.where(edge == 0, 1.0 + k, np.where(edge == 1, 2.0 - 2.0 ** -52 - k, s))


def test_within_the_stated_bound(run):
    rng = np.random.default_rng(11)
    n = 1 << 21
    b = np.ldexp(_significands(rng, n), rng.integers(-300, 301, n)) * rng.choice([-1.0, 1.0], n)
    a = np.ldexp(_significands(rng, n), rng.integers(-300, 301, n)) * rng.choice([-1.0, 1.0], n)
    q, rq, r, rr = run(a, b)
    assert np.abs(rq / b / np.spacing(np.abs(q))).max() <= 0.57
    assert np.abs(rr / b / np.spacing(np.abs(r))).max() <= 0.57
    # and next to the division's result
    assert (np.abs(q - a / b) <= np.spacing(np.abs(q))).all()
    assert (np.abs(r - 1.0 / b) <= np.spacing(np.abs(r))).all()


def test_limits_and_special_values(run):
    """Beyond the limits: the division's bits.  At them: the bound, next to the division."""
    rng = np.random.default_rng(12)
    f = np.array([1, 199, 200, 201, 1023, 1845, 1846, 1847, 2046])
    fa, fb = [x.ravel() for x in np.meshgrid(f, f)]
    near = np.concatenate([np.arange(797, 804), -np.arange(797, 804)])
    fa, fb = np.concatenate([fa, 1023 + near // 2 + near % 2]), np.concatenate([fb, 1023 - near // 2])
    fa, fb = np.repeat(fa, 200), np.repeat(fb, 200)
    a = np.ldexp(_significands(rng, len(fa)), fa - 1023) * rng.choice([-1.0, 1.0], len(fa))
    b = np.ldexp(_significands(rng, len(fa)), fb - 1023)
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        q, _, r, _ = run(a, b)
        div = (np.minimum(fa, fb) < 200) | (np.maximum(fa, fb) > 1846) | (np.abs(fa - fb) > 800)
        assert np.array_equal(q[div], (a / b)[div])
        assert (np.abs(q - a / b)[~div] <= np.spacing(np.abs(q))[~div]).all()
        div = (fb < 200) | (fb > 1846)
        assert np.array_equal(r[div], (1.0 / b)[div])
        assert (np.abs(r - 1.0 / b)[~div] <= np.spacing(np.abs(r))[~div]).all()
    v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1.0, -3.0])
    a, b = [x.ravel() for x in np.meshgrid(v, v)]
    with np.errstate(all="ignore"):
        q, _, r, _ = run(a, b)
        for got, want in ((q, a / b), (r, 1.0 / b)):
            nan = np.isnan(want)
            assert np.array_equal(np.isnan(got), nan)
            assert np.array_equal(got[~nan], want[~nan])
            assert np.array_equal(np.signbit(got[~nan]), np.signbit(want[~nan]))

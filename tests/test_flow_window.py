"""The windows of the on-chip node solves' sums (csrc/cg_window.cuh), compiled for the host and
driven as the kernels drive them: partial sums to limbs, limbs added, total, decision, and the
repeat in the exact windows.  Every sum has to end after one repeat at most, with the integer
sum of the partials.

Tolerance: a partial is truncated below one unit, 2^(top - 1125); equal partials within 2^-32
of the largest lose nothing, and their total is the correctly rounded one (math.fsum).
"""

import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "cg_window.cuh"
using namespace sdc;

static int field(double v) { return flow_max((int)(flow_bits(v) >> 52) & 0x7ff, 1); }

static bool add(const double* v, long n, int top, double& tot) {
    long long s[4] = {0, 0, 0, 0};
    bool below = true, in;
    for (long k = 0; k < n; ++k) {
        int l[4];
        below = flow_limbs(v[k], top, l) && below;
        for (int m = 0; m < 4; ++m) s[m] += l[m];
    }
    tot = flow_value(s[0], s[1], s[2], s[3], top, in);
    return !below || !in;
}

static int largest(const double* v, long n) {
    int f = 1;
    for (long k = 0; k < n; ++k) f = flow_max(f, field(v[k]));
    return f;
}

// One sum of a solve: state as in flow_totals, the totals and the number of repeats.  first: the
// windows of the solve's start (the exact one, and a guess for delta); else those after a
// previous gamma of exponent field prev.  More than five repeats: -1.
extern "C" int solve_sum(const double* a, const double* b, long n, int first, int prev, int head,
                         int drop, double* g, double* d, int* repeats) {
    int ta, tb;
    if (first) {
        const int f = largest(a, n);
        if (f >= 2047) return 2;
        ta = flow_exact_top(f);
        tb = flow_guess_top(f);
    } else {
        ta = tb = flow_next_top(prev, head);
    }
    for (*repeats = 0; *repeats < 5; ++*repeats) {
        const bool xa = add(a, n, ta, *g), xb = add(b, n, tb, *d);
        const int st = flow_decide(xa || xb, *repeats > 0, first != 0, *g, *d, ta, head + drop, 0, 0,
                                   [] { return false; });
        if (st != 3) return st;
        const int fa = largest(a, n), fb = largest(b, n);
        if (fa >= 2047 || fb >= 2047) return 2;
        ta = flow_exact_top(fa);
        tb = flow_exact_top(fb);
    }
    return -1;
}

// The decision on a total alone: sqrt(g) <= thresh, with the kernels' band around thresh^2.
extern "C" int decide(double g, double d, int first, int topa, int fall, double thresh, int* asked) {
    const double q = thresh * thresh;
    const bool normal = q > 1e-280 && q < 1e280;
    const double lo = normal ? q * (1.0 - 0x1p-50) : 0.0, hi = normal ? q * (1.0 + 0x1p-50) : INFINITY;
    *asked = 0;
    return flow_decide(false, false, first != 0, g, d, topa, fall, (long long)flow_bits(lo),
                       (long long)flow_bits(hi), [&] {
                           *asked = 1;
                           return std::sqrt(g) <= thresh;
                       });
}

// The limb sums of v in the window `top`: the total before it is rounded.
extern "C" void limb_sums(const double* v, long n, int top, long long* s) {
    for (int m = 0; m < 4; ++m) s[m] = 0;
    for (long k = 0; k < n; ++k) {
        int l[4];
        flow_limbs(v[k], top, l);
        for (int m = 0; m < 4; ++m) s[m] += l[m];
    }
}

extern "C" void constants(int* c) {
    c[0] = kFlowHead;
    c[1] = kFlowDrop;
    c[2] = kCoarseHead;
    c[3] = kCoarseDrop;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("flow_window")
    src, so = d / "harness.cpp", d / "libharness.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2311_07206_gb300", "csrc"), "-o", str(so), str(src)],
                   check=True)
    return C.CDLL(str(so))


def _sum(lib, a, b, first=True, prev=0, coarse=False):
    c = (C.c_int * 4)()
    lib.constants(c)
    a = np.ascontiguousarray(a, dtype=np.float64)
    b = np.ascontiguousarray(b, dtype=np.float64)
    g, d, rep = C.c_double(), C.c_double(), C.c_int()
    p = lambda x: x.ctypes.data_as(C.c_void_p)
    st = lib.solve_sum(p(a), p(b), C.c_long(len(a)), int(first), prev, c[2 * coarse], c[2 * coarse + 1],
                       C.byref(g),
                       C.byref(d), C.byref(rep))
    return st, g.value, d.value, rep.value


@pytest.mark.parametrize("n", [155_648, 261_120])   # 152 CTAs of 1,024 threads; 255 of them
@pytest.mark.parametrize("first", [True, False])
def test_equal_partials_end(lib, n, first):
    """Uniform residuals: every amplitude of a binade, in the windows of a solve's start and
    after a gamma of a hundredth."""
    for x in np.concatenate([np.linspace(1.0, 2.0, 17)[:-1], [np.nextafter(2.0, 0.0)]]):
        for sign in (1.0, -1.0):
            a = np.full(n, x)
            prev = 1023 + int(math.log2(n * x / 100.0))
            st, g, d, rep = _sum(lib, a, sign * a, first, prev)
            assert st == 0 and rep <= 1, (x, sign, st, rep)
            assert g == math.fsum(a) and d == sign * g


def test_uniform_residual_of_the_slab(lib):
    """442,401 rows on 152 CTAs of 1,024 threads (2,912 rows a CTA): r = const, log-uniform
    amplitudes; delta is 1 % of gamma."""
    n, L, threads = 442_401, 2_912, 1_024
    rows = np.zeros(152 * threads)
    l = np.arange(n) % L
    chunk = l // 32
    wid = (chunk + 1) % 32
    np.add.at(rows, (np.arange(n) // L) * threads + wid * 32 + l % 32, 1.0)
    assert rows.sum() == n
    rng = np.random.default_rng(1)
    for amp in np.exp(rng.uniform(0.0, math.log(2.0), 24)):
        a = rows * (amp * amp)
        st, g, d, rep = _sum(lib, a, 0.01 * a)
        assert st == 0 and rep <= 1
        assert g == math.fsum(a) and d == math.fsum(0.01 * a)


@pytest.mark.parametrize("n", [1, 3, 1_000])
def test_top_of_the_range(lib, n):
    """Totals of 2^1022 to 2^1024: the finite ones are returned, the others end the solve as not
    finite; nothing is repeated for ever."""
    for e in (1021.0, 1022.0, 1022.9, 1023.0, 1023.5, 1023.99, 1024.0, 1025.0):
        x = 2.0 ** (e / 2.0) / n
        x = x * 2.0 ** (e / 2.0)
        if not math.isfinite(x):
            continue
        a = np.full(n, x)
        try:
            want = math.fsum(a)
        except OverflowError:
            want = math.inf
        for first in (True, False):
            st, g, _, rep = _sum(lib, a, a * 1e-3, first, 2046)
            assert rep <= 1
            assert st == (0 if math.isfinite(want) else 2), (e, first)
            if st == 0:
                assert g == want


def test_largest_total_and_non_finite_values(lib):
    """A total one unit below 2^103 units; delta far above its guessed window; infinities and
    NaN in either sum, also where the guessed window reaches the end of the range."""
    # 2^18 partials of 2^85 units less one: one chunk over the largest grid's 261,120 threads
    st, g, _, rep = _sum(lib, np.full(1 << 18, np.nextafter(2.0, 0.0)), np.zeros(1 << 18))
    assert (st, rep) == (0, 0) and g == math.fsum(np.full(1 << 18, np.nextafter(2.0, 0.0)))
    a = np.ones(64)
    st, _, d, rep = _sum(lib, a, a * 2.0 ** 40)
    assert (st, rep) == (0, 1) and d == 64 * 2.0 ** 40
    for bad in (np.inf, -np.inf, np.nan):
        for scale in (1.0, 2.0 ** 1015):
            b = a * scale
            b[5] = bad
            for first in (True, False):
                assert _sum(lib, a * scale, b, first, 1023)[0] == 2
                assert _sum(lib, b, a * scale, first, 1023)[0] == 2


def test_signed_partials(lib):
    """Cancelling partials against exact rationals: off by less than a unit each."""
    from fractions import Fraction
    rng = np.random.default_rng(3)
    a = rng.standard_normal(5_000) * np.exp(rng.uniform(-20, 0, 5_000))
    b = -a[::-1] + 1e-9 * rng.standard_normal(5_000)
    top = 1023 + int(math.floor(math.log2(np.abs(a).max()))) + 22
    for first, prev in ((True, 0), (False, 1023)):
        st, g, d, rep = _sum(lib, a, b, first, prev)
        assert rep <= 1
        for got, v in ((g, a), (d, b)):
            want = sum(Fraction(float(x)) for x in v)
            assert abs(Fraction(got) - want) <= len(v) * Fraction(2) ** (top - 1125) + abs(want) / 2 ** 53


def test_stopping_decision(lib):
    """Converged exactly where 0 <= g and sqrt(g) <= thresh: negative totals, zero, the bound and
    its neighbours, squares beyond the normal range; and a start at gamma = 0 only."""
    lib.decide.argtypes = [C.c_double, C.c_double, C.c_int, C.c_int, C.c_int, C.c_double, C.c_void_p]
    asked = C.c_int()

    def decide(g, thresh, first=False):
        return lib.decide(g, 1.0, int(first), 1, 10_000, thresh, C.addressof(asked))

    for thresh in (1e-10, 0.37, 3.0, 1e-150, 1e150):
        q = thresh * thresh
        gs = [0.0, q, q / 4, q * 4, 5e-324, 1e300]
        for k in (-2, -1, 1, 2):
            gs += [q * (1.0 + k * 2.0 ** -52), q * (1.0 + k * 2.0 ** -49)]
        for g in gs:
            assert decide(g, thresh) == (1 if math.sqrt(g) <= thresh else 0), (g, thresh)
            if g > 0.0:
                assert decide(-g, thresh) == 0, (-g, thresh)
    assert decide(0.0, 0.0) == 1 and decide(1e-300, 0.0) == 0
    for g in (-1.0, -1e-300, 1e-300, 1.0):
        assert decide(g, 1e10, first=True) == 0
    assert decide(0.0, 1e10, first=True) == 1
    assert decide(math.inf, 1.0) == 2 and decide(math.inf, 1.0, first=True) == 2


@pytest.mark.parametrize("coarse", [False, True])
def test_sums_after_a_fall_of_gamma(lib, coarse):
    """gamma 2^1 to 2^40 below the one its window came from, partials over ten orders of
    magnitude on the largest grid of each kernel.  Bound, before the total is rounded: a unit a
    partial, 2^17.3 2^(10 - 102 + 14) = 2^-60.7 of the total for one row a thread, 2^16.8
    2^(20 - 102 + 4) = 2^-61.2 for the two-level kernel; 2^-60."""
    n = 111_872 if coarse else 155_648
    rng = np.random.default_rng(5)
    c = (C.c_int * 4)()
    lib.constants(c)
    for fall in (1, 3, 4, 5, 9, 13, 14, 15, 20, 21, 22, 23, 40):
        a = np.exp(rng.uniform(-23.0, 0.0, n))
        exact = sum(int(math.ldexp(x, 120)) for x in a)
        prev = 1023 + int(math.floor(math.log2(exact))) - 120 + fall
        st, g, d, rep = _sum(lib, a, -a, False, prev, coarse)
        assert st == 0 and rep <= 1 and d == -g
        assert abs(g - math.fsum(a)) <= np.spacing(g)
        top = prev + c[2 * coarse] if rep == 0 else int(np.frexp(a.max())[1]) + 1022 + 18
        limbs = (C.c_longlong * 4)()
        lib.limb_sums(a.ctypes.data_as(C.c_void_p), C.c_long(n), top, limbs)
        got = sum(x << (26 * k) for k, x in enumerate(limbs)) << (top - 1125 + 120)
        assert 0 <= exact - got and (exact - got) << 60 <= exact, (fall, rep)

// Fixed-point windows of the flow kernels' sums (cg_flow.cuh), and what a total leads to.
// Integer arithmetic on bit patterns and a few exact FP64 operations, so that a host compiler
// gives the same results as the device: tests/test_flow_window.py compiles this file.
#pragma once

#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#define SDC_HD __host__ __device__ __forceinline__
#define SDC_HD_COLD __host__ __device__ __noinline__
#else
#define SDC_HD inline
#define SDC_HD_COLD inline
#endif

namespace sdc {
namespace {

typedef unsigned long long u64;

constexpr int kFlowHead = 10;    // growth of gamma over one iteration that fits the window
constexpr int kFlowSumHead = 18; // total over largest partial sum: at most 2^18 partials (155,648
                                 // threads of a launch, 255 CTAs of 1,024), each below 2^85 units
                                 // of a window this far above the largest, so below 2^103
constexpr int kFlowGuessHead = 22; // first delta over gamma's largest partial: |w.r| of a thread
                                   // <= |A| gamma, gamma <= 2^18 largest partials
// Fall of gamma up to which its window serves.  2^17.3 partials truncated at 2^(head - 102) of the
// gamma before it are off by 2^-74.7, and 2^-60.7 of a gamma 2^14 below it: less than the
// partials' own rounding leaves in gamma, and in delta (2^-53 gamma over the root of the terms).
// Slabs, squares and shells fall by 2^2 to 2^6 an iteration; no case took longer than with 2^22.
constexpr int kFlowDrop = 14;
// The same for the two-level solves' gamma = r.u, a sum of terms that cancel against each other
// within a block: more room above, and a repeat for smaller falls (131k rows: no time, and the
// same bits as with 24 and 8).
constexpr int kCoarseHead = 20, kCoarseDrop = 4;

SDC_HD u64 flow_bits(double v) {
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(v);
#else
    u64 b;
    std::memcpy(&b, &v, sizeof b);
    return b;
#endif
}
SDC_HD double flow_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double v;
    std::memcpy(&v, &b, sizeof v);
    return v;
#endif
}
SDC_HD int flow_min(int a, int b) { return a < b ? a : b; }
SDC_HD int flow_max(int a, int b) { return a > b ? a : b; }

// v against a window whose largest exponent field is `top`: |v| = sum_k l[k] 2^(26 k) units
// of 2^(top - 1125), truncated; false when v lies above the window.
SDC_HD bool flow_limbs(double v, int top, int (&l)[4]) {
    const u64 bits = flow_bits(v);
    const int f = (int)(bits >> 52) & 0x7ff;
    const u64 mant = (bits & 0xfffffffffffffull) | (f > 0 ? (1ull << 52) : 0ull);
    const int sh = flow_min(flow_max(f, 1) - top + 50, 50);
    const u64 lo = sh >= 0 ? mant << sh : mant >> flow_min(-sh, 63);
    const u64 hi = sh > 0 ? mant >> (64 - sh) : 0ull;
    const int s = (int)((long long)bits >> 63);   // 0 or -1
    constexpr unsigned m = (1u << 26) - 1u;
    l[0] = ((int)((unsigned)lo & m) ^ s) - s;
    l[1] = ((int)((unsigned)(lo >> 26) & m) ^ s) - s;
    l[2] = ((int)((unsigned)((lo >> 52) | (hi << 12)) & m) ^ s) - s;
    l[3] = ((int)(unsigned)(hi >> 14) ^ s) - s;
    return f <= top;
}

// (out of line: none of its long sequence is to be executed speculatively)
SDC_HD_COLD double flow_ldexp(double v, int e) { return ldexp(v, e); }

// Total of a value's four limb sums in units of 2^(top - 1125), rounded once: the digits are
// carried into A 2^52 + B with -2^51 <= A < 2^51 and 0 <= B < 2^52, which integer additions place
// in the significands of 1.5 2^52 + A and 2^52 + B.  in: false when the total lies outside that
// range, [-2^103, 2^103) units.
SDC_HD double flow_value(long long s0, long long s1, long long s2, long long s3, int top, bool& in) {
    constexpr long long m = (1ll << 26) - 1;
    s1 += s0 >> 26;
    s2 += s1 >> 26;
    s3 += s2 >> 26;
    in = s3 < (1ll << 25) && s3 >= -(1ll << 25);
    const double a = flow_double(0x4338000000000000ll + (s3 * (1ll << 26) + (s2 & m)));
    const double b = flow_double(0x4330000000000000ll + (((s1 & m) << 26) + (s0 & m)));
    const double v = fma(a - 0x1.8p52, 0x1p52, b - 0x1p52);
    // times 2^(top - 1125), in the exponent field where the result is normal
    const long long w = (long long)flow_bits(v);
    const int f = (int)(w >> 52) & 0x7ff, g = f + top - 1125;
    if (f == 0) return 0.0;
    if (g >= 1 && g <= 2046) return flow_double(w + (long long)((u64)(long long)(top - 1125) << 52));
    return flow_ldexp(v, top - 1125);
}

// Tops of the windows.  After a total of exponent field f: room for its growth; a value that is
// not finite must lie above the window, hence the cap.  From the largest field f of the partial
// sums, none of them infinite or NaN: room for the total, with no cap, so that a total near
// the end of the range is summed like any other (and overflows when it is rounded).  guess: from
// the largest field of other values than those summed.
SDC_HD int flow_next_top(int f, int head) { return flow_min(f + head, 2046); }
SDC_HD int flow_exact_top(int f) { return f + kFlowSumHead; }
SDC_HD int flow_guess_top(int f) { return flow_min(f + kFlowGuessHead, 2046); }

// What the totals g (of gamma) and d (of delta) lead to: 0 go on, 1 converged, 2 not finite,
// 3 repeat the sum in the windows of the partial sums' exact exponents.  above: a partial sum or
// a total lies above its window.  A sum is repeated once at most: in the exact windows nothing
// finite lies above.  first: no bound on gamma yet, and no window to fall below.
// close(): sqrt(g) against its bound, where g lies between lo and hi (bit patterns: an FP64
// comparison has 65 cycles latency).  A negative g, which rounding or an indefinite coarse matrix
// can give r.u, is no convergence.
template <class C>
SDC_HD int flow_decide(bool above, bool repeated, bool first, double g, double d, int topa,
                       int fall, long long lo, long long hi, C&& close) {
    if (above) return repeated ? 2 : 3;
    const long long gb = (long long)flow_bits(g);
    const int fg = (int)(gb >> 52) & 0x7ff, fd = (int)(flow_bits(d) >> 52) & 0x7ff;
    if (flow_max(fg, fd) == 0x7ff) return 2;
    if (first) {
        if (gb == 0) return 1;
    } else if (gb >= 0 && gb < hi) {
        if (gb <= lo || close()) return 1;
    }
    if (!repeated && !first && flow_max(fg, 1) < topa - fall) return 3;
    return 0;
}

}  // namespace
}  // namespace sdc

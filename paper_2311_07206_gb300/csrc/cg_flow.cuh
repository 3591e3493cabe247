// Node solves with every vector on chip and no grid barrier in the iteration.
//
// The solves of a step are bound by FP64 issue where a CTA owns many rows and by the
// latency of the iteration's synchronisation chain where it owns few.  Three things
// replace the barrier, the per-block records and their two passes of the other kernels:
//
// 1. Neighbour values travel with their version.  A row's published value and a tag
//    (launch id, iteration) are one 16-byte word, stored and loaded as a single relaxed
//    128-bit access; a consumer re-reads the few words that are not there yet.  No fence
//    and no barrier separate the update from the next product, and the columns a CTA
//    owns itself are read from its shared memory.
// 2. The two dot products are summed in place.  Against an exponent window known from the
//    previous iteration's total a value becomes four signed 26-bit limbs: a warp adds
//    limbs with the integer warp reduction, a CTA adds the warps' limbs, and eight lanes
//    add the CTA's limbs to eight 64-bit words with one relaxed reduction.  A word's top
//    byte counts the arrivals, so the poll that finds all of them has the sum in hand:
//    one store-and-poll round trip for barrier and sum together.  Two sets of words
//    alternate and are never reset: a CTA knows the previous total of a set and takes the
//    difference.  Measured for 152 CTAs: 1,510 cycles for the exchange of eight words,
//    against 2,900 for the release/acquire barrier alone and 8,500 for barrier, block sums
//    and totals of 152 records.
// 3. p and x, which nothing waits for, are updated after the sums are posted.
//
// Integer addition is exact, so a total does not depend on the order of the arrivals, and
// every CTA reads the same total.  The window holds 103 bits from kFlowHead bits above
// the previous gamma down; a partial sum above it, or a total more than kFlowDrop bits
// below the previous one, repeats the exchange once with the exact largest exponents (the
// start of a solve finds its window the same way).  The windows: cg_window.cuh.
#pragma once

#include "cg_window.cuh"
#include "device_common.cuh"

namespace sdc {
namespace {

// A published word: value, tag (12 bits of launch, 20 of iteration; the host clears the words
// when the launch count wraps), 32 spare bits.  Stored and loaded as one relaxed
// single-copy-atomic 128-bit access.  The iteration may wrap: every word is overwritten two
// iterations later, so the only stale one is that of k - 2.
__device__ __forceinline__ unsigned flow_tag(unsigned id, unsigned k) { return id | (k & 0xfffffu); }
__device__ __forceinline__ void pub_store(ulonglong2* p, double v, unsigned tag) {
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p),
                 "l"((u64)__double_as_longlong(v)), "l"((u64)tag)
                 : "memory");
}
__device__ __forceinline__ void pub_load(const ulonglong2* p, u64& v, unsigned& tag) {
    u64 t;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=l"(v), "=l"(t)
                 : "l"(p)
                 : "memory");
    tag = (unsigned)t;
}
// Value of column j: from the CTA's shared memory (32-bit shared address `own` of local row 0)
// when l = j - r0 < nl, else the published word; tag is left alone in the first case.
__device__ __forceinline__ void flow_fetch(unsigned l, unsigned nl, unsigned own, const ulonglong2* p,
                                           u64& v, unsigned& tag) {
    if (l < nl) {
        asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(own + 8u * l) : "memory");
    } else {
        unsigned __int128 w;
        asm volatile("ld.relaxed.gpu.global.b128 %0, [%1];" : "=q"(w) : "l"(p) : "memory");
        v = (u64)w;
        tag = (unsigned)(w >> 64);
    }
}
__device__ __forceinline__ unsigned smem_addr(const double* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ u64 ld_relaxed64(const u64* p) {
    u64 v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ld_relaxed64x2(const u64* p, u64& a, u64& b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void red_add64(u64* p, u64 v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// What warp 0 carries from sum to sum.
struct FlowScalars {
    u64 prev[2][8];           // each set's words before the running sum
    double g, den;            // gamma and gamma / alpha of the last sum
    double inv_g, inv_a;      // 1 / gamma and 1 / alpha of it (0 before the first)
    double thresh, lo, hi;    // stopping test: bound on sqrt(gamma) and a band around its square
    double gamma0, energy;
    int nsum;
};

// Shared state of one CTA.
struct FlowShared {
    alignas(16) int lim[32][8];   // limb sums of each warp: 4 of a, 4 of b
    FlowScalars z;
    double alpha, beta;
    int topa, topb;               // window tops (largest exponent field) of the next sums
    int ovf, ok, state;           // state: 0 go on, 1 converged, 2 non-finite, 3 repeat the sum
    int next;                     // next chunk of rows of the product
    int fmax[64];
};

// Post the CTA's sums of a and b to the words acc[0..7]: every thread calls it; it holds
// one CTA barrier, after which warp 0 adds the warps' limbs and posts them.  A warp without
// rows (warp 0 of a CTA with one row per thread) leaves its zeros of flow_scalars_init.
__device__ __forceinline__ void flow_post(double a, double b, bool rows, FlowShared& S, u64* acc) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (rows) {
        int la[4], lb[4];
        bool in = flow_limbs(a, S.topa, la);
        in = flow_limbs(b, S.topb, lb) && in;
        const bool out = __any_sync(0xffffffffu, !in);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            la[k] = __reduce_add_sync(0xffffffffu, la[k]);
            lb[k] = __reduce_add_sync(0xffffffffu, lb[k]);
        }
        if (lane == 0) {
            *reinterpret_cast<int4*>(&S.lim[wid][0]) = make_int4(la[0], la[1], la[2], la[3]);
            *reinterpret_cast<int4*>(&S.lim[wid][4]) = make_int4(lb[0], lb[1], lb[2], lb[3]);
            if (out) S.ovf = 1;
        }
    }
    __syncthreads();
    if (wid == 0) {
        // lane: limb lane & 7 of warps lane >> 3, + 4, ...; every load before the first add
        const int out0 = S.ovf;
        long long s = S.lim[lane >> 3][lane & 7];   // (rows of warps beyond the block: zero)
        if (nw > 4) {
            int x[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) x[k] = S.lim[(lane >> 3) + 4 * k + 4][lane & 7];
#pragma unroll
            for (int k = 0; k < 7; ++k) s += x[k];
        }
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        // top byte: arrivals; next byte: CTAs with a value above the window
        if (lane < 8) red_add64(acc + lane, (1ull << 56) + ((u64)(out0 != 0) << 48) + (u64)s);
    }
}

// The rare ends of the paths below, kept out of line so that none of their long sequences is
// executed speculatively.
__device__ __noinline__ bool flow_sqrt_at_most(double g, double thresh) { return sqrt(g) <= thresh; }

__device__ __forceinline__ void flow_scalars_init(FlowShared& S) {
    FlowScalars& Z = S.z;
    for (int k = threadIdx.x; k < 256; k += blockDim.x) S.lim[k >> 3][k & 7] = 0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) Z.prev[0][k] = Z.prev[1][k] = 0;
        Z.g = Z.den = 1.0;
        Z.inv_g = Z.inv_a = 0.0;
        Z.thresh = Z.lo = Z.hi = 0.0;
        Z.gamma0 = Z.energy = 0.0;
        Z.nsum = 0;
    }
}

// Warp 0: wait for the sums posted to set `set`, derive alpha and beta (cg_scalars'
// recurrences, den_t = delta_t - beta_t gamma_t / alpha_{t-1}) and the next windows.
// redo: the sum is repeated, in windows from the exact exponents.
// HEAD, DROP: kFlowHead and kFlowDrop.  arrived() runs once the wait is over.
template <int HEAD, int DROP, class A>
__device__ __forceinline__ void flow_totals(FlowShared& S, const u64* acc, int set, int G, bool redo,
                                            long long budget, int* err, A&& arrived) {
    const int lane = threadIdx.x & 31;
    FlowScalars& Z = S.z;
    const double inv_g = Z.inv_g, inv_a = Z.inv_a;
    const long long lo = __double_as_longlong(Z.lo), hi = __double_as_longlong(Z.hi);
    const int nsum = Z.nsum, topa = S.topa, topb = S.topb;
    // lane 0 reads gamma's words, lane 1 delta's: a word with all its arrivals is final
    u64 v[4], d[4];
    u64* const prev = Z.prev[set] + 4 * (lane & 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        d[k] = (1ull << 47) - prev[k];
        v[k] = 0;
    }
    const long long t0 = clock64();
    int ok = 1;
    while (true) {
        bool here = true;
        if (lane < 2) {
            ld_relaxed64x2(acc + 4 * lane, v[0], v[1]);
            ld_relaxed64x2(acc + 4 * lane + 2, v[2], v[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) here = here && ((v[k] + d[k]) >> 56) == (u64)G;
        }
        if (__all_sync(0xffffffffu, here)) break;
        // (a vote: the lanes read different clocks, and must leave the loop together)
        if (__any_sync(0xffffffffu, clock64() - t0 > budget)) {
            ok = 0;
            break;
        }
    }
    if (!ok && lane == 0) {
        raise_error(err, SDC_E_TIMEOUT);
        S.ok = 0;
    }
    arrived();
    if (!ok) return;
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] += v[k];
    bool in;
    const double tot = flow_value((long long)(d[0] & 0xffffffffffffull) - (1ll << 47),
                                  (long long)(d[1] & 0xffffffffffffull) - (1ll << 47),
                                  (long long)(d[2] & 0xffffffffffffull) - (1ll << 47),
                                  (long long)(d[3] & 0xffffffffffffull) - (1ll << 47),
                                  lane ? topb : topa, in);
    const bool above = __any_sync(0xffffffffu, lane < 2 && (!in || ((d[0] >> 48) & 0xff) != 0));
    const double g = __shfl_sync(0xffffffffu, tot, 0), dl = __shfl_sync(0xffffffffu, tot, 1);
    const int fg = xs_field(g);
    const int state = flow_decide(above, redo, nsum == 0, g, dl, topa, HEAD + DROP, lo, hi,
                                  [&] { return flow_sqrt_at_most(g, Z.thresh); });
    const double beta = g * inv_g;
    const double den = fma(-beta, g * inv_a, dl);
    const double alpha = quot(g, den);
    // (a non-finite alpha shows in the next sums, whose exact exponents end the solve)
    if (lane == 0) {
        S.state = state;
        S.ovf = 0;
        if (state != 3) Z.g = g;
        if (state == 0) {
            S.alpha = alpha;
            S.beta = beta;
            Z.den = den;
            S.topa = S.topb = flow_next_top(fg, HEAD);
        }
    }
    if (lane < 2) {
#pragma unroll
        for (int k = 0; k < 4; ++k) prev[k] = v[k];
    }
}

// Once, after the first sum's scalars are out: sqrt(gamma) <= rtol sqrt(gamma_0) is decided by
// comparing gamma with a band of 2^-50 around the squared bound and by the square root
// itself inside it.  Squares that leave the normal range always take the square root.
__device__ __noinline__ void flow_first_bound(FlowScalars& Z, double g, double rtol) {
    const double thresh = rtol * sqrt(g), q = thresh * thresh;
    const bool normal = q > 1e-280 && q < 1e280;
    if ((threadIdx.x & 31) == 0) {
        Z.gamma0 = g;
        Z.thresh = thresh;
        Z.lo = normal ? q * (1.0 - 0x1p-50) : 0.0;
        Z.hi = normal ? q * (1.0 + 0x1p-50) : INFINITY;
    }
}

// Warp 0, off the critical path (the other warps are at the update): what the next sum needs.
__device__ __forceinline__ void flow_next(FlowShared& S, double rtol) {
    const int lane = threadIdx.x & 31;
    FlowScalars& Z = S.z;
    const double g = Z.g, den = Z.den;
    const double q = quot(lane == 0 ? 1.0 : den, g);   // lane 0: 1 / gamma, lane 1: 1 / alpha
    const double e = fma(S.alpha, g, Z.energy);             // x' A x = sum of alpha_t gamma_t
    const int nsum = Z.nsum;
    __syncwarp();
    if (lane == 0) {
        Z.inv_g = q;
        Z.energy = e;
        Z.nsum = nsum + 1;
    }
    if (lane == 1) Z.inv_a = q;
    if (nsum == 0) flow_first_bound(Z, g, rtol);
    __syncwarp();
}

// Windows from the exact largest exponents of the CTAs' partial sums, with a release /
// acquire grid barrier that also publishes every global write before it.  emax words hold
// (generation << 32) | field and only grow.  guess: b is not what the next sum adds as delta
// (the first of a solve), see kFlowGuessHead.  Returns false after a timeout.
__device__ __forceinline__ bool flow_window(double a, double b, FlowShared& S, u64* emax,
                                            unsigned* bar, int G, unsigned& epoch, unsigned gen,
                                            bool guess, long long budget, int* err) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int fa = __reduce_max_sync(0xffffffffu, xs_field(a));
    const int fb = __reduce_max_sync(0xffffffffu, xs_field(b));
    if (lane == 0) {
        S.fmax[wid] = fa;
        S.fmax[32 + wid] = fb;
    }
    __syncthreads();
    epoch += G;
    if (wid == 0) {
        const int ma = __reduce_max_sync(0xffffffffu, lane < nw ? S.fmax[lane] : 1);
        const int mb = __reduce_max_sync(0xffffffffu, lane < nw ? S.fmax[32 + lane] : 1);
        if (lane == 0) {
            atomicMax(emax, ((u64)gen << 32) | (unsigned)ma);
            atomicMax(emax + 1, ((u64)gen << 32) | (unsigned)mb);
            S.ok = barrier_arrive_wait(bar, epoch, budget, err);
            const int ga = (int)(unsigned)ld_relaxed64(emax), gb = (int)(unsigned)ld_relaxed64(emax + 1);
            S.state = ga >= 2047 || gb >= 2047 ? 2 : 0;
            S.topa = flow_exact_top(ga);
            S.topb = guess ? flow_guess_top(gb) : flow_exact_top(gb);
            S.ovf = 0;
        }
    }
    __syncthreads();
    return S.ok != 0;
}

// Off-diagonal product of a row: acc + sum_k v[k vs] x(c[k ld]) over its len slots, in order.
// Columns of this CTA (rows [r0, r0 + nl)) come from shared memory (own), the others from their
// published words, fetched again until they carry `tag` (slots past the row's end fetch row r0:
// with nl = 0 the caller passes a row of its own, whose word is there).  All loads of CH slots are issued
// before the first is used.  The product of a CTA with many rows is bound by instruction
// issue, not by FP64 or latency (two padded slots more per row: 442k rows 13.5 -> 15.2 us per
// iteration), so a slot is kept to a dozen instructions.
template <int CH, bool NC = true>
__device__ __forceinline__ double flow_row_dot(double acc, int len, const int* __restrict__ c, int ld,
                                               const double* v, int vs, int ncol, int r0, int nl,
                                               unsigned own, const ulonglong2* pub, unsigned tag,
                                               int site, FlowShared& S, long long budget, int* err) {
    for (int k0 = 0; k0 < len; k0 += CH) {
        int j[CH];
        double a[CH];
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            j[k] = r0;
            if (k0 + k < len) {
                const int* const q = c + (size_t)k * ld;
                j[k] = sdc_idx(NC ? __ldg(q) : *q, ncol, site);
                a[k] = v[(size_t)k * vs];
            }
        }
        c += (size_t)CH * ld;
        v += (size_t)CH * vs;
        u64 x[CH];
        long long t0 = 0;
        while (true) {
            unsigned bad = 0;
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                unsigned g = tag;
                flow_fetch((unsigned)(j[k] - r0), (unsigned)nl, own, pub + j[k], x[k], g);
                bad |= g ^ tag;
            }
            if (!bad) break;
            if (t0 == 0) t0 = clock64();
            if (clock64() - t0 > budget) {
                raise_error(err, SDC_E_TIMEOUT);
                S.ok = 0;
            }
            if (!*(volatile int*)&S.ok) break;   // a wait of the CTA has run out
        }
#pragma unroll
        for (int k = 0; k < CH; ++k)
            if (k0 + k < len) acc += a[k] * __longlong_as_double((long long)x[k]);
    }
    return acc;
}

// f(l) for the thread's local rows: 32-row chunks over the warps, warp 0 last (a CTA with one
// row per thread leaves it none); the passes that feed the sums use this order.
template <class F>
__device__ __forceinline__ void flow_rows(int nl, F&& f) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = wid == 0 ? nw - 1 : wid - 1; 32 * c < nl; c += nw) {
        const int l = 32 * c + lane;
        if (l < nl) f(l);
    }
}

// The same over the warps but warp 0: p and x, while warp 0 sees to the sums.
template <class F>
__device__ __forceinline__ void flow_rows_px(int nl, F&& f) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (wid == 0) return;
    for (int c = wid - 1; 32 * c < nl; c += nw - 1) {
        const int l = 32 * c + lane;
        if (l < nl) f(l);
    }
}

template <int MAXT>
struct FlowChunk {
    static constexpr int value = MAXT > 768 ? 3 : MAXT > 512 ? 4 : 7;
};

// First phase of a solve on the CTA's rows: s = diag^-1/2, r = s b (and zero vectors), both
// published plainly, then a grid barrier that also finds the first windows, then the scaled
// off-diagonals c s_i a_ij s_j (slot k of local row l at vb[k vs + l]) and
// w = (I + c S K_off S) r.  f(l, r) receives a row's r,
// g(l, w) its w; gamma and delta partial sums in ga, de.  Returns false to leave the kernel.
template <int CH, class F, class H>
__device__ __forceinline__ bool flow_start(const CgParams& P, const FlowParams& Q, FlowShared& S,
                                           int r0, int nl, unsigned short* plen, double* vb, int vs,
                                           unsigned& epoch,
                                           double& ga, double& de, F&& f, H&& h) {
    const int t = threadIdx.x, G = Q.G, ld = P.ld;
    const double c = P.c;
    ga = de = 0.0;
    if (t == 0) {
        S.ok = 1;
        S.ovf = 0;
        S.next = 0;
    }
    if (Q.zero && Q.bidx == 0)
        for (int k = t; k < kFlowWords; k += blockDim.x) Q.zero[k] = 0;
    flow_rows(nl, [&](int l) {
        const int i = r0 + l;
        const double d = P.mc[i] * (1.0 + c * P.J[i]) + c * P.kdc[i];
        double si = 0.0;
        if (!isfinite(d)) raise_error(P.err, SDC_E_NONFINITE);
        else if (!(d > 0.0)) raise_error(P.err, SDC_E_DOMAIN);
        else si = rsqrt(d);
        P.sv[i] = si;
        const double r = si * P.b[i];
        P.u[i] = r;
        ga += r * r;
        f(l, r);
    });
    if (P.inject_fault && Q.bidx == G - 1) {
        // leave without arriving: every other CTA's bounded wait runs out
        if (G == 1 && t == 0) raise_error(P.err, SDC_E_TIMEOUT);
        return false;
    }
    if (!flow_window(ga, ga, S, Q.emax, Q.bar, G, epoch, 1u, true, P.budget, P.err)) return false;
    if (S.state == 2) {
        if (Q.bidx == 0 && t == 0) raise_error(P.err, SDC_E_NONFINITE);
        return false;
    }
    flow_rows(nl, [&](int l) {
        const int i = r0 + l;
        const int len = __ldg(P.alen + i);
        plen[l] = (unsigned short)len;
        const double csi = c * __ldcg(P.sv + i);
        const double ri = __ldcg(P.u + i);
        double acc = ri;
        for (int k0 = 0; k0 < len; k0 += CH) {
            int j[CH];
            double av[CH], sj[CH], uj[CH];
#pragma unroll
            for (int k = 0; k < CH; ++k)
                if (k0 + k < len) {
                    const size_t q = (size_t)(k0 + k) * ld + i;
                    j[k] = sdc_idx(__ldg(P.acol + q), P.n, 44);
                    av[k] = __ldg(P.aval + q);
                }
#pragma unroll
            for (int k = 0; k < CH; ++k)
                if (k0 + k < len) {
                    sj[k] = __ldcg(P.sv + j[k]);
                    uj[k] = __ldcg(P.u + j[k]);
                }
#pragma unroll
            for (int k = 0; k < CH; ++k)
                if (k0 + k < len) {
                    const double a = csi * av[k] * sj[k];
                    vb[(size_t)(k0 + k) * vs + l] = a;
                    acc += a * uj[k];
                }
        }
        h(l, acc);
        de += acc * ri;
    });
    return true;
}

// End of a solve: statistics, x = S x~ on the CTA's rows and the LU-trick coupling, whose
// neighbours' x travel as tagged words.  xt(l): the CTA's x~.
template <int CH, class X>
__device__ __forceinline__ void flow_finish(const CgParams& P, const FlowParams& Q, FlowShared& S,
                                            int r0, int nl, int it, X&& xt) {
    const int ld = P.ld;
    const bool lead = Q.bidx == 0 && threadIdx.x == 0;
    if (S.state == 2) {
        if (lead) raise_error(P.err, SDC_E_NONFINITE);
        return;
    }
    if (lead) {
        *Q.iters_out = it;
        *Q.relres_out = S.z.gamma0 > 0.0 ? sqrt(fabs(S.z.g) / S.z.gamma0) : 0.0;
        if (P.energy_out) *P.energy_out = S.z.energy;
    }
    // the words of iteration it - 1, whose readers are done: their CTAs posted sum `it`
    ulonglong2* const pub = Q.pub + (size_t)((it + 1) & 1) * ld;
    const unsigned tag = flow_tag(Q.id, it + 2u);
    const bool couple = P.epi_lo < P.epi_hi;
    flow_rows(nl, [&](int l) {
        const int i = r0 + l;
        const double x = __ldcg(P.sv + i) * xt(l);
        P.x[i] = x;
        if (couple) pub_store(pub + i, x, tag);
    });
    if (!couple) return;
    flow_rows(nl, [&](int l) {
        const int i = r0 + l;
        const int len = __ldg(P.alen + i);
        const double kx = flow_row_dot<CH>(
            0.0, len, P.acol + i, ld, P.aval + i, ld, P.n, i, 0, 0u, pub, tag, 47, S, P.budget, P.err);
        cg_couple_row(P, i, P.x[i], kx);
    });
}

// ---- pipelined arrangement (see pcg_group), scaled form ------------------------------
// Per iteration: update of z, s, w, r and the two dot products (w published); sums posted;
// p, x (r_old is kept in the other of two r buffers until then); the product
// n = (I + c S K_off S) w on every warp but warp 0, which waits for the sums and derives the
// scalars.  The product's 32-row chunks beyond the first per warp are handed out by a
// counter, so warp 0 takes what is left when it joins.
// Bound by the chain post (1,000 cycles) - poll (1,300-1,900) - scalars (1,200-1,700) - update
// (900-1,800); the product runs beside it.  us per iteration, before (barrier and records, or a
// cluster for up to 10,000 rows) and now: 4,225 rows 4.7 / 2.8, 11.8k 5.2 / 2.8, 58k 6.2 / 3.9,
// 89k 7.5 / 5.1.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_pcg_flow(CgParams P, FlowParams Q) {
    extern __shared__ double sm[];
    __shared__ FlowShared S;
    constexpr int CH = FlowChunk<MAXT>::value;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5;
    const int G = gridDim.x, L = P.L, ld = P.ld;
    Q.G = G;
    Q.bidx = blockIdx.x;
    const int r0 = blockIdx.x * L;
    const int nl = max(0, min(P.n - r0, L));
    const int nch = (nl + 31) >> 5;
    double* rc = sm;             // r, and the r before it
    double* ro = sm + L;
    double* const sw = sm + 2 * L;
    double* const sp = sm + 3 * L;
    double* const ss = sm + 4 * L;
    double* const sz = sm + 5 * L;
    double* const sn = sm + 6 * L;
    double* const xs = Q.x_smem ? sm + 7 * L : P.x + r0;
    // scaled off-diagonals: behind the vectors, or in global memory
    unsigned short* const plen =
        reinterpret_cast<unsigned short*>(sm + (size_t)(7 + Q.x_smem) * L);   // row lengths
    double* const vb = Q.v_smem ? sm + (size_t)(7 + Q.x_smem) * L + L / 4 : P.sval + r0;
    const int vs = Q.v_smem ? L : ld;
    const bool has_rows = wid != 0 || nw <= nch;   // (warps beyond the rows add zeros)
    unsigned epoch = 0, gen = 1;
    double ga, de, alpha = 0.0, beta = 0.0;
    flow_scalars_init(S);
    if (!flow_start<CH>(
            P, Q, S, r0, nl, plen, vb, vs, epoch, ga, de,
            [&](int l, double r) {
                rc[l] = r;
                sp[l] = ss[l] = sz[l] = 0.0;
                xs[l] = 0.0;
            },
            [&](int l, double w) {
                sw[l] = w;
                pub_store(Q.pub + r0 + l, w, Q.id + 1);
            }))
        return;
    int it = 0;
    unsigned npub = 0;
    bool redo = false;
    auto update_px = [&]() {
        flow_rows_px(nl, [&](int l) {
            const double p = ro[l] + beta * sp[l];
            sp[l] = p;
            xs[l] += alpha * p;
        });
    };
    while (true) {
        u64* const acc = Q.acc + 8 * (npub & 1);
        flow_post(ga, de, has_rows, S, acc);
        if (wid == 0)
            flow_totals<kFlowHead, kFlowDrop>(S, acc, npub & 1, G, redo, P.budget, P.err, [] {});
        ++npub;
        if (!redo) {
            if (it > 0) update_px();
            const unsigned tag = flow_tag(Q.id, it + 1u);
            const ulonglong2* const pub = Q.pub + (size_t)(it & 1) * ld;
            int c = wid - 1;
            while (true) {
                if (c < 0) {
                    if (lane == 0) c = atomicAdd(&S.next, 1) + nw - 1;
                    c = __shfl_sync(0xffffffffu, c, 0);
                }
                if (c >= nch) break;
                const int l = 32 * c + lane;
                if (l < nl) {
                    const int i = r0 + l;
                    sn[l] = flow_row_dot<CH>(
                        sw[l], plen[l], P.acol + i, ld, vb + l, vs, P.n, r0, nl, smem_addr(sw), pub, tag,
                        42, S, P.budget, P.err);
                }
                c = -1;
                __syncwarp();
            }
        }
        __syncthreads();
        // (read together: one after the other they cost three shared-memory latencies)
        alpha = S.alpha;
        beta = S.beta;
        if (S.ok - 1 | S.state) {
            if (!S.ok) return;
            if (S.state == 3) {
                if (!flow_window(ga, de, S, Q.emax, Q.bar, G, epoch, ++gen, false, P.budget, P.err))
                    return;
                if (S.state == 0) {
                    redo = true;
                    continue;
                }
            }
            break;
        }
        redo = false;
        if (it >= P.maxit) {
            if (blockIdx.x == 0 && t == 0) raise_error(P.err, SDC_E_CG_NOCONV);
            break;
        }
        ++it;
        if (t == 0) S.next = 0;
        if (wid == 0) flow_next(S, P.rtol);
        const unsigned tag = flow_tag(Q.id, it + 1u);
        ulonglong2* const pub = Q.pub + (size_t)(it & 1) * ld + r0;
        ga = de = 0.0;
        flow_rows(nl, [&](int l) {
            const double w0 = sw[l];
            const double z = sn[l] + beta * sz[l];
            const double s = w0 + beta * ss[l];
            const double w = w0 - alpha * z;
            const double r = rc[l] - alpha * s;
            pub_store(pub + l, w, tag);
            sw[l] = w;
            ro[l] = r;
            sz[l] = z;
            ss[l] = s;
            ga += r * r;
            de += w * r;
        });
        double* const q = rc;
        rc = ro;
        ro = q;
    }
    flow_finish<CH>(P, Q, S, r0, nl, it, [&](int l) { return xs[l]; });
}

// ---- classical arrangement (see pcgc_group), scaled form -----------------------------
// Per iteration: update of s and r (r published), the product w = (I + c S K_off S) r and the
// dot products, the sums posted, and while they are summed p and x.  r_new goes into w's
// place, which s has used up; with three buffers (nbuf = 3) the next w goes into a third, so
// that r_old is still there for p after the product; with two, p and x come before it.
// One group of Q.G CTAs (the launch, or one instance of a batched launch); this CTA, number
// Q.bidx of it, owns rows [r0, r0 + nl), at most P.L.
// Many rows a CTA: bound by FP64 issue (442k rows, 27,400 cycles an iteration: product 15,000 of
// which 11,300 are FP64, update 3,750 of which 2,800, the sums' chain 6,000 with p and x beside
// it); few: by the chain exchange (1,200) - product - post - poll (1,700) - scalars (1,100).
// us per iteration, before and now: 442k 18.3 / 13.2, 813k 30 / 23.5; cell-by-cell 7.7k 6.9 / 2.9,
// 53k 8.7 / 4.1.
template <int CH>
__device__ __forceinline__ void cgc_flow(const CgParams& P, const FlowParams& Q, FlowShared& S, double* sm,
                                         int r0, int nl) {
    const int t = threadIdx.x, wid = t >> 5, nw = blockDim.x >> 5;
    const int G = Q.G, L = P.L, ld = P.ld;
    const int nch = (nl + 31) >> 5;
    const bool late = Q.nbuf == 3;
    double* rb = sm;
    double* wb = sm + L;
    double* const sp = sm + 2 * L;
    double* const ss = sm + 3 * L;
    double* fb = late ? sm + 4 * L : rb;
    double* const xs = Q.x_smem ? sm + 5 * L : P.x + r0;
    unsigned short* const plen =
        reinterpret_cast<unsigned short*>(sm + (size_t)(2 + Q.nbuf + Q.x_smem) * L);
    double* const vb = Q.v_smem ? sm + (size_t)(2 + Q.nbuf + Q.x_smem) * L + L / 4 : P.sval + r0;
    const int vs = Q.v_smem ? L : ld;
    const bool has_rows = wid != 0 || nw <= nch;
    unsigned epoch = 0, gen = 1;
    double ga, de, alpha = 0.0, beta = 0.0;
    flow_scalars_init(S);
    if (!flow_start<CH>(
            P, Q, S, r0, nl, plen, vb, vs, epoch, ga, de,
            [&](int l, double r) {
                rb[l] = r;
                sp[l] = ss[l] = 0.0;
                xs[l] = 0.0;
            },
            [&](int l, double w) { wb[l] = w; }))
        return;
    int it = 0;
    unsigned npub = 0;
    bool redo = false;
    auto px_row = [&](const double* r, int l) {
        const double p = r[l] + beta * sp[l];
        sp[l] = p;
        xs[l] += alpha * p;
    };
    while (true) {
        u64* const acc = Q.acc + 8 * (npub & 1);
        flow_post(ga, de, has_rows, S, acc);
        if (wid == 0)
            flow_totals<kFlowHead, kFlowDrop>(S, acc, npub & 1, G, redo, P.budget, P.err, [] {});
        ++npub;
        if (late && it > 0 && !redo) flow_rows_px(nl, [&](int l) { px_row(fb, l); });
        __syncthreads();
        // (read together: one after the other they cost three shared-memory latencies)
        alpha = S.alpha;
        beta = S.beta;
        if (S.ok - 1 | S.state) {
            if (!S.ok) return;
            if (S.state == 3) {
                if (!flow_window(ga, de, S, Q.emax, Q.bar, G, epoch, ++gen, false, P.budget, P.err))
                    return;
                if (S.state == 0) {
                    redo = true;
                    continue;
                }
            }
            break;
        }
        redo = false;
        if (it >= P.maxit) {
            if (Q.bidx == 0 && t == 0) raise_error(P.err, SDC_E_CG_NOCONV);
            break;
        }
        ++it;
        const unsigned tag = flow_tag(Q.id, it + 1u);
        ulonglong2* const pub = Q.pub + (size_t)(it & 1) * ld;
        flow_rows(nl, [&](int l) {
            const double s = wb[l] + beta * ss[l];
            const double r = rb[l] - alpha * s;
            pub_store(pub + r0 + l, r, tag);
            wb[l] = r;
            ss[l] = s;
        });
        __syncthreads();
        if (wid == 0) flow_next(S, P.rtol);
        // (the thread that writes the row's product over r_old)
        if (!late) flow_rows(nl, [&](int l) { px_row(rb, l); });
        ga = de = 0.0;
        const unsigned own = smem_addr(wb);
        flow_rows(nl, [&](int l) {
            const int i = r0 + l;
            const double r = wb[l];
            const double w = flow_row_dot<CH>(
                r, plen[l], P.acol + i, ld, vb + l, vs, P.n, r0, nl, own, pub, tag, 46, S, P.budget,
                P.err);
            fb[l] = w;
            ga += r * r;
            de += w * r;
        });
        // r <- w's place, w <- the product's, and r_old's is free (two buffers: the same one)
        double* const q = rb;
        rb = wb;
        wb = fb;
        fb = late ? q : rb;
    }
    flow_finish<CH>(P, Q, S, r0, nl, it, [&](int l) { return xs[l]; });
}

template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_cgc_flow(CgParams P, FlowParams Q) {
    extern __shared__ double sm[];
    __shared__ FlowShared S;
    Q.G = gridDim.x;
    Q.bidx = blockIdx.x;
    const int r0 = blockIdx.x * P.L;
    cgc_flow<FlowChunk<MAXT>::value>(P, Q, S, sm, r0, max(0, min(P.n - r0, P.L)));
}

// Batched form: the blocks of an instance are a group with its own sums, barrier and
// iteration count.  Several CTAs share an SM, so that one works while another waits (32
// instances of 20k rows: 5,277 -> 2,493 us per step against the grid-barrier kernel with vectors
// in global memory).  Bound by FP64 issue.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1024 / MAXT)
    k_cgc_flow_batch(CgParams P, FlowParams Q, const SegBlock* __restrict__ tab,
                     int* __restrict__ seg_iters, double* __restrict__ seg_relres) {
    extern __shared__ double sm[];
    __shared__ FlowShared S;
    const SegBlock g = tab[blockIdx.x];
    if (g.nblk == 0) return;   // no group: a planned launch's spare block
    Q.G = g.nblk;
    Q.bidx = (int)blockIdx.x - g.blk0;
    Q.acc += (size_t)g.seg * kFlowWords;
    Q.emax = Q.acc + 16;
    Q.bar = reinterpret_cast<unsigned*>(Q.acc + 32);
    Q.iters_out = seg_iters + g.seg;
    Q.relres_out = seg_relres + g.seg;
    const int Lg = ((g.row1 - g.row0 + g.nblk - 1) / g.nblk + 31) & ~31;
    const int r0 = g.row0 + Q.bidx * Lg;
    cgc_flow<4>(P, Q, S, sm, r0, max(0, min(g.row1 - r0, Lg)));
}

// ---- classical arrangement with the two-level preconditioner --------------------------
// u = r + Y y, y = E^-1 t, t = Y' r, in place of u = r (see k_pcgcs_coarse, whose recurrences for
// t and Y' s this kernel shares: Y' s <- Y' w + beta Y' s, t <- t - alpha Y' s).  The rows are the
// positions of the block order: CTA b owns positions [b L, b L + L), cut at the block boundaries
// into pieces; columns are translated to positions once per solve.  (Carrying y by the same
// recurrences, which would take E^-1 off the critical path, stalls: the rounding of E^-1 Y' w
// is not small against y once the residual has fallen by the condition of E.)
// A piece's sum of Y w is exact: every warp adds its rows of a piece as limbs in a window
// known from the piece's largest term of the iteration before, one warp adds the warps' limbs
// (terms outside the window: that warp adds the rows again, from their largest exponent); the sum travels to
// the other CTAs as a tagged word.  Per iteration: t; y of the own pieces' blocks, s, r; u
// (published); the product, the dot products and the pieces' limbs; while the dot products are
// summed the pieces' sums, p, x and the words of all pieces.
// Before (k_pcgcs_coarse, two grid barriers and vectors in global memory): 16.0 us per
// iteration on 131k rows.
struct CoarseFlowParams {
    int q, qn, ptot, npmax;   // blocks, blocks with active rows, pieces, most pieces of a CTA
    const int* crow;          // [n] compact row of each position
    const int* ipos;          // [n] position of each compact row
    int* pcol;                // [width][ld] columns as positions, in position order
    const int* tp;            // [G + 1] first piece of each CTA
    const int* piece;         // [3 ptot]: block, first and end position
    const int* blk_ptr;       // [q + 1] pieces of each block
    const int* nzb;           // [qn] the blocks with active rows, ascending
    const double* Einv;       // [q][q]
    ulonglong2* words;        // [2][pstride] published piece sums
    int pstride;
    int width;                // (matrix rows on chip) slots of a row
};

// A piece's window: room of the sum over its largest term, growth of the largest term since
// the last sum, and its fall up to which the window keeps 57 bits of it.
constexpr int kPieceHead = 16, kPieceGrow = 10, kPieceFall = 20;

__host__ __device__ inline size_t coarse_flow_smem(int L, int vectors, int qn, int ptot, int npmax) {
    return (size_t)vectors * L * 8 + (size_t)(3 * qn + ptot + npmax) * 8 +
           (size_t)((L + 31) / 32 + npmax) * 16 + 16 + (size_t)(2 * qn + 1 + 5 * npmax) * 4 +
           (size_t)L * 4;
}
// columns and values of a CTA's rows
__host__ __device__ inline size_t coarse_flow_matrix(int L, int width) {
    return 8 + (size_t)L * width * 12;
}

__device__ __forceinline__ void flow_bar_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void flow_bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_cgc2_flow(CgParams P, FlowParams Q, CoarseFlowParams C) {
    extern __shared__ __align__(16) double sm[];
    __shared__ FlowShared S;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5, B = blockDim.x;
    const int G = gridDim.x, L = P.L, ld = P.ld;
    const int r0 = blockIdx.x * L;
    const int nl = max(0, min(P.n - r0, L));
    const int nch = (nl + 31) >> 5;
    const double c = P.c;
    const bool late = Q.nbuf == 3;
    double* ub = sm;
    double* wb = sm + L;
    double* const sr = sm + 2 * L;
    double* const sp = sm + 3 * L;
    double* const ss = sm + 4 * L;
    double* const sy = sm + 5 * L;
    double* ob = late ? sm + 6 * L : nullptr;   // u_old, until p has it
    const int nv = (late ? 7 : 6) + Q.x_smem;
    double* const sx = sm + (size_t)(nv - 1) * L;          // (x_smem)
    double* const tw = sm + (size_t)nv * L;                // [qn] Y' w of the blocks with rows
    double* const ts = tw + C.qn;                          // [qn] Y' s
    double* const tr = ts + C.qn;                          // [qn] t = Y' r
    double* const stp = tr + C.qn;                         // [ptot] the pieces' sums
    double* const ysh = stp + C.ptot;                      // [npmax] y of the own pieces
    int4* const recs = reinterpret_cast<int4*>(
        (reinterpret_cast<uintptr_t>(ysh + C.npmax) + 15) & ~(uintptr_t)15);   // [nch + npmax] limbs
    int* const snz = reinterpret_cast<int*>(recs + (L + 31) / 32 + C.npmax);   // [qn]
    int* const sbp = snz + C.qn;                           // [qn + 1]
    int* const pbeg = sbp + C.qn + 1;                      // [npmax] own pieces: local range, block,
    int* const pend = pbeg + C.npmax;
    int* const pblk = pend + C.npmax;
    int* const ptop = pblk + C.npmax;                      // window, largest exponent of the terms
    int* const pmax = ptop + C.npmax;
    unsigned short* const pid = reinterpret_cast<unsigned short*>(pmax + C.npmax);   // [L]
    unsigned short* const plen = pid + L;                                            // [L]
    const bool has_rows = wid != 0 || nw <= nch;
    const int e0 = C.tp[blockIdx.x], np = C.tp[blockIdx.x + 1] - e0;
    // the CTA's matrix rows, on chip as well where there is room (see coarse_flow_fit)
    double* const sv = reinterpret_cast<double*>(
        (reinterpret_cast<uintptr_t>(plen + L) + 7) & ~(uintptr_t)7);   // [width][L]
    double* const vb = Q.v_smem ? sv : P.sval + r0;
    int* const cb = Q.v_smem ? reinterpret_cast<int*>(sv + (size_t)C.width * L) : C.pcol + r0;
    const int ms = Q.v_smem ? L : ld;
    unsigned epoch = 0, gen = 0;
    flow_scalars_init(S);
    if (t == 0) {
        S.ok = 1;
        S.ovf = 0;
    }
    if (Q.zero && blockIdx.x == 0)
        for (int k = t; k < kFlowWords; k += B) Q.zero[k] = 0;
    for (int m = t; m < C.qn; m += B) {
        const int a = sdc_idx(C.nzb[m], C.q, 73);
        snz[m] = a;
        sbp[m] = C.blk_ptr[a];
    }
    if (t == 0) sbp[C.qn] = C.blk_ptr[C.q];
    for (int a = t; a < np; a += B) {
        const int e = sdc_idx(e0 + a, C.ptot, 74);
        pblk[a] = sdc_idx(C.piece[3 * e], C.q, 75);
        pbeg[a] = C.piece[3 * e + 1] - r0;
        pend[a] = C.piece[3 * e + 2] - r0;
        ptop[a] = 0;         // no window yet: every term lies above it
        pmax[a] = 0;
    }
    __syncthreads();
    for (int l = t; l < nl; l += B) {
        int lo = 0, hi = np - 1;      // the piece that holds position l
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (pend[mid] > l) hi = mid; else lo = mid + 1;
        }
        pid[l] = (unsigned short)lo;
    }
    double* const xs = Q.x_smem ? sx : nullptr;
    auto row_of = [&](int l) { return sdc_idx(C.crow[r0 + l], P.n, 70); };
    flow_rows(nl, [&](int l) {
        const int i = row_of(l);
        const double d = P.mc[i] * (1.0 + c * P.J[i]) + c * P.kdc[i];
        double si = 0.0;
        if (!isfinite(d)) raise_error(P.err, SDC_E_NONFINITE);
        else if (!(d > 0.0)) raise_error(P.err, SDC_E_DOMAIN);
        else si = rsqrt(d);
        P.sv[r0 + l] = si;
        sy[l] = d * si;
        sr[l] = si * P.b[i];
        sp[l] = ss[l] = 0.0;
        plen[l] = (unsigned short)P.alen[i];
        if (xs) xs[l] = 0.0; else P.x[i] = 0.0;
    });
    __syncthreads();
    // a warp's limbs of v over the pieces of chunk k (every lane of the warp calls it)
    auto piece_limbs = [&](int k, double v) {
        const int l = 32 * k + lane;
        const int a0 = pid[32 * k], a1 = pid[min(32 * k + 31, nl - 1)];
        const int mine = l < nl ? (int)pid[l] : -1;
        for (int a = a0; a <= a1; ++a) {
            int q[4];
            const double x = mine == a ? v : 0.0;
            const int top = ptop[a];
            flow_limbs(x, top, q);
            const int f = __reduce_max_sync(0xffffffffu, xs_field(x));
#pragma unroll
            for (int m = 0; m < 4; ++m) q[m] = __reduce_add_sync(0xffffffffu, q[m]);
            if (lane == 0) {
                recs[a + k] = make_int4(q[0], q[1], q[2], q[3]);
                atomicMax(&pmax[a], f);
            }
        }
    };
    // sum of a lane's 64-bit limbs over the warp (each below 2^46)
    auto warp_value = [&](const long long (&x)[4], int top) {
        long long r[4];
#pragma unroll
        for (int m = 0; m < 4; ++m)
            r[m] = ((long long)__reduce_add_sync(0xffffffffu, (int)(x[m] >> 20)) << 20) +
                   __reduce_add_sync(0xffffffffu, (int)(x[m] & 0xfffff));
        bool in;
        return flow_value(r[0], r[1], r[2], r[3], top, in);
    };
    // warps 1..: the own pieces' sums, published with `tag`; term(l): the rows' values
    auto piece_post = [&](ulonglong2* out, unsigned tag, auto&& term) {
        if (wid == 0) return;
        for (int a = wid - 1; a < np; a += nw - 1) {
            long long x[4] = {0, 0, 0, 0};
            const int f = pmax[a], d = ptop[a] - kPieceHead - f;
            int top = ptop[a];
            if (d < 0 || d > kPieceGrow + kPieceFall) {
                top = f + kPieceHead;
                for (int l = pbeg[a] + lane; l < pend[a]; l += 32) {
                    int q[4];
                    flow_limbs(term(l), top, q);
#pragma unroll
                    for (int m = 0; m < 4; ++m) x[m] += q[m];
                }
            } else {
                for (int k = (pbeg[a] >> 5) + lane; k <= (pend[a] - 1) >> 5; k += 32) {
                    const int4 q = recs[a + k];
                    x[0] += q.x;
                    x[1] += q.y;
                    x[2] += q.z;
                    x[3] += q.w;
                }
            }
            const double v = warp_value(x, top);
            if (lane == 0) {
                pub_store(out + e0 + a, v, tag);
                pmax[a] = 0;
                ptop[a] = f + kPieceGrow + kPieceHead;
            }
        }
    };
    // warps 1..: every piece's sum, then Y' w of the blocks with active rows
    auto coarse_in = [&](const ulonglong2* in, unsigned tag) {
        const long long t0 = clock64();
        for (int e = t - 32; e < C.ptot; e += B - 32) {
            u64 v = 0;
            unsigned g = ~tag;
            while (true) {
                pub_load(in + e, v, g);
                if (g == tag) break;
                if (clock64() - t0 > P.budget) {
                    raise_error(P.err, SDC_E_TIMEOUT);
                    S.ok = 0;
                }
                if (!*(volatile int*)&S.ok) break;
            }
            stp[e] = __longlong_as_double((long long)v);
        }
        flow_bar_sync(3, B - 32);
        for (int m = t - 32; m < C.qn; m += B - 32) {
            double a = 0.0;
            for (int e = sbp[m]; e < sbp[m + 1]; ++e) a += stp[e];
            tw[m] = a;
        }
    };
    // y = E^-1 t of the own pieces' blocks, a warp per piece
    auto coarse_y = [&]() {
        for (int a = nw - 1 - wid; a < np; a += nw) {
            const double* row = C.Einv + (size_t)pblk[a] * C.q;
            double pa = 0.0;
            for (int m = lane; m < C.qn; m += 32) pa += __ldg(row + snz[m]) * tr[m];
            const int top = __reduce_max_sync(0xffffffffu, xs_field(pa)) + kPieceHead;
            int q[4];
            flow_limbs(pa, top, q);
            const long long x[4] = {q[0], q[1], q[2], q[3]};
            const double v = warp_value(x, top);
            if (lane == 0) ysh[a] = v;
        }
    };
    // t = Y' r of the initial residual
    for (int k = wid == 0 ? nw - 1 : wid - 1; k < nch; k += nw) {
        const int l = 32 * k + lane;
        piece_limbs(k, l < nl ? sy[l] * sr[l] : 0.0);
    }
    if (!group_barrier(Q.bar, G, epoch, P.budget, P.err, &S.ok)) return;   // diag^-1/2 is out
    piece_post(C.words, Q.id + 1, [&](int l) { return sy[l] * sr[l]; });
    flow_rows(nl, [&](int l) {
        const int i = row_of(l);
        const double csi = c * P.sv[r0 + l];
        const int len = plen[l];
        for (int k = 0; k < len; ++k) {
            const size_t e = (size_t)k * ld;
            const int j = sdc_idx(C.ipos[sdc_idx(P.acol[e + i], P.n, 71)], P.n, 72);
            cb[(size_t)k * ms + l] = j;
            vb[(size_t)k * ms + l] = csi * P.aval[e + i] * __ldcg(P.sv + j);
        }
    });
    if (wid != 0) coarse_in(C.words, Q.id + 1);
    __syncthreads();
    if (!S.ok) return;
    for (int m = t; m < C.qn; m += B) {
        tr[m] = tw[m];
        ts[m] = 0.0;
    }
    __syncthreads();
    coarse_y();
    __syncthreads();
    flow_rows(nl, [&](int l) {
        const double u = sr[l] + sy[l] * ysh[pid[l]];
        ub[l] = u;
        pub_store(Q.pub + r0 + l, u, Q.id + 1);
    });
    __syncthreads();
    int it = 0;
    unsigned npub = 0;
    bool redo = false;
    double ga, de, alpha = 0.0, beta = 0.0;
    auto px_row = [&](const double* u, int l) {
        const double p = u[l] + beta * sp[l];
        sp[l] = p;
        if (xs) xs[l] += alpha * p; else P.x[row_of(l)] += alpha * p;
    };
    while (true) {
        const unsigned wtag = flow_tag(Q.id, it + 2u);
        ulonglong2* const words = C.words + (size_t)((it + 1) & 1) * C.pstride;
        if (!redo) {
            // w = (I + c S K_off S) u, r.u, w.u, Y' w
            const unsigned tag = flow_tag(Q.id, it + 1u);
            const ulonglong2* const pub = Q.pub + (size_t)(it & 1) * ld;
            ga = de = 0.0;
            for (int k = wid == 0 ? nw - 1 : wid - 1; k < nch; k += nw) {
                const int l = 32 * k + lane;
                double v = 0.0;
                if (l < nl) {
                    const double u = ub[l];
                    const double w = flow_row_dot<FlowChunk<MAXT>::value, false>(
                        u, plen[l], cb + l, ms, vb + l, ms, P.n, r0, nl, smem_addr(ub), pub,
                        tag, 76, S, P.budget, P.err);
                    wb[l] = w;
                    ga += sr[l] * u;
                    de += w * u;
                    v = sy[l] * w;
                }
                __syncwarp();
                piece_limbs(k, v);
            }
            if (it == 0) {
                // the windows of the first sums, from the exact exponents
                if (!flow_window(ga, de, S, Q.emax, Q.bar, G, epoch, ++gen, false, P.budget, P.err))
                    return;
                if (S.state == 2) break;
            }
        }
        u64* const acc = Q.acc + 8 * (npub & 1);
        flow_post(ga, de, has_rows, S, acc);
        if (wid == 0) {
            flow_totals<kCoarseHead, kCoarseDrop>(S, acc, npub & 1, G, redo, P.budget, P.err,
                                                  [&] { flow_bar_arrive(2, B); });
        } else {
            if (!redo) {
                piece_post(words, wtag, [&](int l) { return sy[l] * wb[l]; });
                if (late && it > 0) flow_rows_px(nl, [&](int l) { px_row(ob, l); });
            }
            // the words of all pieces follow close on the sums
            flow_bar_sync(2, B);
            if (!redo) coarse_in(words, wtag);
        }
        ++npub;
        __syncthreads();
        alpha = S.alpha;
        beta = S.beta;
        if (S.ok - 1 | S.state) {
            if (!S.ok) return;
            if (S.state == 3) {
                if (!flow_window(ga, de, S, Q.emax, Q.bar, G, epoch, ++gen, false, P.budget, P.err))
                    return;
                if (S.state == 0) {
                    redo = true;
                    continue;
                }
            }
            break;
        }
        redo = false;
        if (it >= P.maxit) {
            if (blockIdx.x == 0 && t == 0) raise_error(P.err, SDC_E_CG_NOCONV);
            break;
        }
        ++it;
        for (int m = B - 1 - t; m < C.qn; m += B) {
            const double sa = tw[m] + beta * ts[m];
            ts[m] = sa;
            tr[m] -= alpha * sa;
        }
        __syncthreads();
        coarse_y();
        flow_rows(nl, [&](int l) {
            const double s = wb[l] + beta * ss[l];
            ss[l] = s;
            sr[l] -= alpha * s;
        });
        __syncthreads();
        const unsigned utag = flow_tag(Q.id, it + 1u);
        ulonglong2* const pub = Q.pub + (size_t)(it & 1) * ld + r0;
        flow_rows(nl, [&](int l) {
            const double u = sr[l] + sy[l] * ysh[pid[l]];
            wb[l] = u;
            pub_store(pub + l, u, utag);
        });
        __syncthreads();
        // (after the barrier: in front of it the other warps waited for its 400 cycles)
        if (wid == 0) flow_next(S, P.rtol);
        if (!late) flow_rows(nl, [&](int l) { px_row(ub, l); });
        // u <- w's place; the next w goes into the third buffer (two: u_old's place)
        double* const o = ub;
        ub = wb;
        wb = late ? ob : o;
        if (late) ob = o;
    }
    if (S.state == 2) {
        if (blockIdx.x == 0 && t == 0) raise_error(P.err, SDC_E_NONFINITE);
        return;
    }
    if (blockIdx.x == 0 && t == 0) {
        *Q.iters_out = it;
        *Q.relres_out = S.z.gamma0 > 0.0 ? sqrt(fabs(S.z.g) / S.z.gamma0) : 0.0;
        if (P.energy_out) *P.energy_out = S.z.energy;
    }
    flow_rows(nl, [&](int l) {
        const int i = row_of(l);
        P.x[i] = P.sv[r0 + l] * (xs ? xs[l] : P.x[i]);
    });
}

}  // namespace
}  // namespace sdc

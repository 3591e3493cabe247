// Discrete adjoint of one adaptive SDC step (Sec. 3.2 eq. final-sdc, Sec. 4.2)
// with the active sets of the forward step held fixed (recorded on a tape).
//
// The forward step is a composition of differentiable maps once the index
// sets I_k are fixed and every node solve is read as the exact solution of its
// linear system.  The reverse pass visits the sweeps k = K-1 .. 0 and, inside a
// sweep, the forward operations backwards:
//   w sweep          pointwise reverse of the LU-trick recursion for w
//   v update         V' = V + dv on I_k: the adjoint passes through
//   node solves      m = M-1 .. 0: A_m bbar_m = dvbar_m (A_m symmetric: the same
//                    restricted Jacobi-PCG), then the coupling into earlier
//                    nodes dvbar_j -= dt Qhat_mj (K bbar_m + mass J_j bbar_m)
//   residual         rbar_m = bbar_m; fbar_j = dt sum_m Q_mj rbar_m; vbar0 +=
//                    mass sum_m rbar_m; Vbar_j -= K fbar_j (full rows: dropped
//                    neighbours receive their share); ionic terms
// followed by the reverse of the predictor (vbar0 += sum_m Vbar_m).
// Parameter gradients: the per-node conductivity scale s enters K through the
// element means sbar_e, so dL/dsbar_e = sum over (u, v) pairs of u_e^T Khat_e v_e
// with Khat_e the unscaled element matrix; the Aliev-Panfilov parameters
// (ga, gs, a) enter I_ion, dI/dv, R and dR/dw pointwise.

#include <algorithm>
#include <vector>

#include "device_common.cuh"
#include "sdc_internal.h"

namespace sdc {
namespace {

constexpr int kAdjBlock = 128;

inline int nb(int n, int b) { return (n + b - 1) / b; }

// Every kernel below is bound by the FP64 pipe (two operations per cycle and SM) or by its
// launch, not by memory: products of constants are folded on the host (dt into Q and Qhat),
// divisions are the three-operation reciprocal, and what several kernels used is computed once.
struct AdjIonic {
    double ga, gs, a, mu2;
    double ga3, gaq, ga6, a1;   // 3 ga, -2 ga (1 + a), 6 ga, 1 + a
    double cmu1, ceps;          // cw mu1, cw eps
};

inline AdjIonic fold_adjoint(const Ionic& p) {
    return AdjIonic{p.ga,       p.gs,           p.a,          p.mu2,         3.0 * p.ga,
                    -2.0 * p.ga * (1.0 + p.a), 6.0 * p.ga, 1.0 + p.a, p.cw * p.mu1,
                    p.cw * p.eps};
}

// Sums of (a, b, c) over the block, added to the block's own three partials: the launches of
// one adjoint follow one another, so a block's partials have one writer at a time and one
// final sum in a fixed order is enough.
__device__ __forceinline__ void block_add3(double a, double b, double c, double* part) {
    __shared__ double sh[3][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    if (lane == 0) {
        sh[0][wid] = a;
        sh[1][wid] = b;
        sh[2][wid] = c;
    }
    __syncthreads();
    if (wid < 3) {
        const double x = warp_sum(lane < nw ? sh[wid][lane] : 0.0);
        if (lane == 0) part[3 * blockIdx.x + wid] += x;
    }
}

// The blocks' partials in a fixed order: 256 strided sums, then the tree of block_add3
// (acc zeroed before).
__global__ void k_sum3(int nblk, const double* __restrict__ part, double* acc) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
        a += part[3 * i];
        b += part[3 * i + 1];
        c += part[3 * i + 2];
    }
    block_add3(a, b, c, acc);
}

__global__ void k_adj_init(int N, int M, const double* __restrict__ lv,
                           const double* __restrict__ lw, double* __restrict__ Vb,
                           double* __restrict__ Wb, double* __restrict__ lv0,
                           double* __restrict__ lw0) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    for (int m = 0; m < M; ++m) {
        Vb[(size_t)i * M + m] = m == M - 1 ? lv[i] : 0.0;
        Wb[(size_t)i * M + m] = m == M - 1 ? lw[i] : 0.0;
    }
    lv0[i] = 0.0;
    lw0[i] = 0.0;
}

// Before the reverse solves of a sweep, on its active rows: the reverse of the pointwise w
// sweep (unless w is frozen), then the compact right-hand sides (Vb), J, mass and K_ii of the
// node solves.  Vo, Wo: state before the sweep, Vn, Wn: after it; Wb is replaced by the adjoint
// of w before the sweep, Vb (adjoint of v after the sweep) and lw0 accumulate.
//   eps_m = N_m / den_m,  N_m = s_m + dt sum_{j<m} Qh_mj R_w,j eps_j,
//   den_m = 1 - dt Qh_mm R_w,m,  s_m = w0 + dt sum_j Q_mj R_j - W_m,  R = cw E G
template <int M>
__global__ void k_adj_prep(int n, const int* __restrict__ act, const double* __restrict__ Vo,
                           const double* __restrict__ Wo, const double* __restrict__ Vn,
                           const double* __restrict__ Wn, const double* __restrict__ kdiag,
                           const double* __restrict__ mass, AdjIonic ion, Coll co, int w_frozen,
                           int reaction_implicit, int ld, double* __restrict__ Vb,
                           double* __restrict__ Wb, double* __restrict__ lw0,
                           double* __restrict__ part3, double* __restrict__ J,
                           double* __restrict__ mc, double* __restrict__ kdc,
                           double* __restrict__ Db, int N) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    double ggs = 0.0, ga_ = 0.0;
    if (p < n) {
        const int g = act ? sdc_idx(act[p], N, 201) : p;
        double wo[M], vb[M];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            wo[m] = Wo[(size_t)g * M + m];
            vb[m] = Vb[(size_t)g * M + m];
        }
        if (!w_frozen) {
            double E[M], u[M], Rv[M], Rw[M], Rwv[M], eps[M], eb[M], sb[M], gb[M], db[M], wb0[M];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const double v = Vn[(size_t)g * M + m], w = wo[m];
                const double inv = recip(v + ion.mu2);
                u[m] = ion.cmu1 * inv;                       // cw dE/dw
                E[m] = fma(u[m], w, ion.ceps);               // cw E
                const double ui = u[m] * inv;                // - cw d2E/dwdv
                const double Ev = -ui * w;
                const double x = v - ion.a1;
                const double G = fma(-ion.gs * v, x, -w);
                const double Gv = -ion.gs * (x + v);
                Rv[m] = fma(Ev, G, E[m] * Gv);
                Rw[m] = fma(u[m], G, -E[m]);
                Rwv[m] = fma(-ui, G, fma(u[m], Gv, -Ev));
                eps[m] = Wn[(size_t)g * M + m] - w;
                wb0[m] = Wb[(size_t)g * M + m];              // adjoint of W' = W + eps
                eb[m] = wb0[m];
                gb[m] = 0.0;
                db[m] = 0.0;
            }
#pragma unroll
            for (int m = M - 1; m >= 0; --m) {
                const double q = co.Qh[m * kMaxM + m];
                sb[m] = eb[m] * recip(fma(-q, Rw[m], 1.0));   // N_m's and s_m's adjoint
                db[m] = fma(sb[m] * eps[m], q, db[m]);
#pragma unroll
                for (int j = 0; j < m; ++j) {
                    const double sq = sb[m] * co.Qh[m * kMaxM + j];
                    db[j] = fma(sq, eps[j], db[j]);
                    eb[j] = fma(sq, Rw[j], eb[j]);
                }
            }
            double w0b = 0.0;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                w0b += sb[m];
#pragma unroll
                for (int j = 0; j < M; ++j) gb[j] = fma(co.Q[m * kMaxM + j], sb[m], gb[j]);
            }
            lw0[g] += w0b;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                // W' = W + eps: direct, - sb (via s), and the chain through R and R_w
                const double v = Vn[(size_t)g * M + m];
                Wb[(size_t)g * M + m] =
                    fma(db[m], -2.0 * u[m], fma(gb[m], Rw[m], wb0[m] - sb[m]));
                vb[m] = fma(db[m], Rwv[m], fma(gb[m], Rv[m], vb[m]));
                Vb[(size_t)g * M + m] = vb[m];
                // dR/dgs = -cw E v (v - a - 1), dR/da = cw E gs v; the same with dE/dw for R_w
                const double t = v * fma(db[m], u[m], gb[m] * E[m]);
                ggs = fma(ion.a1 - v, t, ggs);
                ga_ += t;
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const double v = Vo[(size_t)g * M + m];
            J[(size_t)m * ld + p] =
                reaction_implicit
                    ? fma(v, fma(ion.ga3, v, ion.gaq), fma(ion.ga, ion.a, wo[m])) : 0.0;
            Db[(size_t)m * ld + p] = vb[m];
        }
        mc[p] = mass[g];
        kdc[p] = kdiag[g];
    }
    if (!w_frozen) block_add3(0.0, ggs, ion.gs * ga_, part3);
}

// After the reverse solves (X_m = bbar_m = rbar_m), on the active rows: the reverse of the
// residual and the adjoint of J, which reaches A_m and the couplings of every node m >= j:
//   Jbar_j = - mass D_j sum_{m>=j} dt Qh_mj bbar_m,  D = V' - V
// (one expression over the M solutions: as one pass after each of the M solves it cost four
// microseconds and two launch gaps a node).  Full-length copies of bbar and fbar, node-major.
template <int M>
__global__ void k_adj_residual(int n, const int* __restrict__ act, int ld, int N, Coll co,
                               AdjIonic ion, int reaction_implicit,
                               const double* __restrict__ X, const double* __restrict__ Vo,
                               const double* __restrict__ Wo, const double* __restrict__ Vn,
                               const double* __restrict__ mass, double* __restrict__ Vb,
                               double* __restrict__ Wb, double* __restrict__ lv0,
                               double* __restrict__ bfull, double* __restrict__ ffull,
                               double* __restrict__ part3) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    double gga = 0.0, ga_ = 0.0;
    if (p < n) {
        const int g = act ? sdc_idx(act[p], N, 204) : p;
        const double mi = mass[g];
        double rb[M], fb[M], jb[M];
        double rsum = 0.0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            rb[m] = X[(size_t)m * ld + p];
            bfull[(size_t)g * M + m] = rb[m];
            rsum += rb[m];
            fb[m] = 0.0;
            jb[m] = 0.0;
        }
        lv0[g] = fma(mi, rsum, lv0[g]);
#pragma unroll
        for (int m = 0; m < M; ++m) {
#pragma unroll
            for (int j = 0; j < M; ++j) fb[j] = fma(co.Q[m * kMaxM + j], rb[m], fb[j]);
            if (reaction_implicit) {
#pragma unroll
                for (int j = 0; j <= m; ++j) jb[j] = fma(-co.Qh[m * kMaxM + j], rb[m], jb[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const double v = Vo[(size_t)g * M + j], w = Wo[(size_t)g * M + j];
            if (reaction_implicit) jb[j] *= Vn[(size_t)g * M + j] - v;
            // I = ga v (v - a)(v - 1) + v w; r_j = ... - mass V_j,
            // f_j = -K V_j - mass (I - stim), J_j = dI/dv
            const double vv = v * (v - 1.0);
            const double c1 = fma(3.0, v, -2.0 * ion.a1);
            const double Iv_ga = fma(v, c1, ion.a);
            const double Iv = fma(ion.ga, Iv_ga, w);
            const double Ivv = fma(ion.ga6, v, ion.gaq);
            Vb[(size_t)g * M + j] =
                fma(mi, fma(jb[j], Ivv, -fma(Iv, fb[j], rb[j])), Vb[(size_t)g * M + j]);
            Wb[(size_t)g * M + j] = fma(mi, fma(-v, fb[j], jb[j]), Wb[(size_t)g * M + j]);
            gga = fma(jb[j], Iv_ga, fma(-vv * (v - ion.a), fb[j], gga));
            ga_ = fma(jb[j], fma(-2.0, v, 1.0), fma(vv, fb[j], ga_));
            ffull[(size_t)g * M + j] = fb[j];
        }
        gga *= mi;
        ga_ *= ion.ga * mi;
    }
    block_add3(gga, 0.0, ga_, part3);
}

// Over every row: Vb_j -= K fbar_j (fbar is zero off the active set), and for the conductivity
// gradient the field that bbar_m is paired with in every element,
//   z_m = - dt sum_{j<=m} Qh_mj (V'_j - V_j) - dt sum_j Q_mj V_j
// (the node solves' - K dt Qhat D and, with fbar_j = dt sum_m Q_mj bbar_m, the residual's
// - fbar_j^T K V_j; V' = V off the active set).
template <int M>
__global__ void k_adj_kfull(int N, const double* __restrict__ kval, const int* __restrict__ kcol,
                            const int* __restrict__ klen, int ldk, const double* __restrict__ kdiag,
                            const double* __restrict__ ffull, double* __restrict__ Vb, Coll co,
                            const double* __restrict__ Vo, const double* __restrict__ Vn,
                            double* __restrict__ z) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double acc[M];
#pragma unroll
    for (int m = 0; m < M; ++m) acc[m] = kdiag[i] * ffull[(size_t)i * M + m];
    const int len = klen[i];
    for (int t = 0; t < len; ++t) {
        const double a = kval[(size_t)t * ldk + i];
        const int j = sdc_idx(kcol[(size_t)t * ldk + i], N, 205);
#pragma unroll
        for (int m = 0; m < M; ++m) acc[m] += a * ffull[(size_t)j * M + m];
    }
#pragma unroll
    for (int m = 0; m < M; ++m) Vb[(size_t)i * M + m] -= acc[m];
    if (!z) return;
#pragma unroll
    for (int m = 0; m < M; ++m) acc[m] = 0.0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const double v = Vo[(size_t)i * M + j], d = Vn[(size_t)i * M + j] - v;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            acc[m] = fma(-co.Q[m * kMaxM + j], v, acc[m]);
            if (j <= m) acc[m] = fma(-co.Qh[m * kMaxM + j], d, acc[m]);
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m) z[(size_t)i * M + m] = acc[m];
}

// dL/dsbar_e += sum_m bbar_m^T Khat_e z_m.  The rows and columns of Khat_e sum to zero, so
// with differences to the element's first vertex (u_a = bbar_a - bbar_0, likewise z)
//   sum_m bbar_m^T Khat_e z_m = sum_{a,b>=1} (Khat_e)_ab T_ab,  T_ab = sum_m u_a,m z_b,m .
// T is kept over the sweeps (first: it starts from zero; last: it is contracted with Khat_e),
// so the geometry is formed once per adjoint and not in every sweep, and one pair of fields
// per node is gathered where there were two: 15 FP64 operations per element and node, 115
// for the geometry, where each sweep took 40 a node and 160.  The FP64 pipe bounds both.
template <int DIM, int M>
__global__ void k_adj_elem(int NE, const double* __restrict__ xyz, const int* __restrict__ elem,
                           const double* __restrict__ sig9, const double* __restrict__ esig9,
                           const double* __restrict__ bfull, const double* __restrict__ z,
                           int first, int last, double* __restrict__ T, double* __restrict__ ge) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NE) return;
    constexpr int NV = DIM + 1;
    int vt[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) vt[a] = elem[(size_t)e * NV + a];
    double u[NV][M];
    long long any = 0;
#pragma unroll
    for (int a = 0; a < NV; ++a)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            u[a][m] = bfull[(size_t)vt[a] * M + m];
            any |= __double_as_longlong(u[a][m]) & 0x7fffffffffffffffll;
        }
    if (!any && !first && !last) return;   // no active vertex
    double t[DIM][DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a)
#pragma unroll
        for (int b = 0; b < DIM; ++b)
            t[a][b] = first ? 0.0 : T[(size_t)(a * DIM + b) * NE + e];
    if (any) {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            double dz[DIM];
            const double z0 = z[(size_t)vt[0] * M + m];
#pragma unroll
            for (int b = 0; b < DIM; ++b) dz[b] = z[(size_t)vt[b + 1] * M + m] - z0;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                const double du = u[a + 1][m] - u[0][m];
#pragma unroll
                for (int b = 0; b < DIM; ++b) t[a][b] = fma(du, dz[b], t[a][b]);
            }
        }
    }
    if (!last) {
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = 0; b < DIM; ++b) T[(size_t)(a * DIM + b) * NE + e] = t[a][b];
        return;
    }
    double grad[4][3], vol;
    if (!p1_gradients(DIM, xyz, vt, grad, vol)) return;
    const double* Dm = esig9 ? esig9 + (size_t)e * 9 : sig9;
    // sum_ab t_ab grad_a . D grad_b = sum_r (sum_a grad_a,r sum_b t_ab (D grad_b)_r)
    double acc = 0.0;
#pragma unroll
    for (int r = 0; r < DIM; ++r) {
        double Dg[DIM];
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            Dg[b] = 0.0;
#pragma unroll
            for (int c = 0; c < DIM; ++c) Dg[b] = fma(Dm[r * 3 + c], grad[b + 1][c], Dg[b]);
        }
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            double s = 0.0;
#pragma unroll
            for (int b = 0; b < DIM; ++b) s = fma(t[a][b], Dg[b], s);
            acc = fma(grad[a + 1][r], s, acc);
        }
    }
    ge[e] = fma(vol, acc, ge[e]);
}

// dL/ds_a += sum over elements e containing a of dL/dsbar_e / (d + 1)
__global__ void k_adj_scale_nodes(int N, int nv, const int* __restrict__ n2e_ptr,
                                  const int* __restrict__ n2e, const double* __restrict__ ge,
                                  double* __restrict__ grad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double s = 0.0;
    for (int k = n2e_ptr[i]; k < n2e_ptr[i + 1]; ++k) s += ge[n2e[k]];
    grad[i] += s / nv;
}

__global__ void k_adj_spread_back(int N, int M, const double* __restrict__ Vb,
                                  const double* __restrict__ Wb, double* __restrict__ lv0,
                                  double* __restrict__ lw0) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double a = 0.0, b = 0.0;
    for (int m = 0; m < M; ++m) {
        a += Vb[(size_t)i * M + m];
        b += Wb[(size_t)i * M + m];
    }
    lv0[i] += a;
    lw0[i] += b;
}

__global__ void k_pos_set(int n, const int* __restrict__ act, int* __restrict__ pos, int reset,
                          int N) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    pos[sdc_idx(act[q], N, 206)] = reset ? -1 : q;
}

// restricted matrix of an arbitrary active list, straight from the global K
__global__ void k_extract_global(int n, const int* __restrict__ act, const int* __restrict__ pos,
                                 const double* __restrict__ kval, const int* __restrict__ kcol,
                                 const int* __restrict__ klen, int ldk, double* __restrict__ nval,
                                 int* __restrict__ ncol, int* __restrict__ nlen, int ldn, int N) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int g = sdc_idx(act[q], N, 207);
    const int len = klen[g];
    int c = 0;
    for (int t = 0; t < len; ++t) {
        const int jn = pos[sdc_idx(kcol[(size_t)t * ldk + g], N, 208)];
        if (jn >= 0) {
            nval[(size_t)c * ldn + q] = kval[(size_t)t * ldk + g];
            ncol[(size_t)c * ldn + q] = jn;
            ++c;
        }
    }
    nlen[q] = c;
}

// old compact row -> position in a replayed next list (pos holds that list)
__global__ void k_replay_map(int n_old, const int* __restrict__ act_old,
                             const int* __restrict__ pos, int* __restrict__ map, int N) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_old) return;
    map[p] = pos[act_old ? sdc_idx(act_old[p], N, 209) : p];
}

template <class F>
void dispatch_M(int M, F&& f) {
    switch (M) {
        case 1: f(std::integral_constant<int, 1>()); break;
        case 2: f(std::integral_constant<int, 2>()); break;
        case 3: f(std::integral_constant<int, 3>()); break;
        case 4: f(std::integral_constant<int, 4>()); break;
        case 5: f(std::integral_constant<int, 5>()); break;
        case 6: f(std::integral_constant<int, 6>()); break;
        case 7: f(std::integral_constant<int, 7>()); break;
        case 8: f(std::integral_constant<int, 8>()); break;
        default: break;
    }
}

}  // namespace

void launch_pos_set(int n, const int* act, int* pos, int reset, int N, cudaStream_t s) {
    if (n > 0) k_pos_set<<<nb(n, kAdjBlock), kAdjBlock, 0, s>>>(n, act, pos, reset, N);
}

void launch_replay_map(int n_old, const int* act_old, const int* pos, int* map, int N,
                       cudaStream_t s) {
    if (n_old > 0)
        k_replay_map<<<nb(n_old, kAdjBlock), kAdjBlock, 0, s>>>(n_old, act_old, pos, map, N);
}

void launch_extract_global(int n, const int* act, const int* pos, const Ell& K, Ell& out, int N,
                           cudaStream_t s) {
    if (n > 0)
        k_extract_global<<<nb(n, kAdjBlock), kAdjBlock, 0, s>>>(n, act, pos, K.val, K.col, K.len,
                                                                K.ld, out.val, out.col, out.len,
                                                                out.ld, N);
}

int adjoint_step(const AdjointArgs& a, StepBuffers& B, AdjointBuffers& W, cudaStream_t s) {
    const int N = B.N, M = B.M, ld = B.ld;
    const MeshDev& md = *a.mesh;
    const Ell& K = *a.K;
    const AdjIonic ion = fold_adjoint(a.ion);
    Coll co = a.co;   // times dt
    for (int k = 0; k < kMaxM * kMaxM; ++k) {
        co.Q[k] *= a.dt;
        co.Qh[k] *= a.dt;
    }
    bool first = true;   // no element term yet
    cudaMemsetAsync(W.iacc, 0, 3 * sizeof(double), s);
    cudaMemsetAsync(W.part3, 0, 3 * (size_t)nb(N, kAdjBlock) * sizeof(double), s);
    if (a.grad_scale) cudaMemsetAsync(W.ge, 0, (size_t)md.n_elems * sizeof(double), s);
    k_adj_init<<<nb(N, kAdjBlock), kAdjBlock, 0, s>>>(N, M, a.lam_v, a.lam_w, W.Vb, W.Wb,
                                                     a.lam_v0, a.lam_w0);
    // state before sweep 0: the predictor (spread of v0, w0)
    launch_spread(N, M, a.v0, a.w0, W.V0, W.W0, s);
    int status = SDC_OK;
    for (int k = a.sweeps - 1; k >= 0 && status == SDC_OK; --k) {
        const int n = a.n_active[k];
        if (n == 0) continue;
        const double* Vo = k == 0 ? W.V0 : a.tape_V + (size_t)(k - 1) * N * M;
        const double* Wo = k == 0 ? W.W0 : a.tape_W + (size_t)(k - 1) * N * M;
        const double* Vn = a.tape_V + (size_t)k * N * M;
        const double* Wn = a.tape_W + (size_t)k * N * M;
        const int* act = k == 0 ? nullptr : a.tape_act + (size_t)k * N;
        const int nbk = nb(n, kAdjBlock);
        // restricted matrix of I_k
        const Ell* A = &K;
        if (act) {
            launch_pos_set(n, act, W.pos, 0, N, s);
            launch_extract_global(n, act, W.pos, K, B.A[0], N, s);
            launch_pos_set(n, act, W.pos, 1, N, s);
            A = &B.A[0];
        }
        dispatch_M(M, [&](auto mc) {
            constexpr int MM = decltype(mc)::value;
            k_adj_prep<MM><<<nbk, kAdjBlock, 0, s>>>(n, act, Vo, Wo, Vn, Wn, a.kdiag, a.mass, ion,
                                                     co, a.w_frozen, a.reaction_implicit, ld, W.Vb,
                                                     W.Wb, a.lam_w0, W.part3, B.J, B.mc, B.kdc,
                                                     B.R, N);
        });
        if (n < N) {   // zero off the active set
            cudaMemsetAsync(W.bfull, 0, (size_t)M * N * sizeof(double), s);
            cudaMemsetAsync(W.ffull, 0, (size_t)M * N * sizeof(double), s);
        }
        for (int m = M - 1; m >= 0 && status == SDC_OK; --m) {
            PcgRole role{};
            role.b = B.R + (size_t)m * ld;            // dvbar_m (coupled)
            role.x = W.X + (size_t)m * ld;            // bbar_m
            role.J = B.J + (size_t)m * ld;
            role.Jall = B.J;
            role.R = B.R;
            role.epi_lo = 0;
            role.epi_hi = m;
            role.epi_target_J = 1;
            for (int j = 0; j < kMaxM; ++j) role.qh[j] = j < M ? a.co.Qh[m * kMaxM + j] : 0.0;
            role.c = a.dt * a.co.Qh[m * kMaxM + m];
            role.iters_out = W.iters + (size_t)k * kMaxM + m;
            role.relres_out = W.relres + (size_t)k * kMaxM + m;
            if (launch_pcg_role(n, *A, role, a.dt, M, a.rtol, a.maxit, *a.cfg, B, s) != SDC_OK) {
                status = SDC_E_CUDA;
                break;
            }
        }
        if (status != SDC_OK) break;
        dispatch_M(M, [&](auto mc) {
            constexpr int MM = decltype(mc)::value;
            k_adj_residual<MM><<<nbk, kAdjBlock, 0, s>>>(n, act, ld, N, co, ion,
                                                         a.reaction_implicit, W.X, Vo, Wo, Vn,
                                                         a.mass, W.Vb, W.Wb, a.lam_v0, W.bfull,
                                                         W.ffull, W.part3);
            k_adj_kfull<MM><<<nb(N, kAdjBlock), kAdjBlock, 0, s>>>(
                N, K.val, K.col, K.len, K.ld, a.kdiag, W.ffull, W.Vb, co, Vo, Vn,
                a.grad_scale ? W.z : nullptr);
            if (a.grad_scale) {
                // without the sweeps' T (no memory for it) each sweep is contracted by itself
                const int f = first || !W.T, l = k == 0 || !W.T;
                auto* kern = md.dim == 2 ? k_adj_elem<2, MM> : k_adj_elem<3, MM>;
                kern<<<nb(md.n_elems, 128), 128, 0, s>>>(md.n_elems, md.xyz, md.elem, md.sig,
                                                         md.esig, W.bfull, W.z, f, l, W.T, W.ge);
                first = false;
            }
        });
    }
    if (status != SDC_OK) return status;
    k_sum3<<<1, 256, 0, s>>>(nb(N, kAdjBlock), W.part3, W.iacc);
    k_adj_spread_back<<<nb(N, kAdjBlock), kAdjBlock, 0, s>>>(N, M, W.Vb, W.Wb, a.lam_v0,
                                                            a.lam_w0);
    if (a.grad_scale)
        k_adj_scale_nodes<<<nb(N, kAdjBlock), kAdjBlock, 0, s>>>(N, md.dim + 1, md.n2e_ptr,
                                                                md.n2e, W.ge, a.grad_scale);
    return SDC_OK;
}

}  // namespace sdc

namespace sdc {
SDC_CHECK_READER(check_take_adjoint)
}  // namespace sdc

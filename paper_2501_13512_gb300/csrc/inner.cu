// Persistent block solver for the block-diagonal preconditioner (Eq. 10;
// Section II.B: inner BiCGSTAB-FFT solves with a loose tolerance).
//
// The diagonal blocks are independent (no data exchange between blocks), so one
// thread-block cluster owns one block at a time and runs that block's whole
// BiCGSTAB without any grid-wide synchronisation; clusters take blocks from an
// atomic work counter, longest first. Boxes of up to 16 voxels per axis use the
// parity-split MVM of inner_parity.cuh (whole MVM on chip); for the others each
// inner MVM A_k x = x - G(chi x) is done in three phases over the padded box:
//   XY  for tiles of (component, z) planes: load the box plane with the
//       BiCGSTAB vector update fused in, multiply by chi, zero-pad, row FFTs
//       (x, pruned to the non-zero rows) and column FFTs (y) in shared
//       memory, store the plane spectrum to the block's scratch;
//   Z   for tiles of spectral columns: forward FFT along z, 3x3 symmetric
//       Green multiply, inverse FFT, keep z < bz;
//   XY' inverse column and row FFTs, keep the box, y = mask (x - u), with the
//       inner products of the iteration fused into the store.
// The block scratch ([3][bz][My][Mx]) stays L2-resident for the boxes this
// path accepts. Scalars are FP64; complex64 vectors accumulate products in
// FP32 within a warp and in FP64 across warps and CTAs.
#include <cooperative_groups.h>
#include <stdlib.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "dft_small.cuh"
#include "fft_core.cuh"
#include "vie_internal.cuh"

namespace cg = cooperative_groups;

namespace vie {

template <class C> struct InnerGroup {
    C *b, *x, *r, *rhat, *p, *v, *s, *t;   // [nb][3][bz][by][bx]
    C* w2;                                  // [nb][3][bz][My][Mx]
    const C* chi;                           // [nb][bz][by][bx]
    const uint8_t* mask;                    // [nb][bz][by][bx]
    const C* G;                             // [6][Mz][My][Mx], bit-reversed positions
    const C* const* Gb;                     // optional: one spectrum per box
    const double* tols;                     // optional: one relative tolerance per box
    SegState* st;                           // [nb]
    int nb, bx, by, bz, Mx, My, Mz, lx, ly, lz, lyb;   // lyb = log2 of nextpow2(by)
    int lpt;                                // log2 planes per XY tile
    int ltc;                                // log2 columns per Z tile
    int kb_mvm;                             // profiling: KB moved by one MVM and its fused updates
    int kb_upd;                             // profiling: KB moved by the x/r update pass (shared-memory passes)
    // parity-split MVM (inner_parity.cuh)
    int par;                                // 1: the block uses it
    int ex, ey, ez;                         // the blocks' own extents within the box
    int hx, hy, hz;                         // transform lengths per axis (>= extent)
    int yp;                                 // row pitch in shared memory (ex made odd: no bank conflicts)
    unsigned fd_ex[3], fd_exy[3], fd_hy[3]; // FastDiv constants for ex, ex*ey and hy
    const C* Gq;                            // spectrum [4][hx+1][6][hz/2+1][hy/2+1] (par_spectra)
};

constexpr int kInnerThreads = 256;

__device__ __forceinline__ double2 dcdiv(double2 a, double2 b) {
    double d = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ bool dgood(double2 a) {
    return isfinite(a.x) && isfinite(a.y) && (a.x != 0.0 || a.y != 0.0);
}
template <class C> __device__ __forceinline__ void acc_dot(C& acc, C a, C b) {   // acc += conj(a) b
    acc.x = fma(a.y, b.y, fma(a.x, b.x, acc.x));
    acc.y = fma(-a.y, b.x, fma(a.x, b.y, acc.y));
}

// A block is solved by a team: the R CTAs of one thread-block cluster. Every
// phase splits its rows / columns / planes over the ranks; phases that read
// what other ranks wrote are separated by cluster barriers (release/acquire at
// cluster scope), and sums go CTA -> distributed shared memory in rank order,
// so every CTA gets identical scalars.
__device__ __forceinline__ int team_rank() { return (int)cg::this_cluster().block_rank(); }
__device__ __forceinline__ int team_size() { return (int)cg::this_cluster().num_blocks(); }
__device__ __forceinline__ void team_sync() { cg::this_cluster().sync(); }

// Slot of the next cluster sum; reset to 0 by every CTA at kernel entry so all
// ranks of a cluster flip in step.
__shared__ int team_slot;

template <class T> __device__ __forceinline__ T shfl_dn(T v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }

// Team-wide sums of two complex partials a and b held by every thread (complex64
// or complex128). Each warp adds its lanes in the partials' precision; thread 0
// adds the warps' sums in FP64 in a fixed order (and, for R > 1, the ranks' sums
// in rank order through distributed shared memory), then calls fn(sum_a, sum_b):
// the iteration's FP64 scalar work runs in that one thread and reaches the others
// through the shared state fn writes, published by the closing barrier. Every rank
// computes identical sums. Two rank slots alternate between consecutive sums: a
// slot is rewritten two sums later, after every rank has passed the cluster
// barrier of the sum in between, so one cluster barrier per sum suffices.
template <class C, class Fn>
__device__ __forceinline__ void team_sum(C a, C b, double2* red, Fn fn) {
    constexpr int N = 2;
    C v[N] = {a, b};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) {
            v[i].x += shfl_dn(v[i].x, o);
            v[i].y += shfl_dn(v[i].y, o);
        }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (l == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) red[N * w + i] = make_double2(v[i].x, v[i].y);
    __syncthreads();
    cg::cluster_group cl = cg::this_cluster();
    const unsigned R = cl.num_blocks();
    __shared__ double2 xred[2][N];
    double2 sum[N];
#pragma unroll
    for (int i = 0; i < N; ++i) sum[i] = make_double2(0, 0);
    if (threadIdx.x == 0) {
        for (int k = 0; k < nw; ++k)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                sum[i].x += red[N * k + i].x;
                sum[i].y += red[N * k + i].y;
            }
        if (R > 1) {
            team_slot ^= 1;
#pragma unroll
            for (int i = 0; i < N; ++i) xred[team_slot][i] = sum[i];
        }
    }
    if (R > 1) {
        cl.sync();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int i = 0; i < N; ++i) sum[i] = make_double2(0, 0);
            for (unsigned r = 0; r < R; ++r) {
                const double2* q = cl.map_shared_rank(&xred[team_slot][0], r);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    sum[i].x += q[i].x;
                    sum[i].y += q[i].y;
                }
            }
        }
    }
    if (threadIdx.x == 0) fn(sum[0], sum[1]);
    __syncthreads();
}

enum { IN_P = 0, IN_S = 1 };
enum { OUT_V = 0, OUT_T = 1 };

// Phase XY: plane tiles, fused vector update + chi, 2D forward FFT, store spectrum.
// IN_P: p = r + beta (p - omega v);  IN_S: s = r - alpha v (returns ||s||^2 in .x).
template <class C, int IN>
__device__ C phase_xy(const InnerGroup<C>& g, int64_t voff, C* W, const C* chi, C* sm, const C* tw, C c1, C c2) {
    const int planes = 3 * g.bz, P = g.Mx + 1, pe = g.My * P, tile = 1 << g.lpt;
    const int64_t box = (int64_t)g.bx * g.by * g.bz;
    C acc = czero<C>();
    const int rk = team_rank(), nrk = team_size();
    for (int pl0 = rk * tile; pl0 < planes; pl0 += nrk * tile) {
        const int n = tile * g.My * g.Mx;
        for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
            int xq = idx & (g.Mx - 1), t = idx >> g.lx;
            int yq = t & (g.My - 1), k = t >> g.ly;
            int pl = pl0 + k;
            C val = czero<C>();
            if (pl < planes && xq < g.bx && yq < g.by) {
                int comp = pl / g.bz, z = pl - comp * g.bz;
                int64_t lv = ((int64_t)z * g.by + yq) * g.bx + xq;
                int64_t e = voff + comp * box + lv;
                C in;
                if (IN == IN_P) {
                    in = g.r[e] + cmul(c1, g.p[e] - cmul(c2, g.v[e]));
                    g.p[e] = in;
                } else {
                    in = g.r[e] - cmul(c1, g.v[e]);
                    g.s[e] = in;
                    acc.x += in.x * in.x + in.y * in.y;
                }
                val = cmul(in, chi[lv]);
            }
            sm[k * pe + yq * P + xq] = val;
        }
        __syncthreads();
        smem_fft_g<C, true>(sm, g.lx, 1, g.lyb, P, g.lpt, pe, tw, kLogLmax - g.lx);     // rows (x)
        smem_fft_g<C, true>(sm, g.ly, P, g.lx, 1, g.lpt, pe, tw, kLogLmax - g.ly);      // columns (y)
        for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
            int xq = idx & (g.Mx - 1), t = idx >> g.lx;
            int yq = t & (g.My - 1), k = t >> g.ly;
            int pl = pl0 + k;
            if (pl < planes) W[((int64_t)pl * g.My + yq) * g.Mx + xq] = sm[k * pe + yq * P + xq];
        }
        __syncthreads();
    }
    return acc;   // this thread's partial; the caller folds it into a later sum
}

// Phase Z: forward FFT along z, Green multiply, inverse FFT (columns of the plane spectra).
template <class C>
__device__ void phase_z(const InnerGroup<C>& g, C* W, C* sm, const C* tw) {
    const int TC = 1 << g.ltc, pitch = 3 * TC;
    const int64_t plane = (int64_t)g.My * g.Mx;
    const int64_t cstride = (int64_t)g.bz * plane, gcomp = (int64_t)g.Mz * plane;
    const int L = g.Mz;
    const int rk = team_rank(), nrk = team_size();
    for (int64_t c0 = (int64_t)rk * TC; c0 < plane; c0 += (int64_t)nrk * TC) {
        for (int idx = threadIdx.x; idx < L * 3 * TC; idx += blockDim.x) {
            int c = idx & (TC - 1), t = idx >> g.ltc;
            int comp = t % 3, i = t / 3;
            C v = czero<C>();
            if (i < g.bz && c0 + c < plane) v = W[comp * cstride + i * plane + c0 + c];
            sm[idx] = v;
        }
        __syncthreads();
        smem_fft<C, true, 3>(sm, g.lz, pitch, g.ltc, tw, kLogLmax - g.lz);
        for (int idx = threadIdx.x; idx < L * TC; idx += blockDim.x) {
            int c = idx & (TC - 1), i = idx >> g.ltc;
            if (c0 + c >= plane) continue;
            const C* gp = g.G + i * plane + c0 + c;
            C gxx = gp[0], gxy = gp[gcomp], gxz = gp[2 * gcomp];
            C gyy = gp[3 * gcomp], gyz = gp[4 * gcomp], gzz = gp[5 * gcomp];
            C* q = sm + i * pitch + c;
            C X = q[0], Y = q[TC], Z = q[2 * TC];
            const C e[6] = {gxx, gxy, gxz, gyy, gyz, gzz};
            green3<2, false>(X, Y, Z, e);
            q[0] = X;
            q[TC] = Y;
            q[2 * TC] = Z;
        }
        __syncthreads();
        smem_fft<C, false, 3>(sm, g.lz, pitch, g.ltc, tw, kLogLmax - g.lz);
        for (int idx = threadIdx.x; idx < g.bz * 3 * TC; idx += blockDim.x) {
            int c = idx & (TC - 1), t = idx >> g.ltc;
            int comp = t % 3, i = t / 3;
            if (c0 + c < plane) W[comp * cstride + i * plane + c0 + c] = sm[idx];
        }
        __syncthreads();
    }
}

// Phase XY': inverse 2D FFT of the plane spectra, keep the box, out = mask (in - u).
// OUT_V: in = p, out = v, returns <rhat, v>.  OUT_T: in = s, out = t, returns (<t, s>, <t, t>).
template <class C, int OUT>
__device__ void phase_xy_inv(const InnerGroup<C>& g, int64_t voff, const C* W, const uint8_t* mask, C* sm,
                             const C* tw, C& a1, C& a2) {
    const int planes = 3 * g.bz, P = g.Mx + 1, pe = g.My * P, tile = 1 << g.lpt;
    const int64_t box = (int64_t)g.bx * g.by * g.bz;
    const int rk = team_rank(), nrk = team_size();
    for (int pl0 = rk * tile; pl0 < planes; pl0 += nrk * tile) {
        const int n = tile * g.My * g.Mx;
        for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
            int xq = idx & (g.Mx - 1), t = idx >> g.lx;
            int yq = t & (g.My - 1), k = t >> g.ly;
            int pl = pl0 + k;
            sm[k * pe + yq * P + xq] = pl < planes ? W[((int64_t)pl * g.My + yq) * g.Mx + xq] : czero<C>();
        }
        __syncthreads();
        smem_fft_g<C, false>(sm, g.ly, P, g.lx, 1, g.lpt, pe, tw, kLogLmax - g.ly);     // columns (y)
        smem_fft_g<C, false>(sm, g.lx, 1, g.lyb, P, g.lpt, pe, tw, kLogLmax - g.lx);    // rows (x), y < nextpow2(by)
        const int nb = tile * g.by * g.bx;
        for (int idx = threadIdx.x; idx < nb; idx += blockDim.x) {
            int xq = idx % g.bx, t = idx / g.bx;
            int yq = t % g.by, k = t / g.by;
            int pl = pl0 + k;
            if (pl >= planes) continue;
            int comp = pl / g.bz, z = pl - comp * g.bz;
            int64_t lv = ((int64_t)z * g.by + yq) * g.bx + xq;
            int64_t e = voff + comp * box + lv;
            C u = sm[k * pe + yq * P + xq];
            C in = OUT == OUT_V ? g.p[e] : g.s[e];
            C o = mask[lv] ? in - u : czero<C>();
            if (OUT == OUT_V) {
                g.v[e] = o;
                acc_dot(a1, g.rhat[e], o);
            } else {
                g.t[e] = o;
                acc_dot(a1, o, in);
                a2.x += o.x * o.x + o.y * o.y;
            }
        }
        __syncthreads();
    }
}

// Division by a runtime divisor d (1 <= d < 2^31) of n < 2^31 with a multiply-high
// (Granlund and Montgomery, PLDI 1994): q = (umulhi(n, m) + n) >> s.
struct FastDiv {
    unsigned m, s, d;
};
__device__ __forceinline__ unsigned fdiv(unsigned n, FastDiv f) { return (__umulhi(n, f.m) + n) >> f.s; }
__device__ __forceinline__ FastDiv fd_of(const unsigned (&v)[3]) { return FastDiv{v[0], v[1], v[2]}; }

}  // namespace vie

#include "inner_parity.cuh"

namespace vie {

// BiCGSTAB state of the block being solved, in shared memory: written by thread 0
// inside team_sum (the FP64 scalar work of an iteration runs in that one thread)
// and read by every thread after the sum's closing barrier.
template <class C> struct BiState {
    double2 rho, rho_prev, alpha, omega;
    double tol2, bn2, res2, iters;
    int status, half;
    C cbeta, comega, calpha;                    // coefficients of the vector updates
};

// beta = (rho / rho_prev)(alpha / omega) for the next p update, or a breakdown.
template <class C> __device__ __forceinline__ void next_beta(BiState<C>& S) {
    if (!dgood(S.rho)) {
        S.status = SEG_BREAKDOWN;
        return;
    }
    const double2 beta = cmul(dcdiv(S.rho, S.rho_prev), dcdiv(S.alpha, S.omega));
    S.cbeta = cmk<C>(beta.x, beta.y);
    S.comega = cmk<C>(S.omega.x, S.omega.y);
}

// One block's BiCGSTAB with the MVM through the shared-memory passes above and the block scratch in global memory, for
// boxes of any size whose padded (x, y) plane fits (par_solve of inner_parity.cuh takes the others).
template <class C>
__device__ __forceinline__ void solve_block(const InnerGroup<C>& g, int b, double tol, int maxit, C* sm, const C* tw,
                            double2* red, int* units) {
    const int64_t box = (int64_t)g.bx * g.by * g.bz;
    const int64_t voff = (int64_t)b * 3 * box;
    const int n = 3 * (int)box;                 // elements of the block's vectors, at voff
    C* W = g.w2 + (int64_t)b * 3 * g.bz * g.My * g.Mx;
    const C* chi = g.chi + (int64_t)b * box;
    const uint8_t* mask = g.mask + (int64_t)b * box;
    __shared__ BiState<C> S;

    // x = 0, r = rhat = b, p = v = 0
    const int rk = team_rank(), nrk = team_size();
    const int first = rk * blockDim.x, step = nrk * blockDim.x;
    C acc = czero<C>();
    for (int i = first + threadIdx.x; i < n; i += step) {
        const int64_t e = voff + i;
        const C bv = g.b[e];
        g.x[e] = czero<C>();
        g.r[e] = bv;
        g.rhat[e] = bv;
        g.p[e] = czero<C>();
        g.v[e] = czero<C>();
        acc.x += bv.x * bv.x + bv.y * bv.y;
    }
    team_sum(acc, czero<C>(), red, [&](double2 sa, double2) {
        const double bn2 = sa.x;
        S.bn2 = bn2;
        S.tol2 = tol * tol * bn2;
        S.rho = make_double2(bn2, 0.0);
        S.rho_prev = S.alpha = S.omega = make_double2(1, 0);
        S.iters = 0.0;
        S.res2 = bn2;
        S.half = 0;
        S.status = SEG_ACTIVE;
        if (!(bn2 > 0.0) || !isfinite(bn2)) S.status = bn2 == 0.0 ? SEG_CONVERGED : SEG_BREAKDOWN;
        else if (bn2 <= S.tol2) S.status = SEG_CONVERGED;   // x = 0 meets a tolerance of 1 or more
        else next_beta(S);
    });
    for (int it = 0; it < maxit && S.status == SEG_ACTIVE; ++it) {
        // v = A p, p = r + beta (p - omega v)
        phase_xy<C, IN_P>(g, voff, W, chi, sm, tw, S.cbeta, S.comega);
        team_sync();
        phase_z<C>(g, W, sm, tw);
        team_sync();
        if (units != nullptr && rk == 0 && threadIdx.x == 0) atomicAdd(units, g.kb_mvm);
        C p1 = czero<C>(), p2 = czero<C>();
        phase_xy_inv<C, OUT_V>(g, voff, W, mask, sm, tw, p1, p2);
        team_sum(p1, p2, red, [&](double2 sigma, double2) {
            if (!dgood(sigma)) {
                S.status = SEG_BREAKDOWN;
                return;
            }
            S.alpha = dcdiv(S.rho, sigma);
            S.calpha = cmk<C>(S.alpha.x, S.alpha.y);
        });
        if (S.status != SEG_ACTIVE) break;
        // s = r - alpha v and t = A s; ||s||^2 is summed together with <t,s> and <t,t>, so the
        // half-step test (same value, same decision) costs no reduction of its own
        const C snp = phase_xy<C, IN_S>(g, voff, W, chi, sm, tw, S.calpha, czero<C>());
        team_sync();
        phase_z<C>(g, W, sm, tw);
        team_sync();
        if (units != nullptr && rk == 0 && threadIdx.x == 0) atomicAdd(units, g.kb_mvm + g.kb_upd);
        p1 = czero<C>();
        p2 = czero<C>();
        phase_xy_inv<C, OUT_T>(g, voff, W, mask, sm, tw, p1, p2);
        p2.y = snp.x;                           // the deferred ||s||^2 rides in the unused slot
        team_sum(p1, p2, red, [&](double2 ts, double2 tt) {
            const double sn2 = tt.y;
            if (sn2 <= S.tol2) {
                S.half = 1;
                S.res2 = sn2;
                S.iters += 0.5;
                S.status = SEG_CONVERGED;
                return;
            }
            if (!(tt.x > 0.0) || !isfinite(tt.x)) {
                S.status = SEG_BREAKDOWN;
                return;
            }
            S.omega = make_double2(ts.x / tt.x, ts.y / tt.x);
            S.comega = cmk<C>(S.omega.x, S.omega.y);
        });
        if (S.half) {
            // half-step convergence: x += alpha p (t is not needed)
            const C ac = S.calpha;
            for (int i = first + threadIdx.x; i < n; i += step) {
                const int64_t e = voff + i;
                g.x[e] = g.x[e] + cmul(ac, g.p[e]);
            }
            break;
        }
        if (S.status != SEG_ACTIVE) break;
        // x += alpha p + omega s, r = s - omega t; rho = <rhat, r>, ||r||^2
        const C ac = S.calpha, oc = S.comega;
        C a1 = czero<C>(), a2 = czero<C>();
        for (int i = first + threadIdx.x; i < n; i += step) {
            const int64_t e = voff + i;
            const C sv = g.s[e];
            g.x[e] = g.x[e] + cmul(ac, g.p[e]) + cmul(oc, sv);
            const C rv = sv - cmul(oc, g.t[e]);
            g.r[e] = rv;
            acc_dot(a1, g.rhat[e], rv);
            a2.x += rv.x * rv.x + rv.y * rv.y;
        }
        team_sum(a1, a2, red, [&](double2 r1, double2 r2) {
            S.rho_prev = S.rho;
            S.rho = r1;
            S.res2 = r2.x;
            S.iters += 1.0;
            if (!isfinite(S.res2)) S.status = SEG_BREAKDOWN;
            else if (S.res2 <= S.tol2) S.status = SEG_CONVERGED;
            else if (S.omega.x == 0.0 && S.omega.y == 0.0) S.status = SEG_BREAKDOWN;
            else next_beta(S);
        });
    }
    if (rk == 0 && threadIdx.x == 0) {
        SegState& St = g.st[b];
        St.bnorm2 = S.bn2;
        St.res2 = S.res2;
        St.iters = S.iters;
        St.status = S.status == SEG_ACTIVE ? SEG_MAXIT : S.status;
        St.maxit = maxit;
    }
    __syncthreads();
}

template <int PAR, class C>
__device__ __forceinline__ void solve_dispatch(const InnerGroup<C>& g, int b, double tol, int maxit, C* sm, const C* tw,
                                               double2* red, int* units) {
    if constexpr (PAR) {
        if (PAR == PAR_SMALL || g.par) {           // (the small shape takes no other jobs)
            par_solve<PAR>(g, b, tol, maxit, sm, units);
            return;
        }
    }
    if constexpr (PAR != PAR_SMALL) solve_block<C>(g, b, tol, maxit, sm, tw, red, units);
}

// PAR: the kernel of launches with groups that use the parity-split MVM, in one of its shapes (clusters of
// kParRanks CTAs); otherwise 256 threads and two CTAs per SM.
template <class C, int PAR> __host__ __device__ constexpr int inner_threads() {
    return PAR == PAR_NONE ? kInnerThreads : par_threads<C, PAR>();
}
template <class C, int PAR>
__global__ void __launch_bounds__((inner_threads<C, PAR>()), (PAR == PAR_NONE ? 2 : par_ctas<C, PAR>()))
    k_inner(const InnerGroup<C>* groups, const int2* work, int nwork, int* next, double tol, int maxit, const C* tw,
            int* units) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);
    __shared__ double2 red[2 * (inner_threads<C, PAR>() / 32)];   // per-warp sums
    __shared__ int item;
    cg::cluster_group cl = cg::this_cluster();
    if (threadIdx.x == 0) team_slot = 0;
    __syncthreads();
    for (;;) {
        // rank 0 of the cluster takes the next block; every rank reads it from rank 0's shared memory
        if (cl.block_rank() == 0 && threadIdx.x == 0) item = atomicAdd(next, 1);
        cl.sync();
        const int it = *cl.map_shared_rank(&item, 0);
        cl.sync();
        if (it >= nwork) break;
        const int2 wk = work[it];
        // descriptor in shared memory: fields are reloaded after barriers instead of held in registers
        __shared__ InnerGroup<C> gsh;
        if (threadIdx.x == 0) {
            gsh = groups[wk.x];
            if (gsh.Gb) {
                gsh.G = gsh.Gb[wk.y];
                gsh.Gq = gsh.Gb[wk.y];
            }
        }
        __syncthreads();
        solve_dispatch<PAR>(gsh, wk.y, gsh.tols ? gsh.tols[wk.y] : tol, maxit, sm, tw, red, units);
        __syncthreads();
    }
}

// ---------------------------------------------------------------- host side
static int lg2(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

constexpr size_t kInnerSmemBudget = 96 * 1024;

// CTAs per block (thread-block cluster size) forced by the environment variable
// VIE_INNER_CLUSTER (1, 2, 4 or 8; read once), or 0 when unset.
int inner_cluster_forced() {
    static const int r = [] {
        const char* e = getenv("VIE_INNER_CLUSTER");
        int v = e ? atoi(e) : 0;
        return (v == 1 || v == 2 || v == 4 || v == 8) ? v : 0;
    }();
    return r;
}

// Tiles for one group; false when a single plane does not fit the budget.
static bool inner_tiles(const BoxSet& bs, size_t es, int* lpt, int* ltc, size_t* smem) {
    const size_t pe = (size_t)bs.My * (bs.Mx + 1) * es;
    if (pe > kInnerSmemBudget) return false;
    int l = 0;
    while (((size_t)2 << l) * pe <= kInnerSmemBudget && (1 << (l + 1)) <= 3 * bs.bz * 2 && l < 6) ++l;
    while ((size_t)(1 << l) * pe > kInnerSmemBudget) --l;
    int t = 0;
    while ((size_t)bs.Mz * 3 * ((size_t)2 << t) * es <= kInnerSmemBudget && ((int64_t)2 << t) <= (int64_t)bs.Mx * bs.My &&
           t < 7)
        ++t;
    *lpt = l;
    *ltc = t;
    *smem = std::max((size_t)(1 << l) * pe, (size_t)bs.Mz * 3 * ((size_t)1 << t) * es);
    return true;
}

// m and s of FastDiv for divisor d >= 1: s = ceil(log2 d), m = floor(2^32 (2^s - d) / d) + 1.
static void make_fastdiv(unsigned d, unsigned (&out)[3]) {
    unsigned sh = 0;
    while ((1ull << sh) < d) ++sh;
    unsigned long long m = (((1ull << 32) * ((1ull << sh) - d)) / d) + 1;
    out[0] = (unsigned)m;
    out[1] = sh;
    out[2] = d;
}


// Smallest transform length of the parity-split MVM that holds an extent of b voxels, 0 when none does.
int par_len(int b) {
    for (int h : {2, 4, 6, 8, 10, 12, 16})
        if (b <= h) return h;
    return 0;
}
int par_least(int h) { return par_lo(h) + 1; }
// dynamic shared memory of the parity-split solver: 227 KB less its static part
constexpr size_t kParSmemLimit = 218 * 1024;
bool par_path_ok(const BoxSet& bs) { return par_len(bs.bx) && par_len(bs.by) && par_len(bs.bz); }

bool inner_persistent_ok(const BoxSet& bs, size_t es, bool force) {
    int a, b;
    size_t s;
    return par_path_ok(bs) || ((force || bs.nb >= kInnerMinBlocks) && inner_tiles(bs, es, &a, &b, &s));
}

// FP64 instructions per thread of an H-point transform (dft_small.cuh)
static double dft_ops(int h) {
    return h == 2 ? 4 : h == 4 ? 16 : h == 6 ? 44 : h == 8 ? 56 : h == 10 || h == 12 ? 112 : 168;
}
static int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Microseconds of a complex128 iteration of one block in the parity-split solver: the FP64 instructions of the
// fullest SM quarter (rows of a warp pair, y columns, z columns with the vector updates) over two products, at 64
// clocks each. Within 10 % of the measured time from 4 x 16 x 4 (89 us) to 16 x 16 x 16 voxels (900 us).
static double par_iter_us(const ParClass& c) {
    const double row = ceil_div(ceil_div(c.hz * c.hy, 32), 2) * (6 * dft_ops(c.hx) + 60.0 * c.hx);
    const double y = ceil_div(3 * c.hz * c.ex, 128) * (2 * dft_ops(c.hy) + 8.0 * c.hy);
    const double z = ceil_div(3 * c.ex * c.ey, 512) * (4 * dft_ops(c.hz) + 50.0 * c.hz);
    return std::max(40.0, 0.07 * (row + y + z));
}

// Groups of boxes of at most 16 voxels per axis, by the time of an iteration of all their blocks.
// complex64: the parity-split solver is the fastest way at every number of blocks from 3 x 3 x 3 voxels up (1 to 512
// blocks of 28 shapes). Boxes of up to 128 padded points (2 x 2 x 2, 16 x 1 x 1) use little of a cluster: once
// they outnumber the 152 clusters in flight, one CTA each in the shared-memory passes is faster (4096 blocks of one
// voxel 0.43 against 1.16 ms, 1024 of 2 x 2 x 2 0.34 against 0.69).
// complex128 is bound by the FP64 units, so what counts is how many SMs work:
//   parity-split  38 blocks at a time, each on 4 SMs, no padding: par_iter_us, longer from 48 blocks on;
//   batched       every SM, on padded boxes, a group after the other: 75 us, at least 120, plus per
//                 block 0.1 us and 0.51 (rows of more than 12 voxels) or 0.66 us per 1000 padded points;
//   passes        one CTA per block on padded boxes, 150 at a time: 40 us + 0.13 per padded point.
// The factors are fitted to 28 shapes at 1 to 512 blocks, with equal iterations and converged: the chosen way takes
// 3 % more than the fastest of the three on average, and more than 4 % longer than both the parity-split solver and
// the solver that came before it in none of them. (One 12 x 12 x 16 block 15.3 -> 4.3 ms, 1024 of 4 x 4 x 4
// 12.3 -> 3.1, 256 of 16 x 16 x 2 16.6 -> 7.2.)
void choose_block_paths(std::vector<Group>& groups, int prec, bool batched) {
    const double per_wave = 38.0;
    int nsmall = 0;
    const int64_t small_points = prec == 1 ? 128 : 2048;
    auto small = [&](const Group& g) { return !g.par.empty() && g.bs.spec_elems() <= small_points; };
    for (const Group& g : groups)
        if (small(g)) nsmall += g.bs.nb;
    double t_par_block = 0.0, t_par_sum = 0.0, t_batched = 0.0;
    for (Group& g : groups) {
        if (g.par.empty()) continue;
        g.path[prec] = PATH_PAR;
        if (prec == 1) {
            if (small(g) && nsmall > 152) g.path[prec] = PATH_PASSES;
            continue;
        }
        const double points = (double)g.bs.spec_elems();
        const double tb = std::max(120.0, 75.0 + g.bs.nb * (0.1 + (g.bs.bx > 12 ? 5.1e-4 : 6.6e-4) * points));
        double tp = 0.0, sum = 0.0;
        for (const ParClass& c : g.par) {
            tp = std::max(tp, par_iter_us(c));
            sum += par_iter_us(c) * (double)c.boxes.size();
        }
        const double ts = (40.0 + 0.13 * points) * std::max(1.0, nsmall / 150.0);
        if (small(g) && ts < 1.2 * std::min(tp * std::ceil(nsmall / per_wave), batched ? 1.1 * tb : 1e30)) {
            g.path[prec] = PATH_PASSES;
            continue;
        }
        t_par_block = std::max(t_par_block, tp);
        t_par_sum += sum;
        t_batched += tb;
    }
    if (batched && 1.1 * t_batched < std::max(t_par_block, 0.85 * t_par_sum / per_wave))
        for (Group& g : groups)
            if (!g.par.empty() && g.path[prec] == PATH_PAR) g.path[prec] = PATH_BATCHED;
}

template <class C>
int inner_persistent(const std::vector<InnerJob<C>>& jobs, const int2* d_work, int nwork, int nsingle, void* d_groups,
                     int* d_next, double tol, int maxit, cudaStream_t s, int cluster, const InnerSplit* split) {
    if (jobs.empty() || nwork == 0) return VIE_OK;
    Twiddles tw;
    VIE_TRY(get_twiddles(&tw));
    std::vector<InnerGroup<C>> hg(jobs.size());
    size_t smem = 0, single_smem = 0;
    bool any_par = false, any_pass = false;         // among the jobs that are not single-CTA ones
    int par_points = 0;                             // of the largest parity-split box
    size_t chip_smem = 0;
    for (size_t i = 0; i < jobs.size(); ++i) {
        const InnerJob<C>& j = jobs[i];
        const BoxSet& bs = *j.bs;
        InnerGroup<C>& g = hg[i];
        g.b = j.v.b; g.x = j.v.x; g.r = j.v.r; g.rhat = j.v.rhat; g.p = j.v.p; g.v = j.v.v; g.s = j.v.s; g.t = j.v.t;
        g.w2 = reinterpret_cast<C*>(bs.w2);
        g.chi = j.chi;
        g.mask = bs.mask;
        g.G = j.G;
        g.Gb = j.Gb;
        g.tols = j.tols;
        g.st = j.st;
        g.nb = bs.nb; g.bx = bs.bx; g.by = bs.by; g.bz = bs.bz;
        g.Mx = bs.Mx; g.My = bs.My; g.Mz = bs.Mz; g.lx = bs.lx; g.ly = bs.ly; g.lz = bs.lz;
        g.lyb = lg2(bs.by);
        size_t sm = 0;
        g.par = j.hx > 0 ? 1 : 0;
        if (g.par) {
            any_par = true;
            g.ex = j.ex; g.ey = j.ey; g.ez = j.ez;
            g.hx = j.hx; g.hy = j.hy; g.hz = j.hz;
            g.yp = j.ex | 1;
            g.Gq = j.Gq;
            make_fastdiv((unsigned)g.ex, g.fd_ex);
            make_fastdiv((unsigned)(g.ex * g.ey), g.fd_exy);
            make_fastdiv((unsigned)g.hy, g.fd_hy);
            par_points = std::max(par_points, g.hx * g.hy * g.hz);
            sm = (size_t)par_data_elems(g) * sizeof(C) + (sizeof(C) == 8 ? (size_t)par_rank_spec(g) * sizeof(C) : 0);
            chip_smem = std::max(chip_smem, (size_t)(par_data_elems(g) + par_rank_spec(g)) * sizeof(C) +
                                                (size_t)((3 * g.ez * g.ey * g.ex + kParRanks - 1) / kParRanks) *
                                                    par_chip_bytes<C>());
        } else if (!inner_tiles(bs, sizeof(C), &g.lpt, &g.ltc, &sm)) {
            return fail(VIE_EINVAL, "box too large for the persistent solver");
        }
        // algorithmic bytes of one MVM with its fused vector work: plane spectra written, read and
        // rewritten along z, read back (4 x [3][bz][My][Mx]), the Green spectrum once, chi and mask,
        // and the 4 box vectors the fused update/inverse phases touch; the x/r pass moves 6 vectors.
        const int64_t es = sizeof(C), box = bs.box_elems();
        const int64_t w2b = 3LL * bs.bz * bs.My * bs.Mx * es;
        // parity-split MVM (merged BiCGSTAB): an iteration's two MVMs and fused passes move 17 box vectors
        const int64_t own = (int64_t)j.ex * j.ey * j.ez, oct = (int64_t)(j.hx + 1) * (j.hy + 1) * (j.hz + 1);
        const int64_t mvm = g.par ? 6 * oct * es + own * (es + 1) + 17 * 3 * own * es / 2
                                  : 4 * w2b + 6LL * bs.spec_elems() * es + box * (es + 1) + 4 * 3 * box * es;
        g.kb_mvm = (int)((mvm + 1023) / 1024);
        g.kb_upd = (int)((6 * 3 * box * es + 1023) / 1024);
        any_pass = any_pass || (!g.par && !j.single);
        (j.single ? single_smem : smem) = std::max(j.single ? single_smem : smem, sm);
    }
    const int nmain = nwork - nsingle;
    if (any_par) VIE_TRY(par_twiddles_ready());
    VIE_CK(cudaMemcpyAsync(d_groups, hg.data(), hg.size() * sizeof(InnerGroup<C>), cudaMemcpyHostToDevice, s));
    const bool two = !any_par && nsingle == 0 && split != nullptr && split->nheavy > 0 && split->nheavy < nwork &&
                     !inner_cluster_forced();
    VIE_CK(cudaMemsetAsync(d_next, 0, (two || (nsingle > 0 && nmain > 0) ? 2 : 1) * sizeof(int), s));
    // Shape of a launch with parity-split jobs (complex64). On chip while few blocks queue: a block's own iterations
    // then set the time more than the rate does. How many waves of its 38 clusters may queue depends on the points of
    // a box (one up to 256, two up to 1024, 2.75 above: 96 blocks of 12 x 12 x 16 1.25 ms on chip, 1.47 in the L2 shape;
    // 114 blocks 1.51 and 1.44; 48 blocks of 4 x 4 x 4 0.16 and 0.11). Then the small shape up to 1024 points, L2 above.
    // With boxes over 16 voxels among them three waves on chip, then L2.
    const double waves = any_pass ? 3.0 : par_points <= 256 ? 1.0 : par_points <= 1024 ? 2.0 : 2.75;
    const bool chip = any_par && sizeof(C) == 8 && chip_smem <= kParSmemLimit && nmain <= waves * 38;
    const bool small = any_par && sizeof(C) == 8 && !chip && !any_pass && par_points <= 1024;
    if (chip) smem = std::max(smem, chip_smem);
    auto kern = k_inner<C, PAR_NONE>;
    int threads = kInnerThreads;
    if (chip) {
        if constexpr (sizeof(C) == 8) kern = k_inner<C, PAR_CHIP>;
        threads = par_threads<C, PAR_CHIP>();
    } else if (small) {
        if constexpr (sizeof(C) == 8) kern = k_inner<C, PAR_SMALL>;
        threads = par_threads<C, PAR_SMALL>();
    } else if (any_par) {
        kern = k_inner<C, PAR_L2>;
        threads = par_threads<C, PAR_L2>();
    }
    // one block per cluster of R CTAs; as many clusters as fit at once, pulling blocks from the queue
    auto launch = [&](const int2* work, int n, int* next, int R, cudaStream_t st, int* units) -> int {
        // whatever the size: the default 48 KB limit also counts the static shared memory
        VIE_TRY(raise_dynamic_smem(reinterpret_cast<const void*>(kern), smem));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = R;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(R);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nclusters = 0;
        VIE_CK(cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg));
        if (nclusters < 1) return fail(VIE_EINVAL, "block solver: no cluster of this size fits on the device");
        cfg.gridDim = dim3(std::max(1, std::min(n, nclusters)) * R);
        cudaError_t le = cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<const InnerGroup<C>*>(d_groups), work, n,
                                            next, tol, maxit, tw_of<C>(tw), units);
        if (le != cudaSuccess) return cuda_fail(le, "cudaLaunchKernelEx(k_inner)", __FILE__, __LINE__);
        return VIE_OK;
    };
    const int R = any_par ? kParRanks : inner_cluster_forced() ? inner_cluster_forced() : (cluster > 0 ? cluster : 2);
    // the kernels add the KB they move (per MVM) to one profiling counter; the profiled interval
    // covers both parts of a split launch
    int* units = prof_begin(s, PK_INNER, sizeof(C) == 16 ? VIE_C128 : VIE_C64, 1024, 0, true);
    int rc = VIE_OK;
    if (!two) {
        if (nmain > 0) rc = launch(d_work, nmain, d_next, R, s, units);
        if (!rc && nsingle > 0) {
            kern = k_inner<C, PAR_NONE>;
            threads = kInnerThreads;
            smem = single_smem;
            rc = launch(d_work + nmain, nsingle, d_next + (nmain > 0 ? 1 : 0),
                        inner_cluster_forced() ? inner_cluster_forced() : 1, s, units);
        }
    } else {
        // the heavy part first, so its clusters are resident before the light part fills the GPU
        cudaError_t e = cudaEventRecord(split->fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(split->s2, split->fork, 0);
        if (e != cudaSuccess) rc = cuda_fail(e, "split launch fork", __FILE__, __LINE__);
        if (!rc) rc = launch(d_work, split->nheavy, d_next, split->cluster, s, units);
        if (!rc) rc = launch(d_work + split->nheavy, nwork - split->nheavy, d_next + 1, R, split->s2, units);
        e = cudaEventRecord(split->join, split->s2);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, split->join, 0);
        if (!rc && e != cudaSuccess) rc = cuda_fail(e, "split launch join", __FILE__, __LINE__);
    }
    prof_end(s);
    if (rc) return rc;
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

template int inner_persistent<double2>(const std::vector<InnerJob<double2>>&, const int2*, int, int, void*, int*, double,
                                       int, cudaStream_t, int, const InnerSplit*);
template int inner_persistent<float2>(const std::vector<InnerJob<float2>>&, const int2*, int, int, void*, int*, double, int,
                                      cudaStream_t, int, const InnerSplit*);

// ---------------------------------------------------------------- spectra of the parity-split MVM
// One axis of the real-to-frequency transform of the kernel's octant: sum over offsets |d| < n of
// K(d) exp(-i pi f d / H) for f in [0, H], with K even (K(0) + 2 sum K(d) cos) or odd (-2i sum K(d) sin)
// along the axis, as component c is. AXIS 0: x, from K itself ([c][z][y][x], strides of the padded
// array); 1: y; 2: z, into the layout of the block solver.
struct ParAxis {
    int hx, hy, hz;          // transform lengths
    int nx, ny, nz;          // offsets of each axis (rows beyond them are never read)
    double scale;            // normalisation of the inverse transforms over that of K
    int64_t t1, t2;          // first element of this spectrum in the temporaries of pass x and y
    double2* o128;
    float2* o64;
};
constexpr int kParSetMax = 27;   // lengths 10, 12 or 16 on each axis
struct ParAxisSet {
    ParAxis a[kParSetMax];
};
template <int AXIS>
__global__ void k_par_axis(const double2* __restrict__ in, double2* out, int64_t sy, int64_t sz, int64_t sc, ParAxisSet set) {
    const ParAxis a = set.a[blockIdx.y];
    const int H = AXIS == 0 ? a.hx : AXIS == 1 ? a.hy : a.hz, na = AXIS == 0 ? a.nx : AXIS == 1 ? a.ny : a.nz;
    __shared__ double2 tw[32];                      // exp(-i pi j / H), j < 2H
    if ((int)threadIdx.x < 2 * H) {
        double sn, cs;
        sincospi((double)threadIdx.x / H, &sn, &cs);
        tw[threadIdx.x] = make_double2(cs, -sn);
    }
    __syncthreads();
    if (AXIS > 0) in += AXIS == 1 ? a.t1 : a.t2;
    if (AXIS < 2) out += AXIS == 0 ? a.t1 : a.t2;
    const int nx = a.hx + 1, ny = AXIS == 0 ? a.hy : a.hy + 1, nz = AXIS == 2 ? a.hz + 1 : a.hz;
    const int total = 6 * nz * ny * nx;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int fx = t % nx, y = (t / nx) % ny, z = (t / (nx * ny)) % nz, c = t / (nx * ny * nz);
        if ((AXIS == 0 && y >= a.ny) || (AXIS < 2 && z >= a.nz)) continue;
        const bool odd = AXIS == 0 ? (c == 1 || c == 2) : AXIS == 1 ? (c == 1 || c == 4) : (c == 2 || c == 4);
        const int f = AXIS == 0 ? fx : AXIS == 1 ? y : z;
        const double2* p;
        int64_t st;
        if (AXIS == 0) { p = in + c * sc + z * sz + y * sy; st = 1; }
        else if (AXIS == 1) { p = in + ((int64_t)(c * a.hz + z) * a.hy) * nx + fx; st = nx; }
        else { p = in + ((int64_t)c * a.hz * ny + y) * nx + fx; st = (int64_t)ny * nx; }
        double2 s = odd ? make_double2(0.0, 0.0) : p[0];
        for (int d = 1; d < na; ++d) {
            const double2 w = tw[(f * d) % (2 * H)], k = p[d * st];
            // even: 2 K cos; odd: -2i K sin (w.y = -sin)
            if (odd) s = make_double2(s.x - 2.0 * w.y * k.y, s.y + 2.0 * w.y * k.x);
            else s = make_double2(s.x + 2.0 * w.x * k.x, s.y + 2.0 * w.x * k.y);
        }
        if (AXIS == 0) s = make_double2(s.x * a.scale, s.y * a.scale);
        if (AXIS < 2) {
            out[t] = s;
        } else {
            // frequency k = 2m + parity, folded to [0, H]: entry index m of its parity
            const int pz = z & 1, py = y & 1, iz = z >> 1, iy = y >> 1;
            const int my = a.hy / 2 + 1, mz = a.hz / 2 + 1;
            const int64_t o = ((((int64_t)(2 * pz + py) * nx + fx) * 6 + c) * mz + iz) * my + iy;
            if (a.o128) a.o128[o] = s;
            if (a.o64) a.o64[o] = make_float2((float)s.x, (float)s.y);
        }
    }
}

int64_t par_spectrum_elems(int hx, int hy, int hz) { return 4LL * (hx + 1) * 6 * (hz / 2 + 1) * (hy / 2 + 1); }

// K: lattice samples of the box set's shape (green_octant: [6][bz][by][bx], scaled by 1 / (Mx My Mz)); fills
// the spectra of `out`, all of them in one launch per axis.
int par_spectra(const BoxSet& bs, const double2* K, const std::vector<ParSpec>& out, cudaStream_t s) {
    if (out.empty()) return VIE_OK;
    if ((int)out.size() > kParSetMax) return fail(VIE_EINVAL, "par_spectra: too many classes");
    ParAxisSet set{};
    int64_t n1 = 0, n2 = 0, m1 = 0, m2 = 0, m3 = 0;
    for (size_t k = 0; k < out.size(); ++k) {
        const ParSpec& p = out[k];
        ParAxis& a = set.a[k];
        a.hx = p.hx; a.hy = p.hy; a.hz = p.hz;
        a.nx = std::min(p.hx, bs.bx); a.ny = std::min(p.hy, bs.by); a.nz = std::min(p.hz, bs.bz);
        a.scale = (double)bs.spec_elems() / (8.0 * p.hx * p.hy * p.hz);
        a.t1 = n1; a.t2 = n2;
        a.o128 = p.g128; a.o64 = p.g64;
        const int64_t e1 = 6LL * p.hz * p.hy * (p.hx + 1), e2 = 6LL * p.hz * (p.hy + 1) * (p.hx + 1);
        n1 += e1;
        n2 += e2;
        m1 = std::max(m1, e1);
        m2 = std::max(m2, e2);
        m3 = std::max<int64_t>(m3, 6LL * (p.hz + 1) * (p.hy + 1) * (p.hx + 1));
    }
    double2* tmp = nullptr;
    VIE_CK(cudaMallocAsync((void**)&tmp, (n1 + n2) * sizeof(double2), s));
    const int64_t es = sizeof(double2), sy = bs.bx, sz = (int64_t)bs.bx * bs.by, sc = bs.box_elems();
    auto grid = [&](int64_t n) { return dim3((unsigned)((n + 127) / 128), (unsigned)out.size()); };
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 2 * n1 * es, false);
    k_par_axis<0><<<grid(m1), 128, 0, s>>>(K, tmp, sy, sz, sc, set);
    prof_end(s);
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 2 * n2 * es, false);
    k_par_axis<1><<<grid(m2), 128, 0, s>>>(tmp, tmp + n1, sy, sz, sc, set);
    prof_end(s);
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 2 * n2 * es, false);
    k_par_axis<2><<<grid(m3), 128, 0, s>>>(tmp + n1, nullptr, sy, sz, sc, set);
    prof_end(s);
    const cudaError_t le = cudaGetLastError(), e = cudaFreeAsync(tmp, s);
    if (le != cudaSuccess) return cuda_fail(le, "k_par_axis launch", __FILE__, __LINE__);
    VIE_CK(e);
    return VIE_OK;
}

size_t inner_group_desc_bytes() { return std::max(sizeof(InnerGroup<double2>), sizeof(InnerGroup<float2>)); }

}  // namespace vie

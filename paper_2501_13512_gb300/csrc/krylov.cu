// Batched BiCGSTAB building blocks (Section II.B; van der Vorst's method, ref. [18]).
//
// A "segment" is one independent linear system: the outer system (one
// segment, the whole grid) or one diagonal block A_k of Eq. 10 (one segment
// per block, all blocks of a group stored back to back). Every kernel runs a
// 2D grid (CTAs within a segment) x (segments); each segment's scalars live in
// a SegState on the device, so the host never reads rho, alpha or omega.
//
// Reductions: each CTA writes its partial sums, and the last CTA of the
// segment to arrive (atomic ticket) adds all partials in a fixed order and
// applies the scalar update, so results are deterministic. Complex64 vectors
// are multiplied and summed in FP32 within a thread and in FP64 across
// threads; complex128 vectors use FP64 throughout. Scalars are FP64.
//
// On short segments these kernels are bound by FP64 instructions (two lanes a
// clock and SM, whole warps whatever their active lanes), not by memory: so
// only the sums an operation has are reduced, halved over the lanes, and every
// coefficient is computed once, by the thread that finishes the sum (with
// beta formed by every thread of the p update and 20 additions per warp and
// sum, 13 to 18 us a launch for 8 segments of 24^3 voxels). The sum <rhat, r>
// rides in the x/r update, so an iteration takes five launches beside its
// products.
#include <math.h>

#include "vie_internal.cuh"

namespace vie {

constexpr int kRedThreads = 256;

enum VecOp { OP_INIT = 0, OP_P, OP_S, OP_XHALF, OP_XR, OP_SIGMA, OP_OMEGA };
// real sums of an operation
__host__ __device__ constexpr int op_sums(int op) {
    return op == OP_INIT || op == OP_S ? 1 : op == OP_SIGMA ? 2 : op == OP_XR || op == OP_OMEGA ? 3 : 0;
}

template <class C> struct VecArgs {
    KrylovVecs<C> v;
    SegState* st;
    double2* part;      // [nseg][maxcta][2]
    unsigned* count;    // [nseg]
    int* n_active;
    int64_t seglen;
    int maxcta;
    double tol;
    int maxit;
    int* units;         // profiling: active segments processed
    const double* tols; // optional per-segment relative tolerance (OP_INIT)
};

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double r = 1.0 / (b.x * b.x + b.y * b.y);
    return make_double2((a.x * b.x + a.y * b.y) * r, (a.y * b.x - a.x * b.y) * r);
}
__device__ __forceinline__ float2 to_c64(double2 a) { return make_float2((float)a.x, (float)a.y); }
__device__ __forceinline__ bool cfinite_nz(double2 a) {
    return isfinite(a.x) && isfinite(a.y) && (a.x != 0.0 || a.y != 0.0);
}

// conj(a) * b accumulated into acc (same precision as the vectors)
template <class C> __device__ __forceinline__ void cdot_acc(C& acc, C a, C b) {
    acc.x = fma(a.y, b.y, fma(a.x, b.x, acc.x));
    acc.y = fma(-a.y, b.x, fma(a.x, b.y, acc.y));
}
template <class C> __device__ __forceinline__ C coef(double2 a, float2 a32);
template <> __device__ __forceinline__ double2 coef<double2>(double2 a, float2) { return a; }
template <> __device__ __forceinline__ float2 coef<float2>(double2, float2 a32) { return a32; }

// Block sums of NV (1, 2 or 4) values of every thread; the total of value i is returned to thread i.
template <int NV> __device__ double block_sums(double (&x)[NV]) {
    constexpr int NW = kRedThreads / 32, LG = NV == 4 ? 2 : NV - 1;   // log2 NV
    __shared__ double sh[NV][NW];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (l & o) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double send = up ? x[k] : x[k + h], keep = up ? x[k + h] : x[k];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
    // the lane's value index: its upper log2 NV bits
    if ((l & (31 >> LG)) == 0) sh[l >> (5 - LG)][w] = x[0];
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        if (l < NV * NW) t = sh[l / NW][l % NW];
#pragma unroll
        for (int m = 1; m < NW; m <<= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
        t = __shfl_sync(0xffffffffu, t, (l & (NV - 1)) * NW);
    }
    __syncthreads();
    return t;
}

__device__ __forceinline__ void leave_active(int* n_active) { atomicSub(n_active, 1); }

// Scalar update of one segment, run by thread 0 of the last CTA.
template <int OP>
__device__ void finalize(SegState& s, double2 d1, double2 d2, int* n_active, double tol, int maxit) {
    // (tol already resolved per segment by the caller)
    if (OP == OP_INIT) {
        s.bnorm2 = d1.x;
        s.tol2 = tol * tol * d1.x;
        s.res2 = d1.x;
        s.rho = make_double2(d1.x, 0.0);        // <rhat, r> with rhat = r = b
        s.alpha = s.omega = make_double2(1.0, 0.0);
        s.alpha32 = s.omega32 = make_float2(1.f, 0.f);
        s.beta = make_double2(0.0, 0.0);        // p = v = 0 before the first p update
        s.beta32 = make_float2(0.f, 0.f);
        s.iters = 0.0;
        s.maxit = maxit;
        if (!isfinite(d1.x)) {
            s.status = SEG_BREAKDOWN;
        } else if (d1.x == 0.0 || d1.x <= s.tol2) {   // x0 already meets the tolerance (tol >= 1)
            s.status = SEG_CONVERGED;
        } else {
            s.status = SEG_ACTIVE;
            atomicAdd(n_active, 1);
        }
    } else if (OP == OP_SIGMA) {
        if (!cfinite_nz(d1)) { s.status = SEG_BREAKDOWN; leave_active(n_active); }
        else {
            s.alpha = cdiv(s.rho, d1);
            s.alpha32 = to_c64(s.alpha);
        }
    } else if (OP == OP_OMEGA) {
        if (!(d2.x > 0.0) || !isfinite(d2.x) || !isfinite(d1.x) || !isfinite(d1.y)) {
            s.status = SEG_BREAKDOWN;
            leave_active(n_active);
        } else {
            const double r = 1.0 / d2.x;
            s.omega = make_double2(d1.x * r, d1.y * r);
            s.omega32 = to_c64(s.omega);
        }
    } else if (OP == OP_S) {
        s.res2 = d1.x;
        if (!isfinite(d1.x)) { s.status = SEG_BREAKDOWN; leave_active(n_active); }
        else if (d1.x <= s.tol2) { s.status = SEG_HALF_PENDING; s.iters += 0.5; leave_active(n_active); }
    } else if (OP == OP_XHALF) {
        s.status = SEG_CONVERGED;
    } else if (OP == OP_XR) {                   // d1 = <rhat, r>, d2.x = ||r||^2
        s.res2 = d2.x;
        s.iters += 1.0;
        if (!isfinite(d2.x)) { s.status = SEG_BREAKDOWN; leave_active(n_active); }
        else if (d2.x <= s.tol2) { s.status = SEG_CONVERGED; leave_active(n_active); }
        else if (s.iters >= (double)s.maxit) { s.status = SEG_MAXIT; leave_active(n_active); }
        else if ((s.omega.x == 0.0 && s.omega.y == 0.0) || !cfinite_nz(d1)) { s.status = SEG_BREAKDOWN; leave_active(n_active); }
        else {
            // beta = (rho / rho_prev) (alpha / omega)
            s.beta = cdiv(cmul(d1, s.alpha), cmul(s.rho, s.omega));
            s.beta32 = to_c64(s.beta);
            s.rho = d1;
        }
    }
}

// One fused pass over a segment: vector update and/or up to two inner products.
template <class C, int OP>
__global__ void __launch_bounds__(kRedThreads) k_bicg(VecArgs<C> a) {
    pdl_wait();
    const int seg = blockIdx.y;
    SegState& S = a.st[seg];
    if (OP != OP_INIT) {
        const int need = (OP == OP_XHALF) ? SEG_HALF_PENDING : SEG_ACTIVE;
        if (S.status != need) return;       // same value for every CTA of the segment
    }
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    const int64_t off = (int64_t)seg * a.seglen;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    constexpr int U = 4;                        // elements per thread whose loads are issued together
    C acc1 = czero<C>(), acc2 = czero<C>();
    const C alpha = coef<C>(S.alpha, S.alpha32), omega = coef<C>(S.omega, S.omega32), beta = coef<C>(S.beta, S.beta32);
    const KrylovVecs<C> v = a.v;
    // vectors read by the operation, in order of the argument list of apply
    const C* in0 = OP == OP_INIT ? v.b : OP == OP_P || OP == OP_S ? v.r : OP == OP_XHALF || OP == OP_XR ? v.x
                   : OP == OP_SIGMA ? v.rhat : v.t;
    const C* in1 = OP == OP_P ? v.p : OP == OP_S || OP == OP_SIGMA ? v.v : OP == OP_XHALF || OP == OP_XR ? v.y : v.s;
    const C* in2 = OP == OP_P ? v.v : v.z;
    constexpr int NIN = OP == OP_INIT ? 1 : OP == OP_P ? 3 : OP == OP_XR ? 6 : 2;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < a.seglen; i0 += U * stride) {
        C x[U][NIN];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * stride, k = off + (i < a.seglen ? i : i0);
            x[u][0] = in0[k];
            if constexpr (NIN > 1) x[u][1] = in1[k];
            if constexpr (NIN > 2) x[u][2] = in2[k];
            if constexpr (NIN == 6) {
                x[u][3] = v.s[k];
                x[u][4] = v.t[k];
                x[u][5] = v.rhat[k];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * stride, k = off + i;
            if (i >= a.seglen) break;
            if constexpr (OP == OP_INIT) {
                const C b = x[u][0];
                v.x[k] = czero<C>();
                v.r[k] = b;
                v.rhat[k] = b;
                v.p[k] = czero<C>();
                v.v[k] = czero<C>();
                cdot_acc(acc1, b, b);
            } else if constexpr (OP == OP_P) {
                v.p[k] = x[u][0] + cmul(beta, x[u][1] - cmul(omega, x[u][2]));
            } else if constexpr (OP == OP_S) {
                const C s = x[u][0] - cmul(alpha, x[u][1]);
                v.s[k] = s;
                cdot_acc(acc1, s, s);
            } else if constexpr (OP == OP_XHALF) {
                v.x[k] = x[u][0] + cmul(alpha, x[u][1]);
            } else if constexpr (OP == OP_XR) {
                v.x[k] = x[u][0] + cmul(alpha, x[u][1]) + cmul(omega, x[u][2]);
                const C r = x[u][3] - cmul(omega, x[u][4]);
                v.r[k] = r;
                cdot_acc(acc1, x[u][5], r);
                cdot_acc(acc2, r, r);
            } else if constexpr (OP == OP_SIGMA) {
                cdot_acc(acc1, x[u][0], x[u][1]);
            } else {
                cdot_acc(acc1, x[u][0], x[u][1]);
                cdot_acc(acc2, x[u][0], x[u][0]);
            }
        }
    }
    if constexpr (OP == OP_P) return;
    constexpr int NV = op_sums(OP) == 3 ? 4 : op_sums(OP) == 0 ? 1 : op_sums(OP);
    double d[NV], t = 0.0;
    d[0] = (double)acc1.x;
    if constexpr (NV > 1) d[1] = (double)acc1.y;
    if constexpr (NV == 4) {
        d[2] = (double)acc2.x;
        d[3] = 0.0;
    }
    if constexpr (op_sums(OP) > 0) t = block_sums(d);
    double* part = reinterpret_cast<double*>(a.part + (int64_t)seg * a.maxcta * 2);
    __shared__ bool last;
    if (threadIdx.x < NV) {
        part[4 * blockIdx.x + threadIdx.x] = t;
        __threadfence();
    }
    __syncwarp();
    if (threadIdx.x == 0) last = atomicAdd(&a.count[seg], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // fixed-order sum of the partials of this segment
    if constexpr (op_sums(OP) > 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
            d[i] = threadIdx.x < gridDim.x ? __ldcg(part + 4 * threadIdx.x + i) : 0.0;
        t = block_sums(d);
    }
    if (threadIdx.x < 32) {
        const double t0 = __shfl_sync(0xffffffffu, t, 0), t1 = __shfl_sync(0xffffffffu, t, 1 % NV),
                     t2 = __shfl_sync(0xffffffffu, t, 2 % NV);
        if (threadIdx.x == 0) {
            a.count[seg] = 0;
            finalize<OP>(S, make_double2(t0, NV > 1 ? t1 : 0.0), make_double2(NV == 4 ? t2 : 0.0, 0.0), a.n_active,
                         a.tols ? a.tols[seg] : a.tol, a.maxit);
        }
    }
}

template <class C>
static int launch_bicg(Bicg<C>& k, int op, double tol, int maxit, cudaStream_t s, const double* tols = nullptr) {
    VecArgs<C> a;
    a.tols = tols;
    a.v = k.v;
    a.st = k.st;
    a.part = k.red->part;
    a.count = k.red->count;
    a.n_active = k.red->n_active;
    a.seglen = k.seglen;
    a.maxcta = kMaxCtaPerSeg;
    a.tol = tol;
    a.maxit = maxit;
    int64_t want = (k.seglen + (int64_t)kRedThreads * 4 - 1) / ((int64_t)kRedThreads * 4);
    int nct = (int)std::max<int64_t>(1, std::min<int64_t>(want, kMaxCtaPerSeg));
    dim3 grid(nct, k.nseg);
    // vectors touched per segment by each op (reads + writes)
    static const int nvec[] = {6, 4, 3, 3, 8, 2, 2};
    const bool dot = op == OP_SIGMA || op == OP_OMEGA;
    a.units = prof_begin(s, dot ? PK_BICG_DOT : PK_BICG_UPDATE, sizeof(C) == 16 ? VIE_C128 : VIE_C64,
                         (int64_t)nvec[op] * k.seglen * (int64_t)sizeof(C), 0, true);
    auto kern = k_bicg<C, OP_INIT>;
    switch (op) {
        case OP_INIT: break;
        case OP_P: kern = k_bicg<C, OP_P>; break;
        case OP_S: kern = k_bicg<C, OP_S>; break;
        case OP_XHALF: kern = k_bicg<C, OP_XHALF>; break;
        case OP_XR: kern = k_bicg<C, OP_XR>; break;
        case OP_SIGMA: kern = k_bicg<C, OP_SIGMA>; break;
        case OP_OMEGA: kern = k_bicg<C, OP_OMEGA>; break;
        default: prof_end(s); return fail(VIE_EINVAL, "bad BiCGSTAB op");
    }
    const cudaError_t e = launch_dependent(kern, grid, kRedThreads, 0, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C> int bicg_init(Bicg<C>& k, double tol, int maxit, cudaStream_t s) {
    VIE_CK(cudaMemsetAsync(k.red->n_active, 0, sizeof(int), s));
    return launch_bicg(k, OP_INIT, tol, maxit, s);
}
template <class C> int bicg_init_tols(Bicg<C>& k, const double* tols, int maxit, cudaStream_t s) {
    VIE_CK(cudaMemsetAsync(k.red->n_active, 0, sizeof(int), s));
    return launch_bicg(k, OP_INIT, 0.0, maxit, s, tols);
}
template <class C> int bicg_update_p(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_P, 0, 0, s); }
template <class C> int bicg_sigma(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_SIGMA, 0, 0, s); }
template <class C> int bicg_update_s(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_S, 0, 0, s); }
template <class C> int bicg_x_half(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_XHALF, 0, 0, s); }
template <class C> int bicg_omega(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_OMEGA, 0, 0, s); }
template <class C> int bicg_update_xr(Bicg<C>& k, cudaStream_t s) { return launch_bicg(k, OP_XR, 0, 0, s); }

#define VIE_INST(C)                                                        \
    template int bicg_init<C>(Bicg<C>&, double, int, cudaStream_t);        \
    template int bicg_init_tols<C>(Bicg<C>&, const double*, int, cudaStream_t); \
    template int bicg_update_p<C>(Bicg<C>&, cudaStream_t);                 \
    template int bicg_sigma<C>(Bicg<C>&, cudaStream_t);                    \
    template int bicg_update_s<C>(Bicg<C>&, cudaStream_t);                 \
    template int bicg_x_half<C>(Bicg<C>&, cudaStream_t);                   \
    template int bicg_omega<C>(Bicg<C>&, cudaStream_t);                    \
    template int bicg_update_xr<C>(Bicg<C>&, cudaStream_t);
VIE_INST(double2)
VIE_INST(float2)
#undef VIE_INST

// ---------------------------------------------------------------- plain vector helpers
template <class C>
__global__ void k_copy(const C* a, C* b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = a[i];
}

static unsigned grid_for(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 16));
}

template <class C> int vec_copy(const C* a, C* b, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_FIELD, sizeof(C) == 16 ? VIE_C128 : VIE_C64, 0, 2 * n * (int64_t)sizeof(C), false);
    k_copy<C><<<grid_for(n), 256, 0, s>>>(a, b, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}
template int vec_copy<double2>(const double2*, double2*, int64_t, cudaStream_t);
template int vec_copy<float2>(const float2*, float2*, int64_t, cudaStream_t);

__global__ void k_residual128(const double2* b, const double2* ax, double2* r, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        r[i] = b[i] - ax[i];
}
int vec_residual128(const double2* b, const double2* ax, double2* r, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_FIELD, VIE_C128, 0, 3 * n * 16, false);
    k_residual128<<<grid_for(n), 256, 0, s>>>(b, ax, r, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// ||a||^2 in FP64 into d_out[0] (single segment, deterministic two-level sum).
__global__ void __launch_bounds__(kRedThreads) k_norm2(const double2* a, int64_t n, double2* part, unsigned* count, double* out) {
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = a[i];
        acc[0] = fma(v.y, v.y, fma(v.x, v.x, acc[0]));
    }
    double t = block_sums(acc);
    __shared__ bool last;
    double* pp = reinterpret_cast<double*>(part);
    if (threadIdx.x == 0) {
        pp[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    acc[0] = threadIdx.x < gridDim.x ? __ldcg(pp + threadIdx.x) : 0.0;
    t = block_sums(acc);
    if (threadIdx.x == 0) {
        *count = 0;
        *out = t;
    }
}
int vec_norm2_128(const double2* a, int64_t n, ReduceScratch* red, double* d_out, cudaStream_t s) {
    int64_t want = (n + (int64_t)kRedThreads * 8 - 1) / ((int64_t)kRedThreads * 8);
    int nct = (int)std::max<int64_t>(1, std::min<int64_t>(want, kMaxCtaPerSeg));
    prof_begin(s, PK_FIELD, VIE_C128, 0, n * 16, false);
    k_norm2<<<nct, kRedThreads, 0, s>>>(a, n, red->part, red->count, d_out);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

__global__ void k_sum128(const double2* a, const double2* b, double2* out, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = a[i] + b[i];
}
int vec_sum128(const double2* a, const double2* b, double2* out, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_FIELD, VIE_C128, 0, 3 * n * 16, false);
    k_sum128<<<grid_for(n), 256, 0, s>>>(a, b, out, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// b = a / ||a|| rounded to complex64 (the correction solve's right-hand side).
__global__ void k_scale_to_c64(const double2* a, const double* norm2, float2* b, int64_t n) {
    double inv = 1.0 / sqrt(*norm2);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double2 v = a[i];
        b[i] = make_float2((float)(v.x * inv), (float)(v.y * inv));
    }
}
int vec_scale_to_c64(const double2* a, const double* d_norm2, float2* b, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_FIELD, VIE_C128, 0, n * 24, false);
    k_scale_to_c64<<<grid_for(n), 256, 0, s>>>(a, d_norm2, b, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// x += ||r|| d (FP64 accumulation of a complex64 correction).
__global__ void k_add_scaled_c64(double2* x, const float2* d, const double* norm2, int64_t n) {
    double sc = sqrt(*norm2);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float2 v = d[i];
        double2 xv = x[i];
        x[i] = make_double2(xv.x + sc * (double)v.x, xv.y + sc * (double)v.y);
    }
}
int vec_add_scaled_c64(double2* x, const float2* d, const double* d_norm2, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_FIELD, VIE_C128, 0, n * 40, false);
    k_add_scaled_c64<<<grid_for(n), 256, 0, s>>>(x, d, d_norm2, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

}  // namespace vie

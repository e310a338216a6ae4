// Pencil FFT passes and the FFT-accelerated MVM y = x - G(chi x) (Section I;
// Eq. 4 discretised on the voxel grid).
//
// Every 3D transform is split into three batched 1D passes. Forward passes are
// radix-4 (plus one radix-2) decimation-in-frequency: natural order in,
// bit-reversed order out. Inverse passes are decimation-in-time: bit-reversed
// in, natural out. Intermediate spectra therefore live in bit-reversed
// position order on every axis, and the Green spectrum is generated in the
// same order, so no pass ever reorders data.
//
// One MVM over a batch of boxes (BoxSet; the full grid is the batch of one):
//   pass X  rows of bx -> chi * x, zero-pad to Mx, forward   -> w1 [3][bz][by][Mx]
//   pass Y  columns of by -> zero-pad to My, forward         -> w2 [3][bz][My][Mx]
//   pass Z  columns of bz -> zero-pad to Mz, forward, 3x3 symmetric Green
//           multiply, inverse, keep z < bz                   -> w2 (in place)
//   pass Y' inverse, keep y < by                             -> w1
//   pass X' inverse, keep x < bx, y = x - u (masked)         -> y
// Each pass stages a tile of pencils in shared memory; global accesses are
// along the contiguous x axis in every pass. Most lengths use the two-step
// register transforms of fft_plane.cuh (which also joins x and y of small
// planes) and the z passes below; the radix-4 kernels take the rest.
#include <algorithm>
#include <type_traits>

#include "dft_small.cuh"
#include "fft_core.cuh"
#include "fft_reg.cuh"
#include "vie_internal.cuh"

namespace vie {

constexpr int kThreads = 256;
constexpr int kSmemBudget = 32 * 1024;

__device__ __forceinline__ bool box_active(const SegState* st, int b) {
    return st == nullptr || st[b].status == SEG_ACTIVE;
}

// ---------------------------------------------------------------- pass X (rows)
enum RowMode { ROW_FWD_CHI = 0, ROW_INV_UPDATE = 1, ROW_FWD_PLAIN = 2 };

template <class C> struct RowArgs {
    const C* in;
    C* out;
    const C* chi;        // ROW_FWD_CHI: [nb][bz][by][bx]
    const C* xin;        // ROW_INV_UPDATE: x, same layout as out
    const uint8_t* mask; // ROW_INV_UPDATE: optional [nb][bz][by][bx]
    const SegState* st;  // optional per-box status
    const C* tw;
    int64_t nrows;
    int in_stride, out_stride, n_in, n_out, lL, ltr, twshift;
    int rows_per_box;    // 3 * bz * by
    int plane;           // bz * by
    int bx;
    int* units;          // profiling: boxes processed (null when off)
};

template <class C, int MODE>
__global__ void __launch_bounds__(kThreads) k_rows(RowArgs<C> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int TR = 1 << a.ltr;
    const int pitch = TR + 1;          // odd pitch: conflict-free transposed staging
    const int L = 1 << a.lL;
    const int64_t row0 = (int64_t)blockIdx.x * TR;
    if (a.units != nullptr && threadIdx.x == 0) {
        const int64_t rpb = a.rows_per_box;
        for (int64_t b = (row0 + rpb - 1) / rpb; b * rpb < row0 + TR && b * rpb < a.nrows; ++b)
            if (box_active(a.st, (int)b)) atomicAdd(a.units, 1);
    }

    for (int idx = threadIdx.x; idx < TR * a.n_in; idx += blockDim.x) {
        int r = idx / a.n_in, i = idx - r * a.n_in;
        int64_t row = row0 + r;
        C v = czero<C>();
        if (row < a.nrows) {
            int b = (int)(row / a.rows_per_box);
            if (box_active(a.st, b)) {
                v = a.in[row * a.in_stride + i];
                if (MODE == ROW_FWD_CHI) {
                    int64_t crow = (int64_t)b * a.plane + (row % a.plane);
                    v = cmul(v, a.chi[crow * a.bx + i]);
                }
            }
        }
        buf[i * pitch + r] = v;
    }
    for (int idx = threadIdx.x; idx < TR * (L - a.n_in); idx += blockDim.x) {
        int i = a.n_in + idx / TR, r = idx % TR;
        buf[i * pitch + r] = czero<C>();
    }
    __syncthreads();
    smem_fft<C, MODE != ROW_INV_UPDATE, 1>(buf, a.lL, pitch, a.ltr, a.tw, a.twshift);
    for (int idx = threadIdx.x; idx < TR * a.n_out; idx += blockDim.x) {
        int r = idx / a.n_out, i = idx - r * a.n_out;
        int64_t row = row0 + r;
        if (row >= a.nrows) continue;
        int b = (int)(row / a.rows_per_box);
        if (!box_active(a.st, b)) continue;
        C v = buf[i * pitch + r];
        if (MODE == ROW_INV_UPDATE) {
            int64_t o = row * a.out_stride + i;
            v = a.xin[o] - v;
            if (a.mask != nullptr) {
                int64_t mrow = (int64_t)b * a.plane + (row % a.plane);
                if (!a.mask[mrow * a.bx + i]) v = czero<C>();
            }
            a.out[o] = v;
        } else {
            a.out[row * a.out_stride + i] = v;
        }
    }
}

// ---------------------------------------------------------------- pass Y / spectrum passes (columns)
template <class C> struct ColArgs {
    const C* in;
    C* out;
    const SegState* st;
    const C* tw;
    int ncols, n_in, n_out, lL, ltc, twshift;
    int64_t in_axis, out_axis, in_s1, out_s1, in_s2, out_s2;
    int b2_per_box;      // blockIdx.z / b2_per_box = box index
    int* units;
};

template <class C, bool FWD>
__global__ void __launch_bounds__(kThreads) k_cols(ColArgs<C> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int TC = 1 << a.ltc;
    const int L = 1 << a.lL;
    const int col0 = blockIdx.x * TC;
    if (!box_active(a.st, blockIdx.z / a.b2_per_box)) return;   // uniform per CTA
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 &&
        blockIdx.z % a.b2_per_box == 0)
        atomicAdd(a.units, 1);
    const C* in = a.in + blockIdx.z * a.in_s2 + blockIdx.y * a.in_s1 + col0;
    C* out = a.out + blockIdx.z * a.out_s2 + blockIdx.y * a.out_s1 + col0;
    const int ncol = min(TC, a.ncols - col0);

    for (int idx = threadIdx.x; idx < L * TC; idx += blockDim.x) {
        int i = idx >> a.ltc, c = idx & (TC - 1);
        C v = czero<C>();
        if (i < a.n_in && c < ncol) v = in[i * a.in_axis + c];
        buf[idx] = v;
    }
    __syncthreads();
    smem_fft<C, FWD, 1>(buf, a.lL, TC, a.ltc, a.tw, a.twshift);
    for (int idx = threadIdx.x; idx < a.n_out * TC; idx += blockDim.x) {
        int i = idx >> a.ltc, c = idx & (TC - 1);
        if (c < ncol) out[i * a.out_axis + c] = buf[idx];
    }
}

// ---------------------------------------------------------------- pass Z fused with the Green multiply
template <class C> struct ZArgs {
    C* w;                 // w2 of the BoxSet
    const C* G;           // [6][Mz][My][Mx], or [6][Mz/2+1][My/2+1][Mx/2+1] when oct
    const C* const* Gb;   // optional: one spectrum per box (instances with their own wavenumber)
    const SegState* st;
    const C* tw;
    int ncols, nzb, lL, ltc, twshift;
    int oct, lx, ly;      // octant-compressed spectrum; log2 Mx, log2 My
    int nine;             // nine full spectra G_ab (3a + b), general 3x3 multiply
    int64_t axis, comp_stride, box_stride, gcomp;
    int* units;
};

template <class C>
__global__ void __launch_bounds__(kThreads) k_zgreen(ZArgs<C> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int TC = 1 << a.ltc;
    const int L = 1 << a.lL;
    const int pitch = 3 * TC;
    const int col0 = blockIdx.x * TC;
    const int b = blockIdx.y;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    C* w = a.w + b * a.box_stride + col0;
    const int ncol = min(TC, a.ncols - col0);

    for (int idx = threadIdx.x; idx < L * 3 * TC; idx += blockDim.x) {
        int c = idx & (TC - 1), t = idx >> a.ltc;
        int comp = t % 3, i = t / 3;
        C v = czero<C>();
        if (i < a.nzb && c < ncol) v = w[comp * a.comp_stride + i * a.axis + c];
        buf[idx] = v;     // idx == i * pitch + comp * TC + c
    }
    __syncthreads();
    smem_fft<C, true, 3>(buf, a.lL, pitch, a.ltc, a.tw, a.twshift);
    for (int idx = threadIdx.x; idx < L * TC; idx += blockDim.x) {
        int c = idx & (TC - 1), i = idx >> a.ltc;
        if (c >= ncol) continue;
        const C* g = a.Gb ? a.Gb[b] : a.G;
        bool ux = false, uy = false, uz = false;
        if (a.oct) {
            const int col = col0 + c;
            const int qx = octant_slot(col & ((1 << a.lx) - 1), a.lx, ux);
            const int qy = octant_slot(col >> a.lx, a.ly, uy);
            const int qz = octant_slot(i, a.lL, uz);
            g += ((int64_t)qz * ((1 << a.ly) / 2 + 1) + qy) * ((1 << a.lx) / 2 + 1) + qx;
        } else {
            g += i * a.axis + col0 + c;
        }
        if (a.nine) {
            C* p = buf + i * pitch + c;
            const C X = p[0], Y = p[TC], Z = p[2 * TC];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                p[r * TC] = cmul(g[(3 * r) * a.gcomp], X) + cmul(g[(3 * r + 1) * a.gcomp], Y) +
                            cmul(g[(3 * r + 2) * a.gcomp], Z);
            continue;
        }
        C gxx = g[0], gxy = g[a.gcomp], gxz = g[2 * a.gcomp];
        C gyy = g[3 * a.gcomp], gyz = g[4 * a.gcomp], gzz = g[5 * a.gcomp];
        if (ux != uy) gxy = mk(-gxy.x, -gxy.y);
        if (ux != uz) gxz = mk(-gxz.x, -gxz.y);
        if (uy != uz) gyz = mk(-gyz.x, -gyz.y);
        C* p = buf + i * pitch + c;
        C X = p[0], Y = p[TC], Z = p[2 * TC];
        const C e[6] = {gxx, gxy, gxz, gyy, gyz, gzz};
        green3<2, false>(X, Y, Z, e);
        p[0] = X;
        p[TC] = Y;
        p[2 * TC] = Z;
    }
    __syncthreads();
    smem_fft<C, false, 3>(buf, a.lL, pitch, a.ltc, a.tw, a.twshift);
    for (int idx = threadIdx.x; idx < a.nzb * 3 * TC; idx += blockDim.x) {
        int c = idx & (TC - 1), t = idx >> a.ltc;
        int comp = t % 3, i = t / 3;
        if (c < ncol) w[comp * a.comp_stride + i * a.axis + c] = buf[idx];
    }
}

// Where a column's spectrum entries lie: octant (OCT) or full layout (bit-reversed positions). entry(f) is
// the offset of component xx at the z frequency f in [0, M/2]; the six components are gcomp apart. sxy, sx,
// sy: whether xy, xz and yz change sign with the column's x and y frequencies (octant).
template <class C, bool OCT> struct ZColumn {
    const C* g;
    int64_t row;
    bool sxy, sx, sy;
    __device__ __forceinline__ ZColumn(const ZArgs<C>& a, int b, int col) {
        g = a.Gb ? a.Gb[b] : a.G;
        sxy = sx = sy = false;
        if (OCT) {
            const int hx = (1 << a.lx) / 2 + 1, hy = (1 << a.ly) / 2 + 1;
            bool ux, uy;
            const int qx = octant_slot(col & ((1 << a.lx) - 1), a.lx, ux), qy = octant_slot(col >> a.lx, a.ly, uy);
            g += (int64_t)qy * hx + qx;
            row = (int64_t)hy * hx;
            sx = ux;
            sy = uy;
            sxy = ux != uy;
        } else {
            g += col;
            row = a.axis;
        }
    }
    // the six components at slot q of the z axis (octant_slot / bit-reversed position of the frequency)
    __device__ __forceinline__ void load(C (&v)[6], int q, int64_t gcomp) const {
        const C* p = g + q * row;
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c] = __ldg(p + c * gcomp);
        if (OCT) {
            v[1] = cneg_if(v[1], sxy);
            v[2] = cneg_if(v[2], sx);
            v[4] = cneg_if(v[4], sy);
        }
    }
};

// Pass Z of complex64 MVMs with Mz <= 32, register-resident: each thread
// transforms one (component, column) pencil in registers (pruned: the box
// fills at most the lower half of the padded axis), the three transformed
// components of kZRegCols columns meet in shared memory for the 3x3 Green
// multiply, and each thread transforms its pencil back, keeping z < bz. The
// spectrum is even in z for xx, xy, yy, zz and odd for xz, yz, so one load of
// its six entries serves the z positions of frequencies f and -f. Bound by the
// latency of those loads: entries of two frequencies in flight, 84 -> 68 us at
// 256x256x16 (three 80, six 90: fewer CTAs fit).
constexpr int kZRegCols = 64;
constexpr int kZRegThreads = 3 * kZRegCols;

template <int LZ, bool OCT>
__global__ void __launch_bounds__(kZRegThreads) k_zgreen_reg(ZArgs<float2> a) {
    pdl_wait();
    // the longest CTAs and the most of them: 256x256x16 product 170 us without, 165 with
    if (LZ == 32 && gridDim.x >= 4096) pdl_trigger();
    typedef float2 F;
    constexpr int H = LZ / 2, LGZ = ILog2<LZ>::v;
    static_assert(LZ >= 4, "shorter axes use k_zgreen");
    constexpr int NC = kZRegCols;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    F* sm = reinterpret_cast<F*>(smem_raw);          // [3][LZ][NC]
    const int b = blockIdx.y;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    const int P = a.ncols, bz = a.nzb, c0 = blockIdx.x * NC, t = threadIdx.x;
    const int nc = min(NC, P - c0);
    F* W = a.w + (int64_t)b * a.box_stride + c0;
    const int64_t cs = a.comp_stride;
    const int comp = t / NC, c = t - comp * NC;
    F* S = sm + comp * LZ * NC + c;
    // (radix 2: with the radix-4 transforms of dft_small.cuh 72 us in place of 68 at 256x256x16)
    if (c < nc) {
        const F* src = W + comp * cs + c;
        F v[H], q[H];
#pragma unroll
        for (int j = 0; j < H; ++j) v[j] = j < bz ? src[(int64_t)j * P] : czero<F>();
#pragma unroll
        for (int j = 0; j < H; ++j) q[j] = twc<true>(v[j], j * (kLmax / LZ));
        rfft<H, true>(q, (const F*)nullptr);
#pragma unroll
        for (int m = 0; m < H; ++m) S[(H + m) * NC] = q[m];
        rfft<H, true>(v, (const F*)nullptr);
#pragma unroll
        for (int m = 0; m < H; ++m) S[m * NC] = v[m];
    }
    // Green multiply: thread (comp, c) takes the frequencies f = comp, comp + 3, ... <= LZ / 2 of column c
    // and their mirrors, the spectrum entries of ZU frequencies in flight at once (the first ones before the wait).
    constexpr int NF = (LZ / 2 + 1 + 2) / 3, cst = LZ * NC, ZU = NF < 2 ? NF : 2;
    const ZColumn<F, OCT> zc(a, b, c0 + (c < nc ? c : 0));
#pragma unroll
    for (int k0 = 0; k0 < NF; k0 += ZU) {
        F e[ZU][6];
#pragma unroll
        for (int k = 0; k < ZU; ++k) {
            const int f = min(comp + 3 * (k0 + k), LZ / 2);
            const int i = (int)(__brev((unsigned)f) >> (32 - LGZ));
            const int q = !OCT ? i : f == LZ / 2 ? LZ / 2 : (int)(__brev((unsigned)f) >> (33 - LGZ));
            zc.load(e[k], q, a.gcomp);
        }
        if (k0 == 0) __syncthreads();
#pragma unroll
        for (int k = 0; k < ZU; ++k) {
            const int f = comp + 3 * (k0 + k);
            if (c >= nc || f > LZ / 2) continue;
            const int i = (int)(__brev((unsigned)f) >> (32 - LGZ));
            const int im = (int)(__brev((unsigned)((LZ - f) & (LZ - 1))) >> (32 - LGZ));
            F* q = sm + i * NC + c;
            F X = q[0], Y = q[cst], Z = q[2 * cst];
            green3<2, false>(X, Y, Z, e[k]);
            q[0] = X;
            q[cst] = Y;
            q[2 * cst] = Z;
            if (im != i) {   // frequency -f: xz and yz change sign
                F* m = sm + im * NC + c;
                F X = m[0], Y = m[cst], Z = m[2 * cst];
                green3<2, true>(X, Y, Z, e[k]);
                m[0] = X;
                m[cst] = Y;
                m[2 * cst] = Z;
            }
        }
    }
    __syncthreads();
    if (c >= nc) return;
    F* dst = W + comp * cs + c;
    F u[H], v[H];
#pragma unroll
    for (int m = 0; m < H; ++m) v[m] = S[(H + m) * NC];
    rfft<H, false>(v, (const F*)nullptr);
#pragma unroll
    for (int m = 0; m < H; ++m) u[m] = S[m * NC];
    rfft<H, false>(u, (const F*)nullptr);
#pragma unroll
    for (int j = 0; j < H; ++j)
        if (j < bz) dst[(int64_t)j * P] = u[j] + twc<false>(v[j], j * (kLmax / LZ));
}

// Pass Z of a single plane (Mz = 1): no transform, one thread multiplies a column's three components. Bound by
// its loads; in k_zgreen, through tiles in shared memory, the whole complex64 product of 512 x 512 x 1 voxels took
// 98 us (50 so), complex128 859 (758).
template <class C, bool OCT>
__global__ void __launch_bounds__(kThreads) k_z_one(ZArgs<C> a) {
    pdl_wait();
    const int b = blockIdx.y;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    const int col = blockIdx.x * kThreads + threadIdx.x;
    if (col >= a.ncols) return;
    C* W = a.w + (int64_t)b * a.box_stride + col;
    const ZColumn<C, OCT> zc(a, b, col);
    C e[6];
    zc.load(e, 0, a.gcomp);
    C X = W[0], Y = W[a.comp_stride], Z = W[2 * a.comp_stride];
    green3<2, false>(X, Y, Z, e);
    W[0] = X;
    W[a.comp_stride] = Y;
    W[2 * a.comp_stride] = Z;
}

// exp(-2 pi i m / 1024) at a compile-time m, times or conjugated times v.
template <bool FWD> __device__ __forceinline__ float2 ztw(float2 v, int m, const float2*) { return twc<FWD>(v, m); }
template <bool FWD> __device__ __forceinline__ double2 ztw(double2 v, int m, const double2* tw) { return twmul<FWD>(v, m, tw); }

// Slot of the z frequency f in [0, M/2], M = 1 << l, of a compile-time f.
template <bool OCT> __device__ __forceinline__ int zslot(int f, int l) {
    const int H = (1 << l) >> 1;
    if (!OCT) return (int)bit_reverse((unsigned)f, l);
    return f == H ? H : (l >= 2 ? (int)bit_reverse((unsigned)f, l - 1) : 0);
}

// Pass Z of complex128 MVMs with Mz = 2H <= 32. The zero-padded 2H-point transform of a column of at most H planes is two H-point
// transforms, of the column (even frequencies) and of the column times W_2H^j (odd ones). One thread takes one
// parity of one column, all three components in registers: transform, Green multiply (one load of the six
// entries serves the frequencies k and -k), inverse transform; the odd parity's thread hands its result over
// through shared memory. Two parities per column, kZPairCols columns per CTA.
// (Bound by the FP64 units: no operation is spent on the padding; 256x256x16 2320 -> 1730 us. In complex64 the pencils of k_zgreen_reg
// are faster, 81 against 109 us at 256x256x16: three columns of 16 values do not fit the registers of a
// thread at a useful occupancy.)
constexpr int kZPairCols = 64;

template <class C, int H, bool OCT, int PAR>
__device__ __forceinline__ void z_parity(const ZArgs<C>& a, const ZColumn<C, OCT>& zc, const C* W, C (&v)[3][H]) {
    constexpr int LG = ILog2<2 * H>::v, TS = kLmax / (2 * H);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int j = 0; j < H; ++j) v[c][j] = j < a.nzb ? W[c * a.comp_stride + j * a.axis] : czero<C>();
        if (PAR) {
#pragma unroll
            for (int j = 1; j < H; ++j) v[c][j] = ztw<true>(v[c][j], j * TS, a.tw);
        }
        dft<H, true>(v[c]);
    }
    // frequencies k = 2m + PAR and their mirrors
#pragma unroll
    for (int m = 0; m < (PAR ? H / 2 : H / 2 + 1); ++m) {
        C e[6];
        zc.load(e, zslot<OCT>(2 * m + PAR, LG), a.gcomp);
        const int mm = (H - m - PAR) % H;
        green3<2, false>(v[0][m], v[1][m], v[2][m], e);
        if (mm != m) green3<2, true>(v[0][mm], v[1][mm], v[2][mm], e);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dft<H, false>(v[c]);
        if (PAR) {
#pragma unroll
            for (int j = 1; j < H; ++j) v[c][j] = ztw<false>(v[c][j], j * TS, a.tw);
        }
    }
}

template <class C, int H, bool OCT>
__global__ void __launch_bounds__(2 * kZPairCols, 2) k_z_pair(ZArgs<C> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);      // [3 H][kZPairCols]: the odd parity's results
    const int b = blockIdx.y;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    const int c = threadIdx.x % kZPairCols, odd = threadIdx.x / kZPairCols;   // whole warps per parity
    const int col = blockIdx.x * kZPairCols + c;
    const bool live = col < a.ncols;
    C* W = a.w + (int64_t)b * a.box_stride + col;
    const ZColumn<C, OCT> zc(a, b, live ? col : 0);
    C v[3][H];
    if (odd && live) {
        z_parity<C, H, OCT, 1>(a, zc, W, v);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < H; ++j) sm[(i * H + j) * kZPairCols + c] = v[i][j];
    } else if (live) {
        z_parity<C, H, OCT, 0>(a, zc, W, v);
    }
    __syncthreads();
    if (odd || !live) return;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < H; ++j)
            if (j < a.nzb) W[i * a.comp_stride + j * a.axis] = v[i][j] + sm[(i * H + j) * kZPairCols + c];
}

// Pass Z with Mz = L = A B, 64 to 512 points: n = B n1 + n2, k = k1 + A k2.
//   step A   one thread per (component, column, n2): the A-point transform over n1, whose upper half is
//            padding: two A/2-point transforms as above;                         to shared memory
//   step B   one thread per (column, k1), all components: twiddles W_L^{n2 k1}, B-point transform over n2,
//            Green multiply of its B frequencies, inverse transform, twiddles;   to shared memory
//   step A'  the inverse of step A, planes z < bz kept.
// Four shared-memory accesses per value and no stage over padding, against 2 log4(L) + 4 of the radix-4 form:
// complex64, 128^3 voxels (256 points) 525 -> 194 us, 64^3 (128 points) 62 -> 27 us, 100x37x60 113 -> 45 us (the
// first four frequencies' spectrum entries on their way before the B-point transform: 209 -> 194 us);
// complex128, bound by the FP64 units, 128^3 5970 -> 5220 us with sums as multiply-adds (radd).
template <class C, int A, int B> struct ZFour {
    static constexpr int L = A * B;
    static constexpr int NC = 98304 / (3 * L * (int)sizeof(C)) >= 32 ? 32 : 98304 / (3 * L * (int)sizeof(C));   // columns per CTA
    static constexpr size_t smem = (size_t)3 * L * NC * sizeof(C);
    static constexpr int threads = sizeof(C) == 8 ? 256 : 128;
    static constexpr int ctas = sizeof(C) == 16 || B < 16 ? 2 : 1;
};

template <class C, int A, int B, bool OCT>
__global__ void __launch_bounds__((ZFour<C, A, B>::threads), (ZFour<C, A, B>::ctas)) k_z_four(ZArgs<C> a) {
    pdl_wait();
    constexpr int ZP = sizeof(C) == 8 ? 4 : 1;   // frequencies whose entries are in flight
    constexpr bool AHEAD = sizeof(C) == 8;
    constexpr int L = A * B, HA = A / 2, NC = ZFour<C, A, B>::NC, TS = kLmax / A, LG = ILog2<L>::v;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);      // [3][k1 B + n2][NC]
    const int b = blockIdx.y;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(a.units, 1);
    const int col0 = blockIdx.x * NC, nc = min(NC, a.ncols - col0);
    C* W = a.w + (int64_t)b * a.box_stride + col0;
    for (int task = threadIdx.x; task < 3 * B * NC; task += blockDim.x) {
        const int c = task % NC, n2 = (task / NC) % B, comp = task / (NC * B);
        if (c >= nc) continue;
        const C* src = W + comp * a.comp_stride + c;
        C* S = sm + (comp * L + n2) * NC + c;
        C x[HA], y[HA];
#pragma unroll
        for (int j = 0; j < HA; ++j) {
            const int n = j * B + n2;
            x[j] = n < a.nzb ? src[n * a.axis] : czero<C>();
            y[j] = j ? ztw<true>(x[j], j * TS, a.tw) : x[j];
        }
        dft<HA, true>(x);
        dft<HA, true>(y);
#pragma unroll
        for (int m = 0; m < HA; ++m) {
            S[(2 * m) * B * NC] = x[m];
            S[(2 * m + 1) * B * NC] = y[m];
        }
    }
    __syncthreads();
    for (int task = threadIdx.x; task < A * NC; task += blockDim.x) {
        const int c = task % NC, k1 = task / NC;
        if (c >= nc) continue;
        const ZColumn<C, OCT> zc(a, b, col0 + c);
        const auto entries = [&](C (&e)[6], int k2) {
            const int k = k1 + A * k2, f = k > L / 2 ? L - k : k;
            const int q = !OCT ? (int)(__brev((unsigned)f) >> (32 - LG)) : f == L / 2 ? L / 2 : (int)(__brev((unsigned)f) >> (33 - LG));
            zc.load(e, q, a.gcomp);
            e[2] = cneg_if(e[2], k > L / 2);
            e[4] = cneg_if(e[4], k > L / 2);
        };
        C e[ZP][6];
        if (AHEAD) {
#pragma unroll
            for (int k2 = 0; k2 < ZP; ++k2) entries(e[k2], k2);
        }
        C w[B], v[3][B];
#pragma unroll
        for (int n2 = 1; n2 < B; ++n2) w[n2] = __ldg(a.tw + ((n2 * k1) << (kLogLmax - LG)));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const C* S = sm + (i * L + k1 * B) * NC + c;
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) v[i][n2] = n2 ? cmul(S[n2 * NC], w[n2]) : S[0];
            dft<B, true>(v[i]);
        }
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            if (!AHEAD || k2 >= ZP) entries(e[k2 % ZP], k2);
            green3<2, false>(v[0][k2], v[1][k2], v[2][k2], e[k2 % ZP]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            C* S = sm + (i * L + k1 * B) * NC + c;
            dft<B, false>(v[i]);
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) S[n2 * NC] = n2 ? cmulc(v[i][n2], w[n2]) : v[i][0];
        }
    }
    __syncthreads();
    for (int task = threadIdx.x; task < 3 * B * NC; task += blockDim.x) {
        const int c = task % NC, n2 = (task / NC) % B, comp = task / (NC * B);
        if (c >= nc) continue;
        C* dst = W + comp * a.comp_stride + c;
        const C* S = sm + (comp * L + n2) * NC + c;
        C x[HA], y[HA];
#pragma unroll
        for (int m = 0; m < HA; ++m) {
            x[m] = S[(2 * m) * B * NC];
            y[m] = S[(2 * m + 1) * B * NC];
        }
        dft<HA, false>(x);
        dft<HA, false>(y);
#pragma unroll
        for (int j = 0; j < HA; ++j) {
            const int n = j * B + n2;
            if (n < a.nzb) dst[n * a.axis] = x[j] + (j ? ztw<false>(y[j], j * TS, a.tw) : y[j]);
        }
    }
}

}  // namespace vie

#include "fft_plane.cuh"

namespace vie {

// ---------------------------------------------------------------- four-step register passes (complex64)
// An L = 32 A point transform (A = 2 .. 32) of a line as two register passes
// with one shared-memory exchange, instead of log2 L shared-memory stages.
// Forward (decimation in frequency, natural -> bit-reversed, as smem_fft):
//   step A  thread j < 32 holds the positions j + 32 m (m < A) and applies the
//           radix-2 stages of spans L/2 .. 32; the pair (p, p + S) with p =
//           j + 32 mm (mm < S/32) takes the twiddle W_L^{p L/(2S)}, which is
//           W_Lmax^{16 j / s} W_Lmax^{512 mm / s} with s = S/32: one runtime
//           factor per stage and a compile-time one per pair;
//   step B  thread g < A holds the 32 positions 32 g + r and applies the
//           stages of spans 16 .. 1: a 32-point transform with compile-time
//           twiddles (rfft<32>).
// Inverse (decimation in time, bit-reversed -> natural): step B then step A,
// with conjugate twiddles in reverse span order. Inputs of the forward pass
// are zero beyond L/2 and outputs of the inverse pass beyond L/2 are dropped
// (pruning: a box of n voxels is padded to L >= 2n - 1).
constexpr int kB4 = 32;

template <int A>
__device__ __forceinline__ void step_a_fwd(float2 (&v)[A], int j, const float2* __restrict__ tw) {
#pragma unroll
    for (int sp = A / 2; sp >= 1; sp >>= 1) {
        const float2 wj = __ldg(&tw[(16 * j) / sp]);
#pragma unroll
        for (int m = 0; m < A; ++m) {
            if ((m & sp) != 0) continue;
            const int mm = m & (sp - 1);
            const float2 x0 = v[m], x1 = v[m + sp];
            v[m] = x0 + x1;
            v[m + sp] = twc<true>(cmul(x0 - x1, wj), (512 / sp) * mm);
        }
    }
}

// Inverse step A; only the outputs m < A/2 are formed by the last stage.
template <int A>
__device__ __forceinline__ void step_a_inv(float2 (&v)[A], int j, const float2* __restrict__ tw) {
#pragma unroll
    for (int sp = 1; sp <= A / 2; sp <<= 1) {
        const float2 wj = __ldg(&tw[(16 * j) / sp]);
#pragma unroll
        for (int m = 0; m < A; ++m) {
            if ((m & sp) != 0) continue;
            const int mm = m & (sp - 1);
            const float2 x0 = v[m];
            const float2 x1 = cmulc(twc<false>(v[m + sp], (512 / sp) * mm), wj);
            v[m] = x0 + x1;
            if (sp < A / 2) v[m + sp] = x0 - x1;
        }
    }
}

// shared-memory index of position p of a line: one pad per 32 positions
__device__ __forceinline__ int pad32(int p) { return p + (p >> 5); }

constexpr int kRows4 = 8;   // rows per CTA (256 threads: 8 rows x 32)

// Pass X forward: rows of bx -> chi * x, zero-padded to L = 32 A, forward transform.
template <int A>
__global__ void __launch_bounds__(256, A <= 16 ? 3 : 2) k_rows4_fwd(RowArgs<float2> a) {
    pdl_wait();
    constexpr int L = kB4 * A, LP = L + L / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);     // [kRows4][LP]
    const int64_t row0 = (int64_t)blockIdx.x * kRows4;
    if (a.units != nullptr && threadIdx.x == 0) {
        const int64_t rpb = a.rows_per_box;
        for (int64_t b = (row0 + rpb - 1) / rpb; b * rpb < row0 + kRows4 && b * rpb < a.nrows; ++b)
            if (box_active(a.st, (int)b)) atomicAdd(a.units, 1);
    }
    // warp r owns row r at both ends
    const int r = threadIdx.x >> 5, j = threadIdx.x & 31;
    const int64_t row = row0 + r;
    const int b = row < a.nrows ? (int)(row / a.rows_per_box) : 0;
    const bool live = row < a.nrows && box_active(a.st, b);
    {
        float2 v[A];
        const int64_t crow = live ? (int64_t)b * a.plane + (row % a.plane) : 0;
#pragma unroll
        for (int m = 0; m < A; ++m) {
            v[m] = czero<float2>();
            const int p = j + kB4 * m;
            if (m < A / 2 && live && p < a.n_in) v[m] = cmul(a.in[row * a.in_stride + p], a.chi[crow * a.bx + p]);
        }
        step_a_fwd<A>(v, j, a.tw);
#pragma unroll
        for (int m = 0; m < A; ++m) sm[r * LP + pad32(j + kB4 * m)] = v[m];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kRows4 * A; t += blockDim.x) {
        const int r = t / A, g = t - r * A;
        float2* q = sm + r * LP + g * (kB4 + 1);
        float2 u[kB4];
#pragma unroll
        for (int i = 0; i < kB4; ++i) u[i] = q[i];
        rfft<kB4, true>(u, (const float2*)nullptr);
#pragma unroll
        for (int i = 0; i < kB4; ++i) q[i] = u[i];
    }
    __syncthreads();
    if (!live) return;
    float2* out = a.out + row * a.out_stride;
#pragma unroll
    for (int m = 0; m < A / 2; ++m) {
        const int p = 2 * (j + 32 * m);
        const float2 u = sm[r * LP + pad32(p)], v = sm[r * LP + pad32(p + 1)];
        *reinterpret_cast<float4*>(out + p) = make_float4(u.x, u.y, v.x, v.y);
    }
}

// Pass X inverse: rows of L = 32 A spectrum positions -> keep x < bx, y = mask (x - u).
template <int A>
__global__ void __launch_bounds__(256, A <= 16 ? 3 : 2) k_rows4_inv(RowArgs<float2> a) {
    pdl_wait();
    constexpr int L = kB4 * A, LP = L + L / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);     // [kRows4][LP]
    const int64_t row0 = (int64_t)blockIdx.x * kRows4;
    if (a.units != nullptr && threadIdx.x == 0) {
        const int64_t rpb = a.rows_per_box;
        for (int64_t b = (row0 + rpb - 1) / rpb; b * rpb < row0 + kRows4 && b * rpb < a.nrows; ++b)
            if (box_active(a.st, (int)b)) atomicAdd(a.units, 1);
    }
    // Warp r owns row r at both ends; 16-byte loads, all of a thread's in flight at once. (Element by element,
    // with the box looked up for each, 48 us at 256x256x16; so, 25.)
    const int r = threadIdx.x >> 5, j = threadIdx.x & 31;
    const int64_t row = row0 + r;
    const int b = row < a.nrows ? (int)(row / a.rows_per_box) : 0;
    const bool live = row < a.nrows && box_active(a.st, b);
    {
        const float2* in = a.in + (live ? row : row0) * a.in_stride;
        float4 q[A / 2];
#pragma unroll
        for (int m = 0; m < A / 2; ++m) q[m] = *reinterpret_cast<const float4*>(in + 2 * (j + 32 * m));
#pragma unroll
        for (int m = 0; m < A / 2; ++m) {
            const int p = 2 * (j + 32 * m);
            sm[r * LP + pad32(p)] = make_float2(q[m].x, q[m].y);
            sm[r * LP + pad32(p + 1)] = make_float2(q[m].z, q[m].w);
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kRows4 * A; t += blockDim.x) {
        const int r = t / A, g = t - r * A;
        float2* q = sm + r * LP + g * (kB4 + 1);
        float2 u[kB4];
#pragma unroll
        for (int i = 0; i < kB4; ++i) u[i] = q[i];
        rfft<kB4, false>(u, (const float2*)nullptr);
#pragma unroll
        for (int i = 0; i < kB4; ++i) q[i] = u[i];
    }
    __syncthreads();
    if (!live) return;
    // x and the mask before the last step: loads behind the stores of y would wait for one another
    const int64_t mrow = (int64_t)b * a.plane + (row % a.plane);
    float2 xv[A / 2];
    bool in[A / 2];
#pragma unroll
    for (int m = 0; m < A / 2; ++m) {
        const int p = j + kB4 * m;
        const bool live = p < a.n_out;
        xv[m] = live ? a.xin[row * a.out_stride + p] : czero<float2>();
        in[m] = live && (a.mask == nullptr || a.mask[mrow * a.bx + p]);
    }
    float2 v[A];
#pragma unroll
    for (int m = 0; m < A; ++m) v[m] = sm[r * LP + pad32(j + kB4 * m)];
    step_a_inv<A>(v, j, a.tw);
#pragma unroll
    for (int m = 0; m < A / 2; ++m) {
        const int p = j + kB4 * m;
        if (p < a.n_out) a.out[row * a.out_stride + p] = in[m] ? xv[m] - v[m] : czero<float2>();
    }
}

constexpr int kCols4 = 16;   // columns per CTA (512 threads: 16 columns x 32)

// Pass Y (forward or inverse) over columns of L = 32 A, 16 adjacent columns per CTA.
template <int A, bool FWD>
__global__ void __launch_bounds__(512) k_cols4(ColArgs<float2> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* sm = reinterpret_cast<float2*>(smem_raw);     // [L][kCols4]
    const int col0 = blockIdx.x * kCols4;
    if (!box_active(a.st, blockIdx.z / a.b2_per_box)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 &&
        blockIdx.z % a.b2_per_box == 0)
        atomicAdd(a.units, 1);
    const float2* in = a.in + blockIdx.z * a.in_s2 + blockIdx.y * a.in_s1 + col0;
    float2* out = a.out + blockIdx.z * a.out_s2 + blockIdx.y * a.out_s1 + col0;
    const int ncol = min(kCols4, a.ncols - col0);
    const int c = threadIdx.x % kCols4, k = threadIdx.x / kCols4;    // k: j (step A) or g (step B)
    if (FWD) {
        if (c < ncol) {
            float2 v[A];
#pragma unroll
            for (int m = 0; m < A; ++m) {
                const int p = k + kB4 * m;
                v[m] = (m < A / 2 && p < a.n_in) ? in[p * a.in_axis + c] : czero<float2>();
            }
            step_a_fwd<A>(v, k, a.tw);
#pragma unroll
            for (int m = 0; m < A; ++m) sm[(k + kB4 * m) * kCols4 + c] = v[m];
        }
        __syncthreads();
        if (k < A && c < ncol) {
            float2 u[kB4];
#pragma unroll
            for (int i = 0; i < kB4; ++i) u[i] = sm[(kB4 * k + i) * kCols4 + c];
            rfft<kB4, true>(u, (const float2*)nullptr);
#pragma unroll
            for (int i = 0; i < kB4; ++i)
                if (kB4 * k + i < a.n_out) out[(kB4 * k + i) * a.out_axis + c] = u[i];
        }
    } else {
        if (k < A && c < ncol) {
            float2 u[kB4];
#pragma unroll
            for (int i = 0; i < kB4; ++i) u[i] = in[(kB4 * k + i) * a.in_axis + c];
            rfft<kB4, false>(u, (const float2*)nullptr);
#pragma unroll
            for (int i = 0; i < kB4; ++i) sm[(kB4 * k + i) * kCols4 + c] = u[i];
        }
        __syncthreads();
        if (c < ncol) {
            float2 v[A];
#pragma unroll
            for (int m = 0; m < A; ++m) v[m] = sm[(k + kB4 * m) * kCols4 + c];
            step_a_inv<A>(v, k, a.tw);
#pragma unroll
            for (int m = 0; m < A / 2; ++m) {
                const int p = k + kB4 * m;
                if (p < a.n_out) out[p * a.out_axis + c] = v[m];
            }
        }
    }
}

// ---------------------------------------------------------------- host side
static int ilog2(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

// log2 of the pencils per CTA: as many as fit the shared-memory budget, at most 32.
static int pick_ltile(int lL, size_t esize, int ncomp, int pad) {
    int lt = 5;
    while (lt > 0 && (size_t)((1 << lL)) * (size_t)(ncomp * (1 << lt) + pad) * esize > (size_t)kSmemBudget) --lt;
    return lt;
}

template <class C> static const C* tw_ptr(const Twiddles& t);
template <> const double2* tw_ptr<double2>(const Twiddles& t) { return t.d128; }
template <> const float2* tw_ptr<float2>(const Twiddles& t) { return t.d64; }

template <class K>
static int prep_smem(K kernel, size_t bytes) {
    return bytes > 46 * 1024 ? raise_dynamic_smem(reinterpret_cast<const void*>(kernel), bytes) : VIE_OK;
}

struct Prof {
    int kind;
    int64_t bpu, fixed;
};
template <class C> static int prec_code() { return sizeof(C) == 16 ? VIE_C128 : VIE_C64; }

template <int A, bool FWD>
static int launch_rows4(RowArgs<float2> a, Prof pf, cudaStream_t s) {
    constexpr int L = kB4 * A;
    const size_t smem = (size_t)kRows4 * (L + L / 32) * sizeof(float2);
    auto kern = FWD ? k_rows4_fwd<A> : k_rows4_inv<A>;
    VIE_TRY(prep_smem(kern, smem));
    const int64_t grid = (a.nrows + kRows4 - 1) / kRows4;
    if (grid <= 0) return VIE_OK;
    a.units = prof_begin(s, pf.kind, VIE_C64, pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(kern, dim3((unsigned)grid), 256, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <bool FWD>
static int launch_rows4_any(RowArgs<float2> a, Prof pf, cudaStream_t s) {
    switch (a.lL) {
        case 6: return launch_rows4<2, FWD>(a, pf, s);
        case 7: return launch_rows4<4, FWD>(a, pf, s);
        case 8: return launch_rows4<8, FWD>(a, pf, s);
        case 9: return launch_rows4<16, FWD>(a, pf, s);
        default: return launch_rows4<32, FWD>(a, pf, s);
    }
}

template <class C, int A, int B, bool FWD>
static int launch_line_rows(RowArgs<C> a, Prof pf, cudaStream_t s) {
    constexpr int L = A * B, NR = LineRows<L>::n;
    const size_t smem = (size_t)NR * (L + L / 8 + 8) * sizeof(C);
    VIE_TRY(prep_smem(k_line_rows<C, A, B, FWD>, smem));
    const int64_t grid = (a.nrows + NR - 1) / NR;
    if (grid <= 0) return VIE_OK;
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_line_rows<C, A, B, FWD>, dim3((unsigned)grid), kLineThreadsRow, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, int A, int B, bool FWD>
static int launch_line_cols(ColArgs<C> a, int nb1, int nb2, Prof pf, cudaStream_t s) {
    constexpr int NC = LineCols<C>::n;
    const size_t smem = (size_t)A * B * NC * sizeof(C);
    VIE_TRY(prep_smem(k_line_cols<C, A, B, FWD>, smem));
    dim3 grid((a.ncols + NC - 1) / NC, nb1, nb2);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_line_cols<C, A, B, FWD>, grid, line_threads_col<C>(), smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, int MODE>
static int launch_rows(RowArgs<C> a, Prof pf, cudaStream_t s) {
    if constexpr (std::is_same<C, float2>::value) {
        // four-step register path: complex64 MVM rows of 64 .. 1024, pruned to half the length
        const int L = 1 << a.lL;
        if (a.lL >= 6 && a.lL <= kLogLmax) {
            if (MODE == ROW_FWD_CHI && 2 * a.n_in <= L && a.n_out == L) return launch_rows4_any<true>(a, pf, s);
            if (MODE == ROW_INV_UPDATE && 2 * a.n_out <= L && a.n_in == L) return launch_rows4_any<false>(a, pf, s);
        }
    }
    // complex128 rows of 256 and 512 points, given two waves of CTAs (below that the radix-4 form spreads a row
    // over more threads: 28 against 42 us for 540 rows); complex64 rows are faster in the radix-2 form above
    // (32 and 50 us forward and inverse against 37 and 62 at 256x256x16)
    if constexpr (sizeof(C) == 16) {
        const int L = 1 << a.lL;
        constexpr bool FWD = MODE == ROW_FWD_CHI;
        if ((a.lL == 8 || a.lL == 9) && a.nrows * L >= 2 * 152 * 4096 &&
            (FWD ? 2 * a.n_in <= L && a.n_out == L : MODE == ROW_INV_UPDATE && 2 * a.n_out <= L && a.n_in == L))
            return a.lL == 8 ? launch_line_rows<C, 16, 16, FWD>(a, pf, s) : launch_line_rows<C, 32, 16, FWD>(a, pf, s);
    }
    a.ltr = pick_ltile(a.lL, sizeof(C), 1, 1);
    const int TR = 1 << a.ltr;
    size_t smem = (size_t)(1 << a.lL) * (TR + 1) * sizeof(C);
    VIE_TRY(prep_smem(k_rows<C, MODE>, smem));
    int64_t grid = (a.nrows + TR - 1) / TR;
    if (grid <= 0) return VIE_OK;
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_rows<C, MODE>, dim3((unsigned)grid), kThreads, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <int A, bool FWD>
static int launch_cols4(ColArgs<float2> a, int nb1, int nb2, Prof pf, cudaStream_t s) {
    const size_t smem = (size_t)kB4 * A * kCols4 * sizeof(float2);
    VIE_TRY(prep_smem(k_cols4<A, FWD>, smem));
    dim3 grid((a.ncols + kCols4 - 1) / kCols4, nb1, nb2);
    a.units = prof_begin(s, pf.kind, VIE_C64, pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_cols4<A, FWD>, grid, kB4 * kCols4, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, bool FWD>
static int launch_cols(ColArgs<C> a, int nb1, int nb2, Prof pf, cudaStream_t s) {
    if constexpr (std::is_same<C, float2>::value) {
        // four-step register path: complex64 columns of 1024, pruned to half the length
        const int L = 1 << a.lL;
        if (a.lL == kLogLmax && (FWD ? (2 * a.n_in <= L && a.n_out == L)
                                                   : (2 * a.n_out <= L && a.n_in == L))) {
            return launch_cols4<32, FWD>(a, nb1, nb2, pf, s);
        }
    }
    // two-step register transforms: columns of 64 to 512 points, pruned to half the length; complex128 with a full
    // tile of columns only (one column of 64 voxels: 17 us here, 10 in the radix-4 form, whose stages spread it
    // over all threads)
    if (a.lL >= 6 && a.lL <= 9 && (sizeof(C) == 8 || a.ncols >= LineCols<C>::n) &&
        (FWD ? (2 * a.n_in <= (1 << a.lL) && a.n_out == (1 << a.lL)) : (2 * a.n_out <= (1 << a.lL) && a.n_in == (1 << a.lL))))
        VIE_LONG_LINE_SWITCH(a.lL, return (launch_line_cols<C, AA, BB, FWD>(a, nb1, nb2, pf, s)));
    a.ltc = pick_ltile(a.lL, sizeof(C), 1, 0);
    if ((1 << a.ltc) > a.ncols) a.ltc = ilog2(a.ncols) - ((1 << ilog2(a.ncols)) > a.ncols ? 1 : 0);
    if (a.ltc < 0) a.ltc = 0;
    const int TC = 1 << a.ltc;
    size_t smem = (size_t)(1 << a.lL) * TC * sizeof(C);
    VIE_TRY(prep_smem(k_cols<C, FWD>, smem));
    dim3 grid((a.ncols + TC - 1) / TC, nb1, nb2);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_cols<C, FWD>, grid, kThreads, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <int LZ, bool OCT>
static int launch_zgreen_reg(ZArgs<float2> a, int nb, Prof pf, cudaStream_t s) {
    const size_t smem = (size_t)3 * LZ * kZRegCols * sizeof(float2);
    VIE_TRY(prep_smem(k_zgreen_reg<LZ, OCT>, smem));
    dim3 grid((a.ncols + kZRegCols - 1) / kZRegCols, nb);
    a.units = prof_begin(s, pf.kind, VIE_C64, pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_zgreen_reg<LZ, OCT>, grid, kZRegThreads, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, int H, bool OCT>
static int launch_z_pair(ZArgs<C> a, int nb, Prof pf, cudaStream_t s) {
    const size_t smem = (size_t)3 * H * kZPairCols * sizeof(C);
    VIE_TRY(prep_smem(k_z_pair<C, H, OCT>, smem));
    dim3 grid((a.ncols + kZPairCols - 1) / kZPairCols, nb);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_z_pair<C, H, OCT>, grid, 2 * kZPairCols, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, int A, int B, bool OCT>
static int launch_z_four(ZArgs<C> a, int nb, Prof pf, cudaStream_t s) {
    typedef ZFour<C, A, B> Z;
    VIE_TRY(prep_smem(k_z_four<C, A, B, OCT>, Z::smem));
    dim3 grid((a.ncols + Z::NC - 1) / Z::NC, nb);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_z_four<C, A, B, OCT>, grid, Z::threads, Z::smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, bool OCT>
static int launch_z_one(ZArgs<C> a, int nb, Prof pf, cudaStream_t s) {
    dim3 grid((a.ncols + kThreads - 1) / kThreads, nb);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_z_one<C, OCT>, grid, kThreads, 0, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, bool OCT>
static int launch_z_reg(ZArgs<C> a, int nb, Prof pf, cudaStream_t s) {
    if constexpr (sizeof(C) == 8) {
        switch (a.lL) {
            case 2: return launch_zgreen_reg<4, OCT>(a, nb, pf, s);
            case 3: return launch_zgreen_reg<8, OCT>(a, nb, pf, s);
            case 4: return launch_zgreen_reg<16, OCT>(a, nb, pf, s);
            case 5: return launch_zgreen_reg<32, OCT>(a, nb, pf, s);
            default: break;
        }
    } else {
        switch (a.lL) {
            case 2: return launch_z_pair<C, 2, OCT>(a, nb, pf, s);
            case 3: return launch_z_pair<C, 4, OCT>(a, nb, pf, s);
            case 4: return launch_z_pair<C, 8, OCT>(a, nb, pf, s);
            case 5: return launch_z_pair<C, 16, OCT>(a, nb, pf, s);
            default: break;
        }
    }
    switch (a.lL) {
        case 6: return launch_z_four<C, 8, 8, OCT>(a, nb, pf, s);
        case 7: return launch_z_four<C, 16, 8, OCT>(a, nb, pf, s);
        case 8: return launch_z_four<C, 32, 8, OCT>(a, nb, pf, s);
        default: return launch_z_four<C, 32, 16, OCT>(a, nb, pf, s);
    }
}

template <class C>
static int launch_zgreen(ZArgs<C> a, int nb, Prof pf, cudaStream_t s) {
    // One plane: the multiply alone. Register transforms for 4 to 512 points of the symmetric operator (the box
    // fills at most half of the axis); the radix-4 form for the rest: 1024 points, the nine spectra of the rooftop operator,
    // and complex128 launches of less than two warps' columns per SM, where one thread's serial FP64 work
    // (a column's parity: 84 us at 16^3 against 30 us) sets the time.
    if (!a.nine && a.lL == 0) return a.oct ? launch_z_one<C, true>(a, nb, pf, s) : launch_z_one<C, false>(a, nb, pf, s);
    const bool few = sizeof(C) == 16 && (int64_t)a.ncols * nb < 152 * 64;
    if (!a.nine && !few && a.lL >= 2 && a.lL <= 9 && 2 * a.nzb <= (1 << a.lL))
        return a.oct ? launch_z_reg<C, true>(a, nb, pf, s) : launch_z_reg<C, false>(a, nb, pf, s);
    a.ltc = pick_ltile(a.lL, sizeof(C), 3, 0);
    if ((1 << a.ltc) > a.ncols) a.ltc = ilog2(a.ncols) - ((1 << ilog2(a.ncols)) > a.ncols ? 1 : 0);
    if (a.ltc < 0) a.ltc = 0;
    const int TC = 1 << a.ltc;
    size_t smem = (size_t)(1 << a.lL) * 3 * TC * sizeof(C);
    VIE_TRY(prep_smem(k_zgreen<C>, smem));
    dim3 grid((a.ncols + TC - 1) / TC, nb);
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_zgreen<C>, grid, kThreads, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

template <class C, bool FWD>
static int launch_plane(PlaneArgs<C> a, int nplanes, Prof pf, cudaStream_t s) {
    const size_t smem = (size_t)a.pitch * ((size_t)1 << a.ly) * sizeof(C);
    VIE_TRY(prep_smem(k_plane<C, FWD>, smem));
    a.units = prof_begin(s, pf.kind, prec_code<C>(), pf.bpu, pf.fixed, true);
    const cudaError_t e = launch_dependent(k_plane<C, FWD>, dim3((unsigned)nplanes), a.lx + a.ly <= 10 ? 128 : a.lx + a.ly <= 12 ? 256 : 512, smem, s, a);
    prof_end(s);
    VIE_CK(e);
    return VIE_OK;
}

// x and y transforms of a plane in one launch (k_plane): planes of 4 x 4 to 256 x 256 points that fit shared memory.
// complex128 planes of more than 32 x 32 points need enough CTAs for the FP64 units of every SM (27 planes of
// 32 x 256 points: 145 us against 74 in separate passes).
template <class C> static bool plane_ok(const BoxSet& bs) {
    if (sizeof(C) == 16 && bs.lx + bs.ly > 10 && (int64_t)bs.nb * 3 * bs.bz < 128) return false;
    return bs.lx >= 2 && bs.lx <= 8 && bs.ly >= 2 && bs.ly <= 8 &&
           (size_t)plane_pitch(bs.Mx) * bs.My * sizeof(C) <= (size_t)200 * 1024;
}

template <class C> static const C* chi_ptr(const BoxSet& bs);
template <> const double2* chi_ptr<double2>(const BoxSet& bs) { return bs.chi128; }
template <> const float2* chi_ptr<float2>(const BoxSet& bs) { return bs.chi64; }

template <class C>
int mvm_boxes(const BoxSet& bs, const C* G, const C* x, C* y, const SegState* st, cudaStream_t s,
              const Twiddles* twp, const C* const* Gb, const C* xupd, bool nine) {
    Twiddles tw;
    if (twp) tw = *twp;
    else VIE_TRY(get_twiddles(&tw));
    const C* T = tw_ptr<C>(tw);
    C* w1 = reinterpret_cast<C*>(bs.w1);
    C* w2 = reinterpret_cast<C*>(bs.w2);
    const int64_t planeXY = (int64_t)bs.Mx * bs.My;
    // algorithmic bytes per box of each pass (inputs read + outputs written)
    const int64_t es = sizeof(C);
    const int64_t box = bs.box_elems();
    const int64_t b1 = 3LL * bs.bz * bs.by * bs.Mx * es;          // w1 per box
    const int64_t b2 = 3LL * bs.bz * planeXY * es;                // w2 per box
    const int64_t bv = 3LL * box * es;                            // x or y per box
    const Prof px{PK_X_FWD, bv + box * es + b1, 0};
    const Prof py{PK_Y_FWD, b1 + b2, 0};
    const Prof pz{PK_Z_GREEN, 2 * b2, (nine ? 9LL : 6LL) * (bs.oct ? bs.oct_elems() : bs.spec_elems()) * es};
    const Prof piy{PK_Y_INV, b2 + b1, 0};
    const Prof pix{PK_X_INV, b1 + 2 * bv + (bs.mask ? box : 0), 0};

    const bool planes = plane_ok<C>(bs);
    PlaneArgs<C> pa{};
    RowArgs<C> rx{};
    ColArgs<C> cy{};
    if (planes) {
        pa.in = x; pa.out = w2; pa.chi = chi_ptr<C>(bs); pa.st = st; pa.tw = T;
        pa.bx = bs.bx; pa.by = bs.by; pa.bz = bs.bz; pa.lx = bs.lx; pa.ly = bs.ly; pa.pitch = plane_pitch(bs.Mx);
        VIE_TRY((launch_plane<C, true>(pa, bs.nb * 3 * bs.bz, Prof{PK_X_FWD, bv + box * es + b2, 0}, s)));
    } else {
    // pass X: chi * x, zero-padded forward FFT of every row
    rx.in = x; rx.out = w1; rx.chi = chi_ptr<C>(bs); rx.st = st; rx.tw = T;
    rx.nrows = (int64_t)bs.nb * 3 * bs.bz * bs.by;
    rx.in_stride = bs.bx; rx.out_stride = bs.Mx; rx.n_in = bs.bx; rx.n_out = bs.Mx;
    rx.lL = bs.lx; rx.twshift = kLogLmax - bs.lx;
    rx.rows_per_box = 3 * bs.bz * bs.by; rx.plane = bs.bz * bs.by; rx.bx = bs.bx;
    VIE_TRY((launch_rows<C, ROW_FWD_CHI>(rx, px, s)));

    // pass Y forward
    cy.in = w1; cy.out = w2; cy.st = st; cy.tw = T;
    cy.ncols = bs.Mx; cy.n_in = bs.by; cy.n_out = bs.My; cy.lL = bs.ly; cy.twshift = kLogLmax - bs.ly;
    cy.in_axis = bs.Mx; cy.out_axis = bs.Mx;
    cy.in_s1 = (int64_t)bs.by * bs.Mx; cy.out_s1 = planeXY;
    cy.in_s2 = (int64_t)bs.bz * bs.by * bs.Mx; cy.out_s2 = (int64_t)bs.bz * planeXY;
    cy.b2_per_box = 3;
    VIE_TRY((launch_cols<C, true>(cy, bs.bz, bs.nb * 3, py, s)));
    }

    // pass Z: forward, Green multiply, inverse
    ZArgs<C> z{};
    z.w = w2; z.G = G; z.Gb = Gb; z.st = st; z.tw = T;
    z.ncols = (int)planeXY; z.nzb = bs.bz; z.lL = bs.lz; z.twshift = kLogLmax - bs.lz;
    z.axis = planeXY; z.comp_stride = (int64_t)bs.bz * planeXY; z.box_stride = 3 * z.comp_stride;
    z.gcomp = bs.oct ? bs.oct_elems() : (int64_t)bs.Mz * planeXY;
    z.oct = bs.oct ? 1 : 0; z.lx = bs.lx; z.ly = bs.ly;
    z.nine = nine ? 1 : 0;
    if (nine && bs.oct) return fail(VIE_EINVAL, "mvm_boxes: nine spectra need the full layout");
    VIE_TRY(launch_zgreen<C>(z, bs.nb, pz, s));

    if (planes) {
        pa.in = w2; pa.out = y; pa.xin = xupd ? xupd : x; pa.mask = bs.mask; pa.chi = nullptr;
        return launch_plane<C, false>(pa, bs.nb * 3 * bs.bz, Prof{PK_X_INV, b2 + 2 * bv + (bs.mask ? box : 0), 0}, s);
    }
    // pass Y inverse: keep y < by
    ColArgs<C> iy = cy;
    iy.in = w2; iy.out = w1; iy.n_in = bs.My; iy.n_out = bs.by;
    iy.in_s1 = planeXY; iy.out_s1 = (int64_t)bs.by * bs.Mx;
    iy.in_s2 = (int64_t)bs.bz * planeXY; iy.out_s2 = (int64_t)bs.bz * bs.by * bs.Mx;
    VIE_TRY((launch_cols<C, false>(iy, bs.bz, bs.nb * 3, piy, s)));

    // pass X inverse: keep x < bx, y = x - u
    RowArgs<C> ix = rx;
    ix.in = w1; ix.out = y; ix.xin = xupd ? xupd : x; ix.mask = bs.mask; ix.chi = nullptr;
    ix.in_stride = bs.Mx; ix.out_stride = bs.bx; ix.n_in = bs.Mx; ix.n_out = bs.bx;
    VIE_TRY((launch_rows<C, ROW_INV_UPDATE>(ix, pix, s)));
    return VIE_OK;
}

template <class C>
int spectrum_fft(const BoxSet& bs, C* G, cudaStream_t s, const Twiddles* twp, int ncomp) {
    Twiddles tw;
    if (twp) tw = *twp;
    else VIE_TRY(get_twiddles(&tw));
    const C* T = tw_ptr<C>(tw);
    const int64_t planeXY = (int64_t)bs.Mx * bs.My;
    const int64_t vol = planeXY * bs.Mz;
    const int64_t es = sizeof(C);

    RowArgs<C> rx{};
    rx.in = G; rx.out = G; rx.tw = T;
    rx.nrows = ncomp * (int64_t)bs.Mz * bs.My;
    rx.in_stride = bs.Mx; rx.out_stride = bs.Mx; rx.n_in = bs.Mx; rx.n_out = bs.Mx;
    rx.lL = bs.lx; rx.twshift = kLogLmax - bs.lx;
    rx.rows_per_box = (int)std::min<int64_t>(rx.nrows, 1 << 30); rx.plane = 1; rx.bx = bs.Mx;
    VIE_TRY((launch_rows<C, ROW_FWD_PLAIN>(rx, Prof{PK_SPECTRUM, 12 * vol * es, 0}, s)));

    ColArgs<C> cy{};
    cy.in = G; cy.out = G; cy.tw = T; cy.b2_per_box = 1;
    cy.ncols = bs.Mx; cy.n_in = bs.My; cy.n_out = bs.My; cy.lL = bs.ly; cy.twshift = kLogLmax - bs.ly;
    cy.in_axis = cy.out_axis = bs.Mx;
    cy.in_s1 = cy.out_s1 = planeXY;
    cy.in_s2 = cy.out_s2 = vol;
    VIE_TRY((launch_cols<C, true>(cy, bs.Mz, ncomp, Prof{PK_SPECTRUM, 2 * vol * es, 0}, s)));

    ColArgs<C> cz{};
    cz.in = G; cz.out = G; cz.tw = T; cz.b2_per_box = 1;
    cz.ncols = (int)planeXY; cz.n_in = bs.Mz; cz.n_out = bs.Mz; cz.lL = bs.lz; cz.twshift = kLogLmax - bs.lz;
    cz.in_axis = cz.out_axis = planeXY;
    cz.in_s1 = cz.out_s1 = 0;
    cz.in_s2 = cz.out_s2 = vol;
    VIE_TRY((launch_cols<C, true>(cz, 1, ncomp, Prof{PK_SPECTRUM, 2 * vol * es, 0}, s)));
    return VIE_OK;
}

// One axis of the spectrum of the kernel's octant: each line of n samples K(d), d >= 0, is extended to the
// padded length by its parity (K(M - d) = +-K(d), zero between n and M - n), transformed, and the frequencies
// [0, M/2] kept in octant slot order (octant_freq). AXIS 0: rows along x, [6][bz][by][bx] -> [6][bz][by][hx];
// 1: columns along y -> [6][bz][hy][hx]; 2: columns along z -> [6][hz][hy][hx], also rounded to complex64.
// Against sampling and transforming the full padded array (1/8 of the samples, 1/4 of the lines per axis;
// FP64-bound): 64^3 voxels 2.3 -> 0.6 ms.
struct SpecAxis {
    const double2* in;
    double2* out;
    float2* out64;           // AXIS 2
    const double2* tw;
    int64_t lines;           // lines per component and slice (slices: components x leading extents)
    int64_t in_slice, out_slice;
    int n, lL, ltc, twshift, slices_per_comp;
};

template <int AXIS>
__global__ void __launch_bounds__(kThreads) k_spec_axis(SpecAxis a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const int TC = 1 << a.ltc, L = 1 << a.lL, pitch = AXIS == 0 ? TC + 1 : TC, nf = L / 2 + 1;
    const int slice = blockIdx.y, c = slice / a.slices_per_comp;
    const bool odd = AXIS == 0 ? (c == 1 || c == 2) : AXIS == 1 ? (c == 1 || c == 4) : (c == 2 || c == 4);
    const int64_t l0 = (int64_t)blockIdx.x * TC;
    const int nl = (int)min((int64_t)TC, a.lines - l0);
    const double2* in = a.in + slice * a.in_slice + (AXIS == 0 ? l0 * a.n : l0);
    for (int t = threadIdx.x; t < L * TC; t += blockDim.x) buf[(t >> a.ltc) * pitch + (t & (TC - 1))] = czero<double2>();
    __syncthreads();
    for (int t = threadIdx.x; t < a.n * TC; t += blockDim.x) {
        const int l = AXIS == 0 ? t / a.n : t & (TC - 1), d = AXIS == 0 ? t - l * a.n : t >> a.ltc;
        if (l >= nl) continue;
        const double2 v = AXIS == 0 ? in[t] : in[d * a.lines + l];
        buf[d * pitch + l] = v;
        if (d > 0) buf[(L - d) * pitch + l] = odd ? mk(-v.x, -v.y) : v;
    }
    __syncthreads();
    smem_fft<double2, true, 1>(buf, a.lL, pitch, a.ltc, a.tw, a.twshift);
    const int64_t o0 = slice * a.out_slice + (AXIS == 0 ? l0 * nf : l0);
    for (int t = threadIdx.x; t < nf * TC; t += blockDim.x) {
        const int l = AXIS == 0 ? t / nf : t & (TC - 1), q = AXIS == 0 ? t - l * nf : t >> a.ltc;
        if (l >= nl) continue;
        const double2 v = buf[(int)brev_bits((unsigned)octant_freq(q, a.lL), a.lL) * pitch + l];
        const int64_t o = o0 + (AXIS == 0 ? t : q * a.lines + l);
        if (a.out) a.out[o] = v;
        if (AXIS == 2 && a.out64) a.out64[o] = make_float2((float)v.x, (float)v.y);
    }
}

template <int AXIS>
static int launch_spec_axis(SpecAxis a, int slices, int64_t bytes, cudaStream_t s) {
    a.ltc = pick_ltile(a.lL, sizeof(double2), 1, AXIS == 0 ? 1 : 0);
    const size_t smem = (size_t)(1 << a.lL) * ((1 << a.ltc) + (AXIS == 0 ? 1 : 0)) * sizeof(double2);
    VIE_TRY(prep_smem(k_spec_axis<AXIS>, smem));
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, bytes, false);
    k_spec_axis<AXIS><<<dim3((unsigned)((a.lines + (1 << a.ltc) - 1) >> a.ltc), (unsigned)slices), kThreads, smem, s>>>(a);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// The full layout from the octant: every bit-reversed position takes its folded frequency's entry, negated for
// components odd along an axis in its upper half.
template <class C>
__global__ void k_octant_expand(const double2* oct, C* full, int lx, int ly, int lz) {
    const int hx = (1 << lx) / 2 + 1, hy = (1 << ly) / 2 + 1, hz = (1 << lz) / 2 + 1;
    const int64_t per = (int64_t)hx * hy * hz, vol = (int64_t)1 << (lx + ly + lz);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < vol; t += (int64_t)gridDim.x * blockDim.x) {
        bool ux, uy, uz;
        const int qx = octant_slot((int)(t & ((1 << lx) - 1)), lx, ux), qy = octant_slot((int)((t >> lx) & ((1 << ly) - 1)), ly, uy),
                  qz = octant_slot((int)(t >> (lx + ly)), lz, uz);
        const double2* p = oct + ((int64_t)qz * hy + qy) * hx + qx;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const bool neg = c == 1 ? ux != uy : c == 2 ? ux != uz : c == 4 ? uy != uz : false;
            const double2 v = cneg_if(p[c * per], neg);
            full[c * vol + t] = cmk<C>(v.x, v.y);
        }
    }
}

int spectrum_build(const BoxSet& bs, double k0, double h, const SpecOut& out, cudaStream_t s, const NearRule* near) {
    Twiddles tw;
    VIE_TRY(get_twiddles(&tw));
    const int hx = bs.Mx / 2 + 1, hy = bs.My / 2 + 1, hz = bs.Mz / 2 + 1;
    const int64_t nk = 6 * bs.box_elems(), n1 = 6LL * bs.bz * bs.by * hx, n2 = 6LL * bs.bz * hy * hx, no = 6 * bs.oct_elems();
    const bool full = out.full128 || out.full64, own = full && !out.oct128;
    double2* K = nullptr;
    VIE_CK(cudaMallocAsync((void**)&K, (nk + n1 + n2 + (own ? no : 0)) * sizeof(double2), s));
    double2 *t1 = K + nk, *t2 = t1 + n1, *o128 = own ? t2 + n2 : out.oct128;
    const int64_t es = sizeof(double2);
    int rc = green_octant(bs, k0, h, K, s, near);
    if (!rc && out.par) rc = par_spectra(bs, K, *out.par, s);
    if (!rc) {
        SpecAxis a{};
        a.tw = tw.d128;
        a.in = K; a.out = t1; a.lines = (int64_t)bs.bz * bs.by; a.n = bs.bx; a.lL = bs.lx; a.twshift = kLogLmax - bs.lx;
        a.in_slice = bs.box_elems(); a.out_slice = a.lines * hx; a.slices_per_comp = 1;
        rc = launch_spec_axis<0>(a, 6, (nk + n1) * es, s);
    }
    if (!rc) {
        SpecAxis a{};
        a.tw = tw.d128;
        a.in = t1; a.out = t2; a.lines = hx; a.n = bs.by; a.lL = bs.ly; a.twshift = kLogLmax - bs.ly;
        a.in_slice = (int64_t)bs.by * hx; a.out_slice = (int64_t)hy * hx; a.slices_per_comp = bs.bz;
        rc = launch_spec_axis<1>(a, 6 * bs.bz, (n1 + n2) * es, s);
    }
    if (!rc) {
        SpecAxis a{};
        a.tw = tw.d128;
        a.in = t2; a.out = o128; a.out64 = out.oct64; a.lines = (int64_t)hy * hx; a.n = bs.bz; a.lL = bs.lz; a.twshift = kLogLmax - bs.lz;
        a.in_slice = a.lines * bs.bz; a.out_slice = a.lines * hz; a.slices_per_comp = 1;
        rc = launch_spec_axis<2>(a, 6, (n2 + no) * es, s);
    }
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((bs.spec_elems() + 255) / 256, 152 * 16));
    if (!rc && out.full128) {
        prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 6 * bs.spec_elems() * es, false);
        k_octant_expand<double2><<<grid, 256, 0, s>>>(o128, out.full128, bs.lx, bs.ly, bs.lz);
        prof_end(s);
    }
    if (!rc && out.full64) {
        prof_begin(s, PK_SPECTRUM, VIE_C64, 0, 6 * bs.spec_elems() * es / 2, false);
        k_octant_expand<float2><<<grid, 256, 0, s>>>(o128, out.full64, bs.lx, bs.ly, bs.lz);
        prof_end(s);
    }
    if (!rc && cudaGetLastError() != cudaSuccess) rc = fail(VIE_ECUDA, "spectrum expansion launch failed");
    const cudaError_t e = cudaFreeAsync(K, s);
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "cudaFreeAsync", __FILE__, __LINE__);
    return rc;
}

template int mvm_boxes<double2>(const BoxSet&, const double2*, const double2*, double2*, const SegState*, cudaStream_t,
                                const Twiddles*, const double2* const*, const double2*, bool);
template int mvm_boxes<float2>(const BoxSet&, const float2*, const float2*, float2*, const SegState*, cudaStream_t,
                               const Twiddles*, const float2* const*, const float2*, bool);
template int spectrum_fft<double2>(const BoxSet&, double2*, cudaStream_t, const Twiddles*, int);

}  // namespace vie

// x and y transforms of one padded plane (component, z) in one CTA, for planes that fit shared memory: the
// x and y passes of fft.cu without the intermediate w1, and two launches fewer per product.
//
// Each axis takes L = A B points in two steps (n = B n1 + n2, k = k1 + A k2): A-point transforms over n1,
// whose upper half is padding (two A/2-point transforms, of the line and of the line times W_A^j), then
// twiddles W_L^{n2 k1} and B-point transforms over n2. Rows end up in bit-reversed order in shared memory
// (the order of w2), columns are stored to the bit-reversed row.
//
// Whole complex64 products, separate passes -> planes: 16^3 33.6 -> 17.5 us, 32^3 39.7 -> 21.3, 48^3 83 -> 52,
// 64^3 (planes of 128 x 128, one CTA per SM) 100 -> 74.
#pragma once

#include "dft_small.cuh"

namespace vie {

// log2 L -> (A, B)
#define VIE_LINE_SWITCH(l, CALL)                                                       \
    switch (l) {                                                                       \
        case 2: { constexpr int AA = 2, BB = 2; CALL; } break;                         \
        case 3: { constexpr int AA = 2, BB = 4; CALL; } break;                         \
        case 4: { constexpr int AA = 2, BB = 8; CALL; } break;                         \
        case 5: { constexpr int AA = 4, BB = 8; CALL; } break;                         \
        case 6: { constexpr int AA = 8, BB = 8; CALL; } break;                         \
        case 7: { constexpr int AA = 16, BB = 8; CALL; } break;                        \
        case 8: { constexpr int AA = 32, BB = 8; CALL; } break;                        \
        default: break;                                                                \
    }

template <class C> struct PlaneArgs {
    const C* in;          // forward: x [nb][3][bz][by][bx]; inverse: w2
    C* out;               // forward: w2 [nb][3][bz][My][Mx]; inverse: y
    const C* chi;         // forward: [nb][bz][by][bx]
    const C* xin;         // inverse: the vector of y = mask (xin - u)
    const uint8_t* mask;  // inverse, optional
    const SegState* st;
    const C* tw;
    int bx, by, bz, lx, ly, pitch;
    int* units;
};

// column of position p of a row, one pad per 8 (rows are read and written 8 positions apart)
__device__ __forceinline__ int plane_pad(int p) { return p + (p >> 3); }
// row pitch: consecutive rows start 8 banks (of 8 bytes) apart
inline int plane_pitch(int Mx) {
    const int w = Mx + (Mx >> 3);
    return w + ((24 - (w & 15)) & 15);
}

// A-point step over n1 of one line: get(n) gives input n < L/2, put(position, value) receives k1 B + n2.
template <int A, int B, class C, class Get, class Put>
__device__ __forceinline__ void line_a_fwd(int n2, const C* tw, Get get, Put put) {
    constexpr int HA = A / 2;
    C x[HA], y[HA];
#pragma unroll
    for (int j = 0; j < HA; ++j) {
        x[j] = get(j * B + n2);
        y[j] = j ? ztw<true>(x[j], j * (kLmax / A), tw) : x[j];
    }
    dft<HA, true>(x);
    dft<HA, true>(y);
#pragma unroll
    for (int m = 0; m < HA; ++m) {
        put((2 * m) * B + n2, x[m]);
        put((2 * m + 1) * B + n2, y[m]);
    }
}
// Its inverse: put(n, value) receives the outputs n < L/2.
template <int A, int B, class C, class Get, class Put>
__device__ __forceinline__ void line_a_inv(int n2, const C* tw, Get get, Put put) {
    constexpr int HA = A / 2;
    C x[HA], y[HA];
#pragma unroll
    for (int m = 0; m < HA; ++m) {
        x[m] = get((2 * m) * B + n2);
        y[m] = get((2 * m + 1) * B + n2);
    }
    dft<HA, false>(x);
    dft<HA, false>(y);
#pragma unroll
    for (int j = 0; j < HA; ++j) put(j * B + n2, x[j] + (j ? ztw<false>(y[j], j * (kLmax / A), tw) : y[j]));
}
// B-point step of one k1: v holds n2 = 0 .. B-1 and becomes k2 = 0 .. B-1 (or back).
template <int A, int B, bool FWD, class C> __device__ __forceinline__ void line_b(C (&v)[B], int k1, const C* tw) {
    constexpr int L = A * B;
    if (FWD) {
#pragma unroll
        for (int n2 = 1; n2 < B; ++n2) v[n2] = cmul(v[n2], __ldg(tw + n2 * k1 * (kLmax / L)));
        dft<B, true>(v);
    } else {
        dft<B, false>(v);
#pragma unroll
        for (int n2 = 1; n2 < B; ++n2) v[n2] = cmulc(v[n2], __ldg(tw + n2 * k1 * (kLmax / L)));
    }
}
template <int A, int B> __device__ __forceinline__ int line_brev(int k1, int k2) {
    return (int)(__brev((unsigned)(k1 + A * k2)) >> (32 - ILog2<A * B>::v));
}

// Rows y < by: step A from global memory (x times chi) or to it (y = mask (xin - u)); step B within a row by
// the lanes of one warp, so that it may be reordered in place.
template <int A, int B, class C> __device__ __forceinline__ void plane_rows_fwd(const PlaneArgs<C>& a, C* sm, const C* in,
                                                                                const C* chi) {
    for (int t = threadIdx.x; t < a.by * B; t += blockDim.x) {
        const int n2 = t & (B - 1), y = t / B;
        C* row = sm + y * a.pitch;
        line_a_fwd<A, B>(n2, a.tw,
                         [&](int n) { return n < a.bx ? cmul(in[y * a.bx + n], chi[y * a.bx + n]) : czero<C>(); },
                         [&](int p, C v) { row[plane_pad(p)] = v; });
    }
    __syncthreads();
    const int n = a.by * A;
    for (int t0 = threadIdx.x - (threadIdx.x & 31); t0 < n; t0 += blockDim.x) {
        const int t = t0 + (threadIdx.x & 31), k1 = t & (A - 1);
        C* row = sm + (t < n ? t / A : 0) * a.pitch;
        C v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = row[plane_pad(k1 * B + i)];
        line_b<A, B, true>(v, k1, a.tw);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (t < n) row[plane_pad(line_brev<A, B>(k1, i))] = v[i];
    }
    __syncthreads();
}

template <int A, int B, class C>
__device__ __forceinline__ void plane_rows_inv(const PlaneArgs<C>& a, C* sm, C* out, const C* xin, const uint8_t* mask) {
    const int n = a.by * A;
    for (int t0 = threadIdx.x - (threadIdx.x & 31); t0 < n; t0 += blockDim.x) {
        const int t = t0 + (threadIdx.x & 31), k1 = t & (A - 1);
        C* row = sm + (t < n ? t / A : 0) * a.pitch;
        C v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = row[plane_pad(line_brev<A, B>(k1, i))];
        line_b<A, B, false>(v, k1, a.tw);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (t < n) row[plane_pad(k1 * B + i)] = v[i];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < a.by * B; t += blockDim.x) {
        const int n2 = t & (B - 1), y = t / B;
        const C* row = sm + y * a.pitch;
        // x and the mask first: loads behind the stores of y would wait for one another
        // (complex64; complex128 has no registers left for them)
        constexpr bool AHEAD = sizeof(C) == 8;
        C xv[A / 2];
        bool in[A / 2];
        if (AHEAD) {
#pragma unroll
            for (int j = 0; j < A / 2; ++j) {
                const int x = j * B + n2, o = y * a.bx + x;
                xv[j] = x < a.bx ? xin[o] : czero<C>();
                in[j] = x < a.bx && (mask == nullptr || mask[o]);
            }
        }
        line_a_inv<A, B>(n2, a.tw, [&](int p) { return row[plane_pad(p)]; },
                         [&](int x, C u) {
                             if (x >= a.bx) return;
                             const int o = y * a.bx + x;
                             C v = (AHEAD ? xv[x / B] : xin[o]) - u;
                             if (AHEAD ? !in[x / B] : mask != nullptr && !mask[o]) v = czero<C>();
                             out[o] = v;
                         });
    }
}

// Columns: step A in shared memory, step B to or from the rows of w2.
template <int A, int B, class C> __device__ __forceinline__ void plane_cols_fwd(const PlaneArgs<C>& a, C* sm, C* w) {
    const int Mx = 1 << a.lx;
    for (int t = threadIdx.x; t < Mx * B; t += blockDim.x) {
        const int x = t & (Mx - 1), n2 = t >> a.lx;
        C* col = sm + plane_pad(x);
        line_a_fwd<A, B>(n2, a.tw, [&](int n) { return n < a.by ? col[n * a.pitch] : czero<C>(); },
                         [&](int p, C v) { col[p * a.pitch] = v; });
    }
    __syncthreads();
    for (int t = threadIdx.x; t < Mx * A; t += blockDim.x) {
        const int x = t & (Mx - 1), k1 = t >> a.lx;
        const C* col = sm + plane_pad(x);
        C v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = col[(k1 * B + i) * a.pitch];
        line_b<A, B, true>(v, k1, a.tw);
#pragma unroll
        for (int i = 0; i < B; ++i) w[line_brev<A, B>(k1, i) * Mx + x] = v[i];
    }
}
template <int A, int B, class C> __device__ __forceinline__ void plane_cols_inv(const PlaneArgs<C>& a, C* sm, const C* w) {
    const int Mx = 1 << a.lx;
    for (int t = threadIdx.x; t < Mx * A; t += blockDim.x) {
        const int x = t & (Mx - 1), k1 = t >> a.lx;
        C* col = sm + plane_pad(x);
        C v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = w[line_brev<A, B>(k1, i) * Mx + x];
        line_b<A, B, false>(v, k1, a.tw);
#pragma unroll
        for (int i = 0; i < B; ++i) col[(k1 * B + i) * a.pitch] = v[i];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < Mx * B; t += blockDim.x) {
        const int x = t & (Mx - 1), n2 = t >> a.lx;
        C* col = sm + plane_pad(x);
        line_a_inv<A, B>(n2, a.tw, [&](int p) { return col[p * a.pitch]; },
                         [&](int n, C v) {
                             if (n < a.by) col[n * a.pitch] = v;
                         });
    }
    __syncthreads();
}

template <class C, bool FWD>
__global__ void __launch_bounds__(512) k_plane(PlaneArgs<C> a) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);          // [My][pitch]
    const int pl = blockIdx.x, b = pl / (3 * a.bz), z = pl % a.bz;
    if (!box_active(a.st, b)) return;
    if (a.units != nullptr && threadIdx.x == 0 && pl % (3 * a.bz) == 0) atomicAdd(a.units, 1);
    const int64_t plane = (int64_t)a.by * a.bx, wide = (int64_t)1 << (a.lx + a.ly);
    const int64_t vox = ((int64_t)b * a.bz + z) * plane;
    if (FWD) {
        const C* in = a.in + pl * plane;
        VIE_LINE_SWITCH(a.lx, (plane_rows_fwd<AA, BB>(a, sm, in, a.chi + vox)));
        VIE_LINE_SWITCH(a.ly, (plane_cols_fwd<AA, BB>(a, sm, a.out + pl * wide)));
    } else {
        VIE_LINE_SWITCH(a.ly, (plane_cols_inv<AA, BB>(a, sm, a.in + pl * wide)));
        VIE_LINE_SWITCH(a.lx, (plane_rows_inv<AA, BB>(a, sm, a.out + pl * plane, a.xin + pl * plane,
                                                      a.mask ? a.mask + vox : nullptr)));
    }
}

// ---------------------------------------------------------------- single passes over long lines
// Rows and columns of 64 to 512 points by the same two steps, for planes that do not fit shared memory. Against
// radix-2 stages with a run-time and a compile-time twiddle each, a quarter fewer operations per point: column
// passes in complex64 256x256x16 47 + 53 -> 38 + 46 us, 128^3 120 + 125 -> 55 + 60 us (two 16-point steps keep
// 74 registers; one 32-point step 66 + 72 us), 100x37x60 45 + 39 -> 15 + 16 us; complex128 128^3 1313 -> 1060 us.
template <class C> struct RowArgs;
template <class C> struct ColArgs;
constexpr int kLineThreadsRow = 128;
template <class C> __host__ __device__ constexpr int line_threads_col() { return sizeof(C) == 8 ? 256 : 128; }
template <int L> struct LineRows { static constexpr int n = 4096 / L; };                    // rows per CTA
template <class C> struct LineCols { static constexpr int n = sizeof(C) == 8 ? 16 : 8; };   // columns per CTA: 128 bytes

template <class C, int A, int B, bool FWD>
__global__ void __launch_bounds__(kLineThreadsRow) k_line_rows(RowArgs<C> a) {
    pdl_wait();
    constexpr int L = A * B, NR = LineRows<L>::n, P = L + L / 8 + 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);          // [NR][P]
    const int64_t row0 = (int64_t)blockIdx.x * NR;
    if (a.units != nullptr && threadIdx.x == 0) {
        const int64_t rpb = a.rows_per_box;
        for (int64_t b = (row0 + rpb - 1) / rpb; b * rpb < row0 + NR && b * rpb < a.nrows; ++b)
            if (box_active(a.st, (int)b)) atomicAdd(a.units, 1);
    }
    auto live = [&](int r) { return row0 + r < a.nrows && box_active(a.st, (int)((row0 + r) / a.rows_per_box)); };
    // voxel offset of a row's first element in chi or the mask
    auto vox = [&](int r) {
        const int64_t row = row0 + r, b = row / a.rows_per_box;
        return (b * a.plane + row % a.plane) * a.bx;
    };
    if (FWD) {
        for (int t = threadIdx.x; t < NR * B; t += blockDim.x) {
            const int n2 = t & (B - 1), r = t / B;
            if (!live(r)) continue;
            const C* in = a.in + (row0 + r) * a.in_stride;
            const C* chi = a.chi + vox(r);
            C* row = sm + r * P;
            line_a_fwd<A, B>(n2, a.tw, [&](int n) { return n < a.n_in ? cmul(in[n], chi[n]) : czero<C>(); },
                             [&](int p, C v) { row[plane_pad(p)] = v; });
        }
    } else {
        for (int t = threadIdx.x; t < NR * L; t += blockDim.x) {
            const int r = t / L, p = t - r * L;
            if (live(r)) sm[r * P + plane_pad(p)] = a.in[(row0 + r) * a.in_stride + p];
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < NR * A; t += blockDim.x) {       // whole warps: 32 / A rows each
        const int k1 = t & (A - 1);
        C* row = sm + (t / A) * P;
        C v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = row[plane_pad(FWD ? k1 * B + i : line_brev<A, B>(k1, i))];
        line_b<A, B, FWD>(v, k1, a.tw);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < B; ++i) row[plane_pad(FWD ? line_brev<A, B>(k1, i) : k1 * B + i)] = v[i];
    }
    __syncthreads();
    if (FWD) {
        for (int t = threadIdx.x; t < NR * L; t += blockDim.x) {
            const int r = t / L, p = t - r * L;
            if (live(r)) a.out[(row0 + r) * a.out_stride + p] = sm[r * P + plane_pad(p)];
        }
    } else {
        for (int t = threadIdx.x; t < NR * B; t += blockDim.x) {
            const int n2 = t & (B - 1), r = t / B;
            if (!live(r)) continue;
            const C* row = sm + r * P;
            const C* xin = a.xin + (row0 + r) * a.out_stride;
            C* out = a.out + (row0 + r) * a.out_stride;
            const uint8_t* mask = a.mask ? a.mask + vox(r) : nullptr;
            C xv[A / 2];
            bool in[A / 2];
#pragma unroll
            for (int j = 0; j < A / 2; ++j) {
                const int x = j * B + n2;
                xv[j] = x < a.n_out ? xin[x] : czero<C>();
                in[j] = x < a.n_out && (mask == nullptr || mask[x]);
            }
            line_a_inv<A, B>(n2, a.tw, [&](int p) { return row[plane_pad(p)]; },
                             [&](int x, C u) {
                                 if (x < a.n_out) out[x] = in[x / B] ? xv[x / B] - u : czero<C>();
                             });
        }
    }
}

template <class C, int A, int B, bool FWD>
__global__ void __launch_bounds__(line_threads_col<C>()) k_line_cols(ColArgs<C> a) {
    pdl_wait();
    constexpr int NC = LineCols<C>::n;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* sm = reinterpret_cast<C*>(smem_raw);          // [L][NC]
    if (!box_active(a.st, blockIdx.z / a.b2_per_box)) return;
    if (a.units != nullptr && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z % a.b2_per_box == 0)
        atomicAdd(a.units, 1);
    const int col0 = blockIdx.x * NC, c = threadIdx.x % NC;
    const C* in = a.in + blockIdx.z * a.in_s2 + blockIdx.y * a.in_s1 + col0 + c;
    C* out = a.out + blockIdx.z * a.out_s2 + blockIdx.y * a.out_s1 + col0 + c;
    const bool live = col0 + c < a.ncols;
    C* col = sm + c;
    if (FWD) {
        for (int n2 = threadIdx.x / NC; n2 < B && live; n2 += line_threads_col<C>() / NC)
            line_a_fwd<A, B>(n2, a.tw, [&](int n) { return n < a.n_in ? in[n * a.in_axis] : czero<C>(); },
                             [&](int p, C v) { col[p * NC] = v; });
        __syncthreads();
        for (int k1 = threadIdx.x / NC; k1 < A && live; k1 += line_threads_col<C>() / NC) {
            C v[B];
#pragma unroll
            for (int i = 0; i < B; ++i) v[i] = col[(k1 * B + i) * NC];
            line_b<A, B, true>(v, k1, a.tw);
#pragma unroll
            for (int i = 0; i < B; ++i) out[line_brev<A, B>(k1, i) * a.out_axis] = v[i];
        }
    } else {
        for (int k1 = threadIdx.x / NC; k1 < A && live; k1 += line_threads_col<C>() / NC) {
            C v[B];
#pragma unroll
            for (int i = 0; i < B; ++i) v[i] = in[line_brev<A, B>(k1, i) * a.in_axis];
            line_b<A, B, false>(v, k1, a.tw);
#pragma unroll
            for (int i = 0; i < B; ++i) col[(k1 * B + i) * NC] = v[i];
        }
        __syncthreads();
        for (int n2 = threadIdx.x / NC; n2 < B && live; n2 += line_threads_col<C>() / NC)
            line_a_inv<A, B>(n2, a.tw, [&](int p) { return col[p * NC]; },
                             [&](int n, C v) {
                                 if (n < a.n_out) out[n * a.out_axis] = v;
                             });
    }
}

#define VIE_LONG_LINE_SWITCH(l, CALL)                                                  \
    switch (l) {                                                                       \
        case 6: { constexpr int AA = 8, BB = 8; CALL; }                                \
        case 7: { constexpr int AA = 16, BB = 8; CALL; }                               \
        case 8: { constexpr int AA = 16, BB = 16; CALL; }                              \
        default: { constexpr int AA = 32, BB = 16; CALL; }                             \
    }

}  // namespace vie

// Parity-split block MVM of the persistent block solver (inner.cu): boxes of up to 16 voxels per axis,
// both precisions.
//
// The circulant embedding of an axis of b <= H voxels needs 2H points. The transform of that length of
// a zero-padded line is two H-point transforms: of x_j (the even frequencies) and of x_j W_2H^j (the odd
// ones), and the inverse adds the two halves' results. So the padded 3D product splits into 8
// independent products, one per parity of (kz, ky, kx), each on a dense H_z x H_y x H_x grid no larger
// than the box: no padding is stored, moved or transformed. H is the smallest of 2, 4, 6, 8, 10, 12, 16
// that holds the block's own extent (not the power of two above its group's).
//
// A block is solved by a cluster of 4 CTAs; rank r takes the parities (pz, py) = (r >> 1, r & 1) and both
// parities of x. Per MVM:
//   update   each rank updates its quarter of the Krylov vectors and stores w = chi p into the shared
//            memory of all four ranks;                                            cluster barrier
//   z, y     twisted H-point transforms of the box's columns, in place;
//   x        one thread per (kz, ky) row, parity of x and all three components: transform, 3x3 Green
//            multiply and inverse transform in registers; two warps share 32 rows, the second adds its
//            parity's result to the first's, in place;
//   y, z     inverse transforms, in place;                                        cluster barrier
//   output   each rank adds the four ranks' results for its quarter of the voxels, out = mask (in - u),
//            with the iteration's inner products.
// complex128 is bound by the FP64 units (2 lanes per clock and SM), so there each rank owns a quarter of the
// z columns instead: it transforms its columns to both z parities in registers and stores them into the
// ranks that need them (and back), which halves the z transforms. In complex64 that form leaves three
// quarters of the threads idle in the update and lost (38 us per iteration of a 12 x 12 x 16 box, 28 us with
// elements; complex128 534 and 589 us).
// The spectrum is the octant of the frequencies split by parity: one load of the six components serves the
// frequencies kx and -kx of a row, and the rows of +-ky, +-kz of a warp read the same addresses. The signs
// of components odd along y and z are folded into the y and z transforms of the y and z components
// (diag(1, sy, sz) on both sides), the one along x into the multiply.
#pragma once

#include "dft_small.cuh"

namespace vie {

constexpr int kParRanks = 4;
// Three shapes in complex64. On chip: one CTA of 12 warps per SM, the Krylov vectors and the rank's spectrum in
// shared memory: the shortest iteration of a block (26.4 us for a 12 x 12 x 16 box, 33 us with the vectors in L2).
// L2: two CTAs of 6 warps per SM, which hide each other's barriers: the higher rate when many blocks queue (0.52 us
// per block iteration of the 256 metasurface pillars against 0.65). Small: four CTAs of 4 warps per SM, for boxes
// that leave most threads of more warps idle (256 blocks of 4 x 4 x 4: 38 us an iteration, 55 in the L2 shape; 256 of
// 8 x 8 x 16 88 and 124; 256 of 12 x 12 x 16 212 and 180).
// complex128 (FP64-bound): one CTA of 8 warps of 255 registers. The row stage pairs warps: a multiple of 64.
enum { PAR_NONE = 0, PAR_L2 = 1, PAR_CHIP = 2, PAR_SMALL = 3 };
template <class C, int PAR> __host__ __device__ constexpr int par_threads() {
    return sizeof(C) == 16 ? 256 : PAR == PAR_CHIP ? 384 : PAR == PAR_SMALL ? 128 : 192;
}
template <class C, int PAR> __host__ __device__ constexpr int par_ctas() {
    return sizeof(C) == 16 || PAR == PAR_CHIP ? 1 : PAR == PAR_SMALL ? 4 : 2;
}
// elements per thread whose loads are issued together (vectors in L2: 1, 2, 3 elements 41, 37, 36 us)
template <class C, bool CHIP> __host__ __device__ constexpr int par_batch() { return CHIP ? 1 : 3; }

// Extents below par_lo(H) + 1 take a smaller length: the first par_lo(H) + 1 entries of an axis of length H
// are always inside the block's extent (group_jobs widens extents that run with a larger length).
VIE_HD constexpr int par_lo(int H) { return H == 16 ? 12 : H - 2; }
VIE_HD constexpr int par_slot(int H) { return H == 16 ? 6 : H / 2 - 1; }

// exp(-i pi j / H) per length (par_slot), for the odd frequencies
static __constant__ float2 c_par64[7][16];
static __constant__ double2 c_par128[7][16];
template <class C> __device__ __forceinline__ C par_tw(int slot, int j);
template <> __device__ __forceinline__ float2 par_tw<float2>(int slot, int j) { return c_par64[slot][j]; }
template <> __device__ __forceinline__ double2 par_tw<double2>(int slot, int j) { return c_par128[slot][j]; }

// Whether a rank owns whole z columns (complex128) or single elements (complex64) of the box.
template <class C> __host__ __device__ constexpr bool par_by_column() { return sizeof(C) == 16; }

#define VIE_PAR_SWITCH(h, CALL)                               \
    switch (h) {                                              \
        case 2: { constexpr int HH = 2; CALL; } break;        \
        case 4: { constexpr int HH = 4; CALL; } break;        \
        case 6: { constexpr int HH = 6; CALL; } break;        \
        case 8: { constexpr int HH = 8; CALL; } break;        \
        case 10: { constexpr int HH = 10; CALL; } break;      \
        case 12: { constexpr int HH = 12; CALL; } break;      \
        default: { constexpr int HH = 16; CALL; } break;      \
    }

// Element i of the block's own extents: offset in the group's box vectors, voxel offset (chi, mask) and
// offset in the shared-memory array [3][hz][hy][yp].
struct ParIndex {
    int e, lv, so;
};
// The descriptor's fields that loops over elements need, in registers: stores through generic pointers
// could alias the descriptor in shared memory, which would then be read again for every element.
struct ParMap {
    FastDiv dxy, dx;
    int ex, exy, ez, bx, by, box, hz, hy, yp;
    template <class C> __device__ __forceinline__ explicit ParMap(const InnerGroup<C>& g)
        : dxy(fd_of(g.fd_exy)), dx(fd_of(g.fd_ex)), ex(g.ex), exy(g.ex * g.ey), ez(g.ez), bx(g.bx), by(g.by),
          box(g.bz * g.by * g.bx), hz(g.hz), hy(g.hy), yp(g.yp) {}
    __device__ __forceinline__ ParIndex operator()(int i) const {
        const int pl = (int)fdiv(i, dxy), yx = i - pl * exy;
        const int y = (int)fdiv(yx, dx), x = yx - y * ex;
        const int comp = (pl >= ez ? 1 : 0) + (pl >= 2 * ez ? 1 : 0), z = pl - comp * ez;
        ParIndex k;
        k.lv = (z * by + y) * bx + x;
        k.e = comp * box + k.lv;
        k.so = ((comp * hz + z) * hy + y) * yp + x;
        return k;
    }
};

// Column c (component, y, x) of the block's own extents: offset of its z = 0 element in the group's box
// vectors, in chi and the mask, and in the shared-memory array [3][hz][hy][yp].
struct ParCol {
    int comp, e, lv, so;
};
template <class C> __device__ __forceinline__ ParCol par_col(const InnerGroup<C>& g, int c) {
    const int exy = g.ex * g.ey, comp = (c >= exy ? 1 : 0) + (c >= 2 * exy ? 1 : 0), yx = c - comp * exy;
    const int y = (int)fdiv(yx, fd_of(g.fd_ex)), x = yx - y * g.ex;
    ParCol k;
    k.comp = comp;
    k.lv = y * g.bx + x;
    k.e = comp * g.bz * g.by * g.bx + k.lv;
    k.so = (comp * g.hz * g.hy + y) * g.yp + x;
    return k;
}
// Columns each rank owns.
template <class C> __host__ __device__ __forceinline__ int par_quarter(const InnerGroup<C>& g) {
    return (3 * g.ey * g.ex + kParRanks - 1) / kParRanks;
}
constexpr int kParColsMax = 3 * 16 * 16 / kParRanks;

template <class C> __host__ __device__ __forceinline__ int par_data_elems(const InnerGroup<C>& g) {
    return 3 * g.hz * g.hy * g.yp;
}
template <class C> __host__ __device__ __forceinline__ int par_rank_spec(const InnerGroup<C>& g) {
    return (g.hx + 1) * 6 * (g.hz / 2 + 1) * (g.hy / 2 + 1);
}

// Columns along z (AXIS 2) or y (AXIS 1) of the box in shared memory, H-point transforms in place, with
// the twist of parity p and the sign of the axis's own component. Forward reads the box's extent and
// writes H entries; inverse the other way round.
template <int H, bool FWD, int AXIS, class C>
__device__ __forceinline__ void par_cols(const InnerGroup<C>& g, C* sm, int p) {
    typedef typename real_of<C>::type R;
    constexpr int S = par_slot(H);
    const int zp = g.hy * g.yp;
    // z: every (y, x) of the rows y < ey, pad columns included (their garbage stays in the pad)
    const int cols = AXIS == 2 ? g.ey * g.yp : g.hz * g.ex, step = AXIS == 2 ? zp : g.yp;
    const int ext = AXIS == 2 ? g.ez : g.ey, ex = g.ex, cp = g.hz * zp;
    const FastDiv dx = fd_of(g.fd_ex);
    for (int q = threadIdx.x; q < 3 * cols; q += blockDim.x) {
        const int comp = (q >= cols ? 1 : 0) + (q >= 2 * cols ? 1 : 0);
        C* s;
        if (AXIS == 2) {
            s = sm + comp * cp + (q - comp * cols);
        } else {
            const int pl = (int)fdiv(q, dx);
            s = sm + pl * zp + (q - pl * ex);
        }
        const bool sg = comp == AXIS;
        C a[H];
        if (FWD) {
#pragma unroll
            for (int j = 0; j < H; ++j) a[j] = (j <= par_lo(H) || j < ext) ? s[j * step] : czero<C>();
            if (p) {
#pragma unroll
                for (int j = 1; j < H; ++j) a[j] = cmul(a[j], par_tw<C>(S, j));
            }
            dft<H, true>(a);
#pragma unroll
            for (int j = 0; j < H; ++j) s[j * step] = j >= H / 2 ? cneg_if(a[j], sg) : a[j];
        } else {
#pragma unroll
            for (int j = 0; j < H; ++j) a[j] = j >= H / 2 ? cneg_if(s[j * step], sg) : s[j * step];
            dft<H, false>(a);
            if (p) {
#pragma unroll
                for (int j = 1; j < H; ++j) a[j] = cmulc(a[j], par_tw<C>(S, j));
            }
#pragma unroll
            for (int j = 0; j < H; ++j)
                if (j <= par_lo(H) || j < ext) s[j * step] = a[j];
        }
    }
    __syncthreads();
}

// The frequencies kx = 2m + PX of one row: entries of frequency f = min(kx, 2H - kx) at gp[(6 f + c) n].
template <int H, int PX, class C> __device__ __forceinline__ void par_row_green(C (&a)[3][H], const C* gp, int n) {
    constexpr int NF = PX == 0 ? H / 2 + 1 : H / 2;
    C v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) v[c] = gp[(6 * PX + c) * n];
#pragma unroll
    for (int m = 0; m < NF; ++m) {
        C w[6];
        if (m + 1 < NF) {                         // the next frequency's entries while this one multiplies
#pragma unroll
            for (int c = 0; c < 6; ++c) w[c] = gp[(6 * (2 * (m + 1) + PX) + c) * n];
        }
        const int mm = (H - m - PX) % H;          // the mirror frequency
        green3<0, false>(a[0][m], a[1][m], a[2][m], v);
        if (mm != m) green3<0, true>(a[0][mm], a[1][mm], a[2][mm], v);
        if (m + 1 < NF) {
#pragma unroll
            for (int c = 0; c < 6; ++c) v[c] = w[c];
        }
    }
}

// Barrier of the warp pair that shares 32 rows (ids 1 ...; 0 is __syncthreads).
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

// One parity of x of the rows along x: one thread per (kz, ky) row, all components. Warps 2i and 2i + 1
// take the two parities of the same 32 rows; the even one stores its result, the odd one adds its own.
template <int H, int PX, class C>
__device__ __forceinline__ void par_rows_half(const InnerGroup<C>& g, C* sm, const C* G, int rk) {
    constexpr int S = par_slot(H);
    const int nrow = g.hz * g.hy, cp = nrow * g.yp, ex = g.ex;
    const int ny = g.hy / 2 + 1, nzy = (g.hz / 2 + 1) * ny;
    const int pz = rk >> 1, py = rk & 1;
    const int pair = threadIdx.x >> 6, npair = blockDim.x >> 6;
    for (int q0 = pair * 32; q0 < nrow; q0 += npair * 32) {
        const int q = q0 + (threadIdx.x & 31);
        const bool live = q < nrow;
        C a[3][H];
        C* s = sm + (live ? q : 0) * g.yp;
        const int kz = (int)fdiv(live ? q : 0, fd_of(g.fd_hy)), ky = (live ? q : 0) - kz * g.hy;
        const int iz = kz < g.hz / 2 + 1 - pz ? kz : g.hz - pz - kz;
        const int iy = ky < g.hy / 2 + 1 - py ? ky : g.hy - py - ky;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int j = 0; j < H; ++j) a[c][j] = (j <= par_lo(H) || j < ex) ? s[c * cp + j] : czero<C>();
        }
        pair_sync(1 + pair);                      // both parities hold the rows
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (PX) {
#pragma unroll
                for (int j = 1; j < H; ++j) a[c][j] = cmul(a[c][j], par_tw<C>(S, j));
            }
            dft<H, true>(a[c]);
        }
        par_row_green<H, PX>(a, G + iz * ny + iy, nzy);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dft<H, false>(a[c]);
            if (PX) {
#pragma unroll
                for (int j = 1; j < H; ++j) a[c][j] = cmulc(a[c][j], par_tw<C>(S, j));
            }
        }
        if (!PX && live) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < H; ++j)
                    if (j <= par_lo(H) || j < ex) s[c * cp + j] = a[c][j];
        }
        pair_sync(1 + pair);
        if (PX && live) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int j = 0; j < H; ++j)
                    if (j <= par_lo(H) || j < ex) s[c * cp + j] = s[c * cp + j] + a[c][j];
        }
    }
}

template <int H, bool STG, class C> __device__ __forceinline__ void par_rows(const InnerGroup<C>& g, C* sm, int rk) {
    const C* G = STG ? sm + par_data_elems(g) : g.Gq + (int64_t)rk * par_rank_spec(g);
    if (threadIdx.x & 32) par_rows_half<H, 1>(g, sm, G, rk);
    else par_rows_half<H, 0>(g, sm, G, rk);
    __syncthreads();
}

// The transforms and the Green multiply of this rank's parities, in place.
template <bool STG, class C> __device__ __noinline__ void par_mid(const InnerGroup<C>& g, C* sm, int rk) {
    if (!par_by_column<C>()) VIE_PAR_SWITCH(g.hz, (par_cols<HH, true, 2>(g, sm, rk >> 1)));
    VIE_PAR_SWITCH(g.hy, (par_cols<HH, true, 1>(g, sm, rk & 1)));
    VIE_PAR_SWITCH(g.hx, (par_rows<HH, STG>(g, sm, rk)));
    VIE_PAR_SWITCH(g.hy, (par_cols<HH, false, 1>(g, sm, rk & 1)));
    if (!par_by_column<C>()) VIE_PAR_SWITCH(g.hz, (par_cols<HH, false, 2>(g, sm, rk >> 1)));
}

// ---------------------------------------------------------------- the block's BiCGSTAB
// Team-wide sums of the N complex values v of every thread; fn(sums) runs in warp 0 of every CTA with
// identical arguments and writes the shared state the closing barrier publishes. Each warp halves its
// values over the lanes (2N real values take 2N - 1 + (5 - log2 2N) shuffles, in the vectors' precision),
// its lanes store them into the slot of all four ranks, and after one cluster barrier N warps add the
// warps' and ranks' sums in FP64, one complex value each. What counts there is the number of FP64
// instructions: each holds a quarter SM's unit for 64 clocks whatever the number of active lanes (a serial
// form, thread 0 adding everything, cost 9 us of a 22 us product), so the additions are spread over the
// quarters and lanes, and fn works on real and imaginary parts in different lanes. Two slots alternate: a
// slot is rewritten two sums later, after the cluster barrier of the sum in between.
constexpr int kParWarpsMax = 12;
template <class C> struct ParSums {
    typename real_of<C>::type v[2][kParRanks][kParWarpsMax][8];
    double2 tot[4];
};

template <int NW, int N, class C, class Fn>
__device__ __forceinline__ void par_sum(C (&v)[N], ParSums<C>& xs, int& slot, Fn fn) {
    typedef typename real_of<C>::type R;
    constexpr int NV = 2 * N;
    static_assert(NV == 2 || NV == 8, "par_sum: one or four values");
    R x[NV];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        x[2 * i] = v[i].x;
        x[2 * i + 1] = v[i].y;
    }
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    int o = 16;
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (l & o) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const R send = up ? x[k] : x[k + h], keep = up ? x[k + h] : x[k];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o >= 1; o >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
    // value index of the lane: its upper log2 NV bits; the lanes that share it serve the four ranks
    const int vi = NV == 8 ? l >> 2 : l >> 4, dst = NV == 8 ? l & 3 : l & 15;
    cg::cluster_group cl = cg::this_cluster();
    const int rk = (int)cl.block_rank();
    slot ^= 1;
    if (dst < kParRanks) *cl.map_shared_rank(&xs.v[slot][rk][w][vi], (unsigned)dst) = x[0];
    cl.sync();
    if (w < N) {
        // warp w: complex value w; lane l: component l & 1 of every 16th partial sum, added as a tree
        constexpr int ALL = kParRanks * NW, PER = (ALL + 15) / 16;
        double u[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int k = (l >> 1) + 16 * i;
            u[i] = ALL % 16 == 0 || k < ALL ? (double)xs.v[slot][k & (kParRanks - 1)][k / kParRanks][2 * w + (l & 1)] : 0.0;
        }
#pragma unroll
        for (int h = PER; h > 1; h = (h + 1) / 2) {
#pragma unroll
            for (int i = 0; i < h / 2; ++i) u[i] += u[i + (h + 1) / 2];
        }
        double s = u[0];
#pragma unroll
        for (int m = 2; m < 32; m <<= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        if (l < 2) (l ? xs.tot[w].y : xs.tot[w].x) = s;
        if (N > 1) asm volatile("bar.sync 15, %0;" ::"n"(32 * N) : "memory");
        else __syncwarp();
        if (w == 0) fn(xs.tot, l);
    }
    __syncthreads();
}

// Finite, and not zero: integer tests, an FP64 comparison takes 64 clocks.
__device__ __forceinline__ bool par_finite(double a) { return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool par_zero(double a) { return ((__double2hiint(a) & 0x7fffffff) | __double2loint(a)) == 0; }
__device__ __forceinline__ double par_lane(double a, int lane) { return __shfl_sync(0xffffffffu, a, lane); }
// component c (0, 1) of a complex number
template <class C2, class T> __device__ __forceinline__ void par_put(C2& z, int c, T v) { (c ? z.y : z.x) = v; }

// Scalars of the iteration, written by warp 0 inside par_sum.
template <class C> struct ParState {
    double2 rho, iq;                            // iq = 1 / <rhat, v>
    double tol2, bn2, res2;
    int halves;                                 // half steps done
    int status, half, pend;                     // pend: the last full step's x update is pending
    C cbeta, comega, calpha;                    // coefficients of the vector updates
};

// Where the Krylov vectors of this rank's quarter live while a block is solved. Each thread works on the
// same elements in every phase, so nothing here is shared between threads. CHIP: in shared memory behind
// the data and the spectrum, with chi, the mask and the element's place in the data (complex64 boxes that
// leave room); otherwise in the group's global vectors.
template <class C, bool CHIP> struct ParVecs {
    C *x, *r, *rhat, *p, *v, *s, *t;
    const C* chi;
    const uint8_t* mask;
    unsigned* so;                               // CHIP: place in the data, bit 31: in the block
    int n0, n;                                  // first element of the quarter, elements in it
};
// vectors (and chi) of one element on chip, and its place
template <class C> __host__ __device__ constexpr int par_chip_bytes() { return 8 * (int)sizeof(C) + 4; }

enum { PAR_P = 0, PAR_PX = 1, PAR_S = 2 };

// Update of this rank's quarter (PAR_P: p = r + c1 (p - c2 v); PAR_S: s = r - c1 v; PAR_PX: the previous
// step's r = s - c2 t and x += c3 p + c2 s, then p = r + c1 (p - c2 v)); w = chi in to every rank. Returns
// this thread's part of ||s||^2 (PAR_S).
template <int IN, bool CHIP, class C>
__device__ __forceinline__ typename real_of<C>::type par_update(const InnerGroup<C>& g, const ParVecs<C, CHIP>& Vs, C* sm, C c1,
                                                                C c2, C c3) {
    const ParVecs<C, CHIP> V = Vs;
    const ParMap map(g);
    constexpr int UV = par_batch<C, CHIP>();
    typename real_of<C>::type acc = 0;
    cg::cluster_group cl = cg::this_cluster();
    C* dst[kParRanks];
#pragma unroll
    for (int r = 0; r < kParRanks; ++r) dst[r] = cl.map_shared_rank(sm, (unsigned)r);
    for (int i0 = threadIdx.x; i0 < V.n; i0 += UV * blockDim.x) {
        int e[UV], so[UV];
        C ch[UV], ra[UV], va[UV], pa[UV], ta[UV], xa[UV];
#pragma unroll
        for (int u = 0; u < UV; ++u) {           // every load of the batch first
            const int i = min(i0 + u * (int)blockDim.x, V.n - 1);
            if (CHIP) {
                e[u] = i;
                so[u] = (int)(V.so[i] & 0x7fffffffu);
                ch[u] = V.chi[i];
            } else {
                const ParIndex k = map(V.n0 + i);
                e[u] = k.e;
                so[u] = k.so;
                ch[u] = V.chi[k.lv];
            }
            ra[u] = IN == PAR_PX ? V.s[e[u]] : V.r[e[u]];
            va[u] = V.v[e[u]];
            if (IN != PAR_S) pa[u] = V.p[e[u]];
            if (IN == PAR_PX) {
                ta[u] = V.t[e[u]];
                xa[u] = V.x[e[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < UV; ++u) {
            if (i0 + u * (int)blockDim.x >= V.n) continue;
            C in;
            if (IN == PAR_PX) {
                const C r = ra[u] - cmul(c2, ta[u]);
                V.r[e[u]] = r;
                V.x[e[u]] = xa[u] + cmul(c3, pa[u]) + cmul(c2, ra[u]);
                in = r + cmul(c1, pa[u] - cmul(c2, va[u]));
                V.p[e[u]] = in;
            } else if (IN == PAR_P) {
                in = ra[u] + cmul(c1, pa[u] - cmul(c2, va[u]));
                V.p[e[u]] = in;
            } else {
                in = ra[u] - cmul(c1, va[u]);
                V.s[e[u]] = in;
                acc += in.x * in.x + in.y * in.y;
            }
            const C w = cmul(in, ch[u]);
#pragma unroll
            for (int r = 0; r < kParRanks; ++r) dst[r][so[u]] = w;
        }
    }
    return acc;
}

// Output of this rank's quarter: the four ranks' results added, v = mask (p - u) with <rhat, v> (T false)
// or t = mask (s - u) with <t, s>, <t, t>, <rhat, s>, <rhat, t> (T true). The sum that follows (its cluster
// barrier) also ends every read of the ranks' results.
template <bool T, bool CHIP, class C>
__device__ __forceinline__ void par_output(const InnerGroup<C>& g, const ParVecs<C, CHIP>& Vs, C* sm, C (&acc)[4]) {
    const ParVecs<C, CHIP> V = Vs;
    const ParMap map(g);
    constexpr int UV = par_batch<C, CHIP>();
    cg::cluster_group cl = cg::this_cluster();
    const C* src[kParRanks];
#pragma unroll
    for (int r = 0; r < kParRanks; ++r) src[r] = cl.map_shared_rank(sm, (unsigned)r);
    for (int i0 = threadIdx.x; i0 < V.n; i0 += UV * blockDim.x) {
        int e[UV];
        bool in[UV];
        C ua[UV][kParRanks], ha[UV], ba[UV];
#pragma unroll
        for (int u = 0; u < UV; ++u) {
            const int i = min(i0 + u * (int)blockDim.x, V.n - 1);
            int so;
            if (CHIP) {
                e[u] = i;
                so = (int)(V.so[i] & 0x7fffffffu);
                in[u] = (V.so[i] >> 31) != 0;
            } else {
                const ParIndex k = map(V.n0 + i);
                e[u] = k.e;
                so = k.so;
                in[u] = V.mask[k.lv] != 0;
            }
            ha[u] = V.rhat[e[u]];
            ba[u] = T ? V.s[e[u]] : V.p[e[u]];
#pragma unroll
            for (int r = 0; r < kParRanks; ++r) ua[u][r] = src[r][so];
        }
#pragma unroll
        for (int u = 0; u < UV; ++u) {
            if (i0 + u * (int)blockDim.x >= V.n) continue;
            const C o = in[u] ? ba[u] - ((ua[u][0] + ua[u][1]) + (ua[u][2] + ua[u][3])) : czero<C>();
            if (T) {
                V.t[e[u]] = o;
                acc_dot(acc[0], o, ba[u]);
                acc[1].x += o.x * o.x + o.y * o.y;
                acc_dot(acc[2], ha[u], ba[u]);
                acc_dot(acc[3], ha[u], o);
            } else {
                V.v[e[u]] = o;
                acc_dot(acc[0], ha[u], o);
            }
        }
    }
}

// The same by columns: update, and the z transforms of both parities into the data of the ranks that
// work on them; a column is read and written by its thread alone.
template <int H, int IN, class C>
__device__ __noinline__ typename real_of<C>::type par_update_cols(const InnerGroup<C>& g, const ParVecs<C, false>& Vs, C* sm, C c1, C c2,
                                                             C c3) {
    typedef typename real_of<C>::type R;
    constexpr int S = par_slot(H), B = 4;         // z planes whose loads are issued together
    const ParVecs<C, false> V = Vs;
    R acc = 0;
    cg::cluster_group cl = cg::this_cluster();
    C* dst[kParRanks];
#pragma unroll
    for (int r = 0; r < kParRanks; ++r) dst[r] = cl.map_shared_rank(sm, (unsigned)r);
    const int zp = g.hy * g.yp, ez = g.ez, st = g.by * g.bx;
    for (int c = threadIdx.x; c < V.n; c += blockDim.x) {
        const ParCol k = par_col(g, V.n0 + c);
        const int e0 = k.e, l0 = k.lv;
        C a[H];
#pragma unroll
        for (int j0 = 0; j0 < H; j0 += B) {
            C ra[B], va[B], pa[B], ta[B], xa[B], ch[B];
#pragma unroll
            for (int u = 0; u < B; ++u) {        // every load of the batch first
                const int j = j0 + u, e = e0 + j * st;
                if (j < H && (j <= par_lo(H) || j < ez)) {
                    ra[u] = IN == PAR_PX ? V.s[e] : V.r[e];
                    va[u] = V.v[e];
                    if (IN != PAR_S) pa[u] = V.p[e];
                    if (IN == PAR_PX) {
                        ta[u] = V.t[e];
                        xa[u] = V.x[e];
                    }
                    ch[u] = V.chi[l0 + j * st];
                }
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int j = j0 + u, e = e0 + j * st;
                if (j >= H) continue;
                a[j] = czero<C>();
                if (j <= par_lo(H) || j < ez) {
                    C in;
                    if (IN == PAR_PX) {
                        const C r = ra[u] - cmul(c2, ta[u]);
                        V.r[e] = r;
                        V.x[e] = xa[u] + cmul(c3, pa[u]) + cmul(c2, ra[u]);
                        in = r + cmul(c1, pa[u] - cmul(c2, va[u]));
                        V.p[e] = in;
                    } else if (IN == PAR_P) {
                        in = ra[u] + cmul(c1, pa[u] - cmul(c2, va[u]));
                        V.p[e] = in;
                    } else {
                        in = ra[u] - cmul(c1, va[u]);
                        V.s[e] = in;
                        acc += in.x * in.x + in.y * in.y;
                    }
                    a[j] = cmul(in, ch[u]);
                }
            }
        }
        const bool sg = k.comp == 2;
        C b[H];
#pragma unroll
        for (int j = 0; j < H; ++j) b[j] = a[j];
        dft<H, true>(b);
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const C o = j >= H / 2 ? cneg_if(b[j], sg) : b[j];
            dst[0][k.so + j * zp] = o;
            dst[1][k.so + j * zp] = o;
        }
#pragma unroll
        for (int j = 1; j < H; ++j) a[j] = cmul(a[j], par_tw<C>(S, j));
        dft<H, true>(a);
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const C o = j >= H / 2 ? cneg_if(a[j], sg) : a[j];
            dst[2][k.so + j * zp] = o;
            dst[3][k.so + j * zp] = o;
        }
    }
    return acc;
}

// Output of this rank's columns: the ranks' results of each z parity added, inverse z transforms, parities
// added; v = mask (p - u) with <rhat, v> in acc[0] (T false) or t = mask (s - u) with <t, s>, <t, t>,
// <rhat, s>, <rhat, t> (T true). The sum that follows (its cluster barrier) also ends every read of the
// ranks' results.
template <int H, bool T, class C>
__device__ __noinline__ void par_output_cols(const InnerGroup<C>& g, const ParVecs<C, false>& Vs, C* sm, const unsigned* zmask,
                                        C (&out)[4]) {
    typedef typename real_of<C>::type R;
    constexpr int S = par_slot(H), B = 4;
    const ParVecs<C, false> V = Vs;
    C acc[4] = {czero<C>(), czero<C>(), czero<C>(), czero<C>()};
    cg::cluster_group cl = cg::this_cluster();
    const C* src[kParRanks];
#pragma unroll
    for (int r = 0; r < kParRanks; ++r) src[r] = cl.map_shared_rank(sm, (unsigned)r);
    const int zp = g.hy * g.yp, ez = g.ez, st = g.by * g.bx;
    for (int c = threadIdx.x; c < V.n; c += blockDim.x) {
        const ParCol k = par_col(g, V.n0 + c);
        const int e0 = k.e;
        const bool sg = k.comp == 2;
        C a[H], b[H];
#pragma unroll
        for (int j = 0; j < H; ++j) a[j] = src[0][k.so + j * zp] + src[1][k.so + j * zp];
#pragma unroll
        for (int j = 0; j < H; ++j) b[j] = src[2][k.so + j * zp] + src[3][k.so + j * zp];
#pragma unroll
        for (int j = H / 2; j < H; ++j) {
            a[j] = cneg_if(a[j], sg);
            b[j] = cneg_if(b[j], sg);
        }
        dft<H, false>(a);
        dft<H, false>(b);
        a[0] = a[0] + b[0];
#pragma unroll
        for (int j = 1; j < H; ++j) a[j] = a[j] + cmulc(b[j], par_tw<C>(S, j));
        const unsigned m = zmask[c];
#pragma unroll
        for (int j0 = 0; j0 < H; j0 += B) {
            C ha[B], ba[B];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int j = j0 + u, e = e0 + j * st;
                if (j < H && (j <= par_lo(H) || j < ez)) {
                    ha[u] = V.rhat[e];
                    ba[u] = T ? V.s[e] : V.p[e];
                }
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int j = j0 + u, e = e0 + j * st;
                if (j < H && (j <= par_lo(H) || j < ez)) {
                    const C o = (m >> j) & 1 ? ba[u] - a[j] : czero<C>();
                    if (T) {
                        V.t[e] = o;
                        acc_dot(acc[0], o, ba[u]);
                        acc[1].x += o.x * o.x + o.y * o.y;
                        acc_dot(acc[2], ha[u], ba[u]);
                        acc_dot(acc[3], ha[u], o);
                    } else {
                        V.v[e] = o;
                        acc_dot(acc[0], ha[u], o);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < (T ? 4 : 1); ++i) out[i] = acc[i];
}

// One block's BiCGSTAB from x = 0 to ||r|| <= tol ||b|| on a cluster of kParRanks CTAs, in the merged form:
// r = s - omega t and x += alpha p + omega s are applied in the next p update, and <rhat, r> = <rhat, s> -
// omega <rhat, t> and ||r||^2 = ||s||^2 - |<t, s>|^2 / ||t||^2 come from the sums of the t pass. That difference
// carries the rounding of the sums (in complex64 it can be negative where r is 2e-4 of s), so a block stops on it only
// when ||s|| is near enough to the tolerance; where it does not decide, the next half step does, on ||s||^2 itself.
// (Summing ||r||^2 over r = s - omega t instead, rare as it is, cost 2 to 10 % of every solve in registers.)
template <int PAR, class C>
__device__ __forceinline__ void par_solve(const InnerGroup<C>& g, int b, double tol, int maxit, C* sm, int* units) {
    typedef typename real_of<C>::type R;
    constexpr bool STG = sizeof(C) == 8, COLS = par_by_column<C>(), CHIP = PAR == PAR_CHIP;
    constexpr int NW = par_threads<C, PAR>() / 32;
    // a lone warp would wait in pair_sync for ever; par_sum has a slot for each warp, and four of them add
    static_assert(par_threads<C, PAR>() % 64 == 0 && NW >= 4 && NW <= kParWarpsMax, "par_solve: threads per CTA");
    __shared__ ParState<C> S;
    __shared__ ParSums<C> xs;
    __shared__ ParVecs<C, CHIP> V;
    __shared__ unsigned zmask[COLS ? kParColsMax : 1];
    const int64_t box = (int64_t)g.bx * g.by * g.bz, voff = (int64_t)b * 3 * box;
    const int rk = team_rank();
    int slot = 0;
    if (threadIdx.x == 0) {
        // this rank's quarter, of columns or of elements
        const int all = (COLS ? 1 : g.ez) * 3 * g.ey * g.ex, n4 = (all + kParRanks - 1) / kParRanks;
        V.n0 = rk * n4;
        V.n = max(0, min(all - V.n0, n4));
        if (CHIP) {
            C* p = sm + par_data_elems(g) + par_rank_spec(g);
            V.x = p; V.r = p + n4; V.rhat = p + 2 * n4; V.p = p + 3 * n4; V.v = p + 4 * n4; V.s = p + 5 * n4; V.t = p + 6 * n4;
            V.chi = p + 7 * n4;
            V.so = reinterpret_cast<unsigned*>(p + 8 * n4);
        } else {
            V.x = g.x + voff; V.r = g.r + voff; V.rhat = g.rhat + voff; V.p = g.p + voff; V.v = g.v + voff;
            V.s = g.s + voff; V.t = g.t + voff;
            V.chi = g.chi + (int64_t)b * box;
            V.mask = g.mask + (int64_t)b * box;
        }
    }
    if (STG) {                                  // the rank's spectrum, for every MVM of the block
        const int n = par_rank_spec(g);
        const C* src = g.Gq + (int64_t)rk * n;
        C* dst = sm + par_data_elems(g);
        for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();

    // fn(place in V's vectors, offset in the box vectors, voxel) over this thread's elements
    const ParMap map(g);
    auto own = [&](auto fn) {
        for (int i = threadIdx.x; i < V.n; i += blockDim.x) {
            if constexpr (COLS) {
                const ParCol k = par_col(g, V.n0 + i);
                for (int z = 0; z < g.ez; ++z) {
                    const int o = z * g.by * g.bx;
                    fn(k.e + o, k.e + o, k.lv + o);
                }
            } else {
                const ParIndex k = map(V.n0 + i);
                if (CHIP) V.so[i] = (unsigned)k.so | (g.mask[(int64_t)b * box + k.lv] ? 0x80000000u : 0u);
                fn(CHIP ? i : k.e, k.e, k.lv);
            }
        }
    };
    // x = 0, r = rhat = b, p = v = 0
    C a0[1] = {czero<C>()};
    own([&](int e, int ge, int lv) {
        const C bv = g.b[voff + ge];
        if (CHIP) const_cast<C*>(V.chi)[e] = g.chi[(int64_t)b * box + lv];
        V.x[e] = czero<C>();
        V.r[e] = bv;
        V.rhat[e] = bv;
        V.p[e] = czero<C>();
        V.v[e] = czero<C>();
        a0[0].x += bv.x * bv.x + bv.y * bv.y;
    });
    if constexpr (COLS) {
        for (int c = threadIdx.x; c < V.n; c += blockDim.x) {
            const ParCol k = par_col(g, V.n0 + c);
            unsigned m = 0;
            for (int z = 0; z < g.ez; ++z) m |= (V.mask[k.lv + z * g.by * g.bx] ? 1u : 0u) << z;
            zmask[c] = m;
        }
    }
    par_sum<NW>(a0, xs, slot, [&](const double2* q, int) {
        const double bn2 = q[0].x;
        S.bn2 = bn2;
        S.tol2 = tol * tol * bn2;
        S.rho = make_double2(bn2, 0.0);
        S.comega = cmk<C>(1.0, 0.0);
        S.halves = 0;
        S.res2 = bn2;
        S.half = 0;
        S.pend = 0;
        S.status = SEG_ACTIVE;
        if (!(bn2 > 0.0) || !isfinite(bn2)) S.status = bn2 == 0.0 ? SEG_CONVERGED : SEG_BREAKDOWN;
        else if (bn2 <= S.tol2) S.status = SEG_CONVERGED;   // x = 0 meets a tolerance of 1 or more
        else S.cbeta = cmk<C>(bn2, 0.0);        // (rho / 1) (1 / 1); p = v = 0
    });
    for (int it = 0; it < maxit && S.status == SEG_ACTIVE; ++it) {
        if constexpr (COLS) {
            if (it == 0) {
                VIE_PAR_SWITCH(g.hz, (par_update_cols<HH, PAR_P>(g, V, sm, S.cbeta, S.comega, czero<C>())));
            } else {
                VIE_PAR_SWITCH(g.hz, (par_update_cols<HH, PAR_PX>(g, V, sm, S.cbeta, S.comega, S.calpha)));
            }
        } else {
            if (it == 0) par_update<PAR_P>(g, V, sm, S.cbeta, S.comega, czero<C>());
            else par_update<PAR_PX>(g, V, sm, S.cbeta, S.comega, S.calpha);
        }
        team_sync();                            // the data complete on every rank
        par_mid<STG>(g, sm, rk);
        team_sync();                            // every rank's result in its shared memory
        if (units != nullptr && rk == 0 && threadIdx.x == 0) atomicAdd(units, g.kb_mvm);
        C q4[4] = {czero<C>(), czero<C>(), czero<C>(), czero<C>()};
        if constexpr (COLS) {
            VIE_PAR_SWITCH(g.hz, (par_output_cols<HH, false>(g, V, sm, zmask, q4)));
        } else {
            par_output<false>(g, V, sm, q4);
        }
        C p1[1] = {q4[0]};
        par_sum<NW>(p1, xs, slot, [&](const double2* q, int l) {
            const double2 z = q[0], rho = S.rho;
            const int c = l & 1;                // real and imaginary parts in lanes
            S.pend = 0;                         // the p update took the previous step's x update
            if (!par_finite(z.x) || !par_finite(z.y) || (par_zero(z.x) && par_zero(z.y))) {
                S.status = SEG_BREAKDOWN;
                return;
            }
            const double d = 1.0 / (z.x * z.x + z.y * z.y), iq = (c ? -z.y : z.x) * d;
            const double alpha = fma(rho.x, iq, (c ? rho.y : -rho.y) * __shfl_xor_sync(0xffffffffu, iq, 1));
            if (l < 2) {
                par_put(S.iq, c, iq);
                par_put(S.calpha, c, (R)alpha);
            }
        });
        if (S.status != SEG_ACTIVE) break;
        R sn = 0;
        if constexpr (COLS) {
            VIE_PAR_SWITCH(g.hz, (sn = par_update_cols<HH, PAR_S>(g, V, sm, S.calpha, czero<C>(), czero<C>())));
        } else {
            sn = par_update<PAR_S>(g, V, sm, S.calpha, czero<C>(), czero<C>());
        }
        team_sync();
        par_mid<STG>(g, sm, rk);
        team_sync();
        if (units != nullptr && rk == 0 && threadIdx.x == 0) atomicAdd(units, g.kb_mvm);
        q4[0] = q4[1] = q4[2] = q4[3] = czero<C>();
        if constexpr (COLS) {
            VIE_PAR_SWITCH(g.hz, (par_output_cols<HH, true>(g, V, sm, zmask, q4)));
        } else {
            par_output<true>(g, V, sm, q4);
        }
        q4[1].y = sn;                           // the deferred ||s||^2 rides in the unused slot
        // omega = <t, s> / ||t||^2, rho, ||r||^2 and beta: with alpha = rho_prev / <rhat, v>, beta = (rho / rho_prev)
        // (alpha / omega) = (rho / omega) iq = (<rhat, s> / omega - <rhat, t>) iq. Lanes 0, 1: rho; 2, 3: beta;
        // 4: ||r||^2 (15 FP64 instructions a warp where one thread's scalars took about 60 and 1.3 us).
        par_sum<NW>(q4, xs, slot, [&](const double2* q, int l) {
            const double2 ts = q[0], rs = q[2], rt = q[3], iq = S.iq;
            const double tt = q[1].x, sn2 = q[1].y, tol2 = S.tol2;
            const int c = l & 1, g = l >> 1;
            const double d = 1.0 / (c ? ts.x * ts.x + ts.y * ts.y : tt);
            const double itt = par_lane(d, 0), inn = par_lane(d, 1);
            const double m = (g == 1 ? tt : c ? ts.y : ts.x) * (g == 1 ? inn : itt);     // omega; tt / |ts|^2
            const double ox = par_lane(m, 0), oy = par_lane(m, 1), io = par_lane(m, 2);
            const double w = (c ? -ts.y : ts.x) * io;                                    // 1 / omega
            const double wx = par_lane(w, 0), wy = par_lane(w, 1);
            const double base = g == 0 ? (c ? rs.y : rs.x) : g == 1 ? (c ? -rt.y : -rt.x) : sn2;
            const double m1 = g == 0 ? -ox : g == 1 ? rs.x : -ts.x;
            const double k1 = g == 0 ? (c ? rt.y : rt.x) : g == 1 ? (c ? wy : wx) : ox;
            const double m2 = g == 0 ? (c ? -oy : oy) : g == 1 ? (c ? rs.y : -rs.y) : -ts.y;
            const double k2 = g == 0 ? (c ? rt.x : rt.y) : g == 1 ? (c ? wx : wy) : oy;
            const double v = fma(m2, k2, fma(m1, k1, base));                             // rho; rho / omega; ||r||^2
            const double beta = fma(v, iq.x, (c ? iq.y : -iq.y) * __shfl_xor_sync(0xffffffffu, v, 1));
            const double rhox = par_lane(v, 0), rhoy = par_lane(v, 1);
            const double res2 = par_lane(v, 4);
            const R coef = (R)(g == 0 ? m : beta);
            const unsigned le = __ballot_sync(0xffffffffu, (l == 0 ? sn2 : l == 1 ? res2 : tt) <= (l < 2 ? tol2 : 0.0));
            if (le & 1u) {
                S.half = 1;
                S.res2 = sn2;
                if (l == 0) S.halves += 1;
                S.status = SEG_CONVERGED;
                return;
            }
            if ((le & 4u) || !par_finite(tt)) {
                S.status = SEG_BREAKDOWN;
                return;
            }
            if (g == 0) {
                par_put(S.comega, c, coef);
                par_put(S.rho, c, v);
            } else if (g == 1) {
                par_put(S.cbeta, c, coef);
            }
            S.pend = 1;
            S.res2 = res2;
            if (l == 0) S.halves += 2;
            if (!par_finite(res2)) S.status = SEG_BREAKDOWN;
            // The sums round by 1.3e-5 of ||s||^2 at most in complex64 (24 elements a thread, 5 shuffles, the products;
            // 1e-7 as a rule) and 2.5e-14 in complex128: res2 decides while ||s||^2 is below 2^12 (2^36) times the square
            // of the tolerance. (By the exponents: one FP64 instruction more here cost 1 % of an iteration.)
            else if ((le & 2u) && (__double2hiint(sn2) < __double2hiint(tol2) + ((sizeof(C) == 8 ? 12 : 36) << 20) ||
                                   (par_zero(rhox) && par_zero(rhoy))))
                S.status = SEG_CONVERGED;
            else if ((par_zero(ox) && par_zero(oy)) || !par_finite(rhox) || !par_finite(rhoy) || (par_zero(rhox) && par_zero(rhoy)))
                S.status = SEG_BREAKDOWN;
        });
    }
    // x of a half step (x += alpha p) or of the last full step (no p update followed it)
    const C ac = S.calpha, oc = S.comega;
    own([&](int e, int ge, int) {
        C x = V.x[e];
        if (S.half) x = x + cmul(ac, V.p[e]);
        else if (S.pend) x = x + cmul(ac, V.p[e]) + cmul(oc, V.s[e]);
        g.x[voff + ge] = x;
    });
    if (rk == 0 && threadIdx.x == 0) {
        SegState& St = g.st[b];
        St.bnorm2 = S.bn2;
        St.res2 = S.res2;
        St.iters = 0.5 * S.halves;
        St.status = S.status == SEG_ACTIVE ? SEG_MAXIT : S.status;
        St.maxit = maxit;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- host side and spectra
// exp(-i pi j / H) into this translation unit's constant tables, once per device.
static int par_twiddles_ready() {
    static std::mutex mu;
    static std::vector<int> devs;
    int dev = 0;
    VIE_CK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (std::find(devs.begin(), devs.end(), dev) != devs.end()) return VIE_OK;
    float2 h64[7][16] = {};
    double2 h128[7][16] = {};
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int H : {2, 4, 6, 8, 10, 12, 16})
        for (int j = 0; j < H; ++j) {
            const long double th = pi * j / H;
            h128[par_slot(H)][j] = make_double2((double)cosl(th), (double)-sinl(th));
            h64[par_slot(H)][j] = make_float2((float)cosl(th), (float)-sinl(th));
        }
    VIE_CK(cudaMemcpyToSymbol(c_par64, h64, sizeof(h64)));
    VIE_CK(cudaMemcpyToSymbol(c_par128, h128, sizeof(h128)));
    VIE_CK(cudaDeviceSynchronize());   // a non-blocking stream does not wait for the legacy stream's copies
    devs.push_back(dev);
    return VIE_OK;
}

}  // namespace vie

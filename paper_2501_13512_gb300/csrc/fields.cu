// Field-level kernels: Green-tensor lattice samples (Eq. 1), incident plane
// wave, precision conversion, and the block restriction/prolongation of the
// block-diagonal preconditioner (Eq. 10).
#include <math.h>

#include <cmath>

#include "vie_internal.cuh"

namespace vie {

static unsigned grid_1d(int64_t n, int per_thread = 1) {
    int64_t g = (n + 256LL * per_thread - 1) / (256LL * per_thread);
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 32));
}

// Slot m of an axis of padded length M stores lattice offset m (m < b) or
// m - M (m > M - b); other slots are unused by any product of two in-box
// voxels (circulant embedding of the Toeplitz sum) and hold zero.
__device__ __forceinline__ bool wrap_offset(int m, int M, int b, int& d) {
    if (m < b) { d = m; return true; }
    if (m > M - b) { d = m - M; return true; }
    return false;
}

// The six components of k0^2 G(r) h^3 `scale` at a point r != 0 (Eq. 1:
// k^2 G = g [(k^2 - jk/R - 1/R^2) I + (-k^2 + 3jk/R + 3/R^2) rhat rhat]), added to K.
__device__ __forceinline__ void add_k2G(double rx, double ry, double rz, double k0, double hs, double wgt,
                                        double2 (&K)[6]) {
    const double inv4pi = 0.25 / 3.14159265358979323846;
    const double R2 = rx * rx + ry * ry + rz * rz;
    const double R = sqrt(R2);
    double sn, cs;
    sincos(k0 * R, &sn, &cs);
    // g h^3 scale = e^{-jkR} / (4 pi R) h^3 scale
    const double gm = inv4pi / R * hs * wgt;
    const double2 g = make_double2(cs * gm, -sn * gm);
    const double2 a = make_double2(k0 * k0 - 1.0 / R2, -k0 / R);
    const double2 b = make_double2(-k0 * k0 + 3.0 / R2, 3.0 * k0 / R);
    const double2 ga = cmul(g, a), gb = cmul(g, b);
    const double u[3] = {rx / R, ry / R, rz / R};
    const int P[6] = {0, 0, 0, 1, 1, 2}, Q[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const double uu = u[P[c]] * u[Q[c]];
        double2 v = make_double2(gb.x * uu, gb.y * uu);
        if (P[c] == Q[c]) v = v + ga;
        K[c] = K[c] + v;
    }
}

// K(D) = k0^2 G(D h) h^3 for D != 0 and s_self I at D = 0, times `scale`
// (1 / (Mx My Mz), the inverse-FFT normalisation folded into the spectrum);
// offsets with 0 < max|D| <= near.radius take the mean of k0^2 G over the cube
// of side h around D h instead (tensor Gauss-Legendre rule of order near.q).
// Components xx, xy, xz, yy, yz, zz.
__device__ __forceinline__ void green_entry(int dx, int dy, int dz, double k0, double h, double scale, double2 self,
                                            const NearRule& near, double2 (&K)[6]) {
    for (int c = 0; c < 6; ++c) K[c] = make_double2(0.0, 0.0);
    if (dx == 0 && dy == 0 && dz == 0) {
        const double2 sd = make_double2(self.x * scale, self.y * scale);
        K[0] = sd;
        K[3] = sd;
        K[5] = sd;
        return;
    }
    const double hs = h * h * h * scale;
    const int dmax = max(abs(dx), max(abs(dy), abs(dz)));
    if (dmax <= near.radius) {
        // mean over the cube: weights w_i w_j w_l / 8 of the rule on [-1, 1]^3
        for (int l = 0; l < near.q; ++l)
            for (int j = 0; j < near.q; ++j)
                for (int i = 0; i < near.q; ++i)
                    add_k2G((dx + 0.5 * near.t[i]) * h, (dy + 0.5 * near.t[j]) * h, (dz + 0.5 * near.t[l]) * h, k0, hs,
                            0.125 * near.w[i] * near.w[j] * near.w[l], K);
    } else {
        add_k2G(dx * h, dy * h, dz * h, k0, hs, 1.0, K);
    }
}

// Natural order [6][Mz][My][Mx], zero at offsets that no product uses.
__global__ void k_green_sample(double2* G, int Mx, int My, int Mz, int bx, int by, int bz,
                               double k0, double h, double scale, double2 self, NearRule near) {
    const int64_t vol = (int64_t)Mx * My * Mz;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < vol;
         idx += (int64_t)gridDim.x * blockDim.x) {
        int ix = (int)(idx % Mx);
        int iy = (int)((idx / Mx) % My);
        int iz = (int)(idx / ((int64_t)Mx * My));
        int dx, dy, dz;
        double2 K[6];
        for (int c = 0; c < 6; ++c) K[c] = make_double2(0.0, 0.0);
        if (wrap_offset(ix, Mx, bx, dx) & wrap_offset(iy, My, by, dy) & wrap_offset(iz, Mz, bz, dz))
            green_entry(dx, dy, dz, k0, h, scale, self, near, K);
        for (int c = 0; c < 6; ++c) G[c * vol + idx] = K[c];
    }
}

// The octant of non-negative offsets alone, [6][bz][by][bx]: every component is even or odd along each axis.
__global__ void k_green_octant(double2* G, int bx, int by, int bz, double k0, double h, double scale, double2 self,
                               NearRule near) {
    const int64_t vol = (int64_t)bx * by * bz;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < vol;
         idx += (int64_t)gridDim.x * blockDim.x) {
        double2 K[6];
        green_entry((int)(idx % bx), (int)((idx / bx) % by), (int)(idx / ((int64_t)bx * by)), k0, h, scale, self, near, K);
        for (int c = 0; c < 6; ++c) G[c * vol + idx] = K[c];
    }
}

// Gauss-Legendre rule of order q on [-1, 1]: the nodes are the roots of the Legendre polynomial
// P_q, found by Newton's method from the Chebyshev-like first guesses cos(pi (i + 3/4) / (q + 1/2)),
// with P_q and P_q' from the three-term recurrence; weights 2 / ((1 - t^2) P_q'(t)^2).
int near_rule(int radius, int q, NearRule* out) {
    NearRule r;
    if (radius < 0 || radius > 8) return fail(VIE_EINVAL, "near-field radius must be in [0, 8]");
    r.radius = radius;
    if (radius == 0) {
        *out = r;
        return VIE_OK;
    }
    if (q < 1 || q > kNearMaxOrder) return fail(VIE_EINVAL, "near-field quadrature order must be in [1, 16]");
    r.q = q;
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < q; ++i) {
        double t = std::cos(pi * (i + 0.75) / (q + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = t;                 // P_0, P_1
            for (int n = 2; n <= q; ++n) {
                const double p2 = ((2.0 * n - 1.0) * t * p1 - (n - 1.0) * p0) / n;
                p0 = p1;
                p1 = p2;
            }
            const double pq = q == 1 ? t : p1, pm = q == 1 ? 1.0 : p0;   // P_q, P_{q-1}
            dp = q * (t * pq - pm) / (t * t - 1.0);                      // P_q'
            const double dt = pq / dp;
            t -= dt;
            if (std::fabs(dt) < 1e-16) break;
        }
        // recompute the derivative at the converged node
        double p0 = 1.0, p1 = t;
        for (int n = 2; n <= q; ++n) {
            const double p2 = ((2.0 * n - 1.0) * t * p1 - (n - 1.0) * p0) / n;
            p0 = p1;
            p1 = p2;
        }
        const double pq = q == 1 ? t : p1, pm = q == 1 ? 1.0 : p0;
        dp = q * (t * pq - pm) / (t * t - 1.0);
        r.t[i] = t;
        r.w[i] = 2.0 / ((1.0 - t * t) * dp * dp);
    }
    *out = r;
    return VIE_OK;
}

// equivalent-sphere self term: (2/3)[(1 + jka) e^{-jka} - 1] - 1/3
static double2 self_term(double k0, double h) {
    const double ka = k0 * h * cbrt(3.0 / (4.0 * 3.14159265358979323846));
    const double c = cos(ka), sn = sin(ka);
    // (1 + j ka)(c - j sn) = c + ka sn + j (ka c - sn)
    return make_double2((2.0 / 3.0) * (c + ka * sn - 1.0) - 1.0 / 3.0, (2.0 / 3.0) * (ka * c - sn));
}

int green_sample(const BoxSet& bs, double k0, double h, double2* G, cudaStream_t s, const NearRule* near) {
    const double scale = 1.0 / ((double)bs.Mx * bs.My * bs.Mz);
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 6 * bs.spec_elems() * 16, false);
    const NearRule rule = near ? *near : NearRule();
    k_green_sample<<<grid_1d(bs.spec_elems()), 256, 0, s>>>(G, bs.Mx, bs.My, bs.Mz, bs.bx, bs.by, bs.bz,
                                                            k0, h, scale, self_term(k0, h), rule);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

int green_octant(const BoxSet& bs, double k0, double h, double2* G, cudaStream_t s, const NearRule* near) {
    const double scale = 1.0 / ((double)bs.Mx * bs.My * bs.Mz);
    prof_begin(s, PK_SPECTRUM, VIE_C128, 0, 6 * bs.box_elems() * 16, false);
    const NearRule rule = near ? *near : NearRule();
    k_green_octant<<<grid_1d(bs.box_elems()), 256, 0, s>>>(G, bs.bx, bs.by, bs.bz, k0, h, scale, self_term(k0, h), rule);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

__global__ void k_c128_to_c64(const double2* a, float2* b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = make_float2((float)a[i].x, (float)a[i].y);
}
int convert_c128_to_c64(const double2* a, float2* b, int64_t n, cudaStream_t s) {
    prof_begin(s, PK_SPECTRUM, VIE_C64, 0, n * 24, false);
    k_c128_to_c64<<<grid_1d(n), 256, 0, s>>>(a, b, n);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// E_inc = pol exp(-j k0 khat . r), r the voxel centre relative to the grid centre.
template <class C>
__global__ void k_plane_wave(C* out, int nx, int ny, int nz, double h, double k0, double3 kh,
                             double2 p0, double2 p1, double2 p2) {
    const int64_t N = (int64_t)nx * ny * nz;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N;
         idx += (int64_t)gridDim.x * blockDim.x) {
        int ix = (int)(idx % nx), iy = (int)((idx / nx) % ny), iz = (int)(idx / ((int64_t)nx * ny));
        double x = (ix + 0.5) * h - 0.5 * nx * h;
        double y = (iy + 0.5) * h - 0.5 * ny * h;
        double z = (iz + 0.5) * h - 0.5 * nz * h;
        double sn, cs;
        sincos(k0 * (kh.x * x + kh.y * y + kh.z * z), &sn, &cs);
        double2 ph = make_double2(cs, -sn);
        out[idx] = from_c128<C>(cmul(p0, ph));
        out[N + idx] = from_c128<C>(cmul(p1, ph));
        out[2 * N + idx] = from_c128<C>(cmul(p2, ph));
    }
}

int plane_wave_launch(const vie_grid* g, double k0, const double* khat, const double* pol,
                      int precision, void* out, cudaStream_t s) {
    double3 kh = make_double3(khat[0], khat[1], khat[2]);
    double2 p0 = make_double2(pol[0], pol[1]), p1 = make_double2(pol[2], pol[3]), p2 = make_double2(pol[4], pol[5]);
    prof_begin(s, PK_FIELD, precision, 0, 3 * g->N * (precision == VIE_C128 ? 16 : 8), false);
    if (precision == VIE_C128)
        k_plane_wave<double2><<<grid_1d(g->N), 256, 0, s>>>((double2*)out, g->nx, g->ny, g->nz, g->h, k0, kh, p0, p1, p2);
    else
        k_plane_wave<float2><<<grid_1d(g->N), 256, 0, s>>>((float2*)out, g->nx, g->ny, g->nz, g->h, k0, kh, p0, p1, p2);
    prof_end(s);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

// ---------------------------------------------------------------- block restriction / prolongation
// Groups of blocks of one launch, their box elements numbered one after another from first[i].
constexpr int kBlockTabMax = 16;
template <class C> struct BlockTab {
    int n, nx, ny, nz;
    int64_t first[kBlockTabMax + 1];
    C* vec[kBlockTabMax];                 // b (gather) or x (scatter) of the group, [nb][3][bz][by][bx]
    const uint8_t* mask[kBlockTabMax];
    const int32_t* origin[kBlockTabMax];
    int bx[kBlockTabMax], by[kBlockTabMax], bz[kBlockTabMax];
};

// Element idx of the table: its group i, index j in the group's vectors, mask value and place in the grid.
template <class C>
__device__ __forceinline__ uint8_t block_elem(const BlockTab<C>& t, int64_t idx, int& i, int64_t& j, int64_t& place) {
    i = 0;
    while (i + 1 < t.n && idx >= t.first[i + 1]) ++i;
    j = idx - t.first[i];
    const int bx = t.bx[i], by = t.by[i];
    const int64_t box = (int64_t)bx * by * t.bz[i], bc = j / box;
    const int l = (int)(j - bc * box), c = (int)(bc % 3), b = (int)(bc / 3);
    const uint8_t m = t.mask[i][b * box + l];
    const int32_t* o = t.origin[i] + 3 * b;
    place = c * ((int64_t)t.nx * t.ny * t.nz) +
            ((int64_t)(o[2] + l / (bx * by)) * t.ny + o[1] + (l / bx) % by) * t.nx + o[0] + l % bx;
    return m;
}

// b_k = b restricted to the voxels S_k of block k; zero outside S_k.
template <class C> __global__ void k_gather(const C* src, BlockTab<C> t) {
    pdl_wait();
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < t.first[t.n];
         idx += (int64_t)gridDim.x * blockDim.x) {
        int i;
        int64_t j, p;
        const uint8_t m = block_elem(t, idx, i, j, p);
        t.vec[i][j] = m ? src[p] : czero<C>();
    }
}

// y = x_k on the voxels of block k (mask 1; the blocks are disjoint, so no write conflicts). Halo
// voxels of an expanded block (mask 2) belong to another block or to none and are not written.
// y = b on voxels that belong to no block (identity part of K2), when block_id is given.
template <class C> __global__ void k_scatter(C* y, BlockTab<C> t, const C* b, const int32_t* block_id) {
    pdl_wait();
    const int64_t N = (int64_t)t.nx * t.ny * t.nz, total = t.first[t.n] + (block_id ? N : 0);
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        if (idx < t.first[t.n]) {
            int i;
            int64_t j, p;
            if (block_elem(t, idx, i, j, p) == 1) y[p] = t.vec[i][j];
        } else {
            const int64_t v = idx - t.first[t.n];
            if (block_id[v] < 0) {
                y[v] = b[v];
                y[N + v] = b[N + v];
                y[2 * N + v] = b[2 * N + v];
            }
        }
    }
}

template <class C> static KrylovVecs<C>& vecs_of(Group& gr);
template <> KrylovVecs<double2>& vecs_of<double2>(Group& gr) { return gr.k128; }
template <> KrylovVecs<float2>& vecs_of<float2>(Group& gr) { return gr.k64; }

template <class C> static BlockTab<C> block_tab(vie_grid* g, size_t g0, bool gather) {
    BlockTab<C> t{};
    t.nx = g->nx; t.ny = g->ny; t.nz = g->nz;
    for (size_t i = g0; i < g->groups.size() && t.n < kBlockTabMax; ++i) {
        const BoxSet& bs = g->groups[i].bs;
        const KrylovVecs<C>& v = vecs_of<C>(g->groups[i]);
        t.vec[t.n] = gather ? v.b : v.x;
        t.mask[t.n] = bs.mask;
        t.origin[t.n] = bs.origin;
        t.bx[t.n] = bs.bx; t.by[t.n] = bs.by; t.bz[t.n] = bs.bz;
        t.first[t.n + 1] = t.first[t.n] + bs.nb * bs.vec_elems();
        ++t.n;
    }
    return t;
}

template <class C> int precond_gather(vie_grid* g, const C* b, cudaStream_t s) {
    for (size_t g0 = 0; g0 < g->groups.size(); g0 += kBlockTabMax) {
        const BlockTab<C> t = block_tab<C>(g, g0, true);
        prof_begin(s, PK_FIELD, sizeof(C) == 16 ? VIE_C128 : VIE_C64, 0, 2 * t.first[t.n] * (int64_t)sizeof(C), false);
        const cudaError_t e = launch_dependent(k_gather<C>, dim3(grid_1d(t.first[t.n])), 256, 0, s, b, t);
        prof_end(s);
        VIE_CK(e);
    }
    return VIE_OK;
}

template <class C> int precond_scatter(vie_grid* g, const C* b, C* y, cudaStream_t s) {
    for (size_t g0 = 0; g0 < g->groups.size(); g0 += kBlockTabMax) {
        const BlockTab<C> t = block_tab<C>(g, g0, false);
        const int64_t n = t.first[t.n] + (g0 == 0 ? g->N : 0);
        prof_begin(s, PK_FIELD, sizeof(C) == 16 ? VIE_C128 : VIE_C64, 0,
                   2 * t.first[t.n] * (int64_t)sizeof(C) + (g0 == 0 ? g->N * (4 + 6 * (int64_t)sizeof(C)) : 0), false);
        const cudaError_t e = launch_dependent(k_scatter<C>, dim3(grid_1d(n)), 256, 0, s, y, t, b,
                                               g0 == 0 ? (const int32_t*)g->block_id : (const int32_t*)nullptr);
        prof_end(s);
        VIE_CK(e);
    }
    return VIE_OK;
}

template int precond_gather<double2>(vie_grid*, const double2*, cudaStream_t);
template int precond_gather<float2>(vie_grid*, const float2*, cudaStream_t);
template int precond_scatter<double2>(vie_grid*, const double2*, double2*, cudaStream_t);
template int precond_scatter<float2>(vie_grid*, const float2*, float2*, cudaStream_t);

}  // namespace vie

// Far-zone scattered field and bistatic RCS of a solved total field (the
// far-zone limit of E_s = k0^2 int G chi E dv, Eq. 1 with J = j w eps0 chi E;
// the RCS comparisons of Section III, Figs. 1-2):
//   P(u)     = sum_j chi_j E_j h^3 exp(j k0 u . r_j)
//   sigma(u) = k0^4 / (4 pi) |(I - u u) P(u)|^2
// over voxel centres r_j = ((i + 1/2) h - n h / 2) per axis. The phase is
// separable, exp(j k0 (ux x + uy y + uz z)) = ex(x) ey(y) ez(z), so each CTA
// (ND directions, one slab of z planes) tabulates the three 1D factors in
// shared memory; partial sums are FP64 and are added on the host in a fixed
// order.
//
// Bound by the FP64 units. A thread sums along one axis (y, or z within the
// slab where that is longer) with that axis's factor alone and applies the
// other two factors once per line, and forms chi E once for its ND directions:
// 12 + 12 / ND FP64 instructions per voxel and direction in place of 30
// (64^3 voxels, 181 directions 2.92 -> 1.52 ms; 256 x 256 x 16, 361
// directions 20.6 -> 10.2 ms, on the host with the read-back).
#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "vie_internal.cuh"

namespace vie {
namespace {

constexpr int kFfThreads = 256;
constexpr int kFfSlabs = 16;   // z slabs per direction (CTAs per direction)

// acc += a b
__device__ __forceinline__ void cfma_acc(double2& acc, double2 a, double2 b) {
    acc.x = fma(-a.y, b.y, fma(a.x, b.x, acc.x));
    acc.y = fma(a.y, b.x, fma(a.x, b.y, acc.y));
}

template <int ND>
__global__ void __launch_bounds__(kFfThreads) k_far_field(const double2* E, const double2* chi, const double3* dirs,
                                                           int ndir, int nx, int ny, int nz, double h, double k0,
                                                           double2* partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nf = nx + ny + nz;
    double2* fac = reinterpret_cast<double2*>(smem_raw);    // [ND][ex nx | ey ny | ez nz]
    double2* red = fac + ND * nf;                            // [ND][3][kFfThreads / 32]
    const int d0 = blockIdx.x * ND, slab = blockIdx.y;
    const double kh = k0 * h;
    for (int t = threadIdx.x; t < ND * nf; t += blockDim.x) {
        const int dd = t / nf, i = t - dd * nf;
        const double3 u = dirs[min(d0 + dd, ndir - 1)];
        double w, n, c;
        if (i < nx) { w = u.x; n = nx; c = i; }
        else if (i < nx + ny) { w = u.y; n = ny; c = i - nx; }
        else { w = u.z; n = nz; c = i - nx - ny; }
        double sn, cs;
        sincos(kh * w * (c + 0.5 - 0.5 * n), &sn, &cs);
        fac[t] = make_double2(cs, sn);
    }
    __syncthreads();
    const int z0 = (int)((int64_t)nz * slab / gridDim.y), z1 = (int)((int64_t)nz * (slab + 1) / gridDim.y);
    const int64_t N = (int64_t)nx * ny * nz;
    const int64_t plane = (int64_t)nx * ny;
    // lines along y or z; where they are fewer than threads, each is cut into parts
    const bool alongy = ny >= z1 - z0;
    const int nl = alongy ? ny : z1 - z0, lines = nx * (alongy ? z1 - z0 : ny);
    const int parts = max(1, min(nl, (int)blockDim.x / lines));
    const int64_t step = alongy ? nx : plane;
    double2 acc[ND][3];
#pragma unroll
    for (int dd = 0; dd < ND; ++dd)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[dd][c] = make_double2(0, 0);
    for (int t = threadIdx.x; t < lines * parts; t += blockDim.x) {
        const int part = t / lines, line = t - part * lines, o = line / nx, x = line - o * nx;
        const int64_t l0 = alongy ? (z0 + o) * plane + x : z0 * plane + (int64_t)o * nx + x;
        const double2* fl = fac + (alongy ? nx : nx + ny + z0);                 // factor along the line
        const double2* fo = fac + (alongy ? nx + ny + z0 : nx) + o;             // the other axis's
        double2 sum[ND][3];
#pragma unroll
        for (int dd = 0; dd < ND; ++dd)
#pragma unroll
            for (int c = 0; c < 3; ++c) sum[dd][c] = make_double2(0, 0);
        const int j1 = nl * (part + 1) / parts;
        for (int j = nl * part / parts; j < j1; ++j) {
            const int64_t l = l0 + j * step;
            const double2 ch = chi[l];
            const double2 w[3] = {cmul(ch, E[l]), cmul(ch, E[N + l]), cmul(ch, E[2 * N + l])};
#pragma unroll
            for (int dd = 0; dd < ND; ++dd) {
                const double2 f = fl[dd * nf + j];
#pragma unroll
                for (int c = 0; c < 3; ++c) cfma_acc(sum[dd][c], f, w[c]);
            }
        }
#pragma unroll
        for (int dd = 0; dd < ND; ++dd) {
            const double2 f = cmul(fac[dd * nf + x], fo[dd * nf]);
#pragma unroll
            for (int c = 0; c < 3; ++c) cfma_acc(acc[dd][c], f, sum[dd][c]);
        }
    }
    // CTA sums in a fixed order: warp shuffles, then one thread per component over the warps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int dd = 0; dd < ND; ++dd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double2 v = acc[dd][c];
            for (int o = 16; o > 0; o >>= 1) {
                v.x += __shfl_down_sync(0xffffffffu, v.x, o);
                v.y += __shfl_down_sync(0xffffffffu, v.y, o);
            }
            if (lane == 0) red[(dd * 3 + c) * nw + warp] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < 3 * ND && d0 + (int)threadIdx.x / 3 < ndir) {
        double2 v = make_double2(0, 0);
        for (int k = 0; k < nw; ++k) v = v + red[threadIdx.x * nw + k];
        const int dd = threadIdx.x / 3, c = threadIdx.x - 3 * dd;
        partial[((int64_t)(d0 + dd) * gridDim.y + slab) * 3 + c] = v;
    }
}

template <int ND>
int launch_far_field(const double2* E, const double2* chi, const double3* dirs, int ndir, int slabs, int nx, int ny, int nz,
                     double h, double k0, double2* partial, cudaStream_t s) {
    const size_t smem = (size_t)ND * (nx + ny + nz + 3 * (kFfThreads / 32)) * sizeof(double2);
    if (smem > 46 * 1024) VIE_TRY(raise_dynamic_smem(reinterpret_cast<const void*>(k_far_field<ND>), smem));
    k_far_field<ND><<<dim3((ndir + ND - 1) / ND, slabs), kFfThreads, smem, s>>>(E, chi, dirs, ndir, nx, ny, nz, h, k0, partial);
    VIE_CK(cudaGetLastError());
    return VIE_OK;
}

}  // namespace
}  // namespace vie

using namespace vie;

extern "C" int vie_far_field_rcs(const vie_grid* g, double k0, const void* e_dev, int32_t ndir, const double* dirs_host,
                                 double* rcs_host, vie_stream_t stream) {
    if (!g || !e_dev || !dirs_host || !rcs_host) return fail(VIE_EINVAL, "vie_far_field_rcs: null argument");
    return far_field_rcs_impl(g->nx, g->ny, g->nz, g->h, k0, (const double2*)e_dev, g->full.chi128, nullptr, ndir,
                              dirs_host, rcs_host, (cudaStream_t)stream);
}

namespace vie {

// P(u) = sum_j w_j E_j h^3 exp(j k0 u . (r_j + shift_c e_c)) per component c (w = chi for the
// collocation field; w = 1 and shift = h/2 for rooftop currents on faces), then the RCS.
int far_field_rcs_impl(int nx, int ny, int nz, double h, double k0, const double2* e_dev, const double2* wts,
                       const double* shift, int32_t ndir, const double* dirs_host, double* rcs_host, cudaStream_t s) {
    if (!e_dev || !dirs_host || !rcs_host) return fail(VIE_EINVAL, "vie_far_field_rcs: null argument");
    if (ndir < 1 || ndir > (1 << 20)) return fail(VIE_EINVAL, "vie_far_field_rcs: ndir must be in [1, 2^20]");
    if (!(k0 > 0.0) || !std::isfinite(k0)) return fail(VIE_EINVAL, "vie_far_field_rcs: k0 must be positive");
    std::vector<double3> dirs(ndir);
    for (int i = 0; i < ndir; ++i) {
        const double ux = dirs_host[3 * i], uy = dirs_host[3 * i + 1], uz = dirs_host[3 * i + 2];
        const double n2 = ux * ux + uy * uy + uz * uz;
        if (!(std::fabs(n2 - 1.0) <= 1e-9)) return fail(VIE_EINVAL, "vie_far_field_rcs: directions must be unit vectors");
        dirs[i] = make_double3(ux, uy, uz);
    }
    const int slabs = std::min(kFfSlabs, nz);
    double3* d_dirs = nullptr;
    double2* d_part = nullptr;
    const size_t part_n = (size_t)ndir * slabs * 3;
    VIE_CK(cudaMallocAsync((void**)&d_dirs, ndir * sizeof(double3), s));
    cudaError_t e = cudaMallocAsync((void**)&d_part, part_n * sizeof(double2), s);
    int rc = VIE_OK;
    if (e != cudaSuccess) rc = cuda_fail(e, "cudaMallocAsync", __FILE__, __LINE__);
    std::vector<double2> part(part_n);
    if (!rc) {
        e = cudaMemcpyAsync(d_dirs, dirs.data(), ndir * sizeof(double3), cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) rc = cuda_fail(e, "cudaMemcpyAsync", __FILE__, __LINE__);
    }
    if (!rc) {
        prof_begin(s, PK_FIELD, VIE_C128, 0, (int64_t)ndir * nx * ny * nz * 64, false);
        // four directions per CTA while that leaves two CTAs for each SM (below, the last wave would be uneven)
        rc = (int64_t)((ndir + 3) / 4) * slabs >= 2 * 152
                 ? launch_far_field<4>(e_dev, wts, d_dirs, ndir, slabs, nx, ny, nz, h, k0, d_part, s)
                 : launch_far_field<1>(e_dev, wts, d_dirs, ndir, slabs, nx, ny, nz, h, k0, d_part, s);
        prof_end(s);
    }
    if (!rc) {
        e = cudaMemcpyAsync(part.data(), d_part, part_n * sizeof(double2), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_fail(e, "far-field read-back", __FILE__, __LINE__);
    }
    if (d_part) cudaFreeAsync(d_part, s);
    if (d_dirs) cudaFreeAsync(d_dirs, s);
    if (rc) return rc;
    const double h3 = h * h * h;
    const double pref = k0 * k0 * k0 * k0 / (4.0 * 3.141592653589793238462643383279502884);
    for (int i = 0; i < ndir; ++i) {
        double2 P[3];
        for (int c = 0; c < 3; ++c) {
            P[c] = make_double2(0.0, 0.0);
            for (int sl = 0; sl < slabs; ++sl) P[c] = P[c] + part[((size_t)i * slabs + sl) * 3 + c];
            P[c] = make_double2(P[c].x * h3, P[c].y * h3);
        }
        const double3 u = dirs[i];
        if (shift) {
            const double uc[3] = {u.x, u.y, u.z};
            for (int c = 0; c < 3; ++c) {
                double sn, cs;
                sincos(k0 * uc[c] * shift[c], &sn, &cs);
                P[c] = cmul(P[c], make_double2(cs, sn));
            }
        }
        // (I - u u) P = P - u (u . P)
        const double2 up = make_double2(u.x * P[0].x + u.y * P[1].x + u.z * P[2].x,
                                        u.x * P[0].y + u.y * P[1].y + u.z * P[2].y);
        const double uu[3] = {u.x, u.y, u.z};
        double s2 = 0.0;
        for (int c = 0; c < 3; ++c) {
            const double tx = P[c].x - uu[c] * up.x, ty = P[c].y - uu[c] * up.y;
            s2 += tx * tx + ty * ty;
        }
        rcs_host[i] = pref * s2;
    }
    return VIE_OK;
}

}  // namespace vie

// Register-resident radix-2 FFTs of the complex64 passes (fft.cu), with the
// constant-memory twiddle table that get_twiddles fills.
#pragma once

#include "vie_internal.cuh"

namespace vie {

// Radix-2 FFT of one pencil held in registers, fully unrolled. FWD: natural
// order in, bit-reversed out (decimation in frequency); !FWD: bit-reversed in,
// natural out, unnormalised (decimation in time). Same ordering as the
// shared-memory passes, so spectra from either path are interchangeable.
template <bool FWD, class C>
__device__ __forceinline__ C twmul(C v, int m, const C* __restrict__ tw) {
    if (m == 0) return v;
    if (m == kLmax / 4) return FWD ? mul_mi(v) : mul_i(v);
    C w = __ldg(&tw[m]);
    return FWD ? cmul(v, w) : cmulc(v, w);
}

template <int L> struct ILog2 { static constexpr int v = 1 + ILog2<L / 2>::v; };
template <> struct ILog2<1> { static constexpr int v = 0; };

// Twiddle multiply used by the register FFTs (specialised below per precision).
template <class C> struct TwSel;

// One radix-2 stage of span S (a compile-time constant) on an L-point pencil.
template <int L, int S, bool FWD, class C>
__device__ __forceinline__ void rstage(C (&a)[L], const C* __restrict__ tw) {
#pragma unroll
    for (int g = 0; g < L; g += 2 * S) {
#pragma unroll
        for (int j = 0; j < S; ++j) {
            const int m = j * (kLmax / (2 * S));
            if (FWD) {
                C x0 = a[g + j], x1 = a[g + j + S];
                a[g + j] = x0 + x1;
                a[g + j + S] = TwSel<C>::template apply<true>(x0 - x1, m, tw);
            } else {
                C x0 = a[g + j], x1 = TwSel<C>::template apply<false>(a[g + j + S], m, tw);
                a[g + j] = x0 + x1;
                a[g + j + S] = x0 - x1;
            }
        }
    }
}

// Stages with spans S, S/2, ..., 1 (forward) or S, 2S, ..., L/2 (inverse).
template <int L, int S, bool FWD> struct RStages {
    template <class C> static __device__ __forceinline__ void run(C (&a)[L], const C* __restrict__ tw) {
        rstage<L, S, FWD>(a, tw);
        RStages<L, FWD ? S / 2 : S * 2, FWD>::run(a, tw);
    }
};
template <int L> struct RStages<L, 0, true> {
    template <class C> static __device__ __forceinline__ void run(C (&)[L], const C* __restrict__) {}
};
template <int L> struct RStages<L, L, false> {
    template <class C> static __device__ __forceinline__ void run(C (&)[L], const C* __restrict__) {}
};

template <int L, bool FWD, class C>
__device__ __forceinline__ void rfft(C (&a)[L], const C* __restrict__ tw) {
    if (L < 2) return;
    RStages<L, FWD ? L / 2 : 1, FWD>::run(a, tw);
}

typedef float2 F;

// Twiddles W_Lmax^m of the complex64 register path in constant memory: the
// register FFTs index them with compile-time offsets, so they become constant
// operands instead of loads.
static __constant__ F c_tw64[kLmax];

template <bool FWD>
__device__ __forceinline__ F twc(F v, int m) {
    if (m == 0) return v;
    if (m == kLmax / 4) return FWD ? mul_mi(v) : mul_i(v);
    F w = c_tw64[m];
    return FWD ? cmul(v, w) : cmulc(v, w);
}

template <> struct TwSel<float2> {
    template <bool FWD>
    static __device__ __forceinline__ float2 apply(float2 v, int m, const float2* __restrict__) {
        return twc<FWD>(v, m);
    }
};

// Copies the complex64 twiddles into the constant table of the current device (called by get_twiddles, which
// waits for the copy).
int reg_twiddles_upload(const Twiddles& tw) {
    VIE_CK(cudaMemcpyToSymbol(c_tw64, tw.d64, kLmax * sizeof(float2), 0, cudaMemcpyDeviceToDevice));
    return VIE_OK;
}

}  // namespace vie

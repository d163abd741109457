// Transform plans and stages of the complex64 products on grids that the half-filled
// power-of-two kernels (fft_fast.cuh) do not take: any n <= M / 2, M = 2^a or 3 * 2^a from 16
// to 4096, two or three planes.  As fx.cuh: one stage of radix R0, then q of radix R1, both
// even (the zero half of a padded input and the cropped half of an output are the upper half
// of the registers of the first and last stage), inverse transforms as forward ones with re
// and im exchanged, factors in per-stage tables.
#pragma once

#include "fx.cuh"

namespace die {

// 2^a: eight values per thread on small grids (twice the threads of half the chain), 16 from
// 1024 on.  3 * 2^a: 12 values with radix 4, or 24 with radix 8 from 384 on (three stages
// where radix 4 takes five).
__host__ __device__ constexpr FxPlan gx_plan(int L) {
    switch (L) {
        case 16: return FxPlan{8, 2, 8, 1};
        case 32: return FxPlan{8, 4, 8, 1};
        case 64: return FxPlan{8, 8, 8, 1};
        case 128: return FxPlan{8, 2, 8, 2};
        case 256: return FxPlan{8, 4, 8, 2};
        case 512: return FxPlan{8, 8, 8, 2};
        case 1024: return FxPlan{16, 16, 8, 2};
        case 2048: return FxPlan{16, 8, 16, 2};
        case 4096: return FxPlan{16, 16, 16, 2};
        case 24: return FxPlan{12, 6, 4, 1};
        case 48: return FxPlan{12, 12, 4, 1};
        case 96: return FxPlan{12, 6, 4, 2};
        case 192: return FxPlan{12, 12, 4, 2};
        case 384: return FxPlan{24, 6, 8, 2};
        case 768: return FxPlan{24, 12, 8, 2};
        case 1536: return FxPlan{24, 24, 8, 2};
        default: return FxPlan{24, 6, 8, 3};            // 3072
    }
}

// cos(2 pi m / 24), m = 0 .. 23
__host__ __device__ constexpr float gx_cos24(int m) {
    constexpr float v[7] = {1.f, 0.96592582628906828675f, 0.86602540378443864676f, 0.70710678118654752440f, 0.5f,
                            0.25881904510252076235f, 0.f};
    m = m % 24 < 0 ? m % 24 + 24 : m % 24;
    return m <= 6 ? v[m] : m <= 12 ? -v[12 - m] : m <= 18 ? -v[m - 12] : v[24 - m];
}
// DFT of 3 B values (B = 2, 4, 8): three DFTs of the residues mod 3, then DFT3s.
template <int B> __host__ __device__ __forceinline__ void gx_dft3b(float2* x) {
    float2 e[3][B];
#pragma unroll
    for (int r = 0; r < 3; r++) {
#pragma unroll
        for (int i = 0; i < B; i++) e[r][i] = x[r + 3 * i];
        dft<float2, B, false>(e[r]);
    }
#pragma unroll
    for (int s = 0; s < B; s++) {
        float2 t0 = e[0][s], t1 = e[1][s], t2 = e[2][s];
        if (s > 0) {
            constexpr int u = 8 / B;                    // exp(-2 pi i m / (3 B)) = w24^(u m)
            t1 = cmul(t1, mk(gx_cos24(u * s), -gx_cos24(u * s - 6)));
            t2 = cmul(t2, mk(gx_cos24(2 * u * s), -gx_cos24(2 * u * s - 6)));
        }
        dft3<float2, false>(t0, t1, t2);
        x[s] = t0;
        x[s + B] = t1;
        x[s + 2 * B] = t2;
    }
}
template <int R> __host__ __device__ __forceinline__ void gx_dft(float2* x) {
    if constexpr (R % 3 == 0) gx_dft3b<R / 3>(x);
    else dft<float2, R, false>(x);
}
template <int EPT, int R>
__host__ __device__ __forceinline__ void gx_stage(float2 (&x)[EPT], int Ns, int t, int G, const float2* __restrict__ tw) {
#pragma unroll
    for (int b = 0; b < EPT / R; b++) {
        if (Ns > 1) {
            const int k = mod_ns(t + b * G, Ns);
#pragma unroll
            for (int r = 1; r < R; r++) x[b * R + r] = cmul(x[b * R + r], ld_tw(&tw[r * Ns + k - 1]));
        }
        gx_dft<R>(&x[b * R]);
    }
}

}  // namespace die

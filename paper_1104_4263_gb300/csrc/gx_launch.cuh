// Launchers of the complex64 product passes on any grid (gx_kernels.cuh), one instantiation
// per transform length, compiled in translation units of their own.
#pragma once

#include "gx.cuh"
#include "op.cuh"

namespace die {

template <int LS> struct GxLaunch {
    template <typename IO>
    static void k1(const OpDev<float>& v, const IO* u, const float2* chi, float2* W, const int* skip, cudaStream_t st,
                   int nb);
    static void k2(const OpDev<float>& v, float2* W, const int* skip, cudaStream_t st, int nb);
    template <typename U, typename IO>
    static void k3(const OpDev<float>& v, const float2* W, const U* u, IO* y, const int* skip, cudaStream_t st, int nb);
    template <typename IO>
    static void k3k1(const OpDev<float>& v, float2* W, const IO* u, const float2* chir, float2* vb, const int* skip,
                     cudaStream_t st, int nb);
};

// Calls f with the launchers of a transform length.
template <typename F> inline void gx_for_length(int L, F&& f) {
    switch (L) {
        case 16: f(GxLaunch<16>{}); return;
        case 24: f(GxLaunch<24>{}); return;
        case 32: f(GxLaunch<32>{}); return;
        case 48: f(GxLaunch<48>{}); return;
        case 64: f(GxLaunch<64>{}); return;
        case 96: f(GxLaunch<96>{}); return;
        case 128: f(GxLaunch<128>{}); return;
        case 192: f(GxLaunch<192>{}); return;
        case 256: f(GxLaunch<256>{}); return;
        case 384: f(GxLaunch<384>{}); return;
        case 512: f(GxLaunch<512>{}); return;
        case 768: f(GxLaunch<768>{}); return;
        case 1024: f(GxLaunch<1024>{}); return;
        case 1536: f(GxLaunch<1536>{}); return;
        case 2048: f(GxLaunch<2048>{}); return;
        case 3072: f(GxLaunch<3072>{}); return;
        default: f(GxLaunch<4096>{}); return;
    }
}

}  // namespace die

// Launchers of the FP64 product passes (fx_kernels.cuh), one instantiation per transform
// length, each compiled once in a translation unit of its own.
#pragma once

#include "fx.cuh"

namespace die {

// The device view of an operator's FP64 products.
struct FxDev {
    int n1, n2, M1, M2, Q1, Q2;   // grid, FFT sizes, quarter-spectrum extents (M / 2 + 1)
    int q1, q2;                   // later stages of the transforms along x1 and x2
    const fxw *fx1, *fx2;         // their factors
    const fxw* gx;                // quarter spectra, scaled by 2^(ge + 63) per k1q
    const int* ge;
    const double2* chim;          // magnetic contrast (three planes)
    long xs, ws;                  // batched products: elements per vector and per set of row spectra
    int planes;
    bool apart;                   // no coupling between the planes (TM)
};

// First row pass of a product on a vector that is still to be normalised: v *= *inv in place
// (v is the product's input), with Re - Im of the result in vm (or NULL).  inv NULL: as it is.
struct FxNormalise {
    double2* v = nullptr;
    const double* inv = nullptr;
    double* vm = nullptr;
};

// The passes at one transform length (LS) or, LS = 0, at the lengths R0 4^q; nb vectors per
// launch.
template <int EPT, int R0, int R1, int LS> struct FxLaunch {
    static void k1(const FxDev& v, const double2* u, const double2* chi, double2* W, const FxNormalise& nrm,
                   const int* skip, cudaStream_t st, int nb);
    static void k2(const FxDev& v, double2* W, const int* skip, cudaStream_t st, int nb);
    static void k3(const FxDev& v, const double2* W, const double2* u, double2* y, const int* skip, cudaStream_t st,
                   int nb);
    static void k3k1(const FxDev& v, double2* W, const double2* u, const double2* chir, double2* vb, const int* skip,
                     cudaStream_t st, int nb);
};

template <int LS> using FxLaunch2 = FxLaunch<fx_plan(LS).ept, fx_plan(LS).r0, fx_plan(LS).r1, LS>;    // 2^a
template <int R0> using FxLaunch3 = FxLaunch<12, R0, 4, 0>;                              // 3 * 2^a

}  // namespace die

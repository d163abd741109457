// Fixed-point FFT arithmetic for the FP64 products.
//
// GB300 executes 2 FP64 operations per clock and SM (measured: 2.13 DFMA), but about 55
// 64-bit integer additions and 24 32 x 32 -> 64-bit multiply-adds.  A transform's
// butterflies are additions of numbers that share one scale, so they run here on 64-bit
// integers with one power-of-two scale per transform (a block-floating FFT): an addition
// costs 1/25 of its FP64 form, a complex twiddle product (12 multiply-adds) about 1/4.
//
// Accuracy.  A transform's values are scaled so that no complex value of any stage exceeds
// 2^61: after stage s the values are at most min(g_s max |x|, sum |x|) / 4^s, with g_s the
// product of the radices so far, since the twiddle product of every later stage divides by
// 4 (the high 64 bits of a 64 x 62-bit product).  Every rounding is half a unit; against
// the transform's 2-norm that is 2^-57 ... 2^-53 at lengths 64 ... 4096 on random data, an
// FP64 FFT's rounding or below.  Inputs and outputs are FP64 numbers: the input is rounded
// to the scale once (half a unit), the output to 53 bits.  Contrast products and final
// subtractions stay in FP64.
//
// Inverse transforms run the forward code on values with re and im exchanged.
#pragma once

#include <limits.h>
#include <math.h>

#include "fft.cuh"

namespace die {

struct fxc { long long x, y; };                       // a value of a transform
struct alignas(16) fxw { int xh, xl, yh, yl; };       // a factor: x = xh 2^32 + xl, both parts signed

constexpr int kFxLimit = 61;                          // |complex value| <= 2^kFxLimit in every stage

__host__ __device__ __forceinline__ fxc fadd(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
__host__ __device__ __forceinline__ fxc fsub(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }
// a - i b and a + i b
__host__ __device__ __forceinline__ fxc fadd_mi(fxc a, fxc b) { return fxc{a.x + b.y, a.y - b.x}; }
__host__ __device__ __forceinline__ fxc fadd_pi(fxc a, fxc b) { return fxc{a.x - b.y, a.y + b.x}; }

// a = h 2^32 + l with signed l
__host__ __device__ __forceinline__ void fx_split(long long a, int& h, int& l) {
    l = (int)(unsigned)a;
    h = (int)(a >> 32) + (int)((unsigned)l >> 31);
}
__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
constexpr long long kFxHalf = 1ll << 31;              // rounding of the middle terms

// a w / 2^64, rounded to the nearest but for the dropped low x low term (below one unit).
// |a| <= 2^62 and |w| <= 2^62, or |a| <= 2^62 and w one of the constants below, keep the
// middle sums below 2^63: at most 2^31 (|xh| + |yh|) + 2^30 |(xl, yl)|.
__host__ __device__ __forceinline__ fxc fx_cmul(fxc a, fxw w) {
    int arh, arl, aih, ail;
    fx_split(a.x, arh, arl);
    fx_split(a.y, aih, ail);
    const int nh = -w.yh, nl = -w.yl;
    const long long mr = fx_mad(arh, w.xl, fx_mad(arl, w.xh, fx_mad(aih, nl, fx_mad(ail, nh, kFxHalf))));
    const long long mi = fx_mad(arh, w.yl, fx_mad(arl, w.yh, fx_mad(aih, w.xl, fx_mad(ail, w.xh, kFxHalf))));
    fxc r;
    r.x = fx_mad(arh, w.xh, fx_mad(aih, nh, mr >> 32));
    r.y = fx_mad(arh, w.yh, fx_mad(aih, w.xh, mi >> 32));
    return r;
}
// (c, s) times 2^62 (host)
inline fxw fx_factor(long double c, long double s) {
    fxw w;
    fx_split(llroundl(c * 4611686018427387904.0L), w.xh, w.xl);
    fx_split(llroundl(s * 4611686018427387904.0L), w.yh, w.yl);
    if (w.yl == INT_MIN) w.yl++;          // its negative is formed
    return w;
}
__host__ __device__ __forceinline__ fxw fx_ld(const fxw* p) {
#ifdef __CUDA_ARCH__
    const int4 v = __ldg(reinterpret_cast<const int4*>(p));
    return fxw{v.x, v.y, v.z, v.w};
#else
    return *p;
#endif
}
// a c / 2^63 for a real constant c = ch 2^32 + cl
__host__ __device__ __forceinline__ long long fx_rmul(long long a, int ch, int cl) {
    int h, l;
    fx_split(a + a, h, l);
    const long long m = fx_mad(h, cl, fx_mad(l, ch, kFxHalf));
    return fx_mad(h, ch, m >> 32);
}

// sqrt(1/2), cos(pi/8), sin(pi/8), sqrt(3)/2 times 2^63
constexpr int kR2h = 1518500250, kR2l = -51432894;
constexpr int kC8h = 1984016189, kC8l = -902489949;
constexpr int kS8h = 821806413, kS8l = 1565705635;
constexpr int kH3h = 1859775393, kH3l = 1630710223;

// ------------------------------------------------------------------ small DFTs
__host__ __device__ __forceinline__ void fx_dft2(fxc& x0, fxc& x1) { const fxc t = x0; x0 = fadd(t, x1); x1 = fsub(t, x1); }
__host__ __device__ __forceinline__ void fx_dft4(fxc& x0, fxc& x1, fxc& x2, fxc& x3) {
    const fxc a = fadd(x0, x2), b = fsub(x0, x2), c = fadd(x1, x3), d = fsub(x1, x3);
    x0 = fadd(a, c); x2 = fsub(a, c); x1 = fadd_mi(b, d); x3 = fadd_pi(b, d);
}
// a * exp(-i pi / 4), a * exp(-3 i pi / 4)
__host__ __device__ __forceinline__ fxc fx_w8_1(fxc a) {
    return fxc{fx_rmul(a.x + a.y, kR2h, kR2l), fx_rmul(a.y - a.x, kR2h, kR2l)};
}
__host__ __device__ __forceinline__ fxc fx_w8_3(fxc a) {
    return fxc{fx_rmul(a.y - a.x, kR2h, kR2l), fx_rmul(-a.x - a.y, kR2h, kR2l)};
}
__host__ __device__ __forceinline__ void fx_dft8(fxc* x) {
    fxc e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
    fx_dft4(e0, e1, e2, e3);
    fx_dft4(o0, o1, o2, o3);
    o1 = fx_w8_1(o1);
    o3 = fx_w8_3(o3);
    x[0] = fadd(e0, o0); x[4] = fsub(e0, o0);
    x[1] = fadd(e1, o1); x[5] = fsub(e1, o1);
    x[2] = fadd_mi(e2, o2); x[6] = fadd_pi(e2, o2);
    x[3] = fadd(e3, o3); x[7] = fsub(e3, o3);
}
// a (c - i s), c and s the 2^63-scaled constants
__host__ __device__ __forceinline__ fxc fx_wconst(fxc a, int ch, int cl, int sh, int sl) {
    return fx_cmul(fxc{a.x + a.x, a.y + a.y}, fxw{ch, cl, -sh, -sl});
}
__host__ __device__ __forceinline__ void fx_dft16(fxc* x) {
    fxc e[8], o[8];
#pragma unroll
    for (int i = 0; i < 8; i++) { e[i] = x[2 * i]; o[i] = x[2 * i + 1]; }
    fx_dft8(e);
    fx_dft8(o);
    // y_q = e_q + w^q o_q, w = exp(-i pi / 8)
    o[1] = fx_wconst(o[1], kC8h, kC8l, kS8h, kS8l);
    o[2] = fx_w8_1(o[2]);
    o[3] = fx_wconst(o[3], kS8h, kS8l, kC8h, kC8l);
    o[5] = fx_wconst(o[5], -kS8h, -kS8l, kC8h, kC8l);
    o[6] = fx_w8_3(o[6]);
    o[7] = fx_wconst(o[7], -kC8h, -kC8l, kS8h, kS8l);
#pragma unroll
    for (int q = 0; q < 8; q++) {
        if (q == 4) { x[q] = fadd_mi(e[q], o[q]); x[q + 8] = fadd_pi(e[q], o[q]); }
        else { x[q] = fadd(e[q], o[q]); x[q + 8] = fsub(e[q], o[q]); }
    }
}
__host__ __device__ __forceinline__ long long fx_halve(long long v) { return (v + 1) >> 1; }
__host__ __device__ __forceinline__ void fx_dft3(fxc& x0, fxc& x1, fxc& x2) {
    const fxc s = fadd(x1, x2), d = fsub(x1, x2);
    const fxc m = fxc{x0.x - fx_halve(s.x), x0.y - fx_halve(s.y)};
    const fxc t = fxc{fx_rmul(d.x, kH3h, kH3l), fx_rmul(d.y, kH3h, kH3l)};
    x0 = fadd(x0, s); x1 = fadd_mi(m, t); x2 = fadd_pi(m, t);
}
// a exp(-i pi / 6), a exp(-i pi / 3): the others of a twelfth of a turn follow by -i and -1
__host__ __device__ __forceinline__ fxc fx_w12_1(fxc a) {
    return fxc{fx_rmul(a.x, kH3h, kH3l) + fx_halve(a.y), fx_rmul(a.y, kH3h, kH3l) - fx_halve(a.x)};
}
__host__ __device__ __forceinline__ fxc fx_w12_2(fxc a) {
    return fxc{fx_halve(a.x) + fx_rmul(a.y, kH3h, kH3l), fx_halve(a.y) - fx_rmul(a.x, kH3h, kH3l)};
}
__host__ __device__ __forceinline__ void fx_dft6(fxc* x) {
    fxc e0 = x[0], e1 = x[2], e2 = x[4], o0 = x[1], o1 = x[3], o2 = x[5];
    fx_dft3(e0, e1, e2);
    fx_dft3(o0, o1, o2);
    o1 = fx_w12_2(o1);
    o2 = fx_w12_1(o2);                    // w6^2 = -i w12
    x[0] = fadd(e0, o0); x[3] = fsub(e0, o0);
    x[1] = fadd(e1, o1); x[4] = fsub(e1, o1);
    x[2] = fadd_mi(e2, o2); x[5] = fadd_pi(e2, o2);
}
__host__ __device__ __forceinline__ void fx_dft12(fxc* x) {
    fxc e[6], o[6];
#pragma unroll
    for (int i = 0; i < 6; i++) { e[i] = x[2 * i]; o[i] = x[2 * i + 1]; }
    fx_dft6(e);
    fx_dft6(o);
    o[1] = fx_w12_1(o[1]);
    o[2] = fx_w12_2(o[2]);
    o[4] = fx_w12_1(o[4]);                // w12^4 = -i w12
    o[5] = fx_w12_2(o[5]);                // w12^5 = -i w12^2
#pragma unroll
    for (int q = 0; q < 6; q++) {
        if (q >= 3) { x[q] = fadd_mi(e[q], o[q]); x[q + 6] = fadd_pi(e[q], o[q]); }
        else { x[q] = fadd(e[q], o[q]); x[q + 6] = fsub(e[q], o[q]); }
    }
}
template <int R> __host__ __device__ __forceinline__ void fx_dft(fxc* x) {
    static_assert(R == 2 || R == 4 || R == 6 || R == 8 || R == 12 || R == 16, "radix");
    if constexpr (R == 2) fx_dft2(x[0], x[1]);
    else if constexpr (R == 4) fx_dft4(x[0], x[1], x[2], x[3]);
    else if constexpr (R == 6) fx_dft6(x);
    else if constexpr (R == 8) fx_dft8(x);
    else if constexpr (R == 12) fx_dft12(x);
    else fx_dft16(x);
}

// ----------------------------------------------------------------------- plans
// A transform of length L = R0 R1^q runs one stage of radix R0 and q of radix R1 with EPT
// values per thread (one loop over the equal stages keeps a kernel's code small: the
// unrolled form waited for instructions a third of the time).  R0 and R1 are even, so the
// zero half of a padded input and the cropped half of an output are the upper halves of
// every butterfly of the first and last stage.  Eight values per thread where the grid is
// small: twice the threads of half the serial chain (regularised product with 16 -> 8 values:
// 61^2 70 -> 44 us, 256^2 88 -> 71); 16 from 1024 on, where the fourth stage that 8 values need
// costs more than it hides (512^2 207 against 235 us).
struct FxPlan { int ept, r0, r1, q; };
__host__ __device__ constexpr FxPlan fx_plan(int L) {
    if (L % 3 == 0) {                                   // 3 * 2^a: 12 or 6, then 4
        int a = 0;
        while ((3 << a) < L) a++;
        return (a & 1) ? FxPlan{12, 6, 4, (a - 1) / 2} : FxPlan{12, 12, 4, (a - 2) / 2};
    }
    switch (L) {
        case 16: return FxPlan{8, 2, 8, 1};
        case 32: return FxPlan{8, 4, 8, 1};
        case 64: return FxPlan{8, 8, 8, 1};
        case 128: return FxPlan{8, 2, 8, 2};
        case 256: return FxPlan{8, 4, 8, 2};
        case 512: return FxPlan{8, 8, 8, 2};
        case 1024: return FxPlan{16, 16, 8, 2};
        case 2048: return FxPlan{16, 8, 16, 2};
        default: return FxPlan{16, 16, 16, 2};          // 4096
    }
}
// Register e of a stage of radix R holds the values at t + fx_slot(e) G of the stage's
// input (first stage) or output (last stage).
template <int EPT, int R> __host__ __device__ constexpr int fx_slot(int e) { return e / R + (e % R) * (EPT / R); }
// and the register of slot j
template <int EPT, int R> __host__ __device__ constexpr int fx_reg(int j) {
    return (j % (EPT / R)) * R + j / (EPT / R);
}

__host__ __device__ constexpr float fx_log2(int r) {
    return r == 2 ? 1.f : r == 4 ? 2.f : r == 8 ? 3.f : r == 16 ? 4.f : r == 6 ? 2.5850f : 3.5850f;
}
// Scale of a transform whose values satisfy |x| <= 2^lm and sum |x| <= 2^ls (half: only the
// lower half of the inputs is nonzero, a padded forward transform).  Stage s leaves values
// within 2^(b_s - 2 s), b_s = min(lm + log2 g_s, ls), if nothing is shifted; fx_room(s0) is
// the largest left shift that keeps the stages s >= s0 within 2^kFxLimit.  The inputs are
// scaled by 2^fx_room(0); before the twiddles of stage s the values may go up by
// fx_room(s - 1) - fx_room(s - 2) (what stage s - 1 and all later ones allow).
__host__ __device__ __forceinline__ int fx_room(int r0, int r1, int q, bool half, float lm, float ls, int s0) {
    float g = lm + fx_log2(r0) - (half ? 1.f : 0.f), e = s0 == 0 ? (float)kFxLimit - fminf(g, ls) : 1e30f;
    for (int s = 1; s <= q; s++) {
        g += fx_log2(r1);
        if (s >= s0) e = fminf(e, (float)(kFxLimit + 2 * s) - fminf(g, ls));
    }
    return (int)floorf(e - 0.01f);                      // the bounds' own rounding
}

// ---------------------------------------------------------------------- stages
// A later stage (Ns > 1): twiddles, then the DFTs.  Factors exp(-2 pi i r k / (Ns R)) times
// 2^62 at tw[r Ns + k - 1].
template <int EPT, int R>
__host__ __device__ __forceinline__ void fx_stage(fxc (&x)[EPT], int Ns, int t, int G, const fxw* __restrict__ tw) {
#pragma unroll
    for (int b = 0; b < EPT / R; b++) {
        const int k = mod_ns(t + b * G, Ns);
        x[b * R].x = (x[b * R].x + 2) >> 2;
        x[b * R].y = (x[b * R].y + 2) >> 2;
#pragma unroll
        for (int r = 1; r < R; r++) x[b * R + r] = fx_cmul(x[b * R + r], fx_ld(&tw[r * Ns + k - 1]));
        fx_dft<R>(&x[b * R]);
    }
}
// The first stage (no twiddles).
template <int EPT, int R> __host__ __device__ __forceinline__ void fx_first(fxc (&x)[EPT]) {
#pragma unroll
    for (int b = 0; b < EPT / R; b++) fx_dft<R>(&x[b * R]);
}

}  // namespace die

// Product passes of the FP64 operators on the fixed-point FFT of fx.cuh: the passes K1, K2,
// K3 and K3K1 of matvec_kernels.cuh (same grids, tiles and workspace layout, W in
// complex128), for any grid with n <= M / 2 and two or three planes.
//
// What bounds them: instruction issue and, on one wave of blocks, the serial chain of a
// thread (the FP64 forms were bound by the FP64 pipe).  CUDA-event times per launch, FP64
// form -> this one: 512^2 K1 82.5 -> 29.6 us, K2 290.6 -> 66.2, K3K1 155.5 -> 45.0, K3
// 79.8 -> 26.5 (the regularised product 878 -> 207 us back to back); 61^2 128 -> 44 us; the
// three-plane product at 384^2 476 -> 123 us.  Lengths 3 * 2^a have compile-time plans from
// 48 to 1536 (runtime -> compile time: 96^2 83 -> 61 us, 700^2 700 -> 563).  A product's own rounding (spread of
// y(c x) / c over random factors c) is 3.2e-16 ... 3.9e-16 of it at 61^2 ... 2048 x 1500 on
// noise and wave fields, against 3.5e-16 ... 3.8e-16 of the FP64 form, and 3.3e-16 ...
// 3.9e-16 against 3.9e-16 ... 4.4e-16 for regularised products.
#pragma once

#include "fx_launch.cuh"
#include "matvec_kernels.cuh"

namespace die {

constexpr int kFxTileRows = 2;    // rows per block: 32-byte segments in the transposed accesses

// Magnitudes of a transform's values z: mx >= max (|re| + |im|) and s >= sum (|re| + |im|),
// both times 2^(1023 - e) (FP64 inputs; e is the largest exponent field, 1 where the largest
// number is subnormal, 0 where all are zeros) or over 2^38 (fixed-point values, e unused).
struct FxNorm { int e; float mx, s; };

__device__ __forceinline__ int fx_mag_hi(double v) { return __double2hiint(v) & 0x7fffffff; }
// |v| 2^(1023 - e) rounded up, in FP32 straight from the high word (a conversion instruction
// would run on the FP64 pipe).
__device__ __forceinline__ float fx_mag(double v, int e) {
    return __int_as_float(max(fx_mag_hi(v) + 1 - (e - 127) * (1 << 20), 0) << 3);
}
__device__ __forceinline__ float fx_mag(long long v) {
    const int hi = (int)(v >> 32), ab = hi < 0 ? ~hi : hi;           // at most 2^29
    return __int_as_float(0x4b000000 | (ab >> 6)) - 8388607.0f;      // ceil(|v| / 2^38)
}
// Norm of the values v[e], KEEP(e) true.
template <int EPT, typename K> __device__ __forceinline__ FxNorm fx_norm(const double2 (&v)[EPT], K keep) {
    int m = 0;
#pragma unroll
    for (int e = 0; e < EPT; e++)
        if (keep(e)) m = max(m, max(fx_mag_hi(v[e].x), fx_mag_hi(v[e].y)));
    FxNorm a{m >> 20, 0.f, 0.f};
    if (a.e == 0) {
        int any = m;
#pragma unroll
        for (int e = 0; e < EPT; e++)
            if (keep(e)) any |= __double2loint(v[e].x) | __double2loint(v[e].y);
        if (any) a.e = 1;
    }
#pragma unroll
    for (int e = 0; e < EPT; e++)
        if (keep(e)) {
            const float f = fx_mag(v[e].x, a.e) + fx_mag(v[e].y, a.e);
            a.mx = fmaxf(a.mx, f);
            a.s += f;
        }
    return a;
}
template <int EPT> __device__ __forceinline__ FxNorm fx_norm(const fxc (&v)[EPT]) {
    FxNorm a{0, 0.f, 0.f};
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const float f = fx_mag(v[e].x) + fx_mag(v[e].y);
        a.mx = fmaxf(a.mx, f);
        a.s += f;
    }
    return a;
}
__device__ __forceinline__ float fx_pow2(int e) { return __int_as_float(max(127 + e, 0) << 23); }   // e <= 0
__device__ __forceinline__ FxNorm fx_merge(FxNorm a, FxNorm b, bool add) {
    FxNorm r;
    r.e = max(a.e, b.e);
    const float fa = fx_pow2(a.e - r.e), fb = fx_pow2(b.e - r.e);
    r.mx = fmaxf(a.mx * fa, b.mx * fb);
    r.s = add ? a.s * fa + b.s * fb : fmaxf(a.s * fa, b.s * fb);
    return r;
}

// The norm over the G threads of one transform: inside the warp (segments of G when
// G < 32), then over the transform's warps through red.  All threads of the block call it;
// it holds a barrier (behind the caller's reads of shared memory).
__device__ __forceinline__ FxNorm fx_group_norm(FxNorm a, int G, FxNorm* red) {
    const int live = min(32, (int)blockDim.x - ((int)threadIdx.x & ~31));
    const unsigned mask = live >= 32 ? 0xffffffffu : ((1u << live) - 1u);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (o < G) {
            FxNorm b;
            b.e = __shfl_xor_sync(mask, a.e, o);
            b.mx = __shfl_xor_sync(mask, a.mx, o);
            b.s = __shfl_xor_sync(mask, a.s, o);
            a = fx_merge(a, b, true);
        }
    if (G > 32) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
        __syncthreads();
        const int q0 = (int)(threadIdx.x / G) * (G >> 5);
        a = red[q0];
        for (int q = 1; q < (G >> 5); q++) a = fx_merge(a, red[q0 + q], true);
    } else {
        __syncthreads();
    }
    return a;
}

// Scale of FP64 values: exponent, and what the exponent arithmetic of fx_in and fx_out cannot
// do (bad: a value is not finite; slow: magnitudes near the ends of the range).
struct FxScale { int e; float lm, ls; bool half, bad, slow; };
__device__ __forceinline__ FxScale fx_scale(const FxNorm& a, int r0, int r1, int q, bool half) {
    FxScale s;
    s.half = half;
    s.bad = a.e == 2047;
    s.slow = a.e != 0 && (a.e < 123 || a.e > 1923);
    const float b = (float)(a.e - 1023);
    s.lm = __log2f(a.mx) + b;
    s.ls = __log2f(a.s) + b;
    s.e = a.e == 0 ? 0 : fx_room(r0, r1, q, half, s.lm, s.ls, 0);
    return s;
}

static __device__ __noinline__ long long fx_in_slow(double v, int e) { return __double2ll_rn(scalbn(v, e)); }
static __device__ __noinline__ double fx_out_slow(long long v, int e) { return scalbn(__ll2double_rn(v), -e); }
// round(v 2^e)
__device__ __forceinline__ long long fx_in(double v, int e) {
    const int hi = __double2hiint(v);
    const bool z = (hi & 0x7fffffff) < ((1022 - e) << 20);
    const long long r = __double2ll_rn(__hiloint2double(hi + (e << 20), __double2loint(v)));
    return z ? 0 : r;
}
// v 2^-e
__device__ __forceinline__ double fx_out(long long v, int e) {
    const double d = __ll2double_rn(v);
    return __hiloint2double(v == 0 ? 0 : __double2hiint(d) - (e << 20), __double2loint(d));
}
// All values at once; KEEP(e) false: zero.
template <int EPT, typename K>
__device__ __forceinline__ void fx_load(fxc (&x)[EPT], const double2 (&v)[EPT], const FxScale& s, K keep) {
    if (!s.slow) {
#pragma unroll
        for (int e = 0; e < EPT; e++) x[e] = keep(e) ? fxc{fx_in(v[e].x, s.e), fx_in(v[e].y, s.e)} : fxc{0, 0};
    } else {
#pragma unroll
        for (int e = 0; e < EPT; e++)
            x[e] = keep(e) ? fxc{fx_in_slow(v[e].x, s.e), fx_in_slow(v[e].y, s.e)} : fxc{0, 0};
    }
}
template <int EPT, typename K>
__device__ __forceinline__ void fx_unload(double2 (&v)[EPT], const fxc (&x)[EPT], const FxScale& s, K keep) {
    if (!s.slow && !s.bad) {
#pragma unroll
        for (int e = 0; e < EPT; e++)
            if (keep(e)) v[e] = make_double2(fx_out(x[e].x, s.e), fx_out(x[e].y, s.e));
    } else {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
        for (int e = 0; e < EPT; e++)
            if (keep(e))
                v[e] = s.bad ? make_double2(nan, nan) : make_double2(fx_out_slow(x[e].x, s.e), fx_out_slow(x[e].y, s.e));
    }
}
// v 2^s, 0 <= s <= 31
__device__ __forceinline__ long long fx_shl(long long v, int s) {
    const unsigned lo = (unsigned)v, hi = (unsigned)(v >> 32);
    return (long long)(((unsigned long long)__funnelshift_l(lo, hi, s) << 32) | (lo << s));
}
// round(v 2^-s), 0 <= s <= 31
__device__ __forceinline__ long long fx_shr(long long v, int s) {
    v += (1ll << s) >> 1;
    const unsigned lo = (unsigned)v;
    const int hi = (int)(v >> 32);
    return (long long)(((unsigned long long)(unsigned)(hi >> s) << 32) | __funnelshift_r(lo, (unsigned)hi, s));
}

// The transform of x (first-stage registers, the upper slots possibly constant zeros) into
// last-stage registers; buf: the transform's part of shared memory, free to write; s: the
// values' bounds and scale, the scale updated.  All threads of the block call it.
template <int EPT, int R0, int R1, int LS>
__device__ __forceinline__ void fx_transform(fxc (&x)[EPT], fxc* buf, int q, const fxw* tw, int t, int G, int L,
                                             FxScale& sc) {
    fx_first<EPT, R0>(x);
    stage_store<fxc, EPT, R0>(buf, x, L, 1, t, G);
    __syncthreads();
    int Ns = R0, room = 0;
    const bool rise = q > 1 && !sc.bad;
    if (rise) room = fx_room(R0, R1, q, sc.half, sc.lm, sc.ls, 0);
    auto stage = [&](int s) {
        stage_load<fxc, EPT, R1>(buf, x, L, t, G);
        if (rise && s > 1) {
            const int to = fx_room(R0, R1, q, sc.half, sc.lm, sc.ls, s - 1);
            const int up = max(0, min(to - room, 31));
            room = to;
            if (up) {
#pragma unroll
                for (int e = 0; e < EPT; e++) x[e] = fxc{fx_shl(x[e].x, up), fx_shl(x[e].y, up)};
                sc.e += up;
            }
        }
        fx_stage<EPT, R1>(x, Ns, t, G, tw);
        __syncthreads();
        if (s == q) return;
        stage_store<fxc, EPT, R1>(buf, x, L, Ns, t, G);
        __syncthreads();
        Ns *= R1;
    };
    if constexpr (LS != 0 && R1 == 4) {       // short stages, Ns = 3 * 2^b: divisions by constants
#pragma unroll
        for (int s = 1; s <= fx_plan(LS ? LS : 16).q; s++) stage(s);
    } else {
#pragma unroll 1
        for (int s = 1; s <= q; s++) stage(s);
    }
    sc.e -= 2 * q;
}

template <int EPT> __device__ __forceinline__ void fx_swap(fxc (&x)[EPT]) {
#pragma unroll
    for (int e = 0; e < EPT; e++) { const long long v = x[e].x; x[e].x = x[e].y; x[e].y = v; }
}

// Forward transform of one row (first-stage registers z, the lower half of the slots used)
// into buf as FP64 numbers in natural order.
template <int EPT, int R0, int R1, int LS>
__device__ __forceinline__ void fx_row_forward(double2 (&z)[EPT], fxc* buf, const FxDev& op, int t, int G, int L,
                                               FxNorm* red) {
    constexpr int RL = R1;
    auto low = [](int e) { return fx_slot<EPT, R0>(e) < EPT / 2; };
    const int q = LS ? fx_plan(LS ? LS : 16).q : op.q1;
    FxScale s = fx_scale(fx_group_norm(fx_norm<EPT>(z, low), G, red), R0, R1, q, true);
    fxc x[EPT];
    fx_load<EPT>(x, z, s, low);
    fx_transform<EPT, R0, R1, LS>(x, buf, q, op.fx1, t, G, L, s);
    double2 y[EPT];
    fx_unload<EPT>(y, x, s, [](int) { return true; });
    stage_store<double2, EPT, RL>(reinterpret_cast<double2*>(buf), y, L, L / RL, t, G);
}

// Inverse transform of one row (FP64 numbers in buf, natural order) into last-stage
// registers, the lower half of the slots.
template <int EPT, int R0, int R1, int LS>
__device__ __forceinline__ void fx_row_inverse(fxc* buf, double2 (&y)[EPT], const FxDev& op, int t, int G, int L,
                                               FxNorm* red) {
    constexpr int RL = R1;
    auto all = [](int) { return true; };
    const int q = LS ? fx_plan(LS ? LS : 16).q : op.q1;
    double2 z[EPT];
    stage_load<double2, EPT, R0>(reinterpret_cast<const double2*>(buf), z, L, t, G);
    FxScale s = fx_scale(fx_group_norm(fx_norm<EPT>(z, all), G, red), R0, R1, q, false);
    fxc x[EPT];
    fx_load<EPT>(x, z, s, all);
    fx_swap<EPT>(x);
    fx_transform<EPT, R0, R1, LS>(x, buf, q, op.fx1, t, G, L, s);
    fx_swap<EPT>(x);
    fx_unload<EPT>(y, x, s, [](int e) { return fx_slot<EPT, RL>(e) < EPT / 2; });
}

// The rows of the tile (FP64 numbers) to W[c][k1][row].
__device__ __forceinline__ void fx_store_tile(const double2* tile, double2* __restrict__ W, int c, int i2_0, int L,
                                              int n2, int TR, int Lp) {
    for (int e = threadIdx.x; e < L * TR; e += blockDim.x) {
        const int k1 = e / TR, r = e - k1 * TR;
        if (i2_0 + r < n2) W[((long)c * L + k1) * n2 + i2_0 + r] = tile[r * Lp + pidx(k1)];
    }
}

// ------------------------------------------------------------------------- K1
template <int EPT, int R0, int R1, int LS>
__global__ void __launch_bounds__(512) k1_fx(FxDev op, const double2* u, const double2* __restrict__ chi,
                                             double2* __restrict__ W, FxNormalise nrm, const int* __restrict__ skip) {
    __shared__ FxNorm red[16];
    pdl_wait();
    if (block_flag(skip)) return;
    u += blockIdx.z * op.xs;            // right-hand side of a batched product
    W += blockIdx.z * op.ws;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = LS ? LS : op.M1, G = L / EPT, TR = blockDim.x / G, Lp = tile_stride(L);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    const double2* urow = u + c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
    const double2* crow = (c == 2 ? op.chim : chi) + (long)i2 * op.n1;      // H3 plane: chi_m
    double2 z[EPT];
    if (nrm.inv) {       // the basis vector's normalisation, in the pass that reads it anyway
        const double sc = *nrm.inv;
        const long off = urow - u;
#pragma unroll
        for (int e = 0; e < EPT; e++) {      // all loads before the first store
            const int j = fx_slot<EPT, R0>(e), idx = t + j * G;
            z[e] = j < EPT / 2 && active && idx < op.n1 ? urow[idx] : czero<double2>();
        }
#pragma unroll
        for (int e = 0; e < EPT; e++) {
            const int j = fx_slot<EPT, R0>(e), idx = t + j * G;
            if (j < EPT / 2 && active && idx < op.n1) {
                const double2 v = make_double2(z[e].x * sc, z[e].y * sc);
                nrm.v[off + idx] = v;
                if (nrm.vm) nrm.vm[off + idx] = v.x - v.y;
                z[e] = cmul(v, crow[idx]);
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < EPT; e++) {
            const int j = fx_slot<EPT, R0>(e), idx = t + j * G;
            z[e] = j < EPT / 2 && active && idx < op.n1 ? cmul(urow[idx], crow[idx]) : czero<double2>();
        }
    }
    fx_row_forward<EPT, R0, R1, LS>(z, reinterpret_cast<fxc*>(smem_raw) + rs * Lp, op, t, G, L, red);
    __syncthreads();
    fx_store_tile(reinterpret_cast<const double2*>(smem_raw), W, c, i2_0, L, op.n2, TR, Lp);
}

// ------------------------------------------------------------------------- K3
template <int EPT, int R0, int R1, int LS>
__global__ void __launch_bounds__(512) k3_fx(FxDev op, const double2* __restrict__ W, const double2* __restrict__ u,
                                             double2* __restrict__ y, const int* __restrict__ skip) {
    constexpr int RL = R1;
    __shared__ FxNorm red[16];
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    y += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = LS ? LS : op.M1, G = L / EPT, TR = blockDim.x / G, Lp = tile_stride(L);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    load_tile<double2>(reinterpret_cast<double2*>(smem_raw), W, c, i2_0, L, op.n2, TR);
    double2 z[EPT];
    fx_row_inverse<EPT, R0, R1, LS>(reinterpret_cast<fxc*>(smem_raw) + rs * Lp, z, op, t, G, L, red);
    if (i2 >= op.n2) return;
    const long off = c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, RL>(e), idx = t + j * G;
        if (j < EPT / 2 && idx < op.n1) y[off + idx] = csub(u[off + idx], z[e]);
    }
}

// ----------------------------------------------------------------------- K3K1
template <int EPT, int R0, int R1, int LS>
__global__ void __launch_bounds__(512) k3k1_fx(FxDev op, double2* __restrict__ W, const double2* __restrict__ u,
                                               const double2* __restrict__ chir, double2* __restrict__ vbuf,
                                               const int* __restrict__ skip) {
    constexpr int RL = R1;
    __shared__ FxNorm red[16], red2[16];
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    vbuf += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = LS ? LS : op.M1, G = L / EPT, TR = blockDim.x / G, Lp = tile_stride(L);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    fxc* buf = reinterpret_cast<fxc*>(smem_raw) + rs * Lp;
    load_tile<double2>(reinterpret_cast<double2*>(smem_raw), W, c, i2_0, L, op.n2, TR);
    // Inverse (dir 0), then forward: one copy of the transform's code (see k2_fx).
    auto low = [](int e) { return fx_slot<EPT, R0>(e) < EPT / 2; };
    auto all = [](int) { return true; };
    const int q = LS ? fx_plan(LS ? LS : 16).q : op.q1;
    double2 z[EPT];
    stage_load<double2, EPT, R0>(reinterpret_cast<const double2*>(buf), z, L, t, G);
    FxScale s = fx_scale(fx_group_norm(fx_norm<EPT>(z, all), G, red), R0, R1, q, false);
    fxc x[EPT];
    fx_load<EPT>(x, z, s, all);
    fx_swap<EPT>(x);
#pragma unroll 1
    for (int dir = 0;; dir++) {
        fx_transform<EPT, R0, R1, LS>(x, buf, q, op.fx1, t, G, L, s);
        if (dir) break;
        fx_swap<EPT>(x);
        double2 y[EPT];
        fx_unload<EPT>(y, x, s, [](int e) { return fx_slot<EPT, RL>(e) < EPT / 2; });
        // v = u - y (first product), kept for the final subtraction; then chi' v
        const long off = c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
        const double2* crow = (c == 2 ? op.chim : chir) + (long)i2 * op.n1;     // the regulariser keeps chi_m
#pragma unroll
        for (int e = 0; e < EPT; e++) {
            const int j = fx_slot<EPT, R0>(e), idx = t + j * G;
            if (j < EPT / 2 && active && idx < op.n1) {
                const double2 v = csub(u[off + idx], y[fx_reg<EPT, RL>(j)]);
                vbuf[off + idx] = v;
                z[e] = cmul(v, crow[idx]);
            } else {
                z[e] = czero<double2>();
            }
        }
        s = fx_scale(fx_group_norm(fx_norm<EPT>(z, low), G, red2), R0, R1, q, true);
        fx_load<EPT>(x, z, s, low);
    }
    fx_unload<EPT>(z, x, s, all);
    stage_store<double2, EPT, RL>(reinterpret_cast<double2*>(buf), z, L, L / RL, t, G);
    __syncthreads();
    fx_store_tile(reinterpret_cast<const double2*>(smem_raw), W, c, i2_0, L, op.n2, TR, Lp);
}

// ------------------------------------------------------------------------- K2
// One block per column k1, G threads per plane.  One scale for the planes of the column
// (their products are added; each its own where the planes are not coupled, so that none
// loses bits to a larger one), raised to the largest value before the Green multiply and chosen
// anew for each plane's inverse transform.
// Blocks per SM that keep a thread's registers at 128 (16 warps), or at 80 with 8 values.
constexpr int fx_k2_blocks(int threads, int ept) {
    return threads <= 512 ? (ept == 8 ? 24 : 16) / ((threads + 31) / 32) : 1;
}

template <int P, int EPT, int R0, int R1, int LS, int MAXT>
__global__ void __launch_bounds__(MAXT, fx_k2_blocks(MAXT, EPT)) k2_fx(FxDev op, double2* __restrict__ W, const int* __restrict__ skip) {
    constexpr int RL = R1;
    __shared__ FxNorm red[32], redp[2][3];
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.y * op.ws;            // right-hand side of a batched product
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = LS ? LS : op.M2, G = L / EPT, Lp = padded_len(L);
    const int q = LS ? fx_plan(LS ? LS : 16).q : op.q2;
    fxc* bufs = reinterpret_cast<fxc*>(smem_raw);
    const int comp = threadIdx.x / G, t = threadIdx.x - comp * G;
    fxc* buf = bufs + comp * Lp;
    const int k1 = blockIdx.x;
    double2* col = W + ((long)comp * op.M1 + k1) * op.n2;
    const int h1 = op.M1 >> 1, h2 = L >> 1, Q2 = h2 + 1;
    const int k1q = k1 <= h1 ? k1 : op.M1 - k1;
    const bool neg1 = k1 > h1;
    const long plane = (long)op.Q1 * Q2;
    const fxw* g = op.gx + (long)k1q * Q2;
    auto low = [](int e) { return fx_slot<EPT, R0>(e) < EPT / 2; };
    // the planes' norms, merged over the planes (largest sum); a value that is not finite makes
    // every plane so
    auto over_planes = [&](FxNorm a, FxNorm* rp) {
        if (t == 0) rp[comp] = a;
        __syncthreads();
        FxNorm r = rp[0];
#pragma unroll
        for (int p = 1; p < P; p++) r = fx_merge(r, rp[p], false);
        return P == 2 && op.apart && r.e != 2047 ? a : r;
    };
    fxc x[EPT];
    FxScale s;
    {
        double2 z[EPT];
#pragma unroll
        for (int e = 0; e < EPT; e++) {
            const int idx = t + fx_slot<EPT, R0>(e) * G;
            z[e] = low(e) && idx < op.n2 ? col[idx] : czero<double2>();
        }
        s = fx_scale(over_planes(fx_group_norm(fx_norm<EPT>(z, low), G, red), redp[0]), R0, R1, q, true);
        fx_load<EPT>(x, z, s, low);
    }
    // Both directions run the same code: it is twice as long as what an SM's instruction
    // caches hold when each has a copy.
#pragma unroll 1
    for (int dir = 0;; dir++) {
        fx_transform<EPT, R0, R1, LS>(x, buf, q, op.fx2, t, G, L, s);
        if (dir) break;
        stage_store<fxc, EPT, RL>(buf, x, L, L / RL, t, G);
        const FxNorm ax = over_planes(fx_group_norm(fx_norm<EPT>(x), G, red), redp[1]);
        // bring the largest value up to the limit
        const int up = min(31, max(0, (int)floorf((float)(kFxLimit - 38) - 0.01f - __log2f(ax.mx))));
        // Green-spectrum multiply at the first inverse stage's indices; spectra: planes G11,
        // G22, G12 (G13, G23, G33), of parity -1 in both / x2 / x1 for G12 / G13 / G23
#pragma unroll
        for (int e = 0; e < EPT; e++) {
            const int k2 = t + fx_slot<EPT, R0>(e) * G;
            const bool neg2 = k2 > h2;
            const int k2q = neg2 ? L - k2 : k2;
            fxc acc{0, 0};
#pragma unroll
            for (int p = 0; p < P; p++) {
                const int pl = p == comp ? (p == 2 ? 5 : p) : (p + comp == 1 ? 2 : p + comp + 1);
                const bool neg = p != comp && (p + comp == 1 ? neg1 != neg2 : (p + comp == 2 ? neg2 : neg1));
                const fxw w = fx_ld(&g[pl * plane + k2q]);
                const fxc v = bufs[p * Lp + pidx(k2)];
                const fxc r = fx_cmul(fxc{fx_shl(v.x, up + 1), fx_shl(v.y, up + 1)}, w);
                acc = neg ? fsub(acc, r) : fadd(acc, r);
            }
            x[e] = fxc{acc.y, acc.x};
        }
        s.e += up + op.ge[k1q];
        {   // scale of the inverse transform of this plane
            const FxNorm a = fx_group_norm(fx_norm<EPT>(x), G, red);     // also ends the reads of bufs
            s.half = false;
            s.lm = __log2f(a.mx) + 38.f;
            s.ls = __log2f(a.s) + 38.f;
            const int sh = fx_room(R0, R1, q, false, s.lm, s.ls, 0);
            if (sh >= 0) {
#pragma unroll
                for (int e = 0; e < EPT; e++) x[e] = fxc{fx_shl(x[e].x, min(sh, 31)), fx_shl(x[e].y, min(sh, 31))};
            } else {
#pragma unroll
                for (int e = 0; e < EPT; e++) x[e] = fxc{fx_shr(x[e].x, -sh), fx_shr(x[e].y, -sh)};
            }
            s.e += min(sh, 31);
        }
    }
    fx_swap<EPT>(x);
    s.slow = s.slow || s.e > 900 || s.e < -900;
    double2 z[EPT];
    fx_unload<EPT>(z, x, s, [](int e) { return fx_slot<EPT, RL>(e) < EPT / 2; });
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, RL>(e), idx = t + j * G;
        if (j < EPT / 2 && idx < op.n2) col[idx] = z[e];
    }
}

// --------------------------------------------------------------------- launch
static Launch fx_rows_launch(const FxDev& v, int ept, int nb) {
    const int G = v.M1 / ept;
    // one row per block while that leaves no SM with two
    int TR = (long)v.n2 * v.planes * nb <= 152 ? 1 : kFxTileRows;
    while (TR > 1 && TR * G > kRowsMaxThreads) TR /= 2;
    return Launch{dim3((v.n2 + TR - 1) / TR, v.planes, nb), dim3(TR * G), (size_t)TR * tile_stride(v.M1) * sizeof(fxc)};
}
template <int EPT, int R0, int R1, int LS>
void FxLaunch<EPT, R0, R1, LS>::k1(const FxDev& v, const double2* u, const double2* chi, double2* W,
                                   const FxNormalise& nrm, const int* skip, cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k1_fx<EPT, R0, R1, LS>, a, fx_rows_launch(v, EPT, nb), st, v, u, chi, W, nrm, skip);
}
template <int EPT, int R0, int R1, int LS>
void FxLaunch<EPT, R0, R1, LS>::k3(const FxDev& v, const double2* W, const double2* u, double2* y, const int* skip,
                                   cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k3_fx<EPT, R0, R1, LS>, a, fx_rows_launch(v, EPT, nb), st, v, W, u, y, skip);
}
template <int EPT, int R0, int R1, int LS>
void FxLaunch<EPT, R0, R1, LS>::k3k1(const FxDev& v, double2* W, const double2* u, const double2* chir, double2* vb,
                                     const int* skip, cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k3k1_fx<EPT, R0, R1, LS>, a, fx_rows_launch(v, EPT, nb), st, v, W, u, chir, vb, skip);
}
template <int EPT, int R0, int R1, int LS>
void FxLaunch<EPT, R0, R1, LS>::k2(const FxDev& v, double2* W, const int* skip, cudaStream_t st, int nb) {
    static std::atomic<bool> a2{false}, a3{false};
    const int G = v.M2 / EPT, P = v.planes;
    const Launch l{dim3(v.M1, nb), dim3(P * G), (size_t)P * padded_len(v.M2) * sizeof(fxc)};
    constexpr int T = (LS ? LS : 3072) / EPT;                         // threads per plane, at most
    if (P == 3) launch_kernel(k2_fx<3, EPT, R0, R1, LS, 3 * T>, a3, l, st, v, W, skip);
    else launch_kernel(k2_fx<2, EPT, R0, R1, LS, 2 * T>, a2, l, st, v, W, skip);
}

}  // namespace die

// Product passes of the complex64 operators on any grid (n <= M / 2, M = 2^a or 3 * 2^a, two or
// three planes): the passes K1, K2, K3 and K3K1 of matvec_kernels.cuh, same workspace layout.
// Bound by latency: a pass is one wave of blocks on grids up to about 512^2.
#pragma once

#include "gx_launch.cuh"
#include "matvec_kernels.cuh"

namespace die {

constexpr int kGxTileRows = 4;    // rows per block: 32-byte segments in the transposed accesses

template <int EPT> __device__ __forceinline__ void gx_swap(float2 (&x)[EPT]) {
#pragma unroll
    for (int e = 0; e < EPT; e++) x[e] = make_float2(x[e].y, x[e].x);
}

// The transform of x (first-stage registers) into last-stage registers; buf: the transform's
// part of shared memory, free to write.  All threads of the block call it.
template <int LS> __device__ __forceinline__ void gx_transform(float2 (&x)[gx_plan(LS).ept], float2* buf,
                                                               const float2* tw, int t) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, R0 = p.r0, R1 = p.r1, G = LS / EPT;
    gx_stage<EPT, R0>(x, 1, t, G, tw);
    stage_store<float2, EPT, R0>(buf, x, LS, 1, t, G);
    __syncthreads();
    int Ns = R0;
#pragma unroll
    for (int s = 1; s <= p.q; s++) {
        stage_load<float2, EPT, R1>(buf, x, LS, t, G);
        gx_stage<EPT, R1>(x, Ns, t, G, tw);
        __syncthreads();
        if (s < p.q) {
            stage_store<float2, EPT, R1>(buf, x, LS, Ns, t, G);
            __syncthreads();
        }
        Ns *= R1;
    }
}

// Rows of the tile to / from W[c][k1][row].
__device__ __forceinline__ void gx_store_tile(const float2* tile, float2* __restrict__ W, int c, int i2_0, int L,
                                              int n2, int TR, int Lp) {
    const int sh = 31 - __clz(TR);             // TR = 1, 2, 4 or 8
#pragma unroll 4
    for (int e = threadIdx.x; e < L * TR; e += blockDim.x) {
        const int k1 = e >> sh, r = e & (TR - 1);
        if (i2_0 + r < n2) W[((long)c * L + k1) * n2 + i2_0 + r] = tile[r * Lp + pidx(k1)];
    }
}
__device__ __forceinline__ void gx_load_tile(float2* tile, const float2* __restrict__ W, int c, int i2_0, int L, int n2,
                                             int TR, int Lp) {
    const int sh = 31 - __clz(TR);
#pragma unroll 8
    for (int e = threadIdx.x; e < L * TR; e += blockDim.x) {
        const int k1 = e >> sh, r = e & (TR - 1);
        tile[r * Lp + pidx(k1)] = i2_0 + r < n2 ? W[((long)c * L + k1) * n2 + i2_0 + r] : make_float2(0.f, 0.f);
    }
    __syncthreads();
}

// ------------------------------------------------------------------------- K1
template <typename IO, int LS>
__global__ void __launch_bounds__(512) k1_gx(OpDev<float> op, const IO* __restrict__ u, const float2* __restrict__ chi,
                                             float2* __restrict__ W, const int* __restrict__ skip) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, G = LS / EPT;
    pdl_wait();
    if (block_flag(skip)) return;
    u += blockIdx.z * op.xs;            // right-hand side of a batched product
    W += blockIdx.z * op.ws;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TR = blockDim.x / G, Lp = tile_stride(LS);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    const IO* ur = u + c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
    const float2* cr = (c == 2 ? op.chim : chi) + (long)i2 * op.n1;      // H3 plane: chi_m
    float2* buf = reinterpret_cast<float2*>(smem_raw) + rs * Lp;
    float2 x[EPT];
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r0>(e), idx = t + j * G;
        x[e] = j < EPT / 2 && active && idx < op.n1 ? cmul(cvt<float2>(ur[idx]), cr[idx]) : make_float2(0.f, 0.f);
    }
    gx_transform<LS>(x, buf, op.gx1, t);
    stage_store<float2, EPT, p.r1>(buf, x, LS, LS / p.r1, t, G);
    __syncthreads();
    gx_store_tile(reinterpret_cast<const float2*>(smem_raw), W, c, i2_0, LS, op.n2, TR, Lp);
}

// ------------------------------------------------------------------------- K3
template <typename U, typename IO, int LS>
__global__ void __launch_bounds__(512) k3_gx(OpDev<float> op, const float2* __restrict__ W, const U* __restrict__ u,
                                             IO* __restrict__ y, const int* __restrict__ skip) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, G = LS / EPT;
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    y += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TR = blockDim.x / G, Lp = tile_stride(LS);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    float2* buf = reinterpret_cast<float2*>(smem_raw) + rs * Lp;
    gx_load_tile(reinterpret_cast<float2*>(smem_raw), W, c, i2_0, LS, op.n2, TR, Lp);
    float2 x[EPT];
    stage_load<float2, EPT, p.r0>(buf, x, LS, t, G);
    gx_swap<EPT>(x);
    __syncthreads();
    gx_transform<LS>(x, buf, op.gx1, t);
    if (i2 >= op.n2) return;
    const long off = c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r1>(e), idx = t + j * G;
        if (j < EPT / 2 && idx < op.n1) y[off + idx] = csub(cvt<IO>(u[off + idx]), cvt<IO>(make_float2(x[e].y, x[e].x)));
    }
}

// ----------------------------------------------------------------------- K3K1
// At 256 and 512 (eight values per thread) 40 registers in place of 63, for half again the warps:
// 256 x 1024, 8 products 74 -> 63 us; one product unchanged.
template <typename IO, int LS>
__global__ void __launch_bounds__(512, LS == 256 || LS == 512 ? 3 : 0) k3k1_gx(OpDev<float> op, float2* __restrict__ W, const IO* __restrict__ u,
                                               const float2* __restrict__ chir, float2* __restrict__ vbuf,
                                               const int* __restrict__ skip) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, G = LS / EPT;
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    vbuf += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TR = blockDim.x / G, Lp = tile_stride(LS);
    const int rs = threadIdx.x / G, t = threadIdx.x - rs * G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    float2* buf = reinterpret_cast<float2*>(smem_raw) + rs * Lp;
    gx_load_tile(reinterpret_cast<float2*>(smem_raw), W, c, i2_0, LS, op.n2, TR, Lp);
    float2 x[EPT], z[EPT];
    stage_load<float2, EPT, p.r0>(buf, x, LS, t, G);
    gx_swap<EPT>(x);
    __syncthreads();
    gx_transform<LS>(x, buf, op.gx1, t);
    // v = u - z (first product), kept for the final subtraction; then chi' v
    const long off = c * ((long)op.n1 * op.n2) + (long)i2 * op.n1;
    const float2* cr = (c == 2 ? op.chim : chir) + (long)i2 * op.n1;     // the regulariser keeps chi_m
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r0>(e), idx = t + j * G, f = fx_reg<EPT, p.r1>(j);
        z[e] = make_float2(0.f, 0.f);
        if (j < EPT / 2 && active && idx < op.n1) {
            const float2 v = csub(cvt<float2>(u[off + idx]), make_float2(x[f].y, x[f].x));
            vbuf[off + idx] = v;
            z[e] = cmul(v, cr[idx]);
        }
    }
    gx_transform<LS>(z, buf, op.gx1, t);
    stage_store<float2, EPT, p.r1>(buf, z, LS, LS / p.r1, t, G);
    __syncthreads();
    gx_store_tile(reinterpret_cast<const float2*>(smem_raw), W, c, i2_0, LS, op.n2, TR, Lp);
}

// ------------------------------------------------------------------------- K2
// One block per column k1, G threads per plane; the Green multiply at the first inverse
// stage's indices (planes G11, G22, G12 (G13, G23, G33), of parity -1 in both / x2 / x1 for
// G12 / G13 / G23).
template <int P, int LS>
__global__ void __launch_bounds__(P * (LS / gx_plan(LS).ept)) k2_gx(OpDev<float> op, float2* __restrict__ W,
                                                                 const int* __restrict__ skip) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, G = LS / EPT, Q2 = LS / 2 + 1;
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.y * op.ws;            // right-hand side of a batched product
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Lp = padded_len(LS);
    float2* bufs = reinterpret_cast<float2*>(smem_raw);
    const int comp = threadIdx.x / G, t = threadIdx.x - comp * G;
    float2* buf = bufs + comp * Lp;
    const int k1 = blockIdx.x;
    float2* col = W + ((long)comp * op.M1 + k1) * op.n2;
    const int h1 = op.M1 >> 1;
    const int k1q = k1 <= h1 ? k1 : op.M1 - k1;
    const bool neg1 = k1 > h1;
    const long plane = (long)op.Q1 * Q2;
    const float2* g = op.gq + (long)k1q * Q2;
    float2 x[EPT];
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r0>(e), idx = t + j * G;
        x[e] = j < EPT / 2 && idx < op.n2 ? col[idx] : make_float2(0.f, 0.f);
    }
    gx_transform<LS>(x, buf, op.gx2, t);
    stage_store<float2, EPT, p.r1>(buf, x, LS, LS / p.r1, t, G);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int k2 = t + fx_slot<EPT, p.r0>(e) * G;
        const bool neg2 = k2 > LS / 2;
        const int k2q = neg2 ? LS - k2 : k2;
        float2 acc;
#pragma unroll
        for (int q = 0; q < P; q++) {
            const int pl = q == comp ? (q == 2 ? 5 : q) : (q + comp == 1 ? 2 : q + comp + 1);
            const bool neg = q != comp && (q + comp == 1 ? neg1 != neg2 : (q + comp == 2 ? neg2 : neg1));
            float2 w = __ldg(&g[pl * plane + k2q]);
            if (neg) w = make_float2(-w.x, -w.y);
            const float2 z = cmul(w, bufs[q * Lp + pidx(k2)]);
            acc = q == 0 ? z : cadd(acc, z);
        }
        x[e] = make_float2(acc.y, acc.x);
    }
    __syncthreads();
    gx_transform<LS>(x, buf, op.gx2, t);
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r1>(e), idx = t + j * G;
        if (j < EPT / 2 && idx < op.n2) col[idx] = make_float2(x[e].y, x[e].x);
    }
}

// Two planes with both values of a column index in one thread (G threads per column), where the
// first and the last radix agree: the last forward stage leaves a thread the values that the first
// inverse stage wants, so the Green multiply stays in registers, and a twiddle or Green factor
// is loaded once for both planes.  Large launches of k2_gx are bound by those loads and by its
// shared-memory traffic: 256^2, per launch, one product 9.4 -> 8.2 us, 8 25.6 -> 20.9, 32
// 83 -> 67 (the half-filled kernels of fft_fast.cuh at this length: 10.3, 23.5, 70).
template <int EPT, int R>
__device__ __forceinline__ void gx_stage2(float2 (&x)[EPT], float2 (&y)[EPT], int Ns, int t, int G,
                                          const float2* __restrict__ tw) {
#pragma unroll
    for (int b = 0; b < EPT / R; b++) {
        if (Ns > 1) {
            const int k = mod_ns(t + b * G, Ns);
#pragma unroll
            for (int r = 1; r < R; r++) {
                const float2 w = ld_tw(&tw[r * Ns + k - 1]);
                x[b * R + r] = cmul(x[b * R + r], w);
                y[b * R + r] = cmul(y[b * R + r], w);
            }
        }
        gx_dft<R>(&x[b * R]);
        gx_dft<R>(&y[b * R]);
    }
}
template <int LS> __device__ __forceinline__ void gx_transform2(float2 (&x)[gx_plan(LS).ept], float2 (&y)[gx_plan(LS).ept],
                                                                float2* bx, float2* by, const float2* tw, int t) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, R0 = p.r0, R1 = p.r1, G = LS / EPT;
    gx_stage2<EPT, R0>(x, y, 1, t, G, tw);
    stage_store<float2, EPT, R0>(bx, x, LS, 1, t, G);
    stage_store<float2, EPT, R0>(by, y, LS, 1, t, G);
    __syncthreads();
    int Ns = R0;
#pragma unroll
    for (int s = 1; s <= p.q; s++) {
        stage_load<float2, EPT, R1>(bx, x, LS, t, G);
        stage_load<float2, EPT, R1>(by, y, LS, t, G);
        gx_stage2<EPT, R1>(x, y, Ns, t, G, tw);
        __syncthreads();
        if (s < p.q) {
            stage_store<float2, EPT, R1>(bx, x, LS, Ns, t, G);
            stage_store<float2, EPT, R1>(by, y, LS, Ns, t, G);
            __syncthreads();
        }
        Ns *= R1;
    }
}
// a u + b v, each product rounded before the sum (no multiply-add across it): the results are those
// of k2_gx to the bit.
__device__ __forceinline__ float2 gx_green(float2 a, float2 u, float2 b, float2 v) {
    auto mul = [](float2 p, float2 q) {
        return make_float2(__fmaf_rn(p.x, q.x, -__fmul_rn(p.y, q.y)), __fmaf_rn(p.x, q.y, __fmul_rn(p.y, q.x)));
    };
    const float2 x = mul(a, u), y = mul(b, v);
    return make_float2(__fadd_rn(x.x, y.x), __fadd_rn(x.y, y.y));
}
template <int LS>
__global__ void __launch_bounds__(LS / gx_plan(LS).ept) k2_gx_pair(OpDev<float> op, float2* __restrict__ W,
                                                                   const int* __restrict__ skip) {
    constexpr FxPlan p = gx_plan(LS);
    constexpr int EPT = p.ept, G = LS / EPT, Q2 = LS / 2 + 1;
    static_assert(p.r0 == p.r1, "registers of the last stage are those of the first");
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.y * op.ws;            // right-hand side of a batched product
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf0 = reinterpret_cast<float2*>(smem_raw);
    float2* buf1 = buf0 + padded_len(LS);
    const int t = threadIdx.x, k1 = blockIdx.x;
    float2* col0 = W + (long)k1 * op.n2;
    float2* col1 = W + ((long)op.M1 + k1) * op.n2;
    const int h1 = op.M1 >> 1;
    const int k1q = k1 <= h1 ? k1 : op.M1 - k1;
    const bool neg1 = k1 > h1;
    const long plane = (long)op.Q1 * Q2;
    const float2* g = op.gq + (long)k1q * Q2;
    float2 x[EPT], y[EPT];
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r0>(e), idx = t + j * G;
        const bool in = j < EPT / 2 && idx < op.n2;
        x[e] = in ? col0[idx] : make_float2(0.f, 0.f);
        y[e] = in ? col1[idx] : make_float2(0.f, 0.f);
    }
    gx_transform2<LS>(x, y, buf0, buf1, op.gx2, t);
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int k2 = t + fx_slot<EPT, p.r0>(e) * G;
        const bool neg2 = k2 > LS / 2;
        const int k2q = neg2 ? LS - k2 : k2;
        float2 w = __ldg(&g[2 * plane + k2q]);
        if (neg1 != neg2) w = make_float2(-w.x, -w.y);
        const float2 a = gx_green(__ldg(&g[k2q]), x[e], w, y[e]);
        const float2 b = gx_green(w, x[e], __ldg(&g[plane + k2q]), y[e]);
        x[e] = make_float2(a.y, a.x);
        y[e] = make_float2(b.y, b.x);
    }
    gx_transform2<LS>(x, y, buf0, buf1, op.gx2, t);
#pragma unroll
    for (int e = 0; e < EPT; e++) {
        const int j = fx_slot<EPT, p.r1>(e), idx = t + j * G;
        if (j < EPT / 2 && idx < op.n2) {
            col0[idx] = make_float2(x[e].y, x[e].x);
            col1[idx] = make_float2(y[e].y, y[e].x);
        }
    }
}

// --------------------------------------------------------------------- launch
template <int LS> static Launch gx_rows_launch(const OpDev<float>& v, int nb) {
    constexpr int G = LS / gx_plan(LS).ept;
    // the operator's schedule where it has one (half_filled_rows); else fewer rows per block
    // while that leaves no SM with two blocks
    if (half_filled_rows(v)) {
        int h = v.tr ? v.tr : default_tile_rows_c64(LS);
        // batches at length 256: 64-byte segments once four blocks per SM are left (32 products at
        // 128^2, K1 13.4 -> 12.1 us, K3K1 20.9 -> 18.6; 8 of them 8.2 -> 8.4, 10.2 -> 10.5)
        if (LS == 256 && !v.tr && (long)v.n2 * v.planes * nb >= 8 * 4 * 152) h = 8;
        return Launch{dim3((v.n2 + h - 1) / h, v.planes, nb), dim3(h * G), (size_t)h * tile_stride(LS) * sizeof(float2)};
    }
    int TR = kGxTileRows;
    while (TR > 1 && (TR * G > kRowsMaxThreads || (long)(2 * v.n2 / TR) * v.planes * nb <= 152)) TR /= 2;
    return Launch{dim3((v.n2 + TR - 1) / TR, v.planes, nb), dim3(TR * G), (size_t)TR * tile_stride(LS) * sizeof(float2)};
}
template <int LS> template <typename IO>
void GxLaunch<LS>::k1(const OpDev<float>& v, const IO* u, const float2* chi, float2* W, const int* skip,
                      cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k1_gx<IO, LS>, a, gx_rows_launch<LS>(v, nb), st, v, u, chi, W, skip);
}
template <int LS> template <typename U, typename IO>
void GxLaunch<LS>::k3(const OpDev<float>& v, const float2* W, const U* u, IO* y, const int* skip, cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k3_gx<U, IO, LS>, a, gx_rows_launch<LS>(v, nb), st, v, W, u, y, skip);
}
template <int LS> template <typename IO>
void GxLaunch<LS>::k3k1(const OpDev<float>& v, float2* W, const IO* u, const float2* chir, float2* vb, const int* skip,
                        cudaStream_t st, int nb) {
    static std::atomic<bool> a{false};
    launch_kernel(k3k1_gx<IO, LS>, a, gx_rows_launch<LS>(v, nb), st, v, W, u, chir, vb, skip);
}
template <int LS>
void GxLaunch<LS>::k2(const OpDev<float>& v, float2* W, const int* skip, cudaStream_t st, int nb) {
    static std::atomic<bool> a2{false}, a3{false};
    const Launch l{dim3(v.M1, nb), dim3(v.planes * (LS / gx_plan(LS).ept)),
                   (size_t)v.planes * padded_len(LS) * sizeof(float2)};
    if (v.planes == 3) {
        launch_kernel(k2_gx<3, LS>, a3, l, st, v, W, skip);
    } else if constexpr (LS == 512) {     // equal radices; other such lengths are short or fast_length
        launch_kernel(k2_gx_pair<LS>, a2, Launch{l.grid, dim3(LS / gx_plan(LS).ept), l.smem}, st, v, W, skip);
    } else {
        launch_kernel(k2_gx<2, LS>, a2, l, st, v, W, skip);
    }
}

// Instantiates the launchers of one length.
#define DIE_GX_INSTANTIATE(LS)                                                                                       \
    template void GxLaunch<LS>::k1<float2>(const OpDev<float>&, const float2*, const float2*, float2*, const int*,   \
                                           cudaStream_t, int);                                                      \
    template void GxLaunch<LS>::k1<double2>(const OpDev<float>&, const double2*, const float2*, float2*, const int*, \
                                            cudaStream_t, int);                                                     \
    template void GxLaunch<LS>::k2(const OpDev<float>&, float2*, const int*, cudaStream_t, int);                     \
    template void GxLaunch<LS>::k3<float2, float2>(const OpDev<float>&, const float2*, const float2*, float2*,       \
                                                   const int*, cudaStream_t, int);                                  \
    template void GxLaunch<LS>::k3<double2, double2>(const OpDev<float>&, const float2*, const double2*, double2*,   \
                                                     const int*, cudaStream_t, int);                                \
    template void GxLaunch<LS>::k3<float2, double2>(const OpDev<float>&, const float2*, const float2*, double2*,     \
                                                    const int*, cudaStream_t, int);                                 \
    template void GxLaunch<LS>::k3k1<float2>(const OpDev<float>&, float2*, const float2*, const float2*, float2*,    \
                                             const int*, cudaStream_t, int);                                        \
    template void GxLaunch<LS>::k3k1<double2>(const OpDev<float>&, float2*, const double2*, const float2*, float2*,  \
                                              const int*, cudaStream_t, int);

}  // namespace die

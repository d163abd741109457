// FFT-speed products with the discretised TE operator A = I - G X (Eqs. (4.3)-(4.5)):
// kernels and launchers of the complex64 products, instantiated in matvec_f32.cu (the FP64
// products run the same passes in fixed point, fx_kernels.cuh).
//
// G is block-Toeplitz (its entries depend on x_n - x_m only), so G w is a 2-D
// linear convolution of the 2 x 2 Green's tensor table with the contrast current
// w = chi u; it is computed with zero padding to M1 x M2 >= (2 n1) x (2 n2):
//
//   K1  per grid row i2 and component: w = chi * u, zero-pad to M1, FFT along x1,
//       written transposed: W[c][k1][i2]                    (rows i2 < n2 only)
//   K2  per column k1: FFT along x2 (inputs i2 >= n2 are zero), multiply by the
//       Green spectra  z1 = G11 w1 + G12 w2, z2 = G12 w1 + G22 w2, inverse FFT,
//       keep i2 < n2, written back in place
//   K3  per grid row: inverse FFT along x1, keep i1 < n1, y = u - z
//   K3K1 (regularised product A(chi') A(chi), Section 5) finishes row i2 of the
//       first product (v = u - z, kept in a buffer for the final subtraction) and
//       immediately starts the second product on the same row: chi' * v, FFT.
//
// The spectra are stored for k1 <= M1/2, k2 <= M2/2 only: G11, G22 are even and
// G12 is odd in each offset coordinate (a symmetry of Eqs. (4.3)-(4.5)), so the
// other quadrants follow by sign.  They carry the 1/(M1 M2) of the inverse FFTs.
//
// Here: transforms of length 1024, 2048 and 4096 (rows and columns apart) of two-plane grids,
// on the compile-time stages of fft_fast.cuh; the others take the passes of gx_kernels.cuh.
#pragma once

#include <atomic>
#include <type_traits>

#include "fft_fast.cuh"
#include "gx_launch.cuh"
#include "op.cuh"
#include "prof.cuh"

namespace die {

// Rows per block of the row passes: enough for 32-byte segments in the transposed
// accesses, at most 512 threads per block.
constexpr int kTileRows = 4;
// The column pass stages its Green spectra where that leaves room for two blocks per SM
// (not at length 4096: 119 KB with them, 70 KB without; two blocks of 128 registers there:
// product at 2048^2 770 -> 704 us).
constexpr size_t kStageGreenMaxSmem = 100 * 1024;

template <typename C> __device__ __forceinline__ C czero() { C z; z.x = 0; z.y = 0; return z; }

// Row stride of the row-pass tiles: the padded length plus two slots, so that the TR
// rows (whose lengths are multiples of 128 bytes) start in different banks.
__host__ __device__ __forceinline__ int tile_stride(int L) { return padded_len(L) + 2; }

// Load the transposed tile W[c][0..M1)[i2_0 .. i2_0+TR) into shared memory rows.
template <typename C>
__device__ __forceinline__ void load_tile(C* tile, const C* __restrict__ W, int c, int i2_0, int M1, int n2, int TR) {
    const int Lp = tile_stride(M1);
    for (int e = threadIdx.x; e < M1 * TR; e += blockDim.x) {
        const int k1 = e / TR, r = e - k1 * TR;
        const int row = i2_0 + r;
        tile[r * Lp + pidx(k1)] = row < n2 ? W[((long)c * M1 + k1) * n2 + row] : czero<C>();
    }
    __syncthreads();
}

// ------------------------------------------------------------------ fast path
// Transforms of length L = 1024, 2048 and 4096 (the deflated first row pass: 2^a from 256 on) with
// the compile-time stages of fft_fast.cuh.  The zero inputs (index >= L / 2) of the forward
// transforms and the discarded outputs of the inverse ones are known at compile time; a grid
// that fills less than half of a transform (RAG) checks the others' indices.
template <typename C, int L> constexpr int fast_tr() {
    return kTileRows * (L / 16) <= kRowsMaxThreads ? kTileRows : kRowsMaxThreads / (L / 16);
}
template <int L> constexpr int tile_stride_c() { return L + (L >> 4) + 2; }

// Asynchronous global -> shared copy of one complex value (no register staging), and the
// wait for all of this thread's copies.
template <typename C>
__device__ __forceinline__ void cp_async_elem(C* smem, const C* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    static_assert(sizeof(C) == 8, "complex64");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Transposed tile I/O of the row passes: thread (k0 = tid / TR, r = tid % TR) moves
// elements k1 = k0 + it G, it < 16, of tile row r.
template <typename C, int L, int TR, bool STORE>
__device__ __forceinline__ void tile_io(C* tile, C* __restrict__ W, int c, int i2_0, int n2) {
    constexpr int G = L / 16, Lp = tile_stride_c<L>();
    const int r = threadIdx.x % TR, k0 = threadIdx.x / TR;
    const int row = i2_0 + r;
    C* t = tile + r * Lp + pidx(k0);
    C* g = W + ((long)c * L + k0) * n2 + row;
    const long gs = (long)G * n2;
#pragma unroll
    for (int it = 0; it < 16; it++) {
        const int off = it * G + ((it * G) >> 4);
        if constexpr (STORE) {
            if (row < n2) g[it * gs] = t[off];
        } else {
            t[off] = row < n2 ? g[it * gs] : czero<C>();
        }
    }
}

// RAG: n1 < L / 2 (a run-time row length); the transform still treats its upper half as zero.
template <typename T, typename IO, int L, int TR, bool RAG>
__global__ void __launch_bounds__(512) k1_fast(OpDev<T> op, const IO* __restrict__ u, const C_t<T>* __restrict__ chi,
                                               C_t<T>* __restrict__ W, const int* __restrict__ skip) {
    using C = C_t<T>;
    constexpr int G = L / 16;
    using F0 = typename PlanStage<C, L, false, 0>::St;
    pdl_wait();
    if (block_flag(skip)) return;
    u += blockIdx.z * op.xs;            // right-hand side of a batched product
    W += blockIdx.z * op.ws;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tile = reinterpret_cast<C*>(smem_raw);
    const int rs = threadIdx.x / G, t = threadIdx.x % G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    C* buf = tile + rs * tile_stride_c<L>();
    const int n1 = RAG ? op.n1 : L / 2;
    C x[16];
    if (active) {
        const long N = (long)n1 * op.n2;
        const IO* ur = u + c * N + (long)i2 * n1 + t;
        const C* cr = chi + (long)i2 * n1 + t;
#pragma unroll
        for (int e = 0; e < 16; e++) {
            const int idx = F0::index(e);
            x[e] = idx < L / 2 && (!RAG || t + idx < n1) ? cmul(cvt<C>(ur[idx]), cr[idx]) : czero<C>();
        }
        F0::compute(x, t, op.twx1);
        F0::store(buf, x, t);
    }
    __syncthreads();
    run_fast<C, L, false, 1, P2<L>::fwd.ns, false>(buf, x, t, op.twx1, active);
    tile_io<C, L, TR, true>(tile, W, c, i2_0, op.n2);
}

// First row pass of a deflated FP32-inner product (complex64): per element
// z = v + sum_i V32_i cf_i (v = w / ||w|| written back to the FP64 Arnoldi vector, or
// the complex64 x), stored to zout for the later passes, then chi * z and the forward
// row transform as in k1_fast.  The basis loads go five vectors (40 loads) at a time.
template <int L, int TR>
__global__ void __launch_bounds__(512) k1_defl_fast(OpDev<float> op, DeflIn d, const float2* __restrict__ chi,
                                                    float2* __restrict__ zout, float2* __restrict__ W,
                                                    const int* __restrict__ skip) {
    using C = float2;
    constexpr int G = L / 16, n1 = L / 2;
    using F0 = typename PlanStage<C, L, false, 0>::St;
    __shared__ float2 cs[32];
    pdl_wait();
    if (block_flag(skip)) return;
    for (int i = threadIdx.x; i < d.r; i += blockDim.x) cs[i] = __ldcg(&d.cf[i]);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tile = reinterpret_cast<C*>(smem_raw);
    const int rs = threadIdx.x / G, t = threadIdx.x % G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    C* buf = tile + rs * tile_stride_c<L>();
    __syncthreads();
    C x[16];
    if (active) {
        const long off = c * ((long)n1 * op.n2) + (long)i2 * n1 + t;
        C zq[8];
        if (d.w) {
            const double sc = *d.inv;
#pragma unroll
            for (int e = 0, q = 0; e < 16; e++) {
                const int idx = F0::index(e);
                if (idx < n1) {
                    double2 u = d.w[off + idx];
                    u.x *= sc;
                    u.y *= sc;
                    d.w[off + idx] = u;
                    if (d.wm) d.wm[off + idx] = u.x - u.y;
                    zq[q++] = make_float2((float)u.x, (float)u.y);
                }
            }
        } else {
#pragma unroll
            for (int e = 0, q = 0; e < 16; e++)
                if (F0::index(e) < n1) zq[q++] = d.x[off + F0::index(e)];
        }
        constexpr int VB = 5;                     // basis vectors per round of loads (40 in flight)
        for (int i0 = 0; i0 < d.r; i0 += VB) {
            C a[VB][8];
#pragma unroll
            for (int v = 0; v < VB; v++) {
                const C* p = d.V32 + (long)(i0 + v < d.r ? i0 + v : i0) * d.ld + off;
#pragma unroll
                for (int e = 0, q = 0; e < 16; e++)
                    if (F0::index(e) < n1) a[v][q++] = p[F0::index(e)];
            }
#pragma unroll
            for (int v = 0; v < VB; v++) {
                if (i0 + v < d.r) {
                    const C cv = cs[i0 + v];
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        zq[q].x = fmaf(a[v][q].x, cv.x, zq[q].x);
                        zq[q].x = fmaf(-a[v][q].y, cv.y, zq[q].x);
                        zq[q].y = fmaf(a[v][q].x, cv.y, zq[q].y);
                        zq[q].y = fmaf(a[v][q].y, cv.x, zq[q].y);
                    }
                }
            }
        }
        const C* cr = chi + (long)i2 * n1 + t;
#pragma unroll
        for (int e = 0, q = 0; e < 16; e++) {
            const int idx = F0::index(e);
            if (idx < n1) {
                zout[off + idx] = zq[q];
                x[e] = cmul(zq[q], cr[idx]);
                q++;
            } else {
                x[e] = czero<C>();
            }
        }
        F0::compute(x, t, op.twx1);
        F0::store(buf, x, t);
    }
    __syncthreads();
    run_fast<C, L, false, 1, P2<L>::fwd.ns, false>(buf, x, t, op.twx1, active);
    tile_io<C, L, TR, true>(tile, W, c, i2_0, op.n2);
}

// Complex64 column pass with both components in the same thread (G threads per column):
// the last forward stage leaves each thread's values at the indices where the first
// inverse stage (same radix: the inverse plan is the reversed forward plan) wants them,
// so the 2 x 2 Green multiply is done in registers between the two, with no shared-
// memory round trip, and every twiddle serves both components.
template <typename T, int L, bool RAG>
__global__ void __launch_bounds__(L / 16, (L == 1024 ? 7 : L == 4096 ? 2 : 1)) k2_fast2(OpDev<T> op, C_t<T>* __restrict__ W,
                                                                        int stage_g, const int* __restrict__ skip) {
    using C = C_t<T>;
    constexpr int G = L / 16, Q2 = L / 2 + 1, Lp = L + (L >> 4);
    const int n2 = RAG ? op.n2 : L / 2;
    constexpr int nsf = P2<L>::fwd.ns, nsi = P2<L>::inv.ns;
    using F0 = typename PlanStage<C, L, false, 0>::St;
    using FL = typename PlanStage<C, L, false, nsf - 1>::St;
    using I0 = typename PlanStage<C, L, true, 0>::St;
    using IL = typename PlanStage<C, L, true, nsi - 1>::St;
    static_assert(FL::kR == I0::kR, "the inverse plan is the reversed forward plan");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf0 = reinterpret_cast<C*>(smem_raw);
    C* buf1 = buf0 + Lp;
    C* gs = buf1 + Lp;
    const int t = threadIdx.x;
    W += blockIdx.y * op.ws;            // right-hand side of a batched product
    const int k1 = blockIdx.x;
    C* col0 = W + (long)k1 * n2 + t;
    C* col1 = W + ((long)op.M1 + k1) * n2 + t;
    const int h1 = op.M1 >> 1;
    const int k1q = k1 <= h1 ? k1 : op.M1 - k1;
    const bool neg1 = k1 > h1;
    const long plane = (long)op.Q1 * Q2;
    const C* g = op.gq + (long)k1q * Q2;
    if (stage_g) {   // the column's three quarter-spectrum rows (operator constants), issued
                     // before the wait on the previous kernel; they land during the forward FFT
        for (int e = t; e < 3 * Q2; e += G) {
            const int pl = e / Q2, q = e - pl * Q2;
            cp_async_elem(gs + e, g + pl * plane + q);
        }
    }
    pdl_wait();
    if (block_flag(skip)) {
        cp_async_wait_all();
        return;
    }
    C x0[16], x1[16];
#pragma unroll
    for (int e = 0; e < 16; e++) {
        const int idx = F0::index(e);
        x0[e] = idx < L / 2 && (!RAG || t + idx < n2) ? col0[idx] : czero<C>();
        x1[e] = idx < L / 2 && (!RAG || t + idx < n2) ? col1[idx] : czero<C>();
    }
    F0::compute2(x0, x1, t, op.twx2);
    F0::store(buf0, x0, t);
    F0::store(buf1, x1, t);
    __syncthreads();
    run_fast2<C, L, false, 1, nsf - 1>(buf0, buf1, x0, x1, t, op.twx2);
    FL::load(buf0, x0, t);
    FL::load(buf1, x1, t);
    FL::compute2(x0, x1, t, op.twx2);
    if (stage_g) cp_async_wait_all();
    __syncthreads();             // spectra visible; every thread has read its last forward stage
    {   // 2 x 2 Green-spectrum multiply at k2 = t + c (c = I0::index(e))
        const long ps = stage_g ? (long)Q2 : plane;
        const C* gsrc = stage_g ? gs : g;
        const C* g11p = gsrc + t;           // k2 <= L/2: quarter index k2
        const C* g22p = gsrc + ps + t;
        const C* g12p = gsrc + 2 * ps + t;
        const C* g11m = gsrc - t;           // k2 > L/2: quarter index L - k2
        const C* g22m = gsrc + ps - t;
        const C* g12m = gsrc + 2 * ps - t;
#pragma unroll
        for (int e = 0; e < 16; e++) {
            const int c = I0::index(e);
            C a, b, go;
            bool neg2;
            if (c < L / 2) { a = g11p[c]; b = g22p[c]; go = g12p[c]; neg2 = false; }
            else { a = g11m[L - c]; b = g22m[L - c]; go = g12m[L - c]; neg2 = c > L / 2 || t > 0; }
            if (neg1 != neg2) { go.x = -go.x; go.y = -go.y; }
            const C u0 = x0[e], u1 = x1[e];
            x0[e] = cadd(cmul(a, u0), cmul(go, u1));
            x1[e] = cadd(cmul(go, u0), cmul(b, u1));
        }
    }
    I0::compute2(x0, x1, t, op.twx2);
    I0::store(buf0, x0, t);
    I0::store(buf1, x1, t);
    __syncthreads();
    run_fast2<C, L, true, 1, nsi - 1>(buf0, buf1, x0, x1, t, op.twx2);
    IL::load(buf0, x0, t);
    IL::load(buf1, x1, t);
    IL::compute2(x0, x1, t, op.twx2);
#pragma unroll
    for (int e = 0; e < 16; e++) {
        const int idx = IL::index(e);
        if (idx < L / 2 && (!RAG || t + idx < n2)) { col0[idx] = x0[e]; col1[idx] = x1[e]; }
    }
}

template <typename T, typename U, typename IO, int L, int TR, bool RAG>
__global__ void __launch_bounds__(512) k3_fast(OpDev<T> op, const C_t<T>* __restrict__ W, const U* __restrict__ u,
                                               IO* __restrict__ y, const int* __restrict__ skip) {
    using C = C_t<T>;
    constexpr int G = L / 16, ns = P2<L>::inv.ns;
    const int n1 = RAG ? op.n1 : L / 2;
    using IL = typename PlanStage<C, L, true, ns - 1>::St;
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    y += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tile = reinterpret_cast<C*>(smem_raw);
    const int rs = threadIdx.x / G, t = threadIdx.x % G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    C* buf = tile + rs * tile_stride_c<L>();
    const long off = c * ((long)n1 * op.n2) + (long)(active ? i2 : 0) * n1 + t;
    U up[8];                    // u at this thread's output indices, loaded before the FFT
#pragma unroll
    for (int e = 0, q = 0; e < 16; e++)
        if (IL::index(e) < L / 2) {
            if (!RAG || t + IL::index(e) < n1) up[q] = u[off + IL::index(e)];
            q++;
        }
    tile_io<C, L, TR, false>(tile, const_cast<C*>(W), c, i2_0, op.n2);
    __syncthreads();
    C x[16];
    run_fast<C, L, true, 0, ns - 1, false>(buf, x, t, op.twx1, active);
    if (!active) return;
    IL::load(buf, x, t);
    IL::compute(x, t, op.twx1);
#pragma unroll
    for (int e = 0, q = 0; e < 16; e++) {
        const int idx = IL::index(e);
        if (idx < L / 2) {
            if (!RAG || t + idx < n1) y[off + idx] = csub(cvt<IO>(up[q]), cvt<IO>(x[e]));
            q++;
        }
    }
}

template <typename T, typename IO, int L, int TR, bool RAG>
__global__ void __launch_bounds__(512) k3k1_fast(OpDev<T> op, C_t<T>* __restrict__ W, const IO* __restrict__ u,
                                                 const C_t<T>* __restrict__ chir, C_t<T>* __restrict__ vbuf,
                                                 const int* __restrict__ skip) {
    using C = C_t<T>;
    constexpr int G = L / 16;
    const int n1 = RAG ? op.n1 : L / 2;
    constexpr int nsi = P2<L>::inv.ns, nsf = P2<L>::fwd.ns;
    using IL = typename PlanStage<C, L, true, nsi - 1>::St;
    using F0 = typename PlanStage<C, L, false, 0>::St;
    static_assert(IL::kR == F0::kR, "the inverse plan is the reversed forward plan");
    pdl_wait();
    if (block_flag(skip)) return;
    W += blockIdx.z * op.ws;            // right-hand side of a batched product
    u += blockIdx.z * op.xs;
    vbuf += blockIdx.z * op.xs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tile = reinterpret_cast<C*>(smem_raw);
    const int rs = threadIdx.x / G, t = threadIdx.x % G;
    const int c = blockIdx.y, i2_0 = blockIdx.x * TR, i2 = i2_0 + rs;
    const bool active = i2 < op.n2;
    C* buf = tile + rs * tile_stride_c<L>();
    const long off = c * ((long)n1 * op.n2) + (long)(active ? i2 : 0) * n1 + t;
    const C* cr = chir + (long)(active ? i2 : 0) * n1 + t;
    C up[8], cp[8];             // u and chi' at this thread's indices, loaded before the FFT
#pragma unroll
    for (int e = 0, q = 0; e < 16; e++)
        if (IL::index(e) < L / 2) {
            const bool in = !RAG || t + IL::index(e) < n1;
            up[q] = in ? cvt<C>(u[off + IL::index(e)]) : czero<C>();
            cp[q] = in ? cr[IL::index(e)] : czero<C>();
            q++;
        }
    tile_io<C, L, TR, false>(tile, W, c, i2_0, op.n2);
    __syncthreads();
    C x[16];
    run_fast<C, L, true, 0, nsi - 1, false>(buf, x, t, op.twx1, active);
    if (active) {
        IL::load(buf, x, t);
        IL::compute(x, t, op.twx1);
        // v = u - z (first product), kept for the final subtraction; then chi' v -> FFT
#pragma unroll
        for (int e = 0, q = 0; e < 16; e++) {
            const int idx = IL::index(e);
            if (idx < L / 2) {
                const C v = csub(up[q], x[e]);
                const bool in = !RAG || t + idx < n1;
                if (in) vbuf[off + idx] = v;
                x[e] = in ? cmul(v, cp[q]) : czero<C>();
                q++;
            } else {
                x[e] = czero<C>();
            }
        }
    }
    __syncthreads();            // every thread has read its last inverse stage from the tile
    if (active) {
        F0::compute(x, t, op.twx1);
        F0::store(buf, x, t);
    }
    __syncthreads();
    run_fast<C, L, false, 1, nsf, false>(buf, x, t, op.twx1, active);
    tile_io<C, L, TR, true>(tile, W, c, i2_0, op.n2);
}

// --------------------------------------------------------------------- launch
struct Launch { dim3 grid, block; size_t smem; };
inline Launch with_z(Launch l, int nb) { l.grid.z = nb; return l; }

template <typename T>
inline Launch cols_launch(const OpDev<T>& v, int* stage_g) {
    using C = C_t<T>;
    const size_t base = (size_t)2 * padded_len(v.M2) * sizeof(C);
    const size_t staged = base + (size_t)3 * v.Q2 * sizeof(C);
    *stage_g = staged <= kStageGreenMaxSmem ? 1 : 0;
    return Launch{dim3(v.M1), dim3(v.M2 / 16), *stage_g ? staged : base};
}

// Launch a kernel instantiation, raising its dynamic shared-memory limit on first use
// to what the 227 KB per block leaves beside the kernel's static shared memory.
template <typename K, typename... Args>
inline void launch_kernel(K kernel, std::atomic<bool>& attr_set, const Launch& l, cudaStream_t st, Args... args) {
    if (!attr_set.load(std::memory_order_acquire)) {
        cudaFuncAttributes fa = {};
        const size_t stat = cudaFuncGetAttributes(&fa, kernel) == cudaSuccess ? fa.sharedSizeBytes : 1024;
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(227 * 1024 - stat));
        attr_set.store(true, std::memory_order_release);
    }
    launch_pdl(kernel, l.grid, l.block, l.smem, st, args...);
}

// Transforms on the stages of fft_fast.cuh: two planes, L = 1024, 2048 or 4096 (16 values per
// thread, both components of a column in one thread).  Shorter ones, 3 * 2^a and three planes
// take the any-grid kernels (gx_kernels.cuh), which are faster there: 128^2 24.3 -> 20 us,
// 256^2 29 -> 23; at L = 1024 they take 62 us where these take 46.
inline bool fast_length(int L) { return L == 1024 || L == 2048 || L == 4096; }
template <typename T> inline bool fast_rows(const OpDev<T>& v) { return v.planes == 2 && fast_length(v.M1); }
template <typename T> inline bool fast_cols(const OpDev<T>& v) { return v.planes == 2 && fast_length(v.M2); }
// Grids whose rows fill half of a transform of length 2^a in [256, 4096]: the deflated first
// row pass (k1_defl_fast) and the tile schedule (dieop_autotune).
template <typename T> inline bool half_filled_rows(const OpDev<T>& v) {
    return v.planes == 2 && 2 * v.n1 == v.M1 && v.M1 >= 256 && v.M1 <= 4096 && (v.M1 & (v.M1 - 1)) == 0;
}
template <typename C, int L, int TR> inline Launch rows_launch_fast(int n2) {
    return Launch{dim3((n2 + TR - 1) / TR, 2), dim3(TR * (L / 16)), (size_t)TR * tile_stride_c<L>() * sizeof(C)};
}

#define DIE_FAST_SWITCH(M, CASE)  \
    switch (M) {                  \
        case 1024: CASE(1024); break; \
        case 2048: CASE(2048); break; \
        case 4096: CASE(4096); break; \
        default: break;               \
    }

// Those of half_filled_rows.
#define DIE_HALF_SWITCH(M, CASE)      \
    switch (M) {                      \
        case 256: CASE(256); break;   \
        case 512: CASE(512); break;   \
        default: DIE_FAST_SWITCH(M, CASE); break; \
    }

// Tile height of the fast row passes: the rows of one block (TR).  0 selects fast_tr, the
// default of the length; an operator's schedule (dieop_autotune,
// dieop_set_tile_rows) may pick another valid height for its complex64 passes.  Every row
// is transformed by the same threads and stages whatever TR is, so the products are
// bit-identical for all heights.
template <typename C, int L, int TR> constexpr int tile_of() { return TR == 0 ? fast_tr<C, L>() : TR; }
template <typename C, int L, int TR> constexpr bool tile_ok() {
    return TR == 0 || (TR * (L / 16) <= kRowsMaxThreads && TR != fast_tr<C, L>());
}

// The fast row passes at one tile height (definitions in rows_fast.cuh).
template <typename T, typename IO, int TR>
void rows_fwd_fast(const OpDev<T>& v, const IO* u, const C_t<T>* chi, C_t<T>* W, const int* skip, cudaStream_t st,
                   int nb);
template <typename T, typename U, typename IO, int TR>
void rows_inv_fast(const OpDev<T>& v, const C_t<T>* W, const U* u, IO* y, const int* skip, cudaStream_t st, int nb);
template <typename T, typename IO, int TR>
void rows_inv_fwd_fast(const OpDev<T>& v, C_t<T>* W, const IO* u, const C_t<T>* chir, C_t<T>* vb, const int* skip,
                       cudaStream_t st, int nb);
template <int TR>
void rows_defl_fast(const OpDev<float>& v, const DeflIn& d, const float2* chi, float2* z, float2* W, const int* skip,
                    cudaStream_t st);

// Calls F<TR> with the tile height of the view (the operator's schedule).
template <typename T, typename F>
inline void with_tile_rows(const OpDev<T>& v, F&& f) {
    switch (tile_rows_code(v.tr, v.M1)) {
        case 1: f(std::integral_constant<int, 1>{}); return;
        case 2: f(std::integral_constant<int, 2>{}); return;
        case 8: f(std::integral_constant<int, 8>{}); return;
        default: f(std::integral_constant<int, 0>{});
    }
}

// nb > 1: a batched product over nb right-hand sides (grid z: row passes, grid y: columns).
template <typename T, typename IO>
inline void launch_k1(const OpDev<T>& v, const IO* u, const C_t<T>* chi, C_t<T>* W, const int* skip, cudaStream_t st,
                      int nb = 1) {
    if (fast_rows(v)) {
        with_tile_rows(v, [&](auto tr) { rows_fwd_fast<T, IO, decltype(tr)::value>(v, u, chi, W, skip, st, nb); });
        return;
    }
    DIE_PROF(PK_ROWS_FWD, st, gx_for_length(v.M1, [&](auto l) { l.template k1<IO>(v, u, chi, W, skip, st, nb); }));
}

template <typename T>
inline void launch_k2(const OpDev<T>& v, C_t<T>* W, const int* skip, cudaStream_t st, int nb = 1) {
    if (!fast_cols(v)) {
        DIE_PROF(PK_COLS, st, gx_for_length(v.M2, [&](auto l) { l.k2(v, W, skip, st, nb); }));
        return;
    }
    int sg = 0;
    Launch l = cols_launch(v, &sg);
    l.grid.y = nb;
#define K2F_CASE(LSV)                                                                                    \
    {                                                                                                    \
        static std::atomic<bool> a_{false}, r_{false};                                                   \
        if (2 * v.n2 == LSV) launch_kernel(k2_fast2<T, LSV, false>, a_, l, st, v, W, sg, skip);          \
        else launch_kernel(k2_fast2<T, LSV, true>, r_, l, st, v, W, sg, skip);                           \
    }
    DIE_PROF(PK_COLS, st, DIE_FAST_SWITCH(v.M2, K2F_CASE));
#undef K2F_CASE
}

template <typename T, typename U, typename IO>
inline void launch_k3(const OpDev<T>& v, const C_t<T>* W, const U* u, IO* y, const int* skip, cudaStream_t st,
                      int nb = 1) {
    if (fast_rows(v)) {
        with_tile_rows(v, [&](auto tr) { rows_inv_fast<T, U, IO, decltype(tr)::value>(v, W, u, y, skip, st, nb); });
        return;
    }
    DIE_PROF(PK_ROWS_INV, st, gx_for_length(v.M1, [&](auto l) { l.template k3<U, IO>(v, W, u, y, skip, st, nb); }));
}

template <typename T, typename IO>
inline void launch_k3k1(const OpDev<T>& v, C_t<T>* W, const IO* u, const C_t<T>* chir, C_t<T>* vb, const int* skip,
                        cudaStream_t st, int nb = 1) {
    if (fast_rows(v)) {
        with_tile_rows(v, [&](auto tr) {
            rows_inv_fwd_fast<T, IO, decltype(tr)::value>(v, W, u, chir, vb, skip, st, nb);
        });
        return;
    }
    DIE_PROF(PK_ROWS_INV_FWD, st,
             gx_for_length(v.M1, [&](auto l) { l.template k3k1<IO>(v, W, u, chir, vb, skip, st, nb); }));
}

template <typename T> struct Sel;
template <> struct Sel<float> {
    static const float2* chi(const dieop_s* o, Contrast c) { return c == Contrast::Chi ? o->chi_f : o->chir_f; }
    static OpDev<float> view(const dieop_s* o) { return view_f(o); }
};

template <typename T, typename IO>
die_status apply_op_skip(dieop_s* op, Contrast which, const IO* x, IO* y, const int* skip, cudaStream_t st,
                         const Workspace* ws) {
    if (!ws) ws = &op->ws;
    using C = C_t<T>;
    const OpDev<T> v = Sel<T>::view(op);
    C* W = reinterpret_cast<C*>(ws->W);
    launch_k1<T, IO>(v, x, Sel<T>::chi(op, which), W, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3<T, IO, IO>(v, W, x, y, skip, st);
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

template <typename T, typename IO>
die_status apply_reg_skip(dieop_s* op, const IO* x, IO* y, const int* skip, cudaStream_t st, const Workspace* ws) {
    if (!ws) ws = &op->ws;
    using C = C_t<T>;
    const OpDev<T> v = Sel<T>::view(op);
    C* W = reinterpret_cast<C*>(ws->W);
    C* vb = reinterpret_cast<C*>(ws->v);
    launch_k1<T, IO>(v, x, Sel<T>::chi(op, Contrast::Chi), W, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3k1<T, IO>(v, W, x, Sel<T>::chi(op, Contrast::ChiReg), vb, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3<T, C, IO>(v, W, vb, y, skip, st);
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

// Input and output of different element types (complex64 in, complex128 out: the
// products of the FP32-inner solves whose right preconditioner runs in complex64).
template <typename T, typename IX, typename IY>
die_status apply_op_skip_xy(dieop_s* op, Contrast which, const IX* x, IY* y, const int* skip, cudaStream_t st,
                            const Workspace* ws) {
    if (!ws) ws = &op->ws;
    using C = C_t<T>;
    const OpDev<T> v = Sel<T>::view(op);
    C* W = reinterpret_cast<C*>(ws->W);
    launch_k1<T, IX>(v, x, Sel<T>::chi(op, which), W, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3<T, IX, IY>(v, W, x, y, skip, st);
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

template <typename T, typename IX, typename IY>
die_status apply_reg_skip_xy(dieop_s* op, const IX* x, IY* y, const int* skip, cudaStream_t st,
                             const Workspace* ws) {
    if (!ws) ws = &op->ws;
    using C = C_t<T>;
    const OpDev<T> v = Sel<T>::view(op);
    C* W = reinterpret_cast<C*>(ws->W);
    C* vb = reinterpret_cast<C*>(ws->v);
    launch_k1<T, IX>(v, x, Sel<T>::chi(op, Contrast::Chi), W, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3k1<T, IX>(v, W, x, Sel<T>::chi(op, Contrast::ChiReg), vb, skip, st);
    launch_k2<T>(v, W, skip, st);
    launch_k3<T, C, IY>(v, W, vb, y, skip, st);
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

template <typename T, typename IO>
die_status apply_op(dieop_s* op, Contrast c, const IO* x, IO* y, cudaStream_t st, const Workspace* ws) {
    return apply_op_skip<T, IO>(op, c, x, y, nullptr, st, ws);
}
template <typename T, typename IO>
die_status apply_reg(dieop_s* op, const IO* x, IO* y, cudaStream_t st, const Workspace* ws) {
    return apply_reg_skip<T, IO>(op, x, y, nullptr, st, ws);
}

// nb products y_k = Atilde x_k (Atilde = A_R A when reg, else A) over consecutive field
// vectors, one launch per pass for all of them, with the caller's workspace (nb sets of
// row spectra and, when reg, nb middle vectors).
template <typename T, typename IO>
die_status apply_batch(dieop_s* op, bool reg, const IO* x, IO* y, int nb, void* Wws, void* vws, cudaStream_t st) {
    using C = C_t<T>;
    const OpDev<T> v = Sel<T>::view(op);
    C* W = reinterpret_cast<C*>(Wws);
    C* vb = reinterpret_cast<C*>(vws);
    launch_k1<T, IO>(v, x, Sel<T>::chi(op, Contrast::Chi), W, nullptr, st, nb);
    launch_k2<T>(v, W, nullptr, st, nb);
    if (reg) {
        launch_k3k1<T, IO>(v, W, x, Sel<T>::chi(op, Contrast::ChiReg), vb, nullptr, st, nb);
        launch_k2<T>(v, W, nullptr, st, nb);
        launch_k3<T, C, IO>(v, W, vb, y, nullptr, st, nb);
    } else {
        launch_k3<T, IO, IO>(v, W, x, y, nullptr, st, nb);
    }
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

}  // namespace die

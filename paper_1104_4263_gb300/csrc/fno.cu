// Fourier neural operator forward and backward passes (see include/die_fno.h) as chains
// of tcgen05 BF16 GEMMs (tc_gemm.cuh) and small FP32 elementwise kernels.
//
// Spectral convolution of one layer, for activations h[b][c][y][x] (B x C x H x W),
// m modes, MH = 2 m kept frequencies along y (k_h = 0 .. m-1 and H-m .. H-1, index
// khi), m along x (k_w), NM = MH m modes in all:
//   1  T1[bc][n][y]  = sum_x h[bc][y][x] Fw[n][x]        n = 2 k_w + ri (ri: re / im)
//   2  Z2[bc][k_w][n] = sum_{k=(ri,y)} T1[bc][2 k_w + ri][y] Gh[n][k]   n = 2 khi + ri'
//   3  Zmix[mode][b][ri c]  <- Z2 (the output indices of 2; mode = khi m + k_w)
//   4  Ymix[mode][b][n] = sum_k Zmix[mode][b][k] Rr[mode][n][k]   (the complex channel
//      mixing Y = X R as a real 2C x 2C matrix per mode)
//   5  Y2[bo][k_w][ri khi]  <- Ymix (the output indices of 4)
//   6  T3[bo][y][ri'][k_w] = sum_k Y2[bo][k_w][k] Ginv[2 y + ri'][k]
//   7  out[bo][y][x] += sum_{k=(ri',k_w)} T3[bo][y][k] Fwinv[x][k]
// with Fw, Gh the forward real DFT along x and complex DFT along y restricted to the kept
// modes, Ginv, Fwinv the inverse ones (Fwinv carries c(k_w) / (H W), c = 1 at k_w = 0 and
// 2 otherwise: the inverse real DFT of a half spectrum).  The backward pass runs the
// transposed GEMMs in reverse order; dR comes from dRr = dYmix^T Zmix per mode.
#include <math.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/die_fno.h"
#include "op.cuh"
#include "tc_gemm.cuh"

struct fno_s {
    fno_desc d{};
    int C = 0, H = 0, W = 0, m = 0, MH = 0, NM = 0, HW = 0, L = 0, hid = 0, cin = 0, cout = 0, maxB = 0;
    long np = 0;
    long oP = 0, op = 0, oW[8] = {}, ow[8] = {}, oR1[8] = {}, oR2[8] = {}, oQ1 = 0, oq1 = 0, oQ2 = 0, oq2 = 0;
    float *params = nullptr, *grads = nullptr, *am = nullptr, *av = nullptr;
    long adam_t = 0;
    float *Fw = nullptr, *Gh = nullptr, *Ginv = nullptr, *Fwinv = nullptr;
    float* Rr = nullptr;            // L x NM x (2C)^2
    float* dRr = nullptr;           // NM x (2C)^2
    float* x = nullptr;             // input copy   B x cin x HW
    float* h[9] = {};               // h_0 .. h_{L-1}: B x C x HW (h_L = a_{L-1})
    float* a[8] = {};               // pre-activations
    float *u = nullptr, *s = nullptr;   // B x hid x HW
    float *T1 = nullptr, *Z2 = nullptr, *Ymix = nullptr, *Y2 = nullptr, *T3 = nullptr;
    float* Zmix[8] = {};            // kept for dR
    float *g1 = nullptr, *g2 = nullptr, *g3 = nullptr;   // backward scratch B x max(C, hid) x HW
    float* part = nullptr;          // partial sums of weight and bias gradients
    long part_cap = 0;
    bool expanded = false;          // Rr holds the current parameters: set only by a pass that was
                                    // launched (not recorded) on the parameters, cleared by any error
    bool captured = false;          // a training step was captured: replays change the parameters
                                    // unseen, so Rr is formed on every pass from then on
    cudaStream_t side = nullptr;    // weight gradients of the backward pass
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    int spare = 0;                  // CTA slots the backward pass leaves to the side stream
    float* loss = nullptr;          // device scalar
    float* ytmp = nullptr;          // B x cout x HW (train step)
    float *pin = nullptr, *pout = nullptr;   // preconditioner staging (1 x cin / cout x HW)
    double* rs = nullptr;           // preconditioner: sum of |v|^2 (device)
    int* err = nullptr;
    float* hostbuf = nullptr;
    int lastB = 0;
};

namespace die {
namespace {

constexpr int kT = 256;
// Kernels of a pass are chained by programmatic dependent launches (common.cuh).
template <typename... KArgs, typename... Args>
die_status run(void (*k)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    DIE_CUDA_TRY(launch_pdl(k, grid, dim3(threads), smem, st, args...));
    return DIE_OK;
}
inline int blocks_for(long n) {
    long b = (n + kT - 1) / kT;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

// ------------------------------------------------------------------ elementwise kernels
// Block sum of one value per thread, valid in thread 0 (fixed order).
__device__ __forceinline__ float block_sum(float acc) {
    __shared__ float red[kT];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    return red[0];
}

// part[(b S + s) C + c] = sum of d[b][c][p] over part s of p (grid C x S x B).  A block of
// its own for every (channel, batch entry, part): one block per channel read its 1 MB by
// itself in 454 us at 16 x 128^2.
__global__ void chan_sum_kernel(const float* d, int C, int HW, int S, float* part) {
    pdl_wait();
    const int c = blockIdx.x, sp = blockIdx.y, b = blockIdx.z;
    const int n = (HW + S - 1) / S, p0 = sp * n, p1 = min(HW, p0 + n);
    const float* x = d + ((long)b * C + c) * HW;
    float acc = 0.f;
    if ((reinterpret_cast<uintptr_t>(x + p0) & 15) == 0 && ((p1 - p0) & 3) == 0) {
        const float4* v = reinterpret_cast<const float4*>(x + p0);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int p = threadIdx.x; p < (p1 - p0) / 4; p += blockDim.x) {
            const float4 q = v[p];
            a.x += q.x; a.y += q.y; a.z += q.z; a.w += q.w;
        }
        acc = (a.x + a.y) + (a.z + a.w);
    } else {
        for (int p = p0 + threadIdx.x; p < p1; p += blockDim.x) acc += x[p];
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) part[((long)b * S + sp) * C + c] = acc;
}

// g[e] += sum_b part[b][e], b in order
__global__ void batch_sum_kernel(const float* part, int B, long n, float* g) {
    pdl_wait();
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        float acc = 0.f;
#pragma unroll 8
        for (int b = 0; b < B; b++) acc += part[(long)b * n + e];
        g[e] += acc;
    }
}
// The same for many parts of few entries: a warp per 32 entries and eight slices of b.
__global__ void part_sum_kernel(const float* part, int B, int n, float* g) {
    __shared__ float red[8][32];
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (e < n)
        for (int b = w; b < B; b += 8) acc += part[(long)b * n + e];
    red[w][lane] = acc;
    __syncthreads();
    if (w == 0 && e < n) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < 8; q++) t += red[q][lane];
        g[e] += t;
    }
}

// Real 2C x 2C mixing matrix of every mode from the complex weights R1 / R2 (layout
// [i][o][kh][kw] (re, im)): Rr[mode][ri' C + o][ri C + i] such that
// Yre = sum_i Zre Rre - Zim Rim, Yim = sum_i Zre Rim + Zim Rre.
// A block turns [i][modes] of one o (consecutive in the weights) into [mode][i] (consecutive
// in Rr) through shared memory; element by element, one side of the copy touched a
// 32-byte sector per value.
constexpr int kModeTile = 32;
__global__ void expand_r_kernel(const float* R1, const float* R2, float* Rr, int C, int m, int MH) {
    extern __shared__ float2 tile[];                 // [C][kModeTile + 1]
    pdl_wait();
    const int o = blockIdx.x, q0 = blockIdx.y * kModeTile, half = blockIdx.z;
    const int mm = m * m, nq = min(kModeTile, mm - q0), C2 = 2 * C;
    const float* R = half ? R2 : R1;
    for (int e = threadIdx.x; e < C * kModeTile; e += blockDim.x) {
        const int i = e / kModeTile, q = e % kModeTile;
        const float* p = R + 2 * (((long)i * C + o) * mm + q0 + q);      // any 4-byte alignment
        if (q < nq) tile[i * (kModeTile + 1) + q] = make_float2(p[0], p[1]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nq * C2; e += blockDim.x) {
        const int q = e / C2, k = e % C2, i = k < C ? k : k - C;
        const float2 v = tile[i * (kModeTile + 1) + q];
        float* D = Rr + ((long)half * mm + q0 + q) * C2 * C2;
        D[(long)o * C2 + k] = k < C ? v.x : -v.y;
        D[(long)(C + o) * C2 + k] = k < C ? v.y : v.x;
    }
}

// dR1 / dR2 += fold of dRr (the adjoint of expand_r_kernel, by the same tiles).
__global__ void fold_r_kernel(const float* dRr, float* dR1, float* dR2, int C, int m, int MH) {
    extern __shared__ float2 tile[];
    pdl_wait();
    const int o = blockIdx.x, q0 = blockIdx.y * kModeTile, half = blockIdx.z;
    const int mm = m * m, nq = min(kModeTile, mm - q0), C2 = 2 * C;
    for (int e = threadIdx.x; e < nq * C; e += blockDim.x) {
        const int q = e / C, i = e % C;
        const float* D = dRr + ((long)half * mm + q0 + q) * C2 * C2;
        tile[i * (kModeTile + 1) + q] = make_float2(D[(long)o * C2 + i] + D[(long)(C + o) * C2 + C + i],
                                                    -D[(long)o * C2 + C + i] + D[(long)(C + o) * C2 + i]);
    }
    __syncthreads();
    float* G = half ? dR2 : dR1;
    for (int e = threadIdx.x; e < C * kModeTile; e += blockDim.x) {
        const int i = e / kModeTile, q = e % kModeTile;
        if (q < nq) {
            float* p = G + 2 * (((long)i * C + o) * mm + q0 + q);
            const float2 v = tile[i * (kModeTile + 1) + q];
            p[0] += v.x;
            p[1] += v.y;
        }
    }
}

// g = 2 (y - t) / n and part[block] = the block's sum of (y - t)^2; the last stage adds the
// parts in order: loss = sum / n.
constexpr int kMseBlocks = 256;
__global__ void mse_kernel(const float* y, const float* t, long n, float* g, float* part) {
    pdl_wait();
    float acc = 0.f;
    const float sc = 2.f / (float)n;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        acc += d * d;
        g[i] = sc * d;
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}
__global__ void mse_sum_kernel(const float* part, int np, long n, float* loss) {
    pdl_wait();
    const float s = block_sum((int)threadIdx.x < np ? part[threadIdx.x] : 0.f);
    if (threadIdx.x == 0) *loss = s / (float)n;
}

__global__ void adam_kernel(float* p, const float* g, float* m1, float* m2, long n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
    pdl_wait();
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float a = b1 * m1[i] + (1.f - b1) * gi;
        const float v = b2 * m2[i] + (1.f - b2) * gi * gi;
        m1[i] = a;
        m2[i] = v;
        p[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
    }
}

// --------------------------------------------------------------- preconditioner glue
// sum of |v|^2 over n complex128 entries into *out (one block, fixed order)
__global__ void sumsq_kernel(const double2* v, long n, double* out) {
    __shared__ double red[kT];
    double acc = 0;
    for (long i = threadIdx.x; i < n; i += blockDim.x) acc += v[i].x * v[i].x + v[i].y * v[i].y;
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// x[6][HW] = (Re chi, Im chi, Re v1 / s, Im v1 / s, Re v2 / s, Im v2 / s), s = rms(v)
__global__ void encode_kernel(const double2* chi, const double2* v, const double* ss, long N, float* x) {
    const double s2 = *ss / (2.0 * N);
    const double inv = s2 > 0 ? 1.0 / sqrt(s2) : 1.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const double2 c = chi[i], a = v[i], b = v[N + i];
        x[i] = (float)c.x;
        x[N + i] = (float)c.y;
        x[2 * N + i] = (float)(a.x * inv);
        x[3 * N + i] = (float)(a.y * inv);
        x[4 * N + i] = (float)(b.x * inv);
        x[5 * N + i] = (float)(b.y * inv);
    }
}

// t[4][N] = (u - b) / s, s = rms(b)
__global__ void target_kernel(const double2* b, const double2* u, const double* ss, long N, float* t) {
    const double s2 = *ss / (2.0 * N);
    const double inv = s2 > 0 ? 1.0 / sqrt(s2) : 1.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const double2 a = b[i], c = b[N + i], ua = u[i], uc = u[N + i];
        t[i] = (float)((ua.x - a.x) * inv);
        t[N + i] = (float)((ua.y - a.y) * inv);
        t[2 * N + i] = (float)((uc.x - c.x) * inv);
        t[3 * N + i] = (float)((uc.y - c.y) * inv);
    }
}

// z = v + s d, d = (y0 + i y1, y2 + i y3)
__global__ void decode_kernel(const double2* v, const float* y, const double* ss, long N, double2* z) {
    const double s2 = *ss / (2.0 * N);
    const double s = s2 > 0 ? sqrt(s2) : 0.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const double2 a = v[i], b = v[N + i];
        z[i] = make_double2(a.x + s * y[i], a.y + s * y[N + i]);
        z[N + i] = make_double2(b.x + s * y[2 * N + i], b.y + s * y[3 * N + i]);
    }
}

// ------------------------------------------------------------------ GEMM shorthand
struct Mat {
    const float* p;
    long s0, s1, sb;     // strides of the first index (m or n), of k, of the batch
};

GemmArgs gemm_args(fno_s* f, int M, int N, int K, int batch, Mat A, Mat B, float* C, long scm, long scn, long scb) {
    GemmArgs g;
    g.M = M; g.N = N; g.K = K; g.batch = batch;
    g.A = A.p; g.sam = A.s0; g.sak = A.s1; g.sab = A.sb;
    g.B = B.p; g.sbn = B.s0; g.sbk = B.s1; g.sbb = B.sb;
    g.C = C; g.scm = scm; g.scn = scn; g.scb = scb;
    g.err = f->err;
    g.spare = f->spare;
    return g;
}
die_status gemm(fno_s* f, int M, int N, int K, int batch, Mat A, Mat B, float* C, long scm, long scn, long scb,
                const float* bias, cudaStream_t st) {
    GemmArgs g = gemm_args(f, M, N, K, batch, A, B, C, scm, scn, scb);
    g.bias = bias;
    return tc_gemm(g, st);
}

// grad (M x N) += sum over the batch of A B^T over the H W grid points, one accumulator per
// batch entry.  B tiles of K = H W keep only B CTAs busy, so these run on the side stream
// beside the rest of the backward pass.
die_status gemm_grad(fno_s* f, int M, int N, int B, Mat A, Mat Bm, float* grad) {
    GemmArgs g = gemm_args(f, M, N, f->HW, B, A, Bm, f->part, N, 1, (long)M * N);
    if (M > 32 && N <= 32) {               // the short operand as A (see depth in tc_gemm.cu)
        g = gemm_args(f, N, M, f->HW, B, Bm, A, f->part, 1, N, (long)M * N);
    }
    DIE_TRY(tc_gemm(g, f->side));
    return run(batch_sum_kernel, dim3(blocks_for((long)M * N)), kT, 0, f->side, (const float*)f->part, B, (long)M * N,
               grad);
}
// grad (C) += sums over the batch and the grid of d, on the side stream
die_status chan_sum(fno_s* f, const float* d, int B, int C, float* grad) {
    int S = (608 + B * C - 1) / (B * C);
    if (S > 16) S = 16;
    DIE_TRY(run(chan_sum_kernel, dim3(C, S, B), kT, 0, f->side, d, C, f->HW, S, f->part));
    return run(part_sum_kernel, dim3((C + 31) / 32), kT, 0, f->side, (const float*)f->part, B * S, C, grad);
}
// The side stream waits for what `st` holds so far / the other way round.
die_status fork_side(fno_s* f, cudaStream_t st) {
    DIE_CUDA_TRY(cudaEventRecord(f->ev_fork, st));
    DIE_CUDA_TRY(cudaStreamWaitEvent(f->side, f->ev_fork, 0));
    return DIE_OK;
}
die_status join_side(fno_s* f, cudaStream_t st) {
    DIE_CUDA_TRY(cudaEventRecord(f->ev_join, f->side));
    DIE_CUDA_TRY(cudaStreamWaitEvent(st, f->ev_join, 0));
    return DIE_OK;
}

// ------------------------------------------------------------------ network passes
// a = W h + w (pointwise) + K h (spectral) for layer l, and GELU(a) in hnext (or NULL);
// Zmix[l] kept.
die_status layer_forward(fno_s* f, int l, int B, const float* hin, float* a, float* hnext, cudaStream_t st) {
    const int C = f->C, H = f->H, W = f->W, m = f->m, MH = f->MH, HW = f->HW, C2 = 2 * C;
    const long CHW = (long)C * HW, BC2 = (long)B * C2;
    float* prm = f->params;
    // pointwise
    DIE_TRY(gemm(f, HW, C, C, B, {hin, 1, HW, CHW}, {prm + f->oW[l], C, 1, 0}, a, 1, HW, CHW, prm + f->ow[l], st));
    // 1: along x
    DIE_TRY(gemm(f, H, 2 * m, W, B * C, {hin, W, 1, HW}, {f->Fw, W, 1, 0}, f->T1, 1, H, 2L * m * H, nullptr, st));
    // 2 and 3: along y, written mode by mode: (b, row c m + kw, column 2 khi + ri) goes to
    // ((khi m + kw) B + b) 2C + ri C + c
    GemmArgs g = gemm_args(f, C * m, 2 * MH, 2 * H, B, {f->T1, 2L * H, 1, 2L * C * m * H}, {f->Gh, 2L * H, 1, 0},
                           f->Zmix[l], BC2, C, C2);
    g.mi = m; g.scm2 = 1;
    g.ni = 2; g.scn2 = m * BC2;
    DIE_TRY(tc_gemm(g, st));
    // 4 and 5: channel mixing per mode, written row by row: (mode = khi m + kw, b, column
    // ri C + o) goes to ((b C + o) m + kw) 2MH + ri MH + khi
    g = gemm_args(f, B, C2, C2, f->NM, {f->Zmix[l], C2, 1, BC2}, {f->Rr + (long)l * f->NM * C2 * C2, C2, 1,
                  (long)C2 * C2}, f->Y2, 2L * C * m * MH, 2L * m * MH, 2L * MH);
    g.ni = C; g.scn2 = MH;
    g.bi = m; g.scb2 = 1;
    DIE_TRY(tc_gemm(g, st));
    // 6: inverse along y
    DIE_TRY(gemm(f, m, 2 * H, 2 * MH, B * C, {f->Y2, 2L * MH, 1, 2L * m * MH}, {f->Ginv, 2L * MH, 1, 0}, f->T3, 1, m,
                 2L * H * m, nullptr, st));
    // 7: inverse along x, added to the pointwise part
    g = gemm_args(f, H, W, 2 * m, B * C, {f->T3, 2L * m, 1, 2L * H * m}, {f->Fwinv, 2L * m, 1, 0}, a, W, 1, HW);
    g.beta = 1.f;
    g.gelu = hnext;
    return tc_gemm(g, st);
}

// Backward of layer l given da (B x C x HW): grads of W_l, w_l, R1_l, R2_l accumulated, and
// dh (B x C x HW) written, with the gradient of layer l - 1's pre-activation, dh GELU'(aprev),
// in its place when aprev is given.  dh may equal neither da nor scratch of this pass.
die_status layer_backward(fno_s* f, int l, int B, const float* hin, const float* da, float* dh, const float* aprev,
                          cudaStream_t st) {
    const int C = f->C, H = f->H, W = f->W, m = f->m, MH = f->MH, HW = f->HW, C2 = 2 * C;
    const long CHW = (long)C * HW, BC2 = (long)B * C2;
    float* prm = f->params;
    float* grd = f->grads;
    // the buffer of dh was da of the layer above, read by the side stream until here
    DIE_TRY(join_side(f, st));
    // dW = sum_b da h^T, dw = channel sums
    DIE_TRY(fork_side(f, st));
    DIE_TRY(gemm_grad(f, C, C, B, {da, HW, 1, CHW}, {hin, HW, 1, CHW}, grd + f->oW[l]));
    DIE_TRY(chan_sum(f, da, B, C, grd + f->ow[l]));
    // dh = W^T da
    DIE_TRY(gemm(f, HW, C, C, B, {da, 1, HW, CHW}, {prm + f->oW[l], 1, C, 0}, dh, 1, HW, CHW, nullptr, st));
    // spectral, 7^T: dT3 = da Fwinv
    DIE_TRY(gemm(f, H, 2 * m, W, B * C, {da, W, 1, HW}, {f->Fwinv, 1, 2L * m, 0}, f->T3, 2L * m, 1, 2L * H * m,
                 nullptr, st));
    // 6^T and 5^T: dY2 = dT3 Ginv, written mode by mode (as 2 and 3 of the forward pass, with
    // column ri MH + khi)
    GemmArgs g = gemm_args(f, m, 2 * MH, 2 * H, B * C, {f->T3, 1, m, 2L * H * m}, {f->Ginv, 1, 2L * MH, 0}, f->Ymix,
                           BC2, BC2 * m, 1);
    g.ni = MH; g.scn2 = C;
    g.bi = C; g.scb2 = C2;
    DIE_TRY(tc_gemm(g, st));
    // 4^T: dRr = dYmix^T Zmix, dZmix = dYmix Rr, the latter written row by row: (mode, b, column
    // ri C + c) goes to ((b C + c) m + kw) 2MH + 2 khi + ri
    DIE_TRY(gemm(f, C2, C2, B, f->NM, {f->Ymix, 1, C2, BC2}, {f->Zmix[l], 1, C2, BC2}, f->dRr, C2, 1, (long)C2 * C2,
                 nullptr, st));
    DIE_TRY(run(fold_r_kernel, dim3(C, (m * m + kModeTile - 1) / kModeTile, 2), kT,
                (size_t)C * (kModeTile + 1) * sizeof(float2), st, (const float*)f->dRr, grd + f->oR1[l],
                grd + f->oR2[l], C, m, MH));
    g = gemm_args(f, B, C2, C2, f->NM, {f->Ymix, C2, 1, BC2}, {f->Rr + (long)l * f->NM * C2 * C2, 1, C2, (long)C2 * C2},
                  f->Z2, 2L * C * m * MH, 2L * m * MH, 2L * MH);
    g.ni = C; g.scn2 = 1;
    g.bi = m; g.scb2 = 2;
    DIE_TRY(tc_gemm(g, st));
    // 2^T: dT1 = dZ2 Gh
    DIE_TRY(gemm(f, m, 2 * H, 2 * MH, B * C, {f->Z2, 2L * MH, 1, 2L * m * MH}, {f->Gh, 1, 2L * H, 0}, f->T1, 2L * H, 1,
                 2L * m * H, nullptr, st));
    // 1^T: dh += dT1 Fw
    g = gemm_args(f, H, W, 2 * m, B * C, {f->T1, 1, H, 2L * m * H}, {f->Fw, 1, W, 0}, dh, W, 1, HW);
    g.beta = 1.f;
    g.dgelu = aprev;
    return tc_gemm(g, st);
}

die_status is_capturing(cudaStream_t st, bool* cap) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    DIE_CUDA_TRY(cudaStreamIsCapturing(st, &s));
    *cap = s != cudaStreamCaptureStatusNone;
    return DIE_OK;
}

// Rr from the parameters, once per change of them.  On a capturing stream the work is only
// recorded: it is always part of the recording, and says nothing about Rr's contents.
die_status expand_weights(fno_s* f, cudaStream_t st) {
    bool cap = false;
    DIE_TRY(is_capturing(st, &cap));
    if (f->expanded && !f->captured && !cap) return DIE_OK;
    f->expanded = false;
    const long per = (long)f->NM * 4 * f->C * f->C;
    for (int l = 0; l < f->L; l++)
        DIE_TRY(run(expand_r_kernel, dim3(f->C, (f->m * f->m + kModeTile - 1) / kModeTile, 2), kT,
                    (size_t)f->C * (kModeTile + 1) * sizeof(float2), st, (const float*)f->params + f->oR1[l],
                    (const float*)f->params + f->oR2[l], f->Rr + (long)l * per, f->C, f->m, f->MH));
    f->expanded = !cap;
    return DIE_OK;
}

die_status forward_passes(fno_s* f, int B, const float* x, float* y, cudaStream_t st) {
    const int C = f->C, HW = f->HW;
    const long CHW = (long)C * HW, HHW = (long)f->hid * HW;
    float* prm = f->params;
    DIE_TRY(expand_weights(f, st));
    DIE_CUDA_TRY(cudaMemcpyAsync(f->x, x, (size_t)B * f->cin * HW * sizeof(float), cudaMemcpyDeviceToDevice, st));
    // lifting
    DIE_TRY(gemm(f, HW, C, f->cin, B, {f->x, 1, HW, (long)f->cin * HW}, {prm + f->oP, f->cin, 1, 0}, f->h[0], 1, HW,
                 CHW, prm + f->op, st));
    for (int l = 0; l < f->L; l++)
        DIE_TRY(layer_forward(f, l, B, f->h[l], f->a[l], l < f->L - 1 ? f->h[l + 1] : nullptr, st));
    const float* hL = f->a[f->L - 1];
    GemmArgs g = gemm_args(f, HW, f->hid, C, B, {hL, 1, HW, CHW}, {prm + f->oQ1, C, 1, 0}, f->u, 1, HW, HHW);
    g.bias = prm + f->oq1;
    g.gelu = f->s;
    DIE_TRY(tc_gemm(g, st));
    DIE_TRY(gemm(f, HW, f->cout, f->hid, B, {f->s, 1, HW, HHW}, {prm + f->oQ2, f->hid, 1, 0}, y, 1, HW,
                 (long)f->cout * HW, prm + f->oq2, st));
    f->lastB = B;
    return DIE_OK;
}

die_status forward(fno_s* f, int B, const float* x, float* y, cudaStream_t st) {
    const die_status s = forward_passes(f, B, x, y, st);
    if (s != DIE_OK) f->expanded = false;
    return s;
}

die_status backward_passes(fno_s* f, int B, const float* gy, float* gx, cudaStream_t st) {
    const int C = f->C, HW = f->HW, hid = f->hid;
    const long CHW = (long)C * HW, HHW = (long)hid * HW;
    float* prm = f->params;
    float* grd = f->grads;
    // projection: dQ2, dq2, du = (Q2^T gy) GELU'(u)
    DIE_TRY(fork_side(f, st));
    DIE_TRY(gemm_grad(f, f->cout, hid, B, {gy, HW, 1, (long)f->cout * HW}, {f->s, HW, 1, HHW}, grd + f->oQ2));
    DIE_TRY(chan_sum(f, gy, B, f->cout, grd + f->oq2));
    GemmArgs g = gemm_args(f, HW, hid, f->cout, B, {gy, 1, HW, (long)f->cout * HW}, {prm + f->oQ2, 1, hid, 0}, f->g3, 1,
                           HW, HHW);
    g.dgelu = f->u;
    DIE_TRY(tc_gemm(g, st));
    const float* hL = f->a[f->L - 1];
    DIE_TRY(fork_side(f, st));
    DIE_TRY(gemm_grad(f, hid, C, B, {f->g3, HW, 1, HHW}, {hL, HW, 1, CHW}, grd + f->oQ1));
    DIE_TRY(chan_sum(f, f->g3, B, hid, grd + f->oq1));
    // da of the last layer; then each layer writes the next one's
    float *da = f->g1, *dh = f->g2;
    DIE_TRY(gemm(f, HW, C, hid, B, {f->g3, 1, HW, HHW}, {prm + f->oQ1, 1, C, 0}, da, 1, HW, CHW, nullptr, st));
    for (int l = f->L - 1; l >= 0; l--) {
        DIE_TRY(layer_backward(f, l, B, f->h[l], da, dh, l > 0 ? f->a[l - 1] : nullptr, st));
        float* t = da;
        da = dh;
        dh = t;
    }
    // lifting (da is the gradient of h_0)
    DIE_TRY(fork_side(f, st));
    DIE_TRY(gemm_grad(f, C, f->cin, B, {da, HW, 1, CHW}, {f->x, HW, 1, (long)f->cin * HW}, grd + f->oP));
    DIE_TRY(chan_sum(f, da, B, C, grd + f->op));
    if (gx)
        DIE_TRY(gemm(f, HW, f->cin, C, B, {da, 1, HW, CHW}, {prm + f->oP, 1, f->cin, 0}, gx, 1, HW, (long)f->cin * HW,
                     nullptr, st));
    return DIE_OK;
}

die_status backward(fno_s* f, int B, const float* gy, float* gx, cudaStream_t st) {
    f->spare = B < 64 ? B : 64;
    const die_status s = backward_passes(f, B, gy, gx, st);
    f->spare = 0;
    const die_status j = join_side(f, st);      // at every exit
    return s != DIE_OK ? s : j;
}

// Constant DFT matrices (FP64 on the host, stored FP32).
die_status make_dft(fno_s* f) {
    const int H = f->H, W = f->W, m = f->m, MH = f->MH;
    const double tp = 2.0 * M_PI;
    std::vector<float> Fw((size_t)2 * m * W), Gh((size_t)2 * MH * 2 * H), Gi((size_t)2 * H * 2 * MH),
        Fi((size_t)W * 2 * m);
    for (int kw = 0; kw < m; kw++)
        for (int x = 0; x < W; x++) {
            const double ph = tp * (double)((long)kw * x % W) / W;
            Fw[(size_t)(2 * kw) * W + x] = (float)cos(ph);
            Fw[(size_t)(2 * kw + 1) * W + x] = (float)-sin(ph);
            const double c = (kw == 0 ? 1.0 : 2.0) / ((double)H * W);
            Fi[(size_t)x * 2 * m + kw] = (float)(c * cos(ph));
            Fi[(size_t)x * 2 * m + m + kw] = (float)(-c * sin(ph));
        }
    for (int khi = 0; khi < MH; khi++) {
        const int kh = khi < m ? khi : H - MH + khi;
        for (int y = 0; y < H; y++) {
            const double th = tp * (double)((long)kh * y % H) / H;
            const float c = (float)cos(th), s = (float)sin(th);
            // forward: Zre = sum cos Tre + sin Tim, Zim = sum cos Tim - sin Tre
            Gh[(size_t)(2 * khi) * 2 * H + y] = c;
            Gh[(size_t)(2 * khi) * 2 * H + H + y] = s;
            Gh[(size_t)(2 * khi + 1) * 2 * H + y] = -s;
            Gh[(size_t)(2 * khi + 1) * 2 * H + H + y] = c;
            // inverse: T3re = sum cos Yre - sin Yim, T3im = sum sin Yre + cos Yim
            Gi[(size_t)(2 * y) * 2 * MH + khi] = c;
            Gi[(size_t)(2 * y) * 2 * MH + MH + khi] = -s;
            Gi[(size_t)(2 * y + 1) * 2 * MH + khi] = s;
            Gi[(size_t)(2 * y + 1) * 2 * MH + MH + khi] = c;
        }
    }
    DIE_CUDA_TRY(cudaMemcpy(f->Fw, Fw.data(), Fw.size() * sizeof(float), cudaMemcpyHostToDevice));
    DIE_CUDA_TRY(cudaMemcpy(f->Gh, Gh.data(), Gh.size() * sizeof(float), cudaMemcpyHostToDevice));
    DIE_CUDA_TRY(cudaMemcpy(f->Ginv, Gi.data(), Gi.size() * sizeof(float), cudaMemcpyHostToDevice));
    DIE_CUDA_TRY(cudaMemcpy(f->Fwinv, Fi.data(), Fi.size() * sizeof(float), cudaMemcpyHostToDevice));
    return DIE_OK;
}

void free_fno(fno_s* f) {
    if (!f) return;
    std::vector<void*> ptrs = {f->params, f->grads, f->am, f->av, f->Fw, f->Gh, f->Ginv, f->Fwinv, f->Rr, f->dRr,
                               f->x, f->u, f->s, f->T1, f->Z2, f->Ymix, f->Y2, f->T3, f->g1, f->g2, f->g3, f->part,
                               f->loss, f->ytmp, f->pin, f->pout, f->rs, f->err};
    for (int l = 0; l < 9; l++) ptrs.push_back(f->h[l]);
    for (int l = 0; l < 8; l++) { ptrs.push_back(f->a[l]); ptrs.push_back(f->Zmix[l]); }
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (f->hostbuf) cudaFreeHost(f->hostbuf);
    if (f->side) cudaStreamDestroy(f->side);
    if (f->ev_fork) cudaEventDestroy(f->ev_fork);
    if (f->ev_join) cudaEventDestroy(f->ev_join);
    delete f;
}

die_status create_impl(const fno_desc* d, fno_s* f) {
    f->d = *d;
    f->C = d->width; f->H = d->H; f->W = d->W; f->m = d->modes; f->MH = 2 * d->modes; f->L = d->layers;
    f->hid = d->hidden; f->cin = d->c_in; f->cout = d->c_out; f->maxB = d->max_batch;
    f->HW = f->H * f->W;
    f->NM = f->MH * f->m;
    const int C = f->C, m = f->m;
    long o = 0;
    f->oP = o; o += (long)C * f->cin;
    f->op = o; o += C;
    for (int l = 0; l < f->L; l++) {
        f->oW[l] = o; o += (long)C * C;
        f->ow[l] = o; o += C;
        f->oR1[l] = o; o += 2L * C * C * m * m;
        f->oR2[l] = o; o += 2L * C * C * m * m;
    }
    f->oQ1 = o; o += (long)f->hid * C;
    f->oq1 = o; o += f->hid;
    f->oQ2 = o; o += (long)f->cout * f->hid;
    f->oq2 = o; o += f->cout;
    f->np = o;
    const long B = f->maxB, HW = f->HW, C2 = 2 * C;
    const long wide = (C > f->hid ? C : f->hid);
    // partial sums of one weight gradient (per batch entry) or of channel sums (16 parts each)
    const long widest = wide * (C > f->cin ? (C > f->cout ? C : f->cout) : (f->cin > f->cout ? f->cin : f->cout));
    const long chans = 16 * (wide > f->cout ? wide : f->cout);
    f->part_cap = B * (widest > chans ? widest : chans);
    auto al = [](float** p, long n) { return cudaMalloc((void**)p, (size_t)(n > 0 ? n : 1) * sizeof(float)) == cudaSuccess; };
    bool ok = al(&f->params, f->np) && al(&f->grads, f->np) && al(&f->am, f->np) && al(&f->av, f->np) &&
              al(&f->Fw, 2L * m * f->W) && al(&f->Gh, 2L * f->MH * 2 * f->H) && al(&f->Ginv, 2L * f->H * 2 * f->MH) &&
              al(&f->Fwinv, (long)f->W * 2 * m) && al(&f->Rr, (long)f->L * f->NM * C2 * C2) &&
              al(&f->dRr, (long)f->NM * C2 * C2) && al(&f->x, B * f->cin * HW) && al(&f->u, B * f->hid * HW) &&
              al(&f->s, B * f->hid * HW) && al(&f->T1, B * C * 2 * m * f->H) && al(&f->Z2, B * C * m * 2 * f->MH) &&
              al(&f->Ymix, (long)f->NM * B * C2) && al(&f->Y2, B * C * m * 2 * f->MH) &&
              al(&f->T3, B * C * f->H * 2 * m) && al(&f->g1, B * wide * HW) && al(&f->g2, B * wide * HW) &&
              al(&f->g3, B * wide * HW) &&
              al(&f->part, f->part_cap) &&
              al(&f->loss, 1 + kMseBlocks) && al(&f->ytmp, B * f->cout * HW) && al(&f->pin, (long)f->cin * HW) &&
              al(&f->pout, (long)f->cout * HW);
    for (int l = 0; ok && l < f->L; l++)
        ok = al(&f->h[l], B * C * HW) && al(&f->a[l], B * C * HW) && al(&f->Zmix[l], (long)f->NM * B * C2);
    ok = ok && cudaMalloc((void**)&f->rs, sizeof(double)) == cudaSuccess &&
         cudaMalloc((void**)&f->err, sizeof(int)) == cudaSuccess &&
         cudaHostAlloc((void**)&f->hostbuf, 16 * sizeof(float), cudaHostAllocDefault) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        return DIE_ENOMEM;
    }
    DIE_CUDA_TRY(cudaStreamCreateWithFlags(&f->side, cudaStreamNonBlocking));
    DIE_CUDA_TRY(cudaEventCreateWithFlags(&f->ev_fork, cudaEventDisableTiming));
    DIE_CUDA_TRY(cudaEventCreateWithFlags(&f->ev_join, cudaEventDisableTiming));
    DIE_CUDA_TRY(cudaMemset(f->params, 0, f->np * sizeof(float)));
    DIE_CUDA_TRY(cudaMemset(f->grads, 0, f->np * sizeof(float)));
    DIE_CUDA_TRY(cudaMemset(f->am, 0, f->np * sizeof(float)));
    DIE_CUDA_TRY(cudaMemset(f->av, 0, f->np * sizeof(float)));
    DIE_CUDA_TRY(cudaMemset(f->err, 0, sizeof(int)));
    return make_dft(f);
}

// Reads (and clears) the flag a GEMM sets when one of its bounded waits gave up.  A capturing
// stream refuses the synchronisation; that error is this call's, not one for the next call's
// launch check.
die_status check_err(fno_s* f, cudaStream_t st) {
    int e = 0;
    cudaError_t r = cudaMemcpyAsync(&e, f->err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (r == cudaSuccess) r = cudaStreamSynchronize(st);
    if (r == cudaSuccess && !e) return DIE_OK;
    f->expanded = false;
    if (r != cudaSuccess) {
        cudaGetLastError();
        set_last_cuda_error(r, "network pass", __FILE__, __LINE__);
        return DIE_ECUDA;
    }
    DIE_CUDA_TRY(cudaMemsetAsync(f->err, 0, sizeof(int), st));
    return DIE_ETIMEOUT;
}

}  // namespace
}  // namespace die

using namespace die;

extern "C" die_status die_gemm_bf16(int M, int N, int K, int batch, float alpha, const float* A, long long sam,
                                    long long sak, long long sab, const float* B, long long sbn, long long sbk,
                                    long long sbb, float beta, float* C, long long scm, long long scn, long long scb,
                                    int check, void* stream) {
    GemmArgs g;
    g.M = M; g.N = N; g.K = K; g.batch = batch; g.alpha = alpha; g.beta = beta;
    g.A = A; g.sam = sam; g.sak = sak; g.sab = sab;
    g.B = B; g.sbn = sbn; g.sbk = sbk; g.sbb = sbb;
    g.C = C; g.scm = scm; g.scn = scn; g.scb = scb;
    cudaStream_t st = (cudaStream_t)stream;
    int* err = nullptr;
    if (check) {
        if (cudaMalloc((void**)&err, sizeof(int)) != cudaSuccess) { cudaGetLastError(); return DIE_ENOMEM; }
        if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) { cudaFree(err); return DIE_ECUDA; }
        g.err = err;
    }
    die_status s = tc_gemm(g, st);
    if (s == DIE_OK && check) {
        int e = 0;
        if (cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            s = DIE_ECUDA;
        else if (e)
            s = DIE_ETIMEOUT;
    }
    if (err) cudaFree(err);
    return s;
}

extern "C" die_status fno_create(const fno_desc* d, fno_t* out) {
    if (!d || !out) return DIE_EINVAL;
    *out = nullptr;
    if (d->c_in < 1 || d->c_in > 64 || d->c_out < 1 || d->c_out > 64 || d->width < 1 || d->width > 64 ||
        d->layers < 1 || d->layers > 8 || d->hidden < 1 || d->hidden > 256 || d->H < 2 || d->H > 512 || d->W < 2 ||
        d->W > 512 || d->modes < 1 || 2 * d->modes > d->H || 2 * d->modes > d->W || d->max_batch < 1 ||
        d->max_batch > 256)
        return DIE_EINVAL;
    fno_s* f = new (std::nothrow) fno_s();
    if (!f) return DIE_ENOMEM;
    die_status s;
    try {
        s = create_impl(d, f);
    } catch (...) {
        s = DIE_ENOMEM;
    }
    if (s != DIE_OK) {
        free_fno(f);
        return s;
    }
    *out = f;
    return DIE_OK;
}

extern "C" void fno_destroy(fno_t f) { free_fno(f); }

extern "C" long long fno_param_count(fno_t f) { return f ? f->np : -1; }

extern "C" die_status fno_set_params(fno_t f, const float* host) {
    if (!f || !host) return DIE_EINVAL;
    f->expanded = false;
    DIE_CUDA_TRY(cudaMemcpy(f->params, host, f->np * sizeof(float), cudaMemcpyHostToDevice));
    DIE_CUDA_TRY(cudaMemset(f->am, 0, f->np * sizeof(float)));
    DIE_CUDA_TRY(cudaMemset(f->av, 0, f->np * sizeof(float)));
    f->adam_t = 0;
    return DIE_OK;
}

extern "C" die_status fno_get_params(fno_t f, float* host) {
    if (!f || !host) return DIE_EINVAL;
    DIE_CUDA_TRY(cudaMemcpy(host, f->params, f->np * sizeof(float), cudaMemcpyDeviceToHost));
    return DIE_OK;
}

extern "C" die_status fno_get_grads(fno_t f, float* host) {
    if (!f || !host) return DIE_EINVAL;
    DIE_CUDA_TRY(cudaDeviceSynchronize());
    DIE_CUDA_TRY(cudaMemcpy(host, f->grads, f->np * sizeof(float), cudaMemcpyDeviceToHost));
    return DIE_OK;
}

extern "C" die_status fno_zero_grads(fno_t f, void* stream) {
    if (!f) return DIE_EINVAL;
    DIE_CUDA_TRY(cudaMemsetAsync(f->grads, 0, f->np * sizeof(float), (cudaStream_t)stream));
    return DIE_OK;
}

extern "C" die_status fno_forward(fno_t f, int B, const float* x, float* y, void* stream) {
    if (!f || !x || !y || B < 1 || B > f->maxB) return DIE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    DIE_TRY(forward(f, B, x, y, st));
    return check_err(f, st);
}

extern "C" die_status fno_backward(fno_t f, int B, const float* gy, float* gx, void* stream) {
    if (!f || !gy || B < 1 || B != f->lastB) return DIE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    DIE_TRY(backward(f, B, gy, gx, st));
    return check_err(f, st);
}

extern "C" die_status fno_train_step(fno_t f, int B, const float* x, const float* t, float lr, float* loss,
                                     void* stream) {
    if (!f || !x || !t || B < 1 || B > f->maxB || !(lr >= 0)) return DIE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    bool cap = false;
    DIE_TRY(is_capturing(st, &cap));
    if (cap) f->captured = true;
    const long n = (long)B * f->cout * f->HW;
    DIE_TRY(forward(f, B, x, f->ytmp, st));
    // gradient in place of y
    DIE_TRY(run(mse_kernel, dim3(kMseBlocks), kT, 0, st, (const float*)f->ytmp, t, n, f->ytmp, f->loss + 1));
    DIE_TRY(run(mse_sum_kernel, dim3(1), kT, 0, st, (const float*)f->loss + 1, kMseBlocks, n, f->loss));
    DIE_CUDA_TRY(cudaMemsetAsync(f->grads, 0, f->np * sizeof(float), st));
    DIE_TRY(backward(f, B, f->ytmp, nullptr, st));
    f->adam_t++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)f->adam_t), c2 = 1.f - powf(b2, (float)f->adam_t);
    DIE_TRY(run(adam_kernel, dim3(blocks_for(f->np)), kT, 0, st, f->params, (const float*)f->grads, f->am, f->av, f->np,
                lr, b1, b2, 1e-8f, c1, c2));
    f->expanded = false;
    if (loss) {
        DIE_CUDA_TRY(cudaMemcpyAsync(f->hostbuf, f->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        DIE_TRY(check_err(f, st));
        *loss = f->hostbuf[0];
    }
    return DIE_OK;
}

namespace die {
// z = M(v) = v + s * network(encode(chi, v)) for one field of operator op.
die_status fno_apply_precond(fno_s* f, dieop_s* op, const double2* v, double2* z, cudaStream_t st) {
    const long N = op->N;
    sumsq_kernel<<<1, kT, 0, st>>>(v, 2 * N, f->rs);
    DIE_LAUNCH_CHECK();
    encode_kernel<<<blocks_for(N), kT, 0, st>>>(op->chi_d, v, f->rs, N, f->pin);
    DIE_LAUNCH_CHECK();
    DIE_TRY(forward(f, 1, f->pin, f->pout, st));
    decode_kernel<<<blocks_for(N), kT, 0, st>>>(v, f->pout, f->rs, N, z);
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

bool fno_matches(const fno_s* f, const dieop_s* op) {
    return op->planes == 2 && f->cin == 6 && f->cout == 4 && f->H == op->n2 && f->W == op->n1;
}
}  // namespace die

extern "C" die_status fno_precondition(fno_t f, dieop_t op, const void* v, void* z, void* stream) {
    if (!f || !op || !v || !z || !fno_matches(f, op)) return DIE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    DIE_TRY(fno_apply_precond(f, op, (const double2*)v, (double2*)z, st));
    return check_err(f, st);
}

extern "C" die_status fno_encode_pair(dieop_t op, const void* b, const void* u, float* x, float* t, void* stream) {
    if (!op || !b || !x || (t && !u) || op->planes != 2) return DIE_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const long N = op->N;
    double* ss = nullptr;
    if (cudaMalloc((void**)&ss, sizeof(double)) != cudaSuccess) { cudaGetLastError(); return DIE_ENOMEM; }
    sumsq_kernel<<<1, kT, 0, st>>>((const double2*)b, 2 * N, ss);
    encode_kernel<<<blocks_for(N), kT, 0, st>>>(op->chi_d, (const double2*)b, ss, N, x);
    if (t) target_kernel<<<blocks_for(N), kT, 0, st>>>((const double2*)b, (const double2*)u, ss, N, t);
    const cudaError_t e = cudaGetLastError();
    cudaFree(ss);                 // waits for the kernels
    if (e != cudaSuccess) {
        set_last_cuda_error(e, "fno_encode_pair", __FILE__, __LINE__);
        return DIE_ECUDA;
    }
    return DIE_OK;
}

// tcgen05 BF16 GEMM (see tc_gemm.cuh).
#include <cuda_bf16.h>

#include "tc_gemm.cuh"

namespace die {

namespace {

constexpr int kBM = 128, kBK = 64, kThreads = 256;
constexpr int tile_bytes(int rows) { return rows * kBK * 2; }
constexpr long kWaitLimit = 1L << 26;    // mbarrier polls before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of tcgen05 (no swizzle): start address, leading-
// dimension byte offset (core matrices adjacent in K), stride byte offset (8-row groups
// adjacent in M or N), all in 16-byte units; bits 46-47 hold the descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | (1ull << 46);
}

// Instruction descriptor of tcgen05.mma.kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9 and 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22,
// M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait for the phase `parity` of the barrier to complete; false if it gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (long i = 0; i < kWaitLimit; i++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// 8 consecutive accumulator columns of this thread's TMEM lane (32x32b shape).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

// How an operand is read: k of unit stride, the row index of unit stride (both with
// 16-byte aligned vectors), or any strides.
enum Layout { kAlongK = 0, kAlongR = 1, kAny = 2 };

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// The rows [r0, r0 + R) x k [k0, k0 + 64) of X(r, k) = X[r sr + k sk], zeros outside
// [0, rows) x [0, kend), on their way from global memory (load) to the canonical layout
// (store, tile of TR >= R rows): element (r, k) at byte (k / 8) (TR 16) + (r / 8) 128 +
// (r % 8) 16 + (k % 8) 2.
// kc (a multiple of 16): the columns that are multiplied.
template <int R, int LAY> struct Stage;

// A task is 8 consecutive k of one row.  Eight lanes take eight rows (one 128-byte stretch
// of shared memory), the other lane bits four octets of k (128 bytes of each row).
template <int R> struct Stage<R, kAlongK> {
    static constexpr int kTasks = R * 8, kPer = (kTasks + kThreads - 1) / kThreads;
    float4 v[kPer][2];
    static __device__ __forceinline__ void at(int i, int& r, int& ko) {
        const int e = threadIdx.x + i * kThreads;
        ko = ((e >> 3) & 3) | ((e >> 5) & 1) << 2;
        r = (e >> 6) * 8 + (e & 7);
    }
    __device__ __forceinline__ void load(const float* __restrict__ X, long sr, long, int r0, int k0, int rows, int kend,
                                         int kc) {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            int r, ko;
            at(i, r, ko);
            const int k = k0 + 8 * ko;
            v[i][0] = v[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < R && r0 + r < rows && 8 * ko < kc) {
                const float* p = X + (long)(r0 + r) * sr + k;
                if (k + 8 <= kend) {
                    v[i][0] = load4(p);
                    v[i][1] = load4(p + 4);
                } else {
                    auto part = [&](int q) { return k + q < kend ? p[q] : 0.f; };
                    v[i][0] = make_float4(part(0), part(1), part(2), part(3));
                    v[i][1] = make_float4(part(4), part(5), part(6), part(7));
                }
            }
        }
    }
    template <int TR> __device__ __forceinline__ void store(unsigned char* tile, int kc) const {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            int r, ko;
            at(i, r, ko);
            if (r < R && 8 * ko < kc)
                *reinterpret_cast<uint4*>(tile + ko * (TR * 16) + (r >> 3) * 128 + (r & 7) * 16) =
                    make_uint4(pack2(v[i][0].x, v[i][0].y), pack2(v[i][0].z, v[i][0].w), pack2(v[i][1].x, v[i][1].y),
                               pack2(v[i][1].z, v[i][1].w));
        }
    }
};

// A task is 4 consecutive rows x 8 k; consecutive lanes take consecutive rows.
template <int R> struct Stage<R, kAlongR> {
    static constexpr int kQuads = R / 4, kTasks = kQuads * 8, kPer = (kTasks + kThreads - 1) / kThreads;
    float4 v[kPer][8];
    __device__ __forceinline__ void load(const float* __restrict__ X, long, long sk, int r0, int k0, int rows, int kend,
                                         int kc) {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const int e = threadIdx.x + i * kThreads, r = r0 + 4 * (e % kQuads), ko = e / kQuads;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int k = k0 + 8 * ko + q;
                v[i][q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (e < kTasks && 8 * ko < kc && k < kend) {
                    const float* p = X + (long)k * sk + r;
                    if (r + 4 <= rows) {
                        v[i][q] = load4(p);
                    } else {
                        if (r < rows) v[i][q].x = p[0];
                        if (r + 1 < rows) v[i][q].y = p[1];
                        if (r + 2 < rows) v[i][q].z = p[2];
                    }
                }
            }
        }
    }
    template <int TR> __device__ __forceinline__ void store(unsigned char* tile, int kc) const {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const int e = threadIdx.x + i * kThreads, r = 4 * (e % kQuads), ko = e / kQuads;
            if (e < kTasks && 8 * ko < kc) {
                uint4* p = reinterpret_cast<uint4*>(tile + ko * (TR * 16) + (r >> 3) * 128 + (r & 7) * 16);
                p[0] = make_uint4(pack2(v[i][0].x, v[i][1].x), pack2(v[i][2].x, v[i][3].x), pack2(v[i][4].x, v[i][5].x),
                                  pack2(v[i][6].x, v[i][7].x));
                p[1] = make_uint4(pack2(v[i][0].y, v[i][1].y), pack2(v[i][2].y, v[i][3].y), pack2(v[i][4].y, v[i][5].y),
                                  pack2(v[i][6].y, v[i][7].y));
                p[2] = make_uint4(pack2(v[i][0].z, v[i][1].z), pack2(v[i][2].z, v[i][3].z), pack2(v[i][4].z, v[i][5].z),
                                  pack2(v[i][6].z, v[i][7].z));
                p[3] = make_uint4(pack2(v[i][0].w, v[i][1].w), pack2(v[i][2].w, v[i][3].w), pack2(v[i][4].w, v[i][5].w),
                                  pack2(v[i][6].w, v[i][7].w));
            }
        }
    }
};

// Any strides: the tasks of kAlongK with scalar loads.
template <int R> struct Stage<R, kAny> {
    static constexpr int kTasks = R * 8, kPer = (kTasks + kThreads - 1) / kThreads;
    float v[kPer][8];
    __device__ __forceinline__ void load(const float* __restrict__ X, long sr, long sk, int r0, int k0, int rows,
                                         int kend, int kc) {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            int r, ko;
            Stage<R, kAlongK>::at(i, r, ko);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int k = k0 + 8 * ko + q;
                v[i][q] = r < R && r0 + r < rows && 8 * ko < kc && k < kend ? X[(long)(r0 + r) * sr + (long)k * sk] : 0.f;
            }
        }
    }
    template <int TR> __device__ __forceinline__ void store(unsigned char* tile, int kc) const {
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            int r, ko;
            Stage<R, kAlongK>::at(i, r, ko);
            if (r < R && 8 * ko < kc)
                *reinterpret_cast<uint4*>(tile + ko * (TR * 16) + (r >> 3) * 128 + (r & 7) * 16) =
                    make_uint4(pack2(v[i][0], v[i][1]), pack2(v[i][2], v[i][3]), pack2(v[i][4], v[i][5]),
                               pack2(v[i][6], v[i][7]));
        }
    }
};

__device__ __forceinline__ long two_level(int i, int e, long s, long s2) {
    return e ? (long)(i % e) * s + (long)(i / e) * s2 : (long)i * s;
}

// Eight outputs of one row, columns n .. n + 7 (as far as N goes): everything that is read is
// loaded before the first store (the outputs may be what is read, so the compiler keeps the
// order it is given).
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
    const float4 a = load4(p), b = load4(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void write8(const GemmArgs& g, long rb, int n, float (&v)[8]) {
    const float* Cin = g.Cin ? g.Cin : g.C;
    const bool vec = !g.ni && g.scn == 1 && n + 8 <= g.N && ((rb + n) & 3) == 0 && g.vec16;
    auto at = [&](int i) { return rb + two_level(n + i, g.ni, g.scn, g.scn2); };
    float c[8], d[8];
    if (g.beta != 0.f) {
        if (vec) load8(Cin + rb + n, c);
        else
#pragma unroll
            for (int i = 0; i < 8; i++) c[i] = n + i < g.N ? Cin[at(i)] : 0.f;
    }
    if (g.dgelu) {
        if (vec) load8(g.dgelu + rb + n, d);
        else
#pragma unroll
            for (int i = 0; i < 8; i++) d[i] = n + i < g.N ? g.dgelu[at(i)] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        v[i] = g.alpha * v[i];
        if (g.bias && n + i < g.N) v[i] += g.bias[n + i];
        if (g.beta != 0.f) v[i] += g.beta * c[i];
        if (g.dgelu) v[i] *= gelu_d(d[i]);
    }
    if (vec) store8(g.C + rb + n, v);
    else
#pragma unroll
        for (int i = 0; i < 8; i++)
            if (n + i < g.N) g.C[at(i)] = v[i];
    if (g.gelu) {
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = gelu_f(v[i]);
        if (vec) store8(g.gelu + rb + n, v);
        else
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (n + i < g.N) g.gelu[at(i)] = v[i];
    }
}

// K steps that are loaded, stored and multiplied at a time: as many as the registers of two
// CTAs per SM hold.  Few rows of unit-stride k (weight gradients: one tile per batch entry,
// K = H W) are bound by the chain of loads, barrier and commit of a group: 1.07 us with one
// step of 64 in a group.
template <int RA, int BN, int LA, int LB> constexpr int depth() {
    return RA == 32 && LA != kAlongR && LB != kAlongR ? (BN == 32 ? 4 : 2) : 1;
}

// A CTA works through its tiles (every gridDim.x-th of tiles = tm x tn x outputs): the loads
// of the next step, of this tile or the next one, are in flight while a step is stored and
// multiplied and while a finished tile is written.  RA: rows of A that are staged (32 when
// M <= 32: the accumulator's other rows are never read).
template <int BN, int LA, int LB, int RA>
__global__ void __launch_bounds__(kThreads, 2) tc_gemm_kernel(GemmArgs g, int tm, int tn, int tiles) {
    extern __shared__ __align__(1024) unsigned char smem[];
    // One step's tiles (A packed to RA rows: the rows of the accumulator beyond them come from
    // whatever follows, B's tile at the last, and are never read), D steps to a buffer.
    constexpr int D = depth<RA, BN, LA, LB>(), kStep = tile_bytes(RA) + tile_bytes(BN), kBuf = D * kStep;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + 2 * kBuf);      // one per buffer
    uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + 2 * kBuf + 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar0 = smem_u32(bars);
    if (warp == 0) {
        tmem_alloc(smem_u32(tslot), BN);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    pdl_wait();
    constexpr uint32_t idesc = idesc_bf16(kBM, BN);
    const int groups = g.K > 0 ? (g.K + D * kBK - 1) / (D * kBK) : 1;       // K = 0: one of nothing
    const int mine = blockIdx.x < tiles ? (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const long total = (long)mine * groups;
    auto cols = [&](int i) { return max(0, min(kBK, (g.K - i * kBK + 15) & ~15)); };
    Stage<RA, LA> sa[D];
    Stage<BN, LB> sb[D];
    int lt = 0, li = 0;                        // tile (of mine) and group of the next loads
    auto load = [&] {
        if (lt < mine) {
            const int tile = blockIdx.x + lt * (int)gridDim.x, z = tile / (tm * tn), r = tile % (tm * tn);
#pragma unroll
            for (int d = 0; d < D; d++) {
                const int i = li * D + d;
                sa[d].load(g.A + (long)z * g.sab, g.sam, g.sak, r % tm * kBM, i * kBK, g.M, g.K, cols(i));
                sb[d].load(g.B + (long)z * g.sbb, g.sbn, g.sbk, r / tm * BN, i * kBK, g.N, g.K, cols(i));
            }
            if (++li == groups) { li = 0; lt++; }
        }
    };
    bool ok = true;
    load();
    int ct = 0, ci = 0;                        // tile and group being multiplied
    for (long s = 0; s < total; s++) {
        const int bf = (int)(s & 1);
        unsigned char* buf = smem + bf * kBuf;
        // the buffer's previous tiles are read by the tensor cores until its barrier completes
        if (s >= 2) ok = mbar_wait(bar0 + 8 * bf, (uint32_t)((s >> 1) - 1) & 1) && ok;
#pragma unroll
        for (int d = 0; d < D; d++) {
            sa[d].template store<RA>(buf + d * kStep, cols(ci * D + d));
            sb[d].template store<BN>(buf + d * kStep + tile_bytes(RA), cols(ci * D + d));
        }
        load();
        tc_fence_before();                     // the previous tile's accumulator has been read
        fence_async_smem();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
#pragma unroll
            for (int d = 0; d < D; d++) {
                const uint32_t a0 = smem_u32(buf + d * kStep), b0 = a0 + tile_bytes(RA);
                const int kc = cols(ci * D + d);
                for (int q = 0; q < kc / 16; q++) {
                    const uint64_t ad = smem_desc(a0 + q * 2 * RA * 16, RA * 16, 128);
                    const uint64_t bd = smem_desc(b0 + q * 2 * BN * 16, BN * 16, 128);
                    mma_bf16(tmem, ad, bd, idesc, (ci > 0 || d > 0 || q > 0) ? 1u : 0u);
                }
            }
            mma_commit(bar0 + 8 * bf);
        }
        if (++ci < groups) continue;
        {
            // the tile's last group: its commit covers every MMA before it
            ok = mbar_wait(bar0 + 8 * bf, (uint32_t)(s >> 1) & 1);
            tc_fence_after();
            if (ok) {
                const int tile = blockIdx.x + ct * (int)gridDim.x, z = tile / (tm * tn), r = tile % (tm * tn);
                const int m = r % tm * kBM + 32 * (warp & 3) + lane, n0 = r / tm * BN;
                const long rb = two_level(z, g.bi, g.scb, g.scb2) + two_level(m, g.mi, g.scm, g.scm2);
                constexpr int kHalf = BN / 2;
#pragma unroll 1
                for (int c0 = 0; c0 < kHalf; c0 += 8) {
                    const int cc = (warp >> 2) * kHalf + c0;
                    if (n0 + cc >= g.N) break;         // warp-uniform
                    float v[8];
                    if (g.K > 0) {
                        tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)cc, v);
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; i++) v[i] = 0.f;
                    }
                    if (m < g.M) write8(g, rb, n0 + cc, v);
                }
            }
            ci = 0;                            // a wait that gave up ends the loop at the next barrier
            ct++;
        }
    }
    if (!__syncthreads_and(ok)) {
        if (threadIdx.x == 0 && g.err) atomicExch(g.err, 1);
        // one more bounded wait for the MMAs in flight before the memory is given back
        mbar_wait(bar0, 0);
        mbar_wait(bar0 + 8, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, BN);
    }
}

int sm_count() {
    static int cache[64] = {};       // per device; a benign race writes the same value
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 1; }
    if (!cache[dev] && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) cache[dev] = n;
    return cache[dev] > 0 ? cache[dev] : 1;
}

// Layout of an operand of `rows` rows: vectors of four floats from 16-byte aligned addresses.
Layout layout_of(const float* p, long sr, long sk, long sb, int batch) {
    const bool base = (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (batch == 1 || sb % 4 == 0);
    if (base && sk == 1 && sr % 4 == 0) return kAlongK;
    if (base && sr == 1 && sk % 4 == 0) return kAlongR;
    return kAny;
}

template <int BN, int LA, int LB, int RA> die_status launch(const GemmArgs& g, cudaStream_t st) {
    const size_t smem = 2 * depth<RA, BN, LA, LB>() * (tile_bytes(RA) + tile_bytes(BN)) + 32;
    // the shared-memory limit is raised on every call (a host-side attribute, cheap, and
    // correct on whichever device is current)
    DIE_CUDA_TRY(cudaFuncSetAttribute(tc_gemm_kernel<BN, LA, LB, RA>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int tm = (g.M + kBM - 1) / kBM, tn = (g.N + BN - 1) / BN;
    const long tiles = (long)tm * tn * g.batch;
    if (tiles >= (1l << 30)) return DIE_EINVAL;
    // two resident CTAs per SM, but for those the caller keeps for a concurrent kernel
    const long most = max(2 * sm_count() - g.spare, sm_count());
    DIE_CUDA_TRY(launch_pdl(tc_gemm_kernel<BN, LA, LB, RA>, dim3((unsigned)(tiles < most ? tiles : most)), dim3(kThreads),
                            smem, st, g, tm, tn, (int)tiles));
    return DIE_OK;
}
template <int BN, int RA> die_status launch_l(const GemmArgs& g, Layout la, Layout lb, cudaStream_t st) {
    if (la == kAny) return launch<BN, kAny, kAny, RA>(g, st);
    if (la == kAlongK)
        return lb == kAlongK ? launch<BN, kAlongK, kAlongK, RA>(g, st)
               : lb == kAlongR ? launch<BN, kAlongK, kAlongR, RA>(g, st) : launch<BN, kAlongK, kAny, RA>(g, st);
    return lb == kAlongK ? launch<BN, kAlongR, kAlongK, RA>(g, st)
           : lb == kAlongR ? launch<BN, kAlongR, kAlongR, RA>(g, st) : launch<BN, kAlongR, kAny, RA>(g, st);
}
template <int BN> die_status launch_n(const GemmArgs& g, Layout la, Layout lb, cudaStream_t st) {
    return g.M <= 32 ? launch_l<BN, 32>(g, la, lb, st) : launch_l<BN, 128>(g, la, lb, st);
}

}  // namespace

die_status tc_gemm(const GemmArgs& in, cudaStream_t st) {
    GemmArgs g = in;
    if (g.M < 0 || g.N < 0 || g.K < 0 || g.batch < 1 || g.batch > 65535) return DIE_EINVAL;
    if (g.M == 0 || g.N == 0) return DIE_OK;
    if (!g.A || !g.B || !g.C) return DIE_EINVAL;
    // A batch of few rows against one B (rows one after another): one tall matrix, so that the
    // 128 rows of a tile are used (16-row batches: an eighth of the tiles).
    if (g.batch > 1 && g.sbb == 0 && g.M % kBM != 0 && g.sab == (long)g.M * g.sam && !g.mi && !g.bi &&
        (long)g.M * g.batch < (1l << 30)) {
        g.mi = g.M;
        g.scm2 = g.scb;
        g.M *= g.batch;
        g.batch = 1;
        g.sab = g.scb = 0;
    }
    const Layout la = layout_of(g.A, g.sam, g.sak, g.sab, g.batch), lb = layout_of(g.B, g.sbn, g.sbk, g.sbb, g.batch);
    auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    g.vec16 = aligned(g.C) && aligned(g.Cin) && aligned(g.dgelu) && aligned(g.gelu);
    if (g.N <= 32) return launch_n<32>(g, la, lb, st);
    if (g.N <= 64) return launch_n<64>(g, la, lb, st);
    return launch_n<128>(g, la, lb, st);
}

}  // namespace die

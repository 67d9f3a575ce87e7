// mlp.cu -- the warm-start network: BF16 products on the tcgen05 tensor cores
// with FP32 accumulation in tensor memory, fused epilogues (bias, tanh,
// tanh'), MSE loss, Adam; C ABI in include/mlp.h.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/mlp.h"
#include "pic_device.cuh"

namespace {

using bf16 = __nv_bfloat16;

// ---------------------------------------------------------------------------
// BF16 arrays are the library's own and lie in memory as the tensor core reads them: 8 x 8 core matrices of
// 128 contiguous bytes (row r of one at 16 r bytes), the core matrices of 8 rows one after another. Columns
// are padded to a multiple of 16, rows too, with zeros. Element (r, c) of an array with `ld` columns:
__host__ __device__ inline int pad16(int n) { return (n + 15) / 16 * 16; }
__device__ __forceinline__ size_t cm_index(int r, int c, int ld) {
    return ((size_t)(r >> 3) * (ld >> 3) + (c >> 3)) * 64 + (r & 7) * 8 + (c & 7);
}

// C[M x N] = A(M x K) B(K x N) on the 5th-generation tensor cores (tcgen05). A(m, k) is element (m, k) of
// its array (a_t = 0) or (k, m) (a_t = 1); B(k, n) is (n, k) (b_t = 0) or (k, n) (b_t = 1). The same core
// matrices serve both ways: 8 rows of 8 consecutive k (K-major), or 8 k of 8 consecutive rows (MN-major).
//
// One CTA of 512 threads per 128 x TBN tile of C, K in chunks of 128 in a ring of four stages: 512 of K in
// flight, fetched by bulk copies (one per 8 rows or 8 k of a chunk, issued by one warp, an mbarrier per
// stage); another warp's thread issues the products of a chunk as it lands (tcgen05.mma kind::f16, M 128, N
// TBN, K 16, BF16 operands, FP32 accumulator in tensor memory) and commits them to the stage's second
// mbarrier, after which the stage may be refilled. Every wait is bounded. The epilogue reads the
// accumulator with tcgen05.ld (warp w may read lanes 32 (w % 4) .. + 31, the tile's rows), parks it in
// shared memory, applies the fused bias / tanh / tanh' / squared-error step and writes C row by row.
//
// These products are bounded by latency, far below the tensor rate: a chain of launch, copies, products
// and epilogue in 64 to 130 CTAs. Hence the many threads (epilogue), the narrow tiles (TBN is the narrowest
// of 16, 32, 64 that still gives at most one CTA per SM), and copies that need no thread per 16 bytes (the
// same tile by 16-byte asynchronous copies took 5 us to fetch, by loads through registers, two chunks of 64
// at a time, 20). 256 x 512 x 512, a
// launch (ncu): 27.6 -> 8.1 us, 24 x 512 x 512 23.2 -> 6.9; a training step of the 5-512-512-512-512-768
// network at batch 256: 326 -> 89 us, 11 launches for 28.
enum Epilogue {
    EP_STORE = 0,      // C32 = acc
    EP_BIAS_TANH = 1,  // z = acc + bias; C32 = tanh z; C16 = bf16(C32)
    EP_BIAS = 2,       // C32 = acc + bias
    EP_DTANH = 3,      // C32 = acc (1 - yprev^2); C16 = bf16(C32)
    EP_MSE = 4,        // d = acc + bias - t; C32 = sc d, C16 = bf16(C32); d^2 summed into the loss
};

struct GemmArgs {
    const bf16* A;
    const bf16* B;
    const float* A32;    // FP32 source of A (M rows of K <= TBK, K-major), converted while staged, kept in A16
    bf16* A16;
    int lda, ldb, a_t, b_t;
    int M, N, K;
    int ep;
    const float* bias;
    const float* aux;    // [M x N], ld = ldc: yprev (EP_DTANH) or targets (EP_MSE)
    float* C32;
    bf16* C16;
    int ldc, ldc16;
    float sc;            // 2 / (M N) of the loss
    int tiles;           // CTAs of this product
};
// One launch: a product, optionally a second one (the next CTAs) and column sums (the last CTAs).
struct Launch {
    GemmArgs g[2];
    const float* cs_in;  // column sums of cs_in[cs_rows x cs_cols] (ld cs_cols) to cs_out
    float* cs_out;
    int cs_rows, cs_cols;
    float* part;         // per-CTA sums of d^2, then the loss from them in order by the last CTA
    float* loss;
    unsigned* done;
    unsigned* err;       // set to MLP_ERR_TIMEOUT if a bounded wait gave up
};

constexpr int TBM = 128, TBK = 128, TTHREADS = 512, STAGES = 4;
constexpr unsigned CM = 128;                          // bytes of a core matrix
template <int TBN> __host__ __device__ constexpr unsigned stage_bytes() { return (TBM + TBN) * TBK * 2; }
constexpr unsigned A_BYTES = TBM * TBK * 2;
template <int TBN> constexpr unsigned gemm_smem(int stages) {  // the ring, at least the epilogue's tile
    return stages * stage_bytes<TBN>() > TBM * (TBN + 1) * 4 ? stages * stage_bytes<TBN>() : TBM * (TBN + 1) * 4;
}
constexpr int TC_TRIES = 1 << 20;                     // polls of a bounded mbarrier wait
constexpr unsigned MLP_ERR_TIMEOUT = 1u;

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and B (bits 7-9,
// 10-12 = 1), A, B MN-major (bits 15, 16; 0: K-major), N / 8 in bits 17-22, M / 16 in bits 24-28.
template <int TBN>
__device__ __forceinline__ uint32_t idesc(int a_t, int b_t) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_t << 15) | ((uint32_t)b_t << 16) |
           ((uint32_t)(TBN >> 3) << 17) | ((uint32_t)(TBM >> 4) << 24);
}

__device__ __forceinline__ uint32_t s_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: start address / 16 (bits 0-13), leading-dimension byte offset
// / 16 (16-29: next core matrix along K), stride byte offset / 16 (32-45: next one along M or N), the
// fixed version field 0b001 (46-48), base offset 0, no swizzle (61-63 = 0).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, unsigned lbo, unsigned sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ bool tc_wait(uint32_t mb, unsigned parity) {
    for (int it = 0; it < TC_TRIES; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(mb), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, unsigned bytes, uint32_t mb) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mb)
                 : "memory");
}

// One warp fetches the chunk at k0 (kcs groups of 8 k) of R rows of an operand from row r0; returns the
// bytes requested, the same on every lane. K-major: one copy per 8 rows, in shared memory 8 rows at TBK * 16
// bytes; MN-major: one copy per 8 k, at R * 16 bytes. Rows outside the array (`rows`, padded) stay as they
// are: they only reach results that are not stored.
template <int R>
__device__ __forceinline__ unsigned fetch(uint32_t s, const bf16* X, int ld, int t, int rows, int r0, int k0, int kcs,
                                          uint32_t mb, int lane, bool issue) {
    const int rg = min(R, rows - r0) >> 3;  // groups of 8 rows
    const int copies = t == 0 ? rg : kcs;
    const unsigned bytes = (t == 0 ? kcs : rg) * CM, dstep = t == 0 ? TBK * 16u : R * 16u;
    if (issue)
        for (int i = lane; i < copies; i += 32)
            bulk_copy(s + i * dstep,
                      X + (t == 0 ? (size_t)((r0 >> 3) + i) * (ld >> 3) + (k0 >> 3)
                                  : (size_t)((k0 >> 3) + i) * (ld >> 3) + (r0 >> 3)) * 64,
                      bytes, mb);
    return copies * bytes;
}

// 8 BF16 of row r from column k of an FP32 array of M rows of K (zeros outside).
__device__ __forceinline__ uint4 bf16_group(const float* x, int M, int K, int r, int k) {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (r < M) {
        x += (size_t)r * K + k;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (k + i < K) w[i >> 1] |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[i])) << (16 * (i & 1));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// A from FP32 (K-major, one chunk of kcs groups of 8 k), converted by all threads; the first CTA of a row of
// tiles keeps the converted operand (for the weight gradients), with its padding.
__device__ __forceinline__ void stage_f32(unsigned char* s, const GemmArgs& g, int m0, int kcs, bool keep) {
    const int rows = min(TBM, pad16(g.M) - m0);
#pragma unroll 1
    for (int u = threadIdx.x; u < rows * kcs; u += TTHREADS) {
        const int r = u / kcs, kc = u % kcs;
        const uint4 v = bf16_group(g.A32, g.M, g.K, m0 + r, 8 * kc);
        if (keep) *reinterpret_cast<uint4*>(g.A16 + cm_index(m0 + r, 8 * kc, g.lda)) = v;
        *reinterpret_cast<uint4*>(s + (r >> 3) * (TBK * 16) + kc * CM + (r & 7) * 16) = v;
    }
}

// An input of more than one chunk: converted into core matrices once, by a launch of its own, and fetched
// through the ring like every other operand. (Converted while staged in the product, a chunk had to wait for
// the products of the chunk before, in every column tile again. A forward pass, that way -> this way: 784-512-10
// at batch 4096 99 -> 37 us, at 256 56 -> 18, 4096-4096 at batch 4096 2595 -> 503, 129-64-10 at batch 16,
// two chunks, 10.9 -> 9.2.) A warp takes 8 rows of 4 groups of 8 k: 128 contiguous bytes of each row in, 512
// contiguous bytes out.
__global__ void __launch_bounds__(256) k_input_bf16(const float* x, bf16* x16, int M, int K, int ld) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, groups = ld >> 3, quads = (groups + 3) >> 2;
    const int items = pad16(M) / 8 * quads, step = gridDim.x * 8;
    for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < items; i += step) {
        const int r = i / quads * 8 + (lane & 7), kc = i % quads * 4 + (lane >> 3);
        if (kc < groups) *reinterpret_cast<uint4*>(x16 + cm_index(r, 8 * kc, ld)) = bf16_group(x, M, K, r, 8 * kc);
    }
}

// Sum over the CTA's threads in a fixed tree; thread 0 gets it.
__device__ __forceinline__ float block_sum(float v) {
    __shared__ float s_w[TTHREADS / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.0f;
    if (threadIdx.x == 0)
        for (int k = 0; k < TTHREADS / 32; ++k) t += s_w[k];
    return t;
}

// Column sums of g[rows x cols] (bias gradients): CS_COLS columns x 8 row groups, each thread summing every
// eighth row, then the eight partial sums in order (a fixed order per column).
constexpr int CS_COLS = TTHREADS / 8;
__device__ __forceinline__ void column_sums(const Launch& L, int block) {
    __shared__ float s[8][CS_COLS + 1];
    const int cx = threadIdx.x % CS_COLS, gy = threadIdx.x / CS_COLS, c = block * CS_COLS + cx;
    float acc = 0.0f;
    if (c < L.cs_cols) {
#pragma unroll 16
        for (int r = gy; r < L.cs_rows; r += 8) acc += __ldcg(L.cs_in + (size_t)r * L.cs_cols + c);
    }
    s[gy][cx] = acc;
    __syncthreads();
    if (gy == 0 && c < L.cs_cols) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += s[k][cx];
        L.cs_out[c] = t;
    }
}

template <int TBN>
__global__ void __launch_bounds__(TTHREADS) k_gemm(const __grid_constant__ Launch L, int stages) {
    extern __shared__ __align__(1024) unsigned char smem[];  // the ring: A (128 x 128) then B (TBN x 128) per stage
    __shared__ __align__(8) unsigned long long mbar[2 * STAGES + 1];  // landed, free (per stage), all products done
    __shared__ uint32_t tmem_slot;
    __shared__ int s_fail;  // a wait gave up; then, of the loss: this CTA is the last
    constexpr uint32_t COLS = TBN < 32 ? 32 : TBN;  // tensor-memory columns (a power of two, at least 32)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t landed = s_addr(&mbar[0]), freed = landed + 8 * STAGES, all_done = freed + 8 * STAGES;
    int tile = blockIdx.x;
    const bool second = tile >= L.g[0].tiles;
    if (second) tile -= L.g[0].tiles;
    const GemmArgs& g = L.g[second];
    if (second && tile >= g.tiles) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        column_sums(L, tile - g.tiles);
        return;
    }
    if (warp == 0) {  // tensor memory for the accumulator: one warp allocates, the same warp frees
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(&tmem_slot)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid <= 2 * STAGES) {
        if (tid == 0) s_fail = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(landed + 8u * tid) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int tn = (g.N + TBN - 1) / TBN, m0 = tile / tn * TBM, n0 = tile % tn * TBN;
    const int Kp = pad16(g.K), nk = (Kp + TBK - 1) / TBK;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // nothing above reads what kernels write
    if (g.A32) stage_f32(smem, g, m0, Kp / 8, n0 == 0);  // FP32 input (of one chunk): by all threads
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    // chunk i into stage s: expected bytes first, then the copies
    auto load = [&](int i, int s) {
        const int k0 = i * TBK, kcs = min(TBK, Kp - k0) / 8;
        const uint32_t sa = s_addr(smem) + s * stage_bytes<TBN>(), mb = landed + 8 * s;
        const int ra = g.a_t ? g.lda : (g.M + 7) / 8 * 8, rb = g.b_t ? g.ldb : pad16(g.N);
        unsigned n = g.A32 ? 0u : fetch<TBM>(sa, g.A, g.lda, g.a_t, ra, m0, k0, kcs, mb, lane, false);
        n += fetch<TBN>(sa + A_BYTES, g.B, g.ldb, g.b_t, rb, n0, k0, kcs, mb, lane, false);
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(n) : "memory");
        __syncwarp();
        if (!g.A32) fetch<TBM>(sa, g.A, g.lda, g.a_t, ra, m0, k0, kcs, mb, lane, true);
        fetch<TBN>(sa + A_BYTES, g.B, g.ldb, g.b_t, rb, n0, k0, kcs, mb, lane, true);
    };
    // products of the chunk in stage s, then its commit
    auto products = [&](int i, int s) {
        const int steps = min(TBK, Kp - i * TBK) / 16;
        const unsigned la = g.a_t ? TBM * 16 : CM, sa = g.a_t ? CM : TBK * 16, lb = g.b_t ? TBN * 16 : CM,
                       sb = g.b_t ? CM : TBK * 16;
        const uint32_t a0 = s_addr(smem) + s * stage_bytes<TBN>(), id = idesc<TBN>(g.a_t, g.b_t);
        uint64_t ad = sdesc(a0, la, sa), bd = sdesc(a0 + A_BYTES, lb, sb);
#pragma unroll 1
        for (int q = 0; q < steps; ++q) {  // K 16 per instruction: two core matrices along K
            const uint32_t accumulate = (i > 0 || q > 0) ? 1u : 0u;
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                "l"(ad), "l"(bd), "r"(id), "r"(accumulate)
                : "memory");
            ad += 2 * (la >> 4);
            bd += 2 * (lb >> 4);
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         i + 1 < nk ? freed + 8u * s : all_done)
                     : "memory");
    };
    bool ok = true;
    if (warp == 0) {  // the copies
        int s = 0;
        unsigned phase = 1;
        for (int i = 0; i < nk; ++i) {
            // stage s is free when the products of chunk i - stages are done; a failed wait ends the copies
            // (the products' wait for this chunk then fails too)
            if (i >= stages && !tc_wait(freed + 8u * s, phase)) break;
            load(i, s);
            if (++s == stages) {
                s = 0;
                phase ^= 1u;
            }
        }
    } else if (warp == 1 && lane == 0) {  // the products
        int s = 0;
        unsigned phase = 0;
        for (int i = 0; i < nk; ++i) {
            if (!tc_wait(landed + 8u * s, phase) && !tc_wait(landed + 8u * s, phase)) {
                s_fail = 1;
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(all_done) : "memory");
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            products(i, s);
            if (++s == stages) {
                s = 0;
                phase ^= 1u;
            }
        }
    }
    __syncwarp();
    // the last commit covers every product issued before it; the products' own waits come first, so this one
    // is given as many polls as all of them
    {
        bool done = false;
        for (int i = 0; i <= 2 * nk && !done; ++i) done = tc_wait(all_done, 0u);
        if (__syncthreads_or(!done || s_fail)) ok = false;
    }
    float sum = 0.0f;
    if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // accumulator -> shared tile T[128][TBN + 1] (thread = row: conflict-free with the odd stride)
        float* T = reinterpret_cast<float*>(smem);
        const int row = (warp & 3) * 32 + lane;  // the accumulator rows warp w may read: 32 (w % 4) ..
#pragma unroll 1
        for (int c0 = 16 * (warp >> 2); c0 < TBN; c0 += 16 * (TTHREADS / 128)) {
            uint32_t r[16];
            const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                "[%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                  "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                  "=r"(r[15])
                : "r"(ta));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) T[row * (TBN + 1) + c0 + j] = __uint_as_float(r[j]);
        }
        __syncthreads();
        // row by row: consecutive threads write consecutive columns. Each thread keeps one column (its bias
        // loaded once); the loads of a batch of rows (aux) are all issued before its stores, which the
        // compiler could not reorder (aliasing). The result stays in T for the BF16 copy.
        const int cc = tid % TBN, rb = tid / TBN, n = n0 + cc, rows = min(TBM, g.M - m0);
        const bool nin = n < g.N, aux = g.ep == EP_DTANH || g.ep == EP_MSE;
        const float bn = (nin && g.bias) ? __ldcg(g.bias + n) : 0.0f;
        constexpr int RSTEP = TTHREADS / TBN, BATCH = TBM / RSTEP < 16 ? TBM / RSTEP : 16;
        static_assert(TBM % (RSTEP * BATCH) == 0, "whole batches");
#pragma unroll 1
        for (int r0 = rb; r0 < rows; r0 += RSTEP * BATCH) {
            float y[BATCH];
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int rr = r0 + RSTEP * j;
                y[j] = (aux && nin && rr < rows) ? __ldcg(g.aux + (size_t)(m0 + rr) * g.ldc + n) : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int rr = r0 + RSTEP * j;
                if (!nin || rr >= rows) continue;
                float v = T[rr * (TBN + 1) + cc];
                if (g.ep == EP_BIAS_TANH) v = tanhf(v + bn);
                else if (g.ep == EP_BIAS) v = v + bn;
                else if (g.ep == EP_DTANH) v = v * (1.0f - y[j] * y[j]);
                else if (g.ep == EP_MSE) {
                    const float d = v + bn - y[j];
                    sum += d * d;
                    v = g.sc * d;
                }
                g.C32[(size_t)(m0 + rr) * g.ldc + n] = v;
                if (g.C16) T[rr * (TBN + 1) + cc] = v;
            }
        }
        if (g.C16) {  // BF16 copy in core matrices, 16 bytes per thread, with the zeros of its padding
            __syncthreads();
            const int rows16 = min(TBM, pad16(g.M) - m0), groups = min(TBN, g.ldc16 - n0) / 8;
#pragma unroll 1
            for (int u = tid; u < rows16 * groups; u += TTHREADS) {
                const int r = u / groups, c = 8 * (u % groups);
                uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (r < rows && n0 + c + i < g.N)
                        w[i >> 1] |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(T[r * (TBN + 1) + c + i])) << (16 * (i & 1));
                *reinterpret_cast<uint4*>(g.C16 + cm_index(m0 + r, n0 + c, g.ldc16)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    } else if (tid == 0) {
        atomicOr(L.err, MLP_ERR_TIMEOUT);
        for (int k = 0; k < stages; ++k) tc_wait(landed + 8u * k, 0u);  // a last bounded chance for copies in flight
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
    if (g.ep == EP_MSE) {  // mean squared error: the CTAs' sums, added in a fixed order by the last CTA to finish
        const float b = block_sum(sum);
        if (tid == 0) {
            L.part[blockIdx.x] = b;
            __threadfence();
            s_fail = atomicAdd(L.done, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (s_fail && warp == 0) {
            __threadfence();
            float t = 0.0f;
            for (unsigned k = lane; k < gridDim.x; k += 32) t += __ldcg(L.part + k);
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xFFFFFFFFu, t, o);
            if (lane == 0) {
                *L.loss = t / ((float)g.M * (float)g.N);
                *L.done = 0;
            }
        }
    }
}

// What the parameter kernels need of a layer: its weights and biases in the parameter block, the padded
// BF16 copy.
struct LayerMap {
    long long woff[MLP_MAX_LAYERS], w16off[MLP_MAX_LAYERS];
    int in[MLP_MAX_LAYERS], out[MLP_MAX_LAYERS], ld16[MLP_MAX_LAYERS];
};

// Adam on the FP32 master parameters and the BF16 weight copies in one pass (blockIdx.y = layer; the
// biases follow the weights): 28 bytes read and written per parameter and 2 of the copy.
__global__ void __launch_bounds__(256) k_adam(const __grid_constant__ LayerMap Lm, float* __restrict__ p,
                                              const float* __restrict__ g, float* __restrict__ m,
                                              float* __restrict__ v, bf16* __restrict__ w16, float lr, float b1,
                                              float b2, float eps, float c1, float c2) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int l = blockIdx.y, in = Lm.in[l];
    const int nw = in * Lm.out[l], n = nw + Lm.out[l];
    const long long o = Lm.woff[l];
    for (int k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256) {
        const long long i = o + k;
        const float gi = __ldcg(g + i);
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        m[i] = mi;
        v[i] = vi;
        p[i] = pi;
        if (k < nw) {
            const int r = (int)((unsigned)k / (unsigned)in);
            w16[Lm.w16off[l] + cm_index(r, k - r * in, Lm.ld16[l])] = __float2bfloat16_rn(pi);
        }
    }
}

// BF16 copies of every layer's weights (blockIdx.y = layer).
__global__ void __launch_bounds__(256) k_weights_bf16(const __grid_constant__ LayerMap Lm, const float* __restrict__ p,
                                                      bf16* __restrict__ w16) {
    const int l = blockIdx.y, in = Lm.in[l], nw = in * Lm.out[l];
    for (int k = blockIdx.x * 256 + threadIdx.x; k < nw; k += gridDim.x * 256) {
        const int r = (int)((unsigned)k / (unsigned)in);
        w16[Lm.w16off[l] + cm_index(r, k - r * in, Lm.ld16[l])] = __float2bfloat16_rn(p[Lm.woff[l] + k]);
    }
}

// Glorot-uniform initial weights from Philox (key = seed, counter = (index,
// layer, 0xA0, 0)), zero biases.
__global__ void k_init(float* __restrict__ p, long long off, long long nw, long long nb, int layer, float a,
                       unsigned long long seed) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nw + nb; i += (long long)gridDim.x * blockDim.x) {
        if (i < nw) {
            const pic::U4 r = pic::philox4x32_10((uint32_t)i, (uint32_t)layer, 0xA0u, 0u, (uint32_t)seed,
                                                 (uint32_t)(seed >> 32));
            p[off + i] = a * (2.0f * pic::u01(r.x) - 1.0f);
        } else {
            p[off + i] = 0.0f;
        }
    }
}

}  // namespace

struct mlp_ctx {
    int L = 0;
    int sizes[MLP_MAX_LAYERS + 1] = {};
    int max_batch = 0;
    long long woff[MLP_MAX_LAYERS] = {}, boff[MLP_MAX_LAYERS] = {}, w16off[MLP_MAX_LAYERS] = {};
    int ld[MLP_MAX_LAYERS + 1] = {};  // padded row length of the BF16 arrays of each size
    long long n_params = 0, n_w = 0;
    float* p = nullptr;     // master parameters
    float* grad = nullptr;  // gradients (same layout)
    float* m = nullptr;
    float* v = nullptr;
    bf16* w16 = nullptr;    // weights, packed by layer
    bf16* x16 = nullptr;    // input [max_batch x sizes[0]]
    float* y32[MLP_MAX_LAYERS] = {};
    bf16* y16[MLP_MAX_LAYERS] = {};
    float* g32[2] = {};
    bf16* g16[2] = {};
    float* loss = nullptr;
    float* mse_part = nullptr;  // per-CTA sums of the loss
    unsigned* mse_done = nullptr;
    unsigned* h_err = nullptr;  // mapped pinned word: a product's bounded wait gave up
    unsigned* d_err = nullptr;  // its device address
    int num_sms = 1;
    LayerMap map{};
    long long step = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::vector<void*> allocs;
    std::string err;
};

namespace {

pic_status fail(mlp_ctx* c, pic_status s, const char* what, cudaError_t e = cudaSuccess) {
    if (c) {
        c->err = what;
        if (e != cudaSuccess) {
            c->err += ": ";
            c->err += cudaGetErrorString(e);
        }
    }
    return s;
}

template <typename T>
bool dalloc(mlp_ctx* c, T** p, size_t n) {
    void* q = nullptr;
    if (cudaMalloc(&q, n * sizeof(T)) != cudaSuccess) return false;
    c->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return true;
}

// Launch that may begin while the kernel before it finishes (each waits for it before it reads or writes
// anything kernels share).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(mlp_ctx* c, void (*kern)(KArgs...), dim3 grid, int threads, size_t smem, Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
template <int TBN>
cudaError_t launch_gemm(mlp_ctx* c, const Launch& L, int grid, int nk) {
    const int stages = nk < STAGES ? nk : STAGES;
    return launch_pdl(c, k_gemm<TBN>, dim3(grid), TTHREADS, gemm_smem<TBN>(stages), L, stages);
}
template <int TBN>
cudaError_t gemm_attr() {
    return cudaFuncSetAttribute(k_gemm<TBN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<TBN>(STAGES));
}

int tiles_of(const GemmArgs& g, int tbn) { return ((g.M + TBM - 1) / TBM) * ((g.N + tbn - 1) / tbn); }

// One launch of one or two products and column sums; tile width by the rule above k_gemm.
cudaError_t gemm(mlp_ctx* c, Launch& L) {
    int tbn = 16, grid = 0;
    for (;; tbn *= 2) {
        grid = 0;
        for (GemmArgs& g : L.g) {
            g.tiles = g.M > 0 ? tiles_of(g, tbn) : 0;
            grid += g.tiles;
        }
        if (tbn == 64 || grid <= c->num_sms) break;
    }
    const int nk = std::max((pad16(L.g[0].K) + TBK - 1) / TBK, (pad16(L.g[1].K) + TBK - 1) / TBK);
    grid += (L.cs_cols + CS_COLS - 1) / CS_COLS;
    L.part = c->mse_part;
    L.done = c->mse_done;
    L.err = c->d_err;
    return tbn == 16 ? launch_gemm<16>(c, L, grid, nk) : tbn == 32 ? launch_gemm<32>(c, L, grid, nk)
                                                                   : launch_gemm<64>(c, L, grid, nk);
}

// Synchronises the context's stream and reports a product whose bounded wait gave up.
pic_status sync_checked(mlp_ctx* c, const char* what) {
    const cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return fail(c, PIC_ERR_CUDA, what, e);
    if (*reinterpret_cast<volatile unsigned*>(c->h_err))
        return fail(c, PIC_ERR_TIMEOUT, "a tensor-core product's bounded wait timed out");
    return PIC_OK;
}

int grid_for(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 1024 ? (b > 0 ? b : 1) : 1024);
}

// Blocks per layer of the parameter kernels.
dim3 param_grid(const mlp_ctx* c) {
    long long most = 1;
    for (int l = 0; l < c->L; ++l) most = std::max(most, (long long)(c->sizes[l] + 1) * c->sizes[l + 1]);
    return dim3(grid_for(most), c->L);
}

cudaError_t refresh_bf16(mlp_ctx* c) {
    k_weights_bf16<<<param_grid(c), 256, 0, c->stream>>>(c->map, c->p, c->w16);
    return cudaGetLastError();
}

// Layers 0 .. L - 1 on x; the last layer's outputs to y (EP_BIAS), or with targets t the gradient of the
// loss into g16[0], g32[0] and the loss.
cudaError_t forward(mlp_ctx* c, int batch, const float* x, float* y, const float* t, float* loss) {
    cudaError_t e = cudaSuccess;
    for (int l = 0; l < c->L && e == cudaSuccess; ++l) {
        const int in = c->sizes[l], out = c->sizes[l + 1];
        const bool end = l + 1 == c->L;
        Launch L{};
        GemmArgs& g = L.g[0];
        g.A = l == 0 ? c->x16 : c->y16[l - 1];
        g.lda = c->ld[l];
        if (l == 0 && c->ld[0] <= TBK) {
            g.A32 = x;
            g.A16 = c->x16;
        } else if (l == 0) {
            const int items = pad16(batch) / 8 * ((c->ld[0] / 8 + 3) / 4);  // of a warp, eight warps a CTA
            e = launch_pdl(c, k_input_bf16, dim3(std::min((items + 7) / 8, 8 * c->num_sms)), 256, 0, x, c->x16, batch, in,
                           c->ld[0]);
            if (e != cudaSuccess) break;
        }
        g.B = c->w16 + c->w16off[l];
        g.ldb = c->ld[l];
        g.M = batch;
        g.N = out;
        g.K = in;
        g.bias = c->p + c->boff[l];
        g.ldc = out;
        g.ldc16 = c->ld[l + 1];
        if (!end) {
            g.ep = EP_BIAS_TANH;
            g.C32 = c->y32[l];
            g.C16 = c->y16[l];
        } else if (t) {
            g.ep = EP_MSE;
            g.aux = t;
            g.sc = 2.0f / (float)((long long)batch * out);
            g.C32 = c->g32[0];
            g.C16 = c->g16[0];
            L.loss = loss;
        } else {
            g.ep = EP_BIAS;
            g.C32 = y;
        }
        e = gemm(c, L);
    }
    return e;
}

}  // namespace

extern "C" {

pic_status mlp_create(mlp_ctx** out, int32_t n_layers, const int32_t* sizes, int32_t max_batch, uint64_t seed,
                      void* cuda_stream) {
    if (!out || !sizes || n_layers < 1 || n_layers > MLP_MAX_LAYERS || max_batch < 1) return PIC_ERR_ARG;
    *out = nullptr;
    for (int l = 0; l <= n_layers; ++l)
        if (sizes[l] < 1 || sizes[l] > MLP_MAX_WIDTH) return PIC_ERR_ARG;
    // the ring of operand stages takes more than the default limit of dynamic shared memory
    if (gemm_attr<16>() != cudaSuccess || gemm_attr<32>() != cudaSuccess || gemm_attr<64>() != cudaSuccess)
        return PIC_ERR_CUDA;
    mlp_ctx* c = new mlp_ctx();
    c->L = n_layers;
    c->max_batch = max_batch;
    int wmax = 0;
    for (int l = 0; l <= n_layers; ++l) {
        c->sizes[l] = sizes[l];
        c->ld[l] = pad16(sizes[l]);
        wmax = wmax > c->ld[l] ? wmax : c->ld[l];
    }
    for (int l = 0; l < n_layers; ++l) {
        const long long nw = (long long)sizes[l] * sizes[l + 1];
        c->woff[l] = c->n_params;
        c->boff[l] = c->n_params + nw;
        c->n_params += nw + sizes[l + 1];
        c->w16off[l] = c->n_w;
        c->n_w += (long long)c->ld[l] * pad16(sizes[l + 1]);
        c->map.woff[l] = c->woff[l];
        c->map.w16off[l] = c->w16off[l];
        c->map.in[l] = sizes[l];
        c->map.out[l] = sizes[l + 1];
        c->map.ld16[l] = c->ld[l];
    }
    if (cuda_stream) {
        c->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete c;
            return PIC_ERR_CUDA;
        }
        c->own_stream = true;
    }
    const size_t P = (size_t)c->n_params;
    bool ok = dalloc(c, &c->p, P) && dalloc(c, &c->grad, P) && dalloc(c, &c->m, P) && dalloc(c, &c->v, P) &&
              dalloc(c, &c->w16, (size_t)c->n_w) && dalloc(c, &c->x16, (size_t)pad16(max_batch) * c->ld[0]) &&
              dalloc(c, &c->loss, 1) && dalloc(c, &c->mse_done, 1) &&
              dalloc(c, &c->mse_part, (size_t)((max_batch + TBM - 1) / TBM) * ((wmax + 15) / 16)) &&
              cudaHostAlloc(&c->h_err, sizeof(unsigned), cudaHostAllocMapped) == cudaSuccess &&
              cudaHostGetDevicePointer(&c->d_err, c->h_err, 0) == cudaSuccess;
    // hidden layers' outputs (the last layer writes y or the error; of a single layer, y may go through y32[0])
    for (int l = 0; l < n_layers && ok; ++l) {
        if (l + 1 < n_layers) ok = dalloc(c, &c->y16[l], (size_t)pad16(max_batch) * c->ld[l + 1]);
        if (l + 1 < n_layers || n_layers == 1) ok = ok && dalloc(c, &c->y32[l], (size_t)max_batch * sizes[l + 1]);
    }
    for (int b = 0; b < 2 && ok; ++b)
        ok = dalloc(c, &c->g32[b], (size_t)max_batch * wmax) && dalloc(c, &c->g16[b], (size_t)pad16(max_batch) * wmax);
    if (!ok) {
        mlp_destroy(c);
        return PIC_ERR_CUDA;
    }
    cudaMemsetAsync(c->m, 0, P * sizeof(float), c->stream);
    cudaMemsetAsync(c->v, 0, P * sizeof(float), c->stream);
    cudaMemsetAsync(c->grad, 0, P * sizeof(float), c->stream);
    *c->h_err = 0;
    cudaMemsetAsync(c->mse_done, 0, sizeof(unsigned), c->stream);
    // the weights' padding (that of the activations and gradients is written with them)
    cudaMemsetAsync(c->w16, 0, (size_t)c->n_w * sizeof(bf16), c->stream);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, dev);
    for (int l = 0; l < n_layers; ++l) {
        const long long nw = (long long)sizes[l] * sizes[l + 1];
        const float a = std::sqrt(6.0f / (float)(sizes[l] + sizes[l + 1]));
        k_init<<<grid_for(nw + sizes[l + 1]), 256, 0, c->stream>>>(c->p, c->woff[l], nw, sizes[l + 1], l, a, seed);
    }
    cudaError_t e = refresh_bf16(c);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        mlp_destroy(c);
        return PIC_ERR_CUDA;
    }
    *out = c;
    return PIC_OK;
}

int64_t mlp_param_count(const mlp_ctx* c) { return c ? c->n_params : 0; }

pic_status mlp_set_params(mlp_ctx* c, const float* host) {
    if (!c || !host) return PIC_ERR_ARG;
    cudaError_t e = cudaMemcpyAsync(c->p, host, sizeof(float) * (size_t)c->n_params, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = refresh_bf16(c);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return e == cudaSuccess ? PIC_OK : fail(c, PIC_ERR_CUDA, "set params", e);
}

pic_status mlp_get_params(mlp_ctx* c, float* host) {
    if (!c || !host) return PIC_ERR_ARG;
    cudaError_t e = cudaMemcpyAsync(host, c->p, sizeof(float) * (size_t)c->n_params, cudaMemcpyDeviceToHost, c->stream);
    return e == cudaSuccess ? sync_checked(c, "get params") : fail(c, PIC_ERR_CUDA, "get params", e);
}

pic_status mlp_forward(mlp_ctx* c, int32_t batch, const float* x, float* y) {
    if (!c || !x || !y || batch < 1 || batch > c->max_batch) return PIC_ERR_ARG;
    // A single launch (one layer, its input within one chunk) reads x in every column tile and writes y as
    // tiles finish: if the two overlap, the outputs go through the context's own array. (Otherwise x is read
    // by the first launch and y written by the last.)
    const size_t nx = sizeof(float) * (size_t)batch * c->sizes[0], ny = sizeof(float) * (size_t)batch * c->sizes[c->L];
    const uintptr_t ax = reinterpret_cast<uintptr_t>(x), ay = reinterpret_cast<uintptr_t>(y);
    const bool own = c->L == 1 && c->ld[0] <= TBK && ax < ay + ny && ay < ax + nx;
    cudaError_t e = forward(c, batch, x, own ? c->y32[0] : y, nullptr, nullptr);
    if (e == cudaSuccess && own) e = cudaMemcpyAsync(y, c->y32[0], ny, cudaMemcpyDeviceToDevice, c->stream);
    return e == cudaSuccess ? PIC_OK : fail(c, PIC_ERR_CUDA, "forward", e);
}

pic_status mlp_loss_grad(mlp_ctx* c, int32_t batch, const float* x, const float* t, float* loss) {
    if (!c || !x || !t || batch < 1 || batch > c->max_batch) return PIC_ERR_ARG;
    cudaError_t e = forward(c, batch, x, nullptr, t, loss ? loss : c->loss);
    if (e != cudaSuccess) return fail(c, PIC_ERR_CUDA, "forward", e);
    int cur = 0;
    for (int l = c->L - 1; l >= 0 && e == cudaSuccess; --l) {
        const int in = c->sizes[l], out = c->sizes[l + 1];
        Launch L{};
        // dW_l = G^T X: M = out, N = in, K = batch
        GemmArgs& w = L.g[0];
        w.A = c->g16[cur];
        w.lda = c->ld[l + 1];
        w.a_t = 1;
        w.B = l == 0 ? c->x16 : c->y16[l - 1];
        w.ldb = c->ld[l];
        w.b_t = 1;
        w.M = out;
        w.N = in;
        w.K = batch;
        w.ep = EP_STORE;
        w.C32 = c->grad + c->woff[l];
        w.ldc = in;
        // beside it G_{l-1} = (G W_l) * (1 - y_{l-1}^2): M = batch, N = in, K = out
        if (l > 0) {
            GemmArgs& g = L.g[1];
            g.A = c->g16[cur];
            g.lda = c->ld[l + 1];
            g.B = c->w16 + c->w16off[l];
            g.ldb = c->ld[l];
            g.b_t = 1;
            g.M = batch;
            g.N = in;
            g.K = out;
            g.ep = EP_DTANH;
            g.aux = c->y32[l - 1];
            g.C32 = c->g32[1 - cur];
            g.C16 = c->g16[1 - cur];
            g.ldc = in;
            g.ldc16 = c->ld[l];
        }
        // and the bias gradients
        L.cs_in = c->g32[cur];
        L.cs_out = c->grad + c->boff[l];
        L.cs_rows = batch;
        L.cs_cols = out;
        e = gemm(c, L);
        cur = 1 - cur;
    }
    return e == cudaSuccess ? PIC_OK : fail(c, PIC_ERR_CUDA, "backward", e);
}

pic_status mlp_get_grads(mlp_ctx* c, float* host) {
    if (!c || !host) return PIC_ERR_ARG;
    cudaError_t e =
        cudaMemcpyAsync(host, c->grad, sizeof(float) * (size_t)c->n_params, cudaMemcpyDeviceToHost, c->stream);
    return e == cudaSuccess ? sync_checked(c, "get grads") : fail(c, PIC_ERR_CUDA, "get grads", e);
}

pic_status mlp_adam(mlp_ctx* c, float lr, float beta1, float beta2, float eps) {
    if (!c || !(lr >= 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) return PIC_ERR_ARG;
    c->step += 1;
    const float c1 = (float)(1.0 - std::pow((double)beta1, (double)c->step));
    const float c2 = (float)(1.0 - std::pow((double)beta2, (double)c->step));
    cudaError_t e = launch_pdl(c, k_adam, param_grid(c), 256, 0, c->map, c->p, c->grad, c->m, c->v, c->w16, lr, beta1,
                               beta2, eps, c1, c2);
    return e == cudaSuccess ? PIC_OK : fail(c, PIC_ERR_CUDA, "adam", e);
}

pic_status mlp_train_step(mlp_ctx* c, int32_t batch, const float* x, const float* t, float lr, float* loss) {
    pic_status s = mlp_loss_grad(c, batch, x, t, loss);
    if (s != PIC_OK) return s;
    return mlp_adam(c, lr, 0.9f, 0.999f, 1e-8f);
}

pic_status mlp_sync(mlp_ctx* c) {
    if (!c) return PIC_ERR_ARG;
    return sync_checked(c, "synchronize");
}

void mlp_destroy(mlp_ctx* c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    for (void* q : c->allocs) cudaFree(q);
    if (c->h_err) cudaFreeHost(c->h_err);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
    delete c;
}

const char* mlp_last_error(const mlp_ctx* c) { return c ? c->err.c_str() : "null context"; }

}  // extern "C"

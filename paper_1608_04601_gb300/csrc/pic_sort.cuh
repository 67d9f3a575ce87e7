// pic_sort.cuh -- pieces of the stable counting sort by cell that the context sort (pic_kernels.cu) and
// the allocation-free one (pic_noalloc.cu) share: the tile shape, ranks within a warp, the scans of the
// tile counts and of the cell totals.
#pragma once
#include "pic_internal.h"

namespace pic {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int SORT_BLOCK = 512, SORT_NW = SORT_BLOCK / 32, SORT_R = 8, SORT_TILE = SORT_BLOCK * SORT_R;

// Ranks of a row of 32 slots among the equal cells of its warp so far, and the warp's counters (16 bits per
// cell) advanced. k >= N: not placed. Returns the rank.
__device__ __forceinline__ unsigned row_rank(unsigned short* W, unsigned k, unsigned N, int lane, unsigned lt) {
    const unsigned k0 = __shfl_sync(FULL, k, 0);
    unsigned rank = 0;
    if (__all_sync(FULL, k == k0)) {  // the rule on a nearly sorted store of slow particles
        if (k0 < N) {
            rank = W[k0] + lane;
            __syncwarp();
            if (lane == 31) W[k0] = (unsigned short)(rank + 1);
        }
    } else {
        const unsigned peers = __match_any_sync(FULL, k);
        const unsigned b = k < N ? W[k] : 0u;
        if (k < N) rank = b + __popc(peers & lt);
        __syncwarp();  // of the whole warp: one per group of equal cells runs as many times as there are groups
        if (k < N && lane == __ffs(peers) - 1) W[k] = (unsigned short)(b + __popc(peers));
    }
    __syncwarp();
    return rank;
}

// Exclusive scan of one store's N row totals in place -> the first slot of every cell (1024
// threads; the totals were written by other CTAs of the same grid, so they are read from L2).
__device__ __forceinline__ void cells_scan(unsigned* a, int N) {
    __shared__ unsigned s_v[MAXN];
    __shared__ unsigned s_w[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int j = tid; j < N; j += 1024) s_v[j] = __ldcg(a + j);
    __syncthreads();
    const int per = (N + 1023) / 1024, lo = tid * per, hi = min(N, lo + per);
    unsigned run = 0;
    for (int j = lo; j < hi; ++j) run += s_v[j];
    unsigned x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const unsigned w = s_w[lane];
        unsigned y = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(FULL, y, o);
            if (lane >= o) y += t;
        }
        s_w[lane] = y - w;
    }
    __syncthreads();
    unsigned e = s_w[warp] + x - run;
    for (int j = lo; j < hi; ++j) {
        const unsigned v = s_v[j];
        a[j] = e;
        e += v;
    }
}

// CTA x of ceil(N / 32) of a store, 1024 threads: exclusive scan over the tiles, in place, of the counts
// H[t N + c] of the cells 32 x .. 32 x + 31 (lane = cell, each warp a contiguous range of tiles, so rows are
// read 128 bytes at a time, eight in flight); row totals to tot. The last CTA of the store (*done counts
// them; it is left at 0) turns the totals into the first slot of every cell.
__device__ __forceinline__ void sort_rows(unsigned* __restrict__ H, unsigned Ts, int N, unsigned* __restrict__ tot,
                                          unsigned* done) {
    __shared__ unsigned s_sum[32][33];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
    const unsigned per = (Ts + 31) / 32, t0 = min(Ts, warp * per), t1 = min(Ts, t0 + per);
    unsigned sum = 0;
    if (c < N) {
#pragma unroll 8
        for (unsigned t = t0; t < t1; ++t) sum += H[(size_t)t * N + c];
    }
    s_sum[warp][lane] = sum;
    __syncthreads();
    unsigned pre = 0;
    for (int w = 0; w < warp; ++w) pre += s_sum[w][lane];
    if (warp == 31 && c < N) tot[c] = pre + sum;
    if (c < N)
        for (unsigned t = t0; t < t1; t += 8) {
            unsigned v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = t + q < t1 ? H[(size_t)(t + q) * N + c] : 0u;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (t + q < t1) H[(size_t)(t + q) * N + c] = pre;
                pre += v[q];
            }
        }
    if (warp == 31) __threadfence();  // this CTA's totals, before its count
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == (unsigned)((N + 31) / 32 - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    cells_scan(tot, N);
    if (threadIdx.x == 0) *done = 0;
}

}  // namespace pic

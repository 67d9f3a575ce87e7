// pic_noalloc.cu -- pic_sort_noalloc: the stable sort by cell of one particle
// store, on buffers the caller owns, with no device allocation at all.
//
// Some callers cannot allocate device memory while they run: code that keeps
// its own arena and forbids cudaMalloc/cudaFree (which synchronise the device
// and may fail late), plug-ins that only receive device pointers from a host
// framework, and long-running services that must not fragment or grow memory.
// For them this entry point takes its scratch (per-tile cell counts and cell
// starts) from a fixed array compiled into the library, so a call allocates
// nothing. The array (PIC_NOALLOC_SCRATCH_BYTES) is held by every GPU that
// loads the library until the process exits.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../../include/pic.h"
#include "pic_sort.cuh"

namespace {

using namespace pic;

constexpr long long NA_WORDS = PIC_NOALLOC_SCRATCH_BYTES / 4;

// Shared scratch of every call: [0, N) cell starts, then N x tiles counts (tile-major); the CTAs of the row
// scan that have finished (0 between calls).
static __device__ __align__(256) unsigned g_sort_scratch[NA_WORDS];
static __device__ unsigned g_sort_done;

struct alignas(32) D4 {
    double x, y, z, w;
};

std::mutex g_mu;
void* g_scratch_addr[256] = {};

// Three kernels: tile counts, their scans (sort_rows), scatter. No scratch holds the ranks, so the scatter
// forms them again from the cells. Each waits for the one before it. Bounded by latency at 1e6 particles: the
// loads of a warp's eight rows go out together. 1e6 particles in 512 cells, nearly sorted: 37 -> 21 us a call, in
// random order 55 -> 33 (before: four kernels, one row's loads at a time, two passes over the cells in the
// scatter). The scatter reads a tile's offsets through L1 (plain loads of unrestricted pointers: the row scan
// may still write them when this grid starts); asking L2 for each slot took 61 us in random order.
__global__ void __launch_bounds__(SORT_BLOCK) na_count(const int32_t* __restrict__ c, long long n, int N,
                                                       unsigned* __restrict__ hist, long long Ts) {
    extern __shared__ unsigned s_c[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) g_sort_done = 0;
    for (long long t = blockIdx.x; t < Ts; t += gridDim.x) {
        for (int j = threadIdx.x; j < N; j += SORT_BLOCK) s_c[j] = 0;
        const long long b = t * SORT_TILE + warp * (32 * SORT_R) + lane;
        unsigned k[SORT_R];
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) k[r] = b + 32 * r < n ? (unsigned)c[b + 32 * r] : 0xFFFFFFFFu;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) {
            const unsigned k0 = __shfl_sync(FULL, k[r], 0);
            const bool same = __all_sync(FULL, k[r] == k0);
            if (k[r] < (unsigned)N && (!same || lane == 0)) atomicAdd(&s_c[k[r]], same ? 32u : 1u);
        }
        __syncthreads();
        for (int j = threadIdx.x; j < N; j += SORT_BLOCK) hist[t * N + j] = s_c[j];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) na_rows(unsigned* __restrict__ hist, unsigned Ts, int N, unsigned* __restrict__ tot) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    sort_rows(hist, Ts, N, tot, &g_sort_done);
}

// Per tile: ranks of a warp's slots among its equal cells, prefix of the counts over the warps, placement.
template <typename R>
__global__ void __launch_bounds__(SORT_BLOCK, 2) na_scatter(const int32_t* __restrict__ cs, const R* __restrict__ ps,
                                                         int32_t* __restrict__ cd, R* __restrict__ pd, long long n,
                                                         int N, const unsigned* hist, const unsigned* cstart,
                                                         long long Ts) {
    extern __shared__ __align__(16) unsigned short s_w[];  // [SORT_NW][nw2]
    constexpr int B = sizeof(R) == 16 ? SORT_R / 2 : SORT_R / 4;  // records in flight (at 64 registers)
    const int nw2 = (N + 1) / 2 * 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned short* W = s_w + warp * nw2;
    for (long long t = blockIdx.x; t < Ts; t += gridDim.x) {
        const long long b = t * SORT_TILE + warp * (32 * SORT_R) + lane;
        unsigned k[SORT_R];
        R rec[B];
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) k[r] = b + 32 * r < n ? (unsigned)cs[b + 32 * r] : 0xFFFFu;
#pragma unroll
        for (int r = 0; r < B; ++r)
            if (b + 32 * r < n) rec[r] = ps[b + 32 * r];
        for (int j = tid; j < SORT_NW * nw2 / 2; j += SORT_BLOCK) reinterpret_cast<unsigned*>(s_w)[j] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < SORT_R; ++r) {
            if (k[r] >= (unsigned)N) k[r] = 0xFFFFu;  // past the store, or a cell out of range: not placed
            k[r] |= row_rank(W, k[r], N, lane, lt) << 16;
        }
        __syncthreads();
        for (int j = tid; j < nw2 / 2; j += SORT_BLOCK) {  // two cells per word
            unsigned run = 0;
#pragma unroll
            for (int w = 0; w < SORT_NW; ++w) {
                unsigned* p = reinterpret_cast<unsigned*>(s_w + w * nw2) + j;
                const unsigned v = *p;
                *p = run;
                run += v;
            }
        }
        // the counts of the tile before it and the first slots come from the row scan
        if (t == blockIdx.x) asm volatile("griddepcontrol.wait;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int r0 = 0; r0 < SORT_R; r0 += B) {
            unsigned o[B];
#pragma unroll
            for (int q = 0; q < B; ++q) {
                const unsigned c = k[r0 + q] & 0xFFFFu;
                o[q] = c < (unsigned)N ? cstart[c] + hist[t * N + c] + W[c] + (k[r0 + q] >> 16) : 0xFFFFFFFFu;
                if (r0 > 0 && b + 32 * (r0 + q) < n) rec[q] = ps[b + 32 * (r0 + q)];
            }
#pragma unroll
            for (int q = 0; q < B; ++q)
                if ((long long)o[q] < n) {
                    cd[o[q]] = (int)(k[r0 + q] & 0xFFFFu);
                    pd[o[q]] = rec[q];
                }
        }
        __syncthreads();
    }
}

// Launch that may begin while the kernel before it finishes (it waits itself).
template <typename... KArgs, typename... Args>
cudaError_t launch_after(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Device address of the scratch array for the current device, looked up once
// per device (the host-side name of a __device__ array is not its address).
pic_status scratch_address(unsigned** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return PIC_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_sort_scratch) != cudaSuccess || !p) return PIC_ERR_CUDA;
        g_scratch_addr[dev] = p;
    }
    *out = static_cast<unsigned*>(g_scratch_addr[dev]);
    return PIC_OK;
}

template <typename R>
pic_status run_sort(const int32_t* c_in, const void* rec_in, int32_t* c_out, void* rec_out, long long n, int N,
                    cudaStream_t st, unsigned* scratch) {
    const long long Ts = (n + SORT_TILE - 1) / SORT_TILE;
    unsigned* cstart = scratch;
    unsigned* hist = scratch + N;
    int dev = 0, sms = 1;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return PIC_ERR_CUDA;
    const int grid = (int)(Ts < 3LL * sms ? Ts : 3LL * sms);
    const size_t smem = 2 * (size_t)SORT_NW * ((N + 1) / 2 * 2);
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(na_scatter<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return PIC_ERR_CUDA;
    // each launch is checked on its own, so that a failure is reported by the launch that caused it
    na_count<<<grid, SORT_BLOCK, sizeof(unsigned) * N, st>>>(c_in, n, N, hist, Ts);
    if (cudaGetLastError() != cudaSuccess) return PIC_ERR_CUDA;
    if (launch_after(na_rows, (N + 31) / 32, 1024, 0, st, hist, (unsigned)Ts, N, cstart) != cudaSuccess) return PIC_ERR_CUDA;
    if (launch_after(na_scatter<R>, grid, SORT_BLOCK, smem, st, c_in, static_cast<const R*>(rec_in), c_out,
                     static_cast<R*>(rec_out), n, N, hist, cstart, Ts) != cudaSuccess)
        return PIC_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

}  // namespace

extern "C" pic_status pic_sort_noalloc(const int32_t* c_in, const void* rec_in, int32_t* c_out, void* rec_out,
                                       int64_t n, int32_t n_cells, int32_t precision, void* cuda_stream) {
    if (n < 0 || n_cells < 1 || n_cells > PIC_MAX_CELLS || (precision != PIC_FP32 && precision != PIC_FP64))
        return PIC_ERR_ARG;
    if (n > 0 && (!c_in || !rec_in || !c_out || !rec_out)) return PIC_ERR_ARG;
    // the kernels move records as float4 (16 bytes) or as 32-byte groups of four doubles, and cells
    // as int32: a misaligned buffer is rejected here, before any launch
    const size_t rec_align = precision == PIC_FP64 ? sizeof(D4) : sizeof(float4);
    if (n > 0 && (!aligned(rec_in, rec_align) || !aligned(rec_out, rec_align) || !aligned(c_in, 4) ||
                  !aligned(c_out, 4)))
        return PIC_ERR_ARG;
    const long long tiles = (n + SORT_TILE - 1) / SORT_TILE;
    if ((long long)n_cells + (long long)n_cells * tiles > NA_WORDS) return PIC_ERR_CAPACITY;
    // an error left over from the caller's earlier work is not this call's: report it without
    // clearing it and launch nothing
    if (n > 0 && cudaPeekAtLastError() != cudaSuccess) return PIC_ERR_CUDA;
    unsigned* scratch = nullptr;
    pic_status s = scratch_address(&scratch);
    if (s != PIC_OK || n == 0) return s;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (precision == PIC_FP64) return run_sort<D4>(c_in, rec_in, c_out, rec_out, n, n_cells, st, scratch);
    return run_sort<float4>(c_in, rec_in, c_out, rec_out, n, n_cells, st, scratch);
}

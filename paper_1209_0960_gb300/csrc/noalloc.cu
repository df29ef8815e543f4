// amg_residual_norm_noalloc: ||b - A x||_2 for a CSR matrix in device memory,
// computed without allocating any memory.
//
// Why: some callers cannot call cudaMalloc at the point where they need a
// residual check.  cudaMalloc and cudaFree may synchronise the whole device,
// which a latency-bound loop sharing the GPU with other streams cannot afford;
// an allocator hook or callback must not re-enter the allocator; and a
// process that has handed all device memory to a pool it does not control has
// nothing left to allocate from.  This entry point needs no context and no
// allocation: the per-block partial sums of its deterministic two-stage
// reduction live in a fixed file-scope device array.
//
// The array holds kMaxBlocks partial sums, one per 256 rows where a thread takes
// a row (the other kernel has at most five blocks per SM), so matrices of up to
// kMaxBlocks * 256 = 16,777,216 rows are accepted and larger ones are rejected
// with AMG_EINVAL.  Every GPU that loads the library holds the array (512 KiB
// plus a counter) until the process exits.  All calls share it and it keeps the
// last call's contents; each call clears the arrival counter before its kernel
// runs.  Calls that overlap on the GPU (concurrent streams, or several host
// threads) race on the array and must be serialised by the caller.
//
// Set-up: the first call on each device looks up the array's device address
// with cudaGetSymbolAddress while that device is current, and caches it for
// the life of the process (a device reset invalidates it).
//
// Every pointer argument is checked with cudaPointerGetAttributes (a query,
// not an allocation): it must be device or managed memory of the current
// device, else the call returns AMG_EINVAL before anything is launched.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "device.h"
#include "device_util.cuh"
#include "row_tiles.h"

namespace amg {

namespace {

constexpr int kNaBlock = 256;
constexpr int kMaxBlocks = 65536;
constexpr int64_t kMaxRows = (int64_t)kMaxBlocks * kNaBlock;
constexpr int kMaxDevices = 64;

struct NoAllocScratch {
    double partial[kMaxBlocks];   // one partial sum per block
    unsigned int counter;         // blocks finished; reset by the last one and before each call
};

static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

std::mutex g_scratch_mu;
NoAllocScratch* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once
// per device; the symbol's host-side name is not a device address).
NoAllocScratch* scratch_for_current_device() {
    int dev = 0;
    AMG_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) throw Error{AMG_EINVAL, "device index out of range"};
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess)
            throw Error{AMG_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e)};
        g_scratch_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    return g_scratch_ptr[dev];
}

// Reject anything but device or managed memory: a host pointer handed to the
// kernel would fault or read the wrong memory.  Returns the device that owns
// device memory, -1 for managed memory (reachable from every device).
int device_of_pointer(const void* p, const char* name) {
    cudaPointerAttributes at{};
    const cudaError_t e = cudaPointerGetAttributes(&at, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw Error{AMG_EINVAL, std::string(name) + ": cannot query the pointer (" +
                                    cudaGetErrorString(e) + ")"};
    }
    if (at.type == cudaMemoryTypeManaged) return -1;
    if (at.type != cudaMemoryTypeDevice) throw Error{AMG_EINVAL, std::string(name) + " is not device memory"};
    return at.device;
}

constexpr int kNaWarps = kNaBlock / 32;

// The sum of v over all threads: per block in a fixed order, then the last block
// to finish adds the block sums in index order and writes the square root.
__device__ __forceinline__ void finish_norm(double v, NoAllocScratch* __restrict__ scratch,
                                            double* __restrict__ out) {
    __shared__ double sh[kNaWarps];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double q = 0.0;
        for (int w = 0; w < kNaWarps; ++w) q += sh[w];
        scratch->partial[blockIdx.x] = q;
        __threadfence();
        last = atomicAdd(&scratch->counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    double a = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kNaBlock) a += __ldcg(scratch->partial + i);
    for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    __syncthreads();
    if (lane == 0) sh[warp] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double q = 0.0;
        for (int w = 0; w < kNaWarps; ++w) q += sh[w];
        *out = sqrt(q);
        scratch->counter = 0u;
    }
}

// ||b - A x||^2 over the rows, a warp per 32 consecutive rows at a time.
//
// One thread per row reading its CSR row directly touches a different line per
// lane and entry, and summing the squares of every 32 rows costs five warp-wide
// float64 additions where the rows themselves cost eight: on GB300, whose
// float64 pipe takes about as long for this kernel as HBM does, that was half
// the copy rate (97 us for 3.0M rows, 312 MB; now 81 us).  Here the entries of a
// warp's 32 rows, which are contiguous, are copied line by line into shared memory
// with cp.async, the next 32 rows' while the current ones are summed, and each
// thread adds its squares over all its rows before one reduction per block at the
// end.
// Every row is still b_i - A_i0 x_0 - ... in stored order.
//
// Rows are read in tiles of kNaTile entries per warp (row_tiles.h): 32 rows of a
// 7-point stencil.
__device__ __forceinline__ void copy_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__global__ void __launch_bounds__(kNaBlock) k_csr_residual_norm(
    int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
    const double* __restrict__ va, const double* __restrict__ b, const double* __restrict__ x,
    NoAllocScratch* __restrict__ scratch, double* __restrict__ out) {
    __shared__ double sv[kNaWarps][2][kNaTile];
    __shared__ int32_t sc[kNaWarps][2][kNaTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int groups = (n + 31) >> 5, stride = (int)gridDim.x * kNaWarps;
    const int g0 = (int)blockIdx.x * kNaWarps + warp;
    // the entries [k0, k1) of this lane's row in group g (empty past the matrix)
    auto row_range = [&](int g, int& k0, int& k1) {
        const int64_t row = (int64_t)g * 32 + lane;
        k0 = g < groups ? rp[min(row, (int64_t)n)] : 0;
        k1 = g < groups ? rp[min(row + 1, (int64_t)n)] : 0;
    };
    // copy the entries [s, min(s + kNaTile, e)) into buffer `buf`
    auto fetch = [&](int buf, int s, int e) {
        const int m = min(kNaTile, e - s);
        for (int i = lane; i < m; i += 32) {
            copy_async8(&sv[warp][buf][i], va + s + i);
            copy_async4(&sc[warp][buf][i], ci + s + i);
        }
    };
    double acc = 0.0;
    int k0, k1, k0n, k1n;
    row_range(g0, k0, k1);
    row_range(g0 + stride, k0n, k1n);
    int s = __shfl_sync(0xffffffffu, k0, 0), e = __shfl_sync(0xffffffffu, k1, 31);
    fetch(0, s, e);
    copy_commit();
    int buf = 0;
    for (int g = g0; g < groups; g += stride, buf ^= 1) {
        const int row = g * 32 + lane;
        const int sn = __shfl_sync(0xffffffffu, k0n, 0), en = __shfl_sync(0xffffffffu, k1n, 31);
        fetch(buf ^ 1, sn, en);   // nothing past the last group
        copy_commit();
        int k0f, k1f;
        row_range(g + 2 * stride < groups ? g + 2 * stride : groups, k0f, k1f);
        double t = row < n ? b[row] : 0.0;
        copy_wait<1>();
        __syncwarp();
        int k = max(k0, s);   // (never left of the tile, also for a malformed row_ptr)
        RowTiles tile(s, e);
        for (;;) {
            const int base = tile.base, end = tile.end_in_tile(k1);
#pragma unroll 4
            for (; k < end; ++k)
                t = __fma_rn(-sv[warp][buf][k - base], x[sc[warp][buf][k - base]], t);
            if (!tile.next()) break;
            __syncwarp();
            fetch(buf, tile.base, e);
            copy_commit();
            copy_wait<0>();
            __syncwarp();
        }
        acc = __fma_rn(t, t, acc);
        __syncwarp();   // the buffer is filled again in the next round
        k0 = k0n, k1 = k1n, k0n = k0f, k1n = k1f, s = sn, e = en;
    }
    finish_norm(acc, scratch, out);
}

// The same norm with one thread per row reading its CSR row directly: rows of
// more than kNaTile / 32 entries on the mean.  There a tile holds the rows of a
// few lanes only, the float64 pipe takes a warp's instruction at the same rate
// however few of its lanes are active, and the tiles after a group's first are
// waited for.  A longer row also uses more of each line it touches.  Tiled
// kernel against this one (GB300): 27 entries a row, 2.1M rows 415 against 232 us
// and 262k rows 66 against 38; 12.5 a row, 300k rows 34.5 against 29; 9 a row, 1M
// rows 53 against 47; the other way round 7 a row, 3.0M rows 81 against 97; 5 a
// row, 1M rows 26 against 37; 3 a row, 3M rows 48 against 75; rows of uneven
// length, 5.9 a row on the mean, 300k rows 20.7 against 21.8.
__global__ void __launch_bounds__(kNaBlock) k_csr_residual_norm_rows(
    int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
    const double* __restrict__ va, const double* __restrict__ b, const double* __restrict__ x,
    NoAllocScratch* __restrict__ scratch, double* __restrict__ out) {
    const int row = blockIdx.x * kNaBlock + threadIdx.x;
    double v = 0.0;
    if (row < n) {
        double t = b[row];
        for (int k = rp[row]; k < rp[row + 1]; ++k) t = __fma_rn(-va[k], x[ci[k]], t);
        v = t * t;
    }
    finish_norm(v, scratch, out);
}

}  // namespace
}  // namespace amg

using namespace amg;

extern "C" int amg_residual_norm_noalloc(const amg_csr* A, const double* b_dev,
                                         const double* x_dev, double* norm_dev,
                                         void* cuda_stream) {
    try {
        if (!A || !b_dev || !x_dev || !norm_dev) throw Error{AMG_EINVAL, "null argument"};
        if (!A->on_device) throw Error{AMG_EINVAL, "the matrix must be in device memory (on_device = 1)"};
        if (A->n <= 0 || !A->row_ptr || !A->col || !A->val) throw Error{AMG_EINVAL, "empty or null matrix"};
        if ((int64_t)A->n > kMaxRows)
            throw Error{AMG_EINVAL, "n = " + std::to_string(A->n) +
                                        " exceeds the fixed scratch of this entry point (at most " +
                                        std::to_string(kMaxRows) + " rows)"};
        const void* ptrs[] = {A->row_ptr, A->col, A->val, b_dev, x_dev, norm_dev};
        const char* names[] = {"A->row_ptr", "A->col", "A->val", "b_dev", "x_dev", "norm_dev"};
        int owner[6];
        for (int k = 0; k < 6; ++k) owner[k] = device_of_pointer(ptrs[k], names[k]);
        int dev = 0;
        AMG_CUDA_TRY(cudaGetDevice(&dev));
        for (int k = 0; k < 6; ++k)
            if (owner[k] >= 0 && owner[k] != dev)
                throw Error{AMG_EINVAL, std::string(names[k]) + " belongs to device " +
                                            std::to_string(owner[k]) + ", not the current device " +
                                            std::to_string(dev)};
        NoAllocScratch* scratch = scratch_for_current_device();
        cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
        AMG_CUDA_TRY(cudaMemsetAsync(&scratch->counter, 0, sizeof(unsigned int), s));
        const int blocks = (A->n + kNaBlock - 1) / kNaBlock;   // at most kMaxBlocks
        if ((int64_t)A->nnz * 32 > (int64_t)A->n * kNaTile) {
            k_csr_residual_norm_rows<<<blocks, kNaBlock, 0, s>>>(A->n, A->row_ptr, A->col, A->val, b_dev,
                                                                 x_dev, scratch, norm_dev);
        } else {
            // as many blocks as are resident at once (five per SM by their
            // shared memory), each taking every grid-th 256 rows
            int sms = 0;
            AMG_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            const int grid = std::min(blocks, std::max(1, 5 * sms));
            k_csr_residual_norm<<<grid, kNaBlock, 0, s>>>(A->n, A->row_ptr, A->col, A->val, b_dev, x_dev,
                                                          scratch, norm_dev);
        }
        AMG_CUDA_TRY(cudaGetLastError());
        set_last_error("");
        return AMG_OK;
    } catch (const Error& e) {
        set_last_error(e.msg);
        return e.code;
    }
}

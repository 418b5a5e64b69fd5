// noalloc.cu -- one plain ST-BIEM step from caller-provided buffers, without any allocation.
//
// Some callers cannot allocate device memory at all: code that runs inside another runtime's
// memory pool, inside a stream-ordered region where a cudaMalloc would synchronise the device,
// or in a process whose allocator is owned and budgeted by someone else.  For them,
// fdph_plain_step_noalloc evaluates T_n = sum_{k <= min(n, W-1)} K_k D_{n-k} (Eq. 4) from a
// kernel tensor and a slip-rate history they already hold, and keeps its split-k partial sums
// in the file-scope array below instead of in allocated scratch.  The array lives on every GPU
// that loads the library until the process exits.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "../../include/fdph.h"
#include "internal.h"

namespace {

const int kTile = 32;          // receivers per work item
const int kSteps = 64;         // kernel steps per work item of the documented size limit
const int kWarps = 8;
const int kThreads = 32 * kWarps;

// Shared by every call on a device; each call overwrites the slots it uses.
static __device__ __align__(256) double g_noalloc_partials[FDPH_NOALLOC_MAX_PARTIALS];

std::mutex g_mu;
double* g_addr[64] = {nullptr};   // device address of the array, per device ordinal

__device__ __forceinline__ int ring_slot(long long t, int L) {
    long long r = t % L;
    return (int)(r < 0 ? r + L : r);
}

// The kernel tensor is kmax n rows (k, j) of n receivers, each read once: a stream, as long as enough of
// it is in flight (134 MB at n = W = 256: 20 us at the copy rate; the 1.7e7 FP64 multiply-adds take 27 us at
// two a clock and SM).  Work item = (receiver tile, range of rows); lane = receiver, the warps take
// contiguous parts of the range, eight rows in flight each.  The ranges are as many as fill the GPU
// (kFill CTAs), where the partial sums have room.  One item per 64 kernel steps, as before, left most
// of the GPU idle: 1000 us at n = W = 256.
__global__ void __launch_bounds__(kThreads) noalloc_partial_kernel(const double* __restrict__ K, int n, long long rows,
                                                                   const double* __restrict__ D, int hist_len,
                                                                   int step, int nsplit, double* partial) {
    __shared__ double red[kWarps][kTile];
    const int tile = blockIdx.x / nsplit, part = blockIdx.x % nsplit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = tile * kTile + lane;
    const long long w = (long long)part * kWarps + warp, nw = (long long)nsplit * kWarps;
    const long long r0 = rows * w / nw, r1 = rows * (w + 1) / nw;
    const double* Ki = K + (i < n ? i : n - 1);   // lanes past n read the last receiver, unused
    double s0 = 0.0, s1 = 0.0;
    long long k = r0 / n;
    int j = (int)(r0 - k * n);
    for (long long r = r0; r < r1; ++k, j = 0) {
        const double* Dk = D + (size_t)ring_slot((long long)step - k, hist_len) * n;
        const long long e = min(r1, (k + 1) * n);   // the rows of kernel step k
        for (; r + 8 <= e; r += 8, j += 8) {
            double x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = __ldcs(Ki + (size_t)(r + q) * n);
#pragma unroll
            for (int q = 0; q < 8; q += 2) {
                s0 = fma(x[q], Dk[j + q], s0);
                s1 = fma(x[q + 1], Dk[j + q + 1], s1);
            }
        }
        for (; r < e; ++r, ++j) s0 = fma(__ldcs(Ki + (size_t)r * n), Dk[j], s0);
    }
    red[warp][lane] = s0 + s1;
    __syncthreads();
    if (warp == 0) {
        double s = 0.0;
        for (int q = 0; q < kWarps; ++q) s += red[q][lane];
        partial[(size_t)blockIdx.x * kTile + lane] = s;   // every slot of the item is written
    }
}

// one warp per receiver
__global__ void noalloc_reduce_kernel(const double* partial, int n, int nsplit, double* T) {
    const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    cudaGridDependencySynchronize();   // the partial sums are complete
    if (i >= n) return;
    const int tile = i / kTile, q = i % kTile;
    double s = 0.0;
    for (int c = lane; c < nsplit; c += 32) s += partial[((size_t)tile * nsplit + c) * kTile + q];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) T[i] = s;
}

const int kFill = 152 * 4;   // CTAs that fill the GPU

}  // namespace

extern "C" int fdph_plain_step_noalloc(const double* K, int32_t n, int32_t W, const double* D_hist,
                                       int32_t hist_len, int32_t step, double* T, void* stream) {
    if (!K || !D_hist || !T || n <= 0 || W <= 0 || hist_len <= 0 || step < 0) {
        fdph::set_error("fdph_plain_step_noalloc: null pointer or non-positive size");
        return FDPH_E_ARG;
    }
    const int kmax = step + 1 < W ? step + 1 : W;
    if (hist_len < kmax) {
        fdph::set_error("fdph_plain_step_noalloc: hist_len must cover min(step + 1, W) steps");
        return FDPH_E_ARG;
    }
    // sizes in 64-bit arithmetic: n + kTile - 1 would overflow int32 for n near INT32_MAX
    const long long tiles = ((long long)n + kTile - 1) / kTile;
    const long long nchunks = ((long long)kmax + kSteps - 1) / kSteps;
    if (tiles * nchunks * kTile > FDPH_NOALLOC_MAX_PARTIALS) {
        fdph::set_error("fdph_plain_step_noalloc: ceil(n/32) * ceil(min(step+1, W)/64) * 32 = " +
                        std::to_string(tiles * nchunks * kTile) + " exceeds FDPH_NOALLOC_MAX_PARTIALS = " +
                        std::to_string(FDPH_NOALLOC_MAX_PARTIALS));
        return FDPH_E_ARG;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        fdph::set_error("fdph_plain_step_noalloc: no current CUDA device");
        return FDPH_E_CUDA;
    }
    double* partial = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_addr[dev]) {
            // first call on this device: host code must ask the runtime for the array's device
            // address (its host-side name is only a stand-in)
            cudaError_t e = cudaGetSymbolAddress((void**)&g_addr[dev], g_noalloc_partials);
            if (e != cudaSuccess) {
                g_addr[dev] = nullptr;
                fdph::set_error(std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
                return FDPH_E_CUDA;
            }
        }
        partial = g_addr[dev];
    }
    cudaStream_t s = (cudaStream_t)stream;
    // parts of the rows: enough to fill the GPU, at least 8 rows a warp, no more than the array holds
    const long long rows = (long long)kmax * n;
    long long nsplit = std::min((kFill + tiles - 1) / tiles, rows / (8 * kWarps));
    nsplit = std::max(1LL, std::min(nsplit, FDPH_NOALLOC_MAX_PARTIALS / (tiles * kTile)));
    noalloc_partial_kernel<<<(unsigned)(tiles * nsplit), kThreads, 0, s>>>(K, n, rows, D_hist, hist_len, step, (int)nsplit,
                                                                           partial);
    // the reduction's launch does not wait for the sums to end: its CTAs start as theirs exit, and wait on the device
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(((long long)n * 32 + kThreads - 1) / kThreads));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, noalloc_reduce_kernel, (const double*)partial, (int)n, (int)nsplit, T);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        fdph::set_error(std::string("fdph_plain_step_noalloc launch: ") + cudaGetErrorString(e));
        return FDPH_E_CUDA;
    }
    return FDPH_OK;
}

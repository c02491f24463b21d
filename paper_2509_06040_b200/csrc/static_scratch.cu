// bgrpo_reward_mse_static: the -MSE row reduction of the leaf-reward kernel for callers that cannot hand the
// library a scratch buffer.  Rows are added up in shared memory, long ones over a fixed array that is part of the
// loaded library image on every GPU, so the call needs no cudaMalloc from anybody.  The paper has no counterpart;
// this is a deployment convenience.
#include <mutex>

#include "internal.h"

namespace bgrpo {
namespace {

constexpr int kStaticVec = kChunkVec / kStreamThreads;                       // float4 per thread
constexpr int kWarps = kStreamThreads / 32;
// A row of up to kClusterCtas * kClusterChunks chunks (262 144 elements) is one thread-block cluster's, which adds it up in
// shared memory: no state outside the call, and one launch.  A longer row is cut over the whole grid; a second launch adds the
// partials up, which wait in the built-in array.  Nothing in that array has to have been left in some state by the call
// before (a ticket per row for the last CTA to add up had to be zero: calls that overlapped, though they may not, spoilt
// every later call).
constexpr int kClusterCtas = 8, kClusterChunks = 8;
constexpr size_t kPartialSlots = (BGRPO_STATIC_SCRATCH_BYTES - BGRPO_STATIC_MAX_ROWS * sizeof(unsigned int)) / sizeof(double);   // as the header states the limit

static __device__ __align__(256) unsigned char g_static_scratch[BGRPO_STATIC_SCRATCH_BYTES];     // one double per (row, chunk) of long rows

// The squared differences of one chunk, one warp's share: thread sums are float over 16 elements, double above that.
__device__ __forceinline__ void load_chunk(const float4* __restrict__ z, const float4* __restrict__ tg, int64_t D4, int chunk,
                                           float4 (&a)[kStaticVec], float4 (&t)[kStaticVec]) {
#pragma unroll
    for (int k = 0; k < kStaticVec; ++k) {      // all loads before the first use; past the row both are zero
        const int64_t e = static_cast<int64_t>(chunk) * kChunkVec + k * kStreamThreads + threadIdx.x;
        a[k] = e < D4 ? __ldcs(z + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        t[k] = e < D4 ? __ldg(tg + e) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
__device__ __forceinline__ double warp_squares(const float4 (&a)[kStaticVec], const float4 (&t)[kStaticVec]) {
    float acc = 0.0f;
#pragma unroll
    for (int k = 0; k < kStaticVec; ++k) {
        const float dx = a[k].x - t[k].x, dy = a[k].y - t[k].y, dz = a[k].z - t[k].z, dw = a[k].w - t[k].w;
        acc = fmaf(dx, dx, acc);
        acc = fmaf(dy, dy, acc);
        acc = fmaf(dz, dz, acc);
        acc = fmaf(dw, dw, acc);
    }
    double s = static_cast<double>(acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}
__device__ __forceinline__ double sum_of_warps(const double* red) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += red[w];
    return s;
}
// One warp: a row's chunks in index order within each lane, then a fixed shuffle tree; lane 0 writes the reward.
__device__ __forceinline__ void write_reward(const double* chunks, int nchunks, double inv_D, float* r) {
    const int lane = threadIdx.x & 31;
    double tot = 0.0;
    for (int c = lane; c < nchunks; c += 32) tot += chunks[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
    if (lane == 0) *r = static_cast<float>(-tot * inv_D);
}

// A cluster of p CTAs per row: CTA q takes the chunks q, q + p, ... (the next one's loads under way while one is added up)
// and leaves each chunk's sum in the shared memory of the first CTA.
__global__ void __launch_bounds__(kStreamThreads)
reward_mse_cluster_kernel(const float* __restrict__ rows, const float* __restrict__ target, float* __restrict__ r_out, int64_t D,
                          int32_t nchunks, int32_t ctas, double inv_D) {
    __shared__ double red[kClusterChunks][kWarps], s_chunk[kClusterCtas * kClusterChunks];
    pdl_release();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // every CTA of the cluster has started
    const int row = blockIdx.x / ctas, rank = blockIdx.x - row * ctas;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t D4 = D >> 2;
    const float4* __restrict__ z = reinterpret_cast<const float4*>(rows + static_cast<int64_t>(row) * D);
    const float4* __restrict__ tg = reinterpret_cast<const float4*>(target);
    pdl_wait();
    float4 a[kStaticVec], t[kStaticVec], an[kStaticVec], tn[kStaticVec];
    load_chunk(z, tg, D4, rank, a, t);
    int mine = 0;
    for (int chunk = rank; chunk < nchunks; chunk += ctas, ++mine) {
        if (chunk + ctas < nchunks) load_chunk(z, tg, D4, chunk + ctas, an, tn);
        const double s = warp_squares(a, t);
        if (lane == 0) red[mine][warp] = s;
#pragma unroll
        for (int k = 0; k < kStaticVec; ++k) { a[k] = an[k]; t[k] = tn[k]; }
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x < mine) {
        const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(&s_chunk[rank + threadIdx.x * ctas]));
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(0u));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(sum_of_warps(red[threadIdx.x])) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank == 0 && warp == 0) write_reward(s_chunk, nchunks, inv_D, r_out + row);
}

// Long rows: one CTA per (row, chunk), then one warp per row.
__global__ void __launch_bounds__(kStreamThreads)
reward_mse_chunk_kernel(const float* __restrict__ rows, const float* __restrict__ target, double* __restrict__ partials, int64_t D, int32_t nchunks) {
    __shared__ double red[kWarps];
    pdl_release();
    const int chunk = blockIdx.x % nchunks, row = blockIdx.x / nchunks;
    pdl_wait();
    float4 a[kStaticVec], t[kStaticVec];
    load_chunk(reinterpret_cast<const float4*>(rows + static_cast<int64_t>(row) * D), reinterpret_cast<const float4*>(target), D >> 2, chunk, a, t);
    const double s = warp_squares(a, t);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) partials[blockIdx.x] = sum_of_warps(red);
}
__global__ void __launch_bounds__(kStreamThreads)
reward_mse_finish_kernel(const double* __restrict__ partials, float* __restrict__ r_out, int32_t n_rows, int32_t nchunks, double inv_D) {
    pdl_release();
    pdl_wait();
    const int row = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (row < n_rows) write_reward(partials + static_cast<int64_t>(row) * nchunks, nchunks, inv_D, r_out + row);
}

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
unsigned char* g_scratch_addr[kMaxDevices] = {nullptr};

// Device address of g_static_scratch on the current device.  In host code the symbol's name is only a handle, not an
// address a kernel can use; the address is asked for once per device, with that device current, and remembered.
cudaError_t static_scratch_address(unsigned char** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = static_cast<unsigned char*>(ptr);
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace bgrpo

extern "C" {

bgrpo_status bgrpo_reward_mse_static(const float* rows_dev, const float* target_dev, int32_t n_rows, int64_t D,
                                     float* r_out_dev, void* stream) {
    using namespace bgrpo;
    if (!rows_dev || !target_dev || !r_out_dev) return BGRPO_ERR_INVALID_ARG;   // NULL pointer
    if ((reinterpret_cast<uintptr_t>(rows_dev) | reinterpret_cast<uintptr_t>(target_dev)) % 16 != 0)
        return BGRPO_ERR_INVALID_ARG;   // rows_dev and target_dev must be 16-byte aligned
    if (n_rows < 1 || D < 4 || D % 4 != 0) return BGRPO_ERR_INVALID_ARG;   // n_rows must be >= 1 and D a positive multiple of 4
    if (n_rows > BGRPO_STATIC_MAX_ROWS)
        return BGRPO_ERR_CAPACITY;   // n_rows exceeds BGRPO_STATIC_MAX_ROWS: split the call or use bgrpo_leaf_reward_mse
    const int64_t nchunks = (D / 4 + kChunkVec - 1) / kChunkVec;
    if (static_cast<uint64_t>(n_rows) * static_cast<uint64_t>(nchunks) > kPartialSlots)
        return BGRPO_ERR_CAPACITY;   // n_rows * ceil(D/4096) exceeds the built-in scratch: split the call or use bgrpo_leaf_reward_mse
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int32_t chunks = static_cast<int32_t>(nchunks);
    const double inv_D = 1.0 / static_cast<double>(D);
    cudaError_t e;
    if (chunks <= kClusterCtas * kClusterChunks) {
        const int ctas = chunks < kClusterCtas ? chunks : kClusterCtas;
        e = launch_overlapped_clusters(reward_mse_cluster_kernel, static_cast<unsigned int>(n_rows * ctas), kStreamThreads, 0, s, ctas,
                                       rows_dev, target_dev, r_out_dev, D, chunks, ctas, inv_D);
        return e == cudaSuccess ? BGRPO_OK : BGRPO_ERR_CUDA;
    }
    unsigned char* scratch = nullptr;
    e = static_scratch_address(&scratch);
    if (e != cudaSuccess) return BGRPO_ERR_CUDA;
    double* partials = reinterpret_cast<double*>(scratch);
    e = launch_overlapped(reward_mse_chunk_kernel, static_cast<unsigned int>(n_rows) * chunks, kStreamThreads, 0, s, rows_dev, target_dev, partials, D, chunks);
    if (e == cudaSuccess)
        e = launch_overlapped(reward_mse_finish_kernel, (static_cast<unsigned int>(n_rows) + kWarps - 1) / kWarps, kStreamThreads, 0, s,
                              static_cast<const double*>(partials), r_out_dev, n_rows, chunks, inv_D);
    if (e != cudaSuccess) return BGRPO_ERR_CUDA;
    return BGRPO_OK;
}

}  // extern "C"

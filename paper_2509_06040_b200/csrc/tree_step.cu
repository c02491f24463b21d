// Streaming kernels of the rollout: root initialisation, the fused gather / fork / Euler-Maruyama update /
// log-prob step (Eq. 2 and the appendix's Euler-Maruyama form).  Every latent element is read or written once,
// with 128-bit accesses, and the noise is generated in registers.
//
// Sums over a row are integers, so results do not depend on scheduling.
#include "internal.h"
#include "philox.cuh"

namespace bgrpo {
namespace {

constexpr int kVecPerThread = kChunkVec / kStreamThreads;   // 4
// ---------------------------------------------------------------------------------------------------------------
// Root: z_0 ~ N(0, I) from the ROOT stream, node-table row of the root, and a clean scratch (row sums, status).
__global__ void __launch_bounds__(kStreamThreads)
root_kernel(float* latents, int32_t* table, float* logp, unsigned long long* row_sums, int32_t* status, int64_t D,
            int32_t n_trees, int32_t nodes_cap, int32_t nchunks, uint32_t node_id_base, const __grid_constant__ PhiloxKeys keys) {
    pdl_release();
    const int chunk = blockIdx.x % nchunks;
    const int tree = blockIdx.x / nchunks;
    const int64_t D4 = D >> 2;
    if (!BGRPO_IN_BOUNDS(status, tree < n_trees && static_cast<int64_t>(chunk) * kChunkVec < D4)) return;
    float4* z = reinterpret_cast<float4*>(latents + static_cast<int64_t>(tree) * nodes_cap * D);
    const uint32_t gid = node_id_base + static_cast<uint32_t>(tree) * nodes_cap;
    float4 noise[kVecPerThread];
#pragma unroll
    for (int k = 0; k < kVecPerThread; ++k)
        noise[k] = noise4(static_cast<uint32_t>(chunk) * kChunkVec + k * kStreamThreads + threadIdx.x, gid, 0u, BGRPO_TAG_ROOT, keys);
    pdl_wait();           // the buffers may still be read by the kernels of the previous pass
#pragma unroll
    for (int k = 0; k < kVecPerThread; ++k) {
        const int64_t e = static_cast<int64_t>(chunk) * kChunkVec + k * kStreamThreads + threadIdx.x;
        if (e < D4) z[e] = noise[k];
    }
    const int64_t rows = static_cast<int64_t>(n_trees) * nodes_cap;
    if (chunk == 0) {
        for (int n = threadIdx.x; n < nodes_cap; n += kStreamThreads) row_sums[static_cast<int64_t>(tree) * nodes_cap + n] = 0ull;
        if (threadIdx.x == 0) {
            const int64_t r = static_cast<int64_t>(tree) * nodes_cap;
            table[r] = -1;
            table[rows + r] = 0;
            table[2 * rows + r] = -1;
            table[3 * rows + r] = 0;
            logp[r] = 0.0f;
            if (tree == 0) *status = 0;
        }
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Fused step.  One CTA per work item (tree, parent, chunk of kStepChunkVec float4): kStepThreads threads of kStepVec float4,
// or kStepThreadsSmall threads of half of that where the launch is less than one wave (step_threads()).
//
// A thread issues the 128-bit loads of its kStepVec float4 of the parent tile and of the operand tile (velocity or
// target mean) first, then generates the noise of all its elements - Philox and Box-Muller depend on indices only,
// so kStepVec independent chains per child are in flight while the loads travel - and only then touches the loaded
// values: mean once per parent element, then for each of the K children z' = mean + g xi (128-bit store) and the
// squares of the noise.  The parent is read once however many children it has.
//
// Log-prob: a warp adds its squares per child as integers (philox.cuh) and stores one number per (child row, chunk, warp).
// Nothing waits for those stores: the sums over chunks and warps are taken by the NEXT launch on the stream (FinalizeDesc), or
// by the flush kernel when the tree is complete, so the kernel has no fence and no atomic.  One of the launch's first CTAs adds
// a row up, behind its own loads.  (One warp per row, 16 steps of a video tree: 589 us for 574, and 605 ahead of the loads, as
// launches of one wave wait for it; the CTA of the row's own first chunk, four image trees: 161 us for 149, as the last rows'
// come in the last wave; one number per CTA, which takes a barrier at its end, 32 image trees: 1 157 us for 1 120.)
//
// FAN children per parent; SHARED: xi_b mixes a per-parent xi_0 (finite s at a split step); FULL: the tile holds
// kStepChunkVec float4, so no element needs a bounds test; NOISY = false: a deterministic step (sigma = 0) of the
// hybrid schedule, no noise is generated at all.

template <int THREADS, bool FULL>
__device__ __forceinline__ void load_tile(const float4* __restrict__ zp, const float4* __restrict__ xop, bool streamed,
                                          uint32_t vecs, float4 (&z)[kStepChunkVec / THREADS], float4 (&x)[kStepChunkVec / THREADS]) {
#pragma unroll
    for (int k = 0; k < kStepChunkVec / THREADS; ++k) {
        const uint32_t t = threadIdx.x + k * THREADS;
        if (FULL || t < vecs) {
            z[k] = __ldcs(zp + t);                                   // read once: evict first
            x[k] = streamed ? __ldcs(xop + t) : __ldg(xop + t);      // the target mean is shared by the whole level
        }
    }
}

// The noise of a parent's children for one float4 of elements; adds its squares.
template <int FAN, bool SHARED>
struct StepNoise {
    NoiseNode shared_node, node[FAN];
    __device__ __forceinline__ StepNoise(const StepLaunch& p, uint32_t gid_parent, uint32_t gid_child0) {
        if (SHARED) shared_node = noise_node(gid_parent, p.step, p.keys);
#pragma unroll
        for (int b = 0; b < FAN; ++b) node[b] = noise_node(gid_child0 + b, p.step, p.keys);
    }
    __device__ __forceinline__ void draw(const StepLaunch& p, uint32_t e, float4 (&xi)[FAN], uint32_t (&acc)[FAN]) const {
        float squares;
        float4 xi0;
        if (SHARED) xi0 = mul4(p.mix_shared, normal4(philox_from(noise_element(e, BGRPO_TAG_SHARED, p.keys), shared_node, p.keys), squares));
        const NoiseElement el = noise_element(e, BGRPO_TAG_INNOV, p.keys);
#pragma unroll
        for (int b = 0; b < FAN; ++b) {
            xi[b] = normal4(philox_from(el, node[b], p.keys), squares);
            if (SHARED) {
                xi[b] = fma4(p.mix_innov, xi[b], xi0);
                squares = squares_of(xi[b]);
            }
            // z' - mean is g xi up to the rounding of z' (relative 6e-8 of |z'|, far below the 1e-5 the log-prob
            // is good to)
            acc[b] += quantized_squares(squares);
        }
    }
};

template <int FAN, bool NOISY>
__device__ __forceinline__ void store_children(const StepLaunch& p, float4 z, float4 x, const float4 (&xi)[FAN], float4* zc, uint32_t D4) {
    const float4 m = fma4(p.ca, z, mul4(p.cb, x));
#pragma unroll
    for (int b = 0; b < FAN; ++b)       // deterministic step: the child is the mean
        zc[static_cast<size_t>(b) * D4] = NOISY ? fma4(p.g, xi[b], m) : m;
}

template <int FAN, bool SHARED, int THREADS, bool FULL, bool NOISY>
__device__ __forceinline__ void compute_tile(const StepLaunch& p, const float4 (&z)[kStepChunkVec / THREADS], const float4 (&x)[kStepChunkVec / THREADS],
                                             uint32_t vecs, uint32_t e_base, uint32_t D4, float4* zc, const StepNoise<FAN, SHARED>& noise,
                                             uint32_t (&acc)[FAN]) {
#pragma unroll
    for (int k = 0; k < kStepChunkVec / THREADS; ++k) {
        const uint32_t t = threadIdx.x + k * THREADS;
        if (FULL || t < vecs) {
            float4 xi[FAN];
            if (NOISY) noise.draw(p, e_base + t, xi, acc);
            store_children<FAN, NOISY>(p, z[k], x[k], xi, zc + e_base + t, D4);
        }
    }
}

template <int FAN, bool SHARED, bool NOISY, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == kStepThreads ? step_ctas_per_sm(FAN, SHARED) : kStepCtasPerSmSmall)
step_kernel(const __grid_constant__ StepLaunch p) {
    constexpr int kWarps = THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_release();
    // The parents, the velocity and the pending partial sums come from earlier kernels.  A launch of many waves waits for
    // them here: its loads travel while the noise is generated.
    if (THREADS == kStepThreads) pdl_wait();

    const int chunk = blockIdx.x % p.nchunks;
    const int row = blockIdx.x / p.nchunks;             // tree * W_in + j
    const int tree = row / p.W_in;
    const int j = row - tree * p.W_in;
    const uint32_t D4 = static_cast<uint32_t>(p.D >> 2);
    const uint32_t e_base = static_cast<uint32_t>(chunk) * kStepChunkVec;
    const uint32_t vecs = min(static_cast<uint32_t>(kStepChunkVec), D4 - e_base);
    const int64_t tree_row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    const int parent = p.off_in + j;
    const int child0 = p.off_out + j * FAN;
    const bool streamed = (p.v != nullptr);
    if (!BGRPO_IN_BOUNDS(p.status, tree < p.n_trees && parent < p.nodes_cap && child0 + FAN <= p.nodes_cap && e_base < D4 &&
                                       2 * (chunk + 1) * kWarps <= p.per_row)) return;
    const float4* __restrict__ zp = reinterpret_cast<const float4*>(p.latents + (tree_row0 + parent) * p.D) + e_base;
    const float4* __restrict__ xop = (streamed ? reinterpret_cast<const float4*>(p.v + static_cast<int64_t>(row) * p.D)
                                               : reinterpret_cast<const float4*>(p.mu + static_cast<int64_t>(tree) * p.D)) + e_base;
    float4* zc = reinterpret_cast<float4*>(p.latents + (tree_row0 + child0) * p.D);
    const uint32_t gid_parent = p.node_id_base + static_cast<uint32_t>(tree_row0 + parent);
    const uint32_t gid_child0 = p.node_id_base + static_cast<uint32_t>(tree_row0 + child0);

    // the parents' own log-probs, from the sums the launch before left: a row for each of the first CTAs
    __shared__ unsigned long long s_sum[kWarps];
    auto finalize_previous = [&] {
        if (p.prev.logp_out == nullptr || blockIdx.x >= p.n_trees * p.prev.W) return;
        const int t = blockIdx.x / p.prev.W;
        if (BGRPO_IN_BOUNDS(p.status, p.prev.W == p.W_in && p.prev.off == p.off_in && 2 * p.prev.per_row <= p.per_row))
            finalize_row<THREADS>(p.prev, static_cast<int64_t>(t) * p.nodes_cap + p.prev.off + (blockIdx.x - t * p.prev.W), p.half_per, threadIdx.x, s_sum);
    };
    uint32_t acc[FAN];
#pragma unroll
    for (int b = 0; b < FAN; ++b) acc[b] = 0u;
    float4 z[kStepChunkVec / THREADS], x[kStepChunkVec / THREADS];
    const StepNoise<FAN, SHARED> noise(p, gid_parent, gid_child0);
    if (THREADS == kStepThreadsSmall) {
        // A launch of less than a wave sits through the end of the kernel before it: the noise, which needs nothing but
        // indices, is drawn before the wait, and what is left behind it is a load, a few FMAs and a store (16 steps of one
        // tree of 256 tokens, each after the MLP stage: 249 -> 235 us for the pass).
        float4 xi[kStepChunkVec / THREADS][FAN];
        if (NOISY) {
#pragma unroll
            for (int k = 0; k < kStepChunkVec / THREADS; ++k)
                if (threadIdx.x + k * THREADS < vecs) noise.draw(p, e_base + threadIdx.x + k * THREADS, xi[k], acc);
        }
        pdl_wait();
        load_tile<THREADS, false>(zp, xop, streamed, vecs, z, x);
        finalize_previous();
#pragma unroll
        for (int k = 0; k < kStepChunkVec / THREADS; ++k) {
            const uint32_t t = threadIdx.x + k * THREADS;
            if (t < vecs) store_children<FAN, NOISY>(p, z[k], x[k], xi[k], zc + e_base + t, D4);
        }
    } else if (vecs == kStepChunkVec) {
        load_tile<THREADS, true>(zp, xop, streamed, vecs, z, x);
        finalize_previous();
        compute_tile<FAN, SHARED, THREADS, true, NOISY>(p, z, x, vecs, e_base, D4, zc, noise, acc);
    } else {
        load_tile<THREADS, false>(zp, xop, streamed, vecs, z, x);
        finalize_previous();
        compute_tile<FAN, SHARED, THREADS, false, NOISY>(p, z, x, vecs, e_base, D4, zc, noise, acc);
    }
    // one number per (child row, chunk, warp): a lane's sum takes up to 30 bits, so its halves are added apart
#pragma unroll
    for (int b = 0; b < FAN; ++b) {
        const uint32_t lo = __reduce_add_sync(0xffffffffu, acc[b] & 0xffffu), hi = __reduce_add_sync(0xffffffffu, acc[b] >> 16);
        if (lane == 0)
            p.partials[(tree_row0 + child0 + b) * (p.per_row >> 1) + chunk * kWarps + warp] = (static_cast<unsigned long long>(hi) << 16) + lo;
    }
    if (chunk == 0 && threadIdx.x < FAN) {      // node-table rows of the new children
        const int b = threadIdx.x;
        const int64_t rows = static_cast<int64_t>(p.n_trees) * p.nodes_cap;
        const int64_t r = tree_row0 + child0 + b, rp = tree_row0 + parent;
        p.table[r] = parent;
        p.table[rows + r] = p.step + 1;
        p.table[2 * rows + r] = p.is_split ? p.step : p.table[2 * rows + rp];
        p.table[3 * rows + r] = p.is_split ? b : p.table[3 * rows + rp];
    }
}

// Flush: adds up a pending level outside a step launch (the tree is complete, or its record is saved): THREADS threads per row.
template <int THREADS>
__global__ void __launch_bounds__(kStreamThreads)
finalize_kernel(const FinalizeDesc f, int32_t n_trees, int32_t nodes_cap, double half_per, int32_t* status, int32_t per_row_cap) {
    __shared__ unsigned long long s_sum[kStreamThreads / 32];
    pdl_release();
    pdl_wait();
    const int idx = blockIdx.x * (kStreamThreads / THREADS) + threadIdx.x / THREADS;
    if (idx >= n_trees * f.W) return;
    const int tree = idx / f.W;
    if (!BGRPO_IN_BOUNDS(status, f.off + f.W <= nodes_cap && 2 * f.per_row <= per_row_cap)) return;
    finalize_row<THREADS>(f, static_cast<int64_t>(tree) * nodes_cap + f.off + (idx - tree * f.W), half_per, threadIdx.x % THREADS, s_sum);
}

__global__ void philox_words_kernel(const __grid_constant__ PhiloxKeys keys, uint32_t node, uint32_t step, uint32_t tag, uint4* out, int64_t nblk) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < nblk) out[i] = philox4x32_10(make_uint4(static_cast<uint32_t>(i), node, step, tag), keys);
}
__global__ void philox_normals_kernel(const __grid_constant__ PhiloxKeys keys, uint32_t node, uint32_t step, uint32_t tag, float4* out, int64_t nblk) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < nblk) out[i] = noise4(static_cast<uint32_t>(i), node, step, tag, keys);
}

__global__ void debug_trip_kernel(int32_t* status) {
    if (!BGRPO_IN_BOUNDS(status, threadIdx.x > 0)) return;      // thread 0 fails the test; nothing is accessed
}

template <int FAN, int THREADS>
cudaError_t launch_step_fan(const StepLaunch& p, unsigned int grid, cudaStream_t s) {
    if (p.g == 0.0f) return launch_overlapped(step_kernel<FAN, false, false, THREADS>, grid, THREADS, 0, s, p);     // ODE step
    if (p.shared_noise) return launch_overlapped(step_kernel<FAN, true, true, THREADS>, grid, THREADS, 0, s, p);
    return launch_overlapped(step_kernel<FAN, false, true, THREADS>, grid, THREADS, 0, s, p);
}
template <int THREADS>
cudaError_t launch_step_threads(const StepLaunch& p, unsigned int grid, cudaStream_t s) {
    switch (p.fan) {
        case 1: return launch_step_fan<1, THREADS>(p, grid, s);
        case 2: return launch_step_fan<2, THREADS>(p, grid, s);
        case 3: return launch_step_fan<3, THREADS>(p, grid, s);
        case 4: return launch_step_fan<4, THREADS>(p, grid, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_debug_trip(int32_t* status, cudaStream_t s) {
    debug_trip_kernel<<<1, 32, 0, s>>>(status);
    return count_launch(cudaGetLastError());
}

cudaError_t launch_root(const bgrpo_tree* t, cudaStream_t s) {
    const unsigned int grid = static_cast<unsigned int>(t->desc.n_trees) * t->nchunks;
    return launch_overlapped(root_kernel, grid, kStreamThreads, 0, s, t->buf.latents, t->buf.node_table, t->buf.logp, t->row_sums,
                             t->status, t->D, t->desc.n_trees, t->desc.nodes_cap, t->nchunks,
                             static_cast<uint32_t>(t->desc.tree_id_base * t->desc.nodes_cap), make_philox_keys(t->desc.seed));
}

cudaError_t launch_step(const StepLaunch& p0, cudaStream_t s) {
    StepLaunch p = p0;
    p.half_per = logp_half_per(p.D);
    const int64_t items = static_cast<int64_t>(p.n_trees) * p.W_in * p.nchunks;
    if (items <= 0 || items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const unsigned int grid = static_cast<unsigned int>(items);
    return step_threads(items) == kStepThreads ? launch_step_threads<kStepThreads>(p, grid, s) : launch_step_threads<kStepThreadsSmall>(p, grid, s);
}

cudaError_t launch_finalize(const bgrpo_tree* t, const FinalizeDesc& f, cudaStream_t s) {
    const int rows = t->desc.n_trees * f.W, row_threads = f.per_row >= 512 ? kStreamThreads : 32;
    const int grid = (rows + kStreamThreads / row_threads - 1) / (kStreamThreads / row_threads);
    return launch_overlapped(row_threads == 32 ? finalize_kernel<32> : finalize_kernel<kStreamThreads>, grid < 1 ? 1 : grid, kStreamThreads, 0, s, f,
                             t->desc.n_trees, t->desc.nodes_cap, logp_half_per(t->D), t->status, static_cast<int32_t>(partials_per_row(t->D)));
}

cudaError_t launch_philox_words(uint64_t seed, uint32_t node, uint32_t step, uint32_t tag, uint32_t* out, int64_t nblk, cudaStream_t s) {
    if (nblk <= 0) return cudaSuccess;
    philox_words_kernel<<<static_cast<unsigned int>((nblk + 255) / 256), 256, 0, s>>>(
        make_philox_keys(seed), node, step, tag, reinterpret_cast<uint4*>(out), nblk);
    return count_launch(cudaGetLastError());
}
cudaError_t launch_philox_normals(uint64_t seed, uint32_t node, uint32_t step, uint32_t tag, float* out, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t nblk = n / 4;
    philox_normals_kernel<<<static_cast<unsigned int>((nblk + 255) / 256), 256, 0, s>>>(
        make_philox_keys(seed), node, step, tag, reinterpret_cast<float4*>(out), nblk);
    return count_launch(cudaGetLastError());
}

}  // namespace bgrpo

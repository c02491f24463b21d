// Log-probs of stored edges under a given velocity (the numerator of rho_e in Eq. 5): per edge the mean squared distance of
// the stored child from the Euler-Maruyama mean of its parent.  HBM-bound.
//
// All edges under the closed-form velocity: every latent is read once, 4 bytes per element and edge.  A CTA takes one chunk of the row for one *family*: a node, its F children and the only children below each of them down
// to the next fork.  It keeps the parent's piece in registers and walks down, so a node is read once although it is child
// of one edge and parent of the next; the next node's loads are issued before the current one is used.  A small kernel with
// one warp per row adds the chunks up.  On a video tree of 111 nodes x 2.1 M elements: 155 us (6.06 TB/s) for the whole
// tree, where one launch per level, each reading parents and children, took 290 us.
//
// One step's edges under a given velocity (12 bytes per element and edge without a fork): one CTA per parent and chunk, all
// its loads issued before the first is used.
//
// The sums of squares are float32 inside a warp's elements of a chunk (512, or 1024 for one step's edges), double from there
// on, added in chunk order.
#include "internal.h"

namespace bgrpo {
namespace {

constexpr int kThreads = 128, kWarps = kThreads / 32;
constexpr int kVec = kLogprobChunkVec / kThreads;            // float4 per thread
constexpr int kMaxSeq = BGRPO_MAX_K * BGRPO_MAX_T;           // nodes of a family below its parent

template <bool FULL>
__device__ __forceinline__ void load(float4 (&r)[kVec], const float4* __restrict__ src, uint32_t vecs) {
#pragma unroll
    for (int k = 0; k < kVec; ++k) {
        const uint32_t t = threadIdx.x + k * kThreads;
        r[k] = (FULL || t < vecs) ? __ldcs(src + t) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// The family below a node of depth d0: children b = 0 .. fan-1 (index j0 + b of depth d0 + 1), each followed by len - 1
// only children.  Pieces past the row are zero everywhere and add nothing.
template <bool FULL>
__device__ __forceinline__ void walk(const LogprobLaunch& p, const float4* __restrict__ zp, const float4* __restrict__ xp, uint32_t vecs,
                                     const float4* __restrict__ tree_base, size_t D4, uint32_t e_base, int d0, int j0, int fan, int len,
                                     float (*acc_out)[kWarps]) {
    float4 parent[kVec], x[kVec], prev[kVec], cur[kVec], next[kVec];
    auto node = [&](int i) {       // node i of the family: child i / len, depth d0 + 1 + i % len
        const int b = i / len, d = i - b * len;
        return tree_base + static_cast<size_t>(p.off[d0 + 1 + d] + j0 + b) * D4 + e_base;
    };
    load<FULL>(cur, node(0), vecs);
    load<FULL>(parent, zp, vecs);
    load<FULL>(x, xp, vecs);
    const int n = fan * len;
    for (int i = 0, d = 0; i < n; ++i) {
        if (i + 1 < n) load<FULL>(next, node(i + 1), vecs);
        const float ca = p.ca[d0 + d], cb = p.cb[d0 + d];
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < kVec; ++k) {
            const float4 z = d == 0 ? parent[k] : prev[k];
            const float dx = cur[k].x - fmaf(ca, z.x, cb * x[k].x), dy = cur[k].y - fmaf(ca, z.y, cb * x[k].y);
            const float dz = cur[k].z - fmaf(ca, z.z, cb * x[k].z), dw = cur[k].w - fmaf(ca, z.w, cb * x[k].w);
            acc = fmaf(dx, dx, acc);
            acc = fmaf(dy, dy, acc);
            acc = fmaf(dz, dz, acc);
            acc = fmaf(dw, dw, acc);
            prev[k] = cur[k];
            cur[k] = next[k];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) acc_out[i][threadIdx.x >> 5] = acc;
        if (++d == len) d = 0;
    }
}

__global__ void __launch_bounds__(kThreads, 5)
logprob_tree_kernel(const __grid_constant__ LogprobLaunch p) {
    __shared__ float s_acc[kMaxSeq][kWarps];
    pdl_release();
    pdl_wait();
    const int chunk = blockIdx.x % p.nchunks;
    int f = blockIdx.x / p.nchunks;                         // family, the last run's first (they are the longest)
    const int tree = f / p.families;
    f -= tree * p.families;
    int r = p.n_runs - 1;
    while (r > 0 && f >= p.run_families[r]) f -= p.run_families[r--];
    const int d0 = p.run_d0[r], fan = p.run_fan[r], len = p.run_len[r];
    const int j0 = f * fan;                                 // first child's index within its depth
    const uint32_t D4 = static_cast<uint32_t>(p.D >> 2);
    const uint32_t e_base = static_cast<uint32_t>(chunk) * kLogprobChunkVec;
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    const int parent = p.off[d0] + f;
    if (!BGRPO_IN_BOUNDS(p.status, tree < p.n_trees && f < p.run_families[r] && e_base < D4 && fan * len <= kMaxSeq && parent < p.off[d0 + 1] &&
                                       p.off[d0 + len] + j0 + fan <= p.nodes_cap && p.nchunks * 2 <= p.per_row)) return;
    const uint32_t vecs = min(static_cast<uint32_t>(kLogprobChunkVec), D4 - e_base);
    const float4* tree_base = reinterpret_cast<const float4*>(p.latents + row0 * p.D);
    const float4* zp = tree_base + static_cast<size_t>(parent) * D4 + e_base;
    const float4* xp = reinterpret_cast<const float4*>(p.mu + static_cast<int64_t>(tree) * p.D) + e_base;
    if (vecs == kLogprobChunkVec) walk<true>(p, zp, xp, vecs, tree_base, D4, e_base, d0, j0, fan, len, s_acc);
    else walk<false>(p, zp, xp, vecs, tree_base, D4, e_base, d0, j0, fan, len, s_acc);
    __syncthreads();
    for (int i = threadIdx.x; i < fan * len; i += kThreads) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += static_cast<double>(s_acc[i][w]);
        const int b = i / len, d = i - b * len;
        p.partials[(row0 + p.off[d0 + 1 + d] + j0 + b) * p.nchunks + chunk] = s;
    }
}

// One step's edges: parent, velocity and first child of a chunk are loaded together, further children one after the other.
constexpr int kEdgeThreads = 64, kEdgeVec = kLogprobChunkVec / kEdgeThreads, kEdgeWarps = kEdgeThreads / 32;

template <bool FULL>
__device__ __forceinline__ void score_chunk(const float4* __restrict__ zp, const float4* __restrict__ xp, const float4* __restrict__ cp, size_t D4,
                                            uint32_t vecs, int fan, float ca, float cb, double* out, int parts) {
    float4 m[kEdgeVec], x[kEdgeVec], c[kEdgeVec];
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kEdgeVec; ++k) {
        const uint32_t t = threadIdx.x + k * kEdgeThreads;
        const bool in = FULL || t < vecs;
        m[k] = in ? __ldcs(zp + t) : zero;
        x[k] = in ? __ldcs(xp + t) : zero;
        c[k] = in ? __ldcs(cp + t) : zero;
    }
#pragma unroll
    for (int k = 0; k < kEdgeVec; ++k)
        m[k] = make_float4(fmaf(ca, m[k].x, cb * x[k].x), fmaf(ca, m[k].y, cb * x[k].y), fmaf(ca, m[k].z, cb * x[k].z), fmaf(ca, m[k].w, cb * x[k].w));
    for (int b = 0; b < fan; ++b) {
        if (b > 0) {
#pragma unroll
            for (int k = 0; k < kEdgeVec; ++k) {
                const uint32_t t = threadIdx.x + k * kEdgeThreads;
                c[k] = (FULL || t < vecs) ? __ldcs(cp + b * D4 + t) : zero;
            }
        }
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < kEdgeVec; ++k) {
            const float dx = c[k].x - m[k].x, dy = c[k].y - m[k].y, dz = c[k].z - m[k].z, dw = c[k].w - m[k].w;
            acc = fmaf(dx, dx, acc);
            acc = fmaf(dy, dy, acc);
            acc = fmaf(dz, dz, acc);
            acc = fmaf(dw, dw, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) out[static_cast<int64_t>(b) * parts] = static_cast<double>(acc);
    }
}

__global__ void __launch_bounds__(kEdgeThreads, 8)
logprob_step_kernel(const __grid_constant__ LogprobStepLaunch p) {
    pdl_release();
    pdl_wait();
    const int chunk = blockIdx.x % p.nchunks;
    const int row = blockIdx.x / p.nchunks;                 // tree * W + j
    const int tree = row / p.W, j = row - tree * p.W;
    const uint32_t D4 = static_cast<uint32_t>(p.D >> 2), e = static_cast<uint32_t>(chunk) * kLogprobChunkVec;
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap, child = row0 + p.off_child + j * p.fan;
    const int parts = p.nchunks * kEdgeWarps;
    if (!BGRPO_IN_BOUNDS(p.status, tree < p.n_trees && e < D4 && p.off + j < p.off_child && p.off_child + (j + 1) * p.fan <= p.nodes_cap &&
                                       parts * 2 <= p.per_row)) return;
    const float4* zp = reinterpret_cast<const float4*>(p.latents + (row0 + p.off + j) * p.D) + e;
    const float4* cp = reinterpret_cast<const float4*>(p.latents + child * p.D) + e;
    const float4* xp = (p.v != nullptr ? reinterpret_cast<const float4*>(p.v + static_cast<int64_t>(row) * p.D)
                                       : reinterpret_cast<const float4*>(p.mu + static_cast<int64_t>(tree) * p.D)) + e;
    double* out = p.partials + child * parts + chunk * kEdgeWarps + (threadIdx.x >> 5);
    if (D4 - e >= kLogprobChunkVec) score_chunk<true>(zp, xp, cp, D4, kLogprobChunkVec, p.fan, p.ca, p.cb, out, parts);
    else score_chunk<false>(zp, xp, cp, D4, D4 - e, p.fan, p.ca, p.cb, out, parts);
}

// One warp: a row's partials in index order within each lane, then a fixed shuffle tree; lane 0 writes the log-prob.
__device__ __forceinline__ void finish_row(const double* q, int n, float g, double scale, float logp_const, float* out) {
    double s = 0.0;
#pragma unroll 4
    for (int c = threadIdx.x & 31; c < n; c += 32) s += __ldcg(q + c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0)
        *out = (g == 0.0f) ? 0.0f : static_cast<float>(static_cast<double>(logp_const) - s * scale);
}

__global__ void __launch_bounds__(256)
logprob_step_finish_kernel(const __grid_constant__ LogprobStepLaunch p) {
    pdl_release();
    pdl_wait();
    const int w = blockIdx.x * 8 + (threadIdx.x >> 5), W = p.W * p.fan;
    if (w >= p.n_trees * W) return;
    const int tree = w / W, parts = p.nchunks * kEdgeWarps;
    const int64_t row = static_cast<int64_t>(tree) * p.nodes_cap + p.off_child + (w - tree * W);
    if (!BGRPO_IN_BOUNDS(p.status, p.off_child + W <= p.nodes_cap && parts * 2 <= p.per_row)) return;
    finish_row(p.partials + row * parts, parts, p.g, p.scale, p.logp_const, p.logp_out + row);
}

// All edges: one warp per non-root row.
__global__ void __launch_bounds__(256)
logprob_tree_finish_kernel(const __grid_constant__ LogprobLaunch p) {
    pdl_release();
    pdl_wait();
    const int edges = p.off[p.depth + 1] - 1;
    const int64_t w = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
    if (w >= static_cast<int64_t>(p.n_trees) * edges) return;
    const int tree = static_cast<int>(w / edges);
    const int local = 1 + static_cast<int>(w - static_cast<int64_t>(tree) * edges);
    int step = 0;                                           // the node's depth is step + 1
    while (step + 1 < p.depth && local >= p.off[step + 2]) ++step;
    const int64_t row = static_cast<int64_t>(tree) * p.nodes_cap + local;
    if (!BGRPO_IN_BOUNDS(p.status, local < p.nodes_cap && p.nchunks * 2 <= p.per_row)) return;
    finish_row(p.partials + row * p.nchunks, p.nchunks, p.g[step], p.scale[step], p.logp_const[step], p.logp_out + row);
}

}  // namespace

cudaError_t launch_logprob_tree(const LogprobLaunch& p, cudaStream_t s) {
    const int64_t items = static_cast<int64_t>(p.n_trees) * p.families * p.nchunks;
    if (items == 0) return cudaSuccess;
    if (items < 0 || items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const cudaError_t e = launch_overlapped(logprob_tree_kernel, static_cast<unsigned int>(items), kThreads, 0, s, p);
    if (e != cudaSuccess) return e;
    const int64_t rows = static_cast<int64_t>(p.n_trees) * (p.off[p.depth + 1] - 1);
    return launch_overlapped(logprob_tree_finish_kernel, static_cast<unsigned int>((rows + 7) / 8), 256, 0, s, p);
}

cudaError_t launch_logprob_step(const LogprobStepLaunch& p, cudaStream_t s) {
    const int64_t items = static_cast<int64_t>(p.n_trees) * p.W * p.nchunks;
    if (items <= 0 || items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const cudaError_t e = launch_overlapped(logprob_step_kernel, static_cast<unsigned int>(items), kEdgeThreads, 0, s, p);
    if (e != cudaSuccess) return e;
    const int64_t rows = static_cast<int64_t>(p.n_trees) * p.W * p.fan;
    return launch_overlapped(logprob_step_finish_kernel, static_cast<unsigned int>((rows + 7) / 8), 256, 0, s, p);
}

}  // namespace bgrpo

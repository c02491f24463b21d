// Whole-tree rollout in one launch, for velocities that act on each latent element by itself (the closed-form linear
// Gaussian-target velocity).  With such a velocity an element's trajectory through the tree never looks at any other
// element, so a thread can carry its elements from the root through every depth in registers, depth first, and
// write each node's latent exactly once: the parent read of the level-by-level step kernel disappears (4 bytes per
// element and node-step instead of 8) and the T launches become one.  The saving the Branch Rollout Algorithm draws
// from shared prefixes is taken literally: a prefix is computed once and never re-read.
//
// Every node gets exactly the value the level-by-level path gives it: the same Philox counters (element block, global
// node id, step, tag), the same float32 expressions (mean = ca z + cb mu, child = g xi + mean, Eq. 2 noise mixing), the same
// integer sums of squares for the log-probs (philox.cuh).
//
// Bound: the noise, that is the FMA pipe: one of Philox' wide multiplies takes it four cycles, Box-Muller's and the update's
// float32 operations one each, and they do not overlap; a register-only loop draws 1.18 T normals a second.  So everything
// around the noise is kept small.  The walk is one loop with one copy of the noise code, not a recursion over split levels
// (which took 113-168 registers, spilled, and did not fit the instruction cache): a node's local index, written in base K,
// is the path that leads to it, and the means of the open forks wait in shared memory.  A thread takes four float4 of long rows
// (24 instructions per element, one: 42), the first two Philox rounds are split into a part per element
// and a part per node.  Video tree (110 edges x 2.1 M elements): 379 -> 249 us, 0.93 T normals/s; four trees of 129 600
// elements: 162 -> 102 us; one: 103 -> 40 us.
//
// A tree of few elements gives too few CTAs, so the first forks can be dealt out to the grid as well: a CTA then walks the
// subtree of one assignment of the first p.par forks, recomputing the prefix that leads to it; of the CTAs that share a
// prefix node, the one whose remaining assignments are all zero writes it.
#include "internal.h"
#include "philox.cuh"

namespace bgrpo {
namespace {

constexpr uint32_t kNotMine = 0xffffffffu;          // no sum of a warp, or with shared noise of half a warp
static_assert(32 * 4 * kMostSquares * kSquareScale < 4294967295.0, "a warp's sum in 32 bits");
static_assert(32 * 2 * 2 * kMostSquares * kSquareScale < 4294967295.0, "with shared noise a warp's at two float4 a thread,");
static_assert(16 * 4 * 2 * kMostSquares * kSquareScale < 4294967295.0, "and a half-warp's at four");

// VEC: float4 per thread.
template <bool SHARED, int VEC>
__global__ void __launch_bounds__(kFusedThreads, kFusedCtasPerSm)
rollout_fused_kernel(const __grid_constant__ FusedLaunch p) {
    constexpr int WORDS = fused_words_per_cta(SHARED, VEC);
    extern __shared__ float4 s_stack[];             // [open fork][VEC] means, SHARED: and as many xi_0; rows of one CTA: the sums of all nodes
    pdl_release();
    const int chunk = blockIdx.x % p.nchunks;
    const int group = blockIdx.x / p.nchunks;       // (tree, assignment of the first forks)
    const int tree = group / p.subtrees;
    int sub = group - tree * p.subtrees;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    const uint32_t gid0 = p.node_id_base + static_cast<uint32_t>(row0);
    const uint32_t D4 = static_cast<uint32_t>(p.D >> 2);
    float4* const tree_base = reinterpret_cast<float4*>(p.latents + row0 * p.D);
    const float4* __restrict__ mu_row = reinterpret_cast<const float4*>(p.mu + static_cast<int64_t>(tree) * p.D);
    const bool writes_table = chunk == 0 && threadIdx.x == 0;
    // nodes below this many forks are this CTA's to write
    int emit_from = p.par;
    for (int s = sub; emit_from > 0 && s % p.K == 0; s /= p.K) --emit_from;

    uint32_t e[VEC];
    bool live[VEC];
    NoiseElement el[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        e[k] = (static_cast<uint32_t>(chunk) * VEC + k) * kFusedThreads + threadIdx.x;
        live[k] = e[k] < D4;
        el[k] = noise_element(e[k], BGRPO_TAG_INNOV, p.keys);
    }
    if (!BGRPO_IN_BOUNDS(p.status, tree < p.n_trees && static_cast<uint32_t>(chunk) * VEC * kFusedThreads < D4 && (chunk + 1) * WORDS <= p.per_row &&
                                       p.per_row <= p.per_row_cap)) return;
    uint32_t* const partials = p.partials + row0 * p.per_row + chunk * WORDS + warp * (WORDS * 32 / kFusedThreads);
    // a row that is one CTA's alone: its sums stay here and the CTA writes the log-probs of the nodes it makes
    uint32_t (*const s_sums)[WORDS] = p.sums_at > 0 ? reinterpret_cast<uint32_t (*)[WORDS]>(s_stack + p.sums_at - 1) : nullptr;
    if (s_sums) {
        for (int n = threadIdx.x; n < p.nodes; n += kFusedThreads) s_sums[n][0] = kNotMine;
        __syncthreads();
    }
    pdl_wait();
    float4 mu[VEC], m[VEC], xi0[VEC];               // m: the mean of the next child, xi0: mix_shared times the shared noise of its fork
    FusedStep st = p.step[0];
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        mu[k] = live[k] ? __ldg(mu_row + e[k]) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 z = live[k] ? __ldcs(tree_base + e[k]) : make_float4(0.f, 0.f, 0.f, 0.f);       // root latent (row 0 of the tree)
        m[k] = fma4(st.ca, z, mul4(st.cb, mu[k]));
        xi0[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int i = 0;                                      // the node about to be made: child of step i (st),
    uint32_t j = 0, parent = 0;                     // with index j in its depth, below the local node parent
    int forks = 0;                                  // forks on its path, the one of step i included
    // Step i forks: chooses the first child to make below index j and keeps what its siblings need.
    auto open_fork = [&]() {
        if (SHARED && st.g != 0.0f) {
            const NoiseNode node = noise_node_of(gid0 + parent, st.px, st.ph, p.keys);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                float squares;
                xi0[k] = mul4(p.mix_shared, normal4(philox_from(noise_element(e[k], BGRPO_TAG_SHARED, p.keys), node, p.keys), squares));
            }
        }
        j *= p.K;
        if (forks < p.par) {
            int div = 1;
            for (int q = forks + 1; q < p.par; ++q) div *= p.K;
            j += (sub / div) % p.K;
        } else {
            const int level = forks - p.par;
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                s_stack[(level * VEC + k) * kFusedThreads + threadIdx.x] = m[k];
                if (SHARED) s_stack[((p.levels + level) * VEC + k) * kFusedThreads + threadIdx.x] = xi0[k];
            }
        }
        ++forks;
    };
    if (st.child0 & kForks) open_fork();
    while (true) {
        const uint32_t child = (st.child0 & ~kForks) + j;
        if (!BGRPO_IN_BOUNDS(p.status, child > 0 && child < static_cast<uint32_t>(p.nodes_cap))) return;
        const bool emit = forks >= emit_from;
        uint32_t acc = 0u;
        float4 z[VEC];
        if (st.g != 0.0f) {
            const NoiseNode node = noise_node_of(gid0 + child, st.px, st.ph, p.keys);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                float squares;
                float4 xi = normal4(philox_from(el[k], node, p.keys), squares);
                if (SHARED && (st.child0 & kForks)) {
                    xi = fma4(p.mix_innov, xi, xi0[k]);
                    squares = squares_of(xi);
                }
                z[k] = fma4(st.g, xi, m[k]);
                acc += live[k] ? quantized_squares(squares) : 0u;
            }
        } else {
#pragma unroll
            for (int k = 0; k < VEC; ++k) z[k] = m[k];
        }
        if (emit) {
            float4* row = tree_base + static_cast<uint64_t>(child) * D4;
#pragma unroll
            for (int k = 0; k < VEC; ++k)
                if (live[k]) __stcs(row + e[k], z[k]);
            if (WORDS > kFusedThreads / 32) {
                const uint32_t low = __reduce_add_sync(0xffffffffu, lane < 16 ? acc : 0u), high = __reduce_add_sync(0xffffffffu, lane < 16 ? 0u : acc);
                if (lane == 0) {
                    uint32_t* const out = s_sums ? s_sums[child] + 2 * warp : partials + static_cast<uint64_t>(child) * static_cast<uint32_t>(p.per_row);
                    out[0] = low;
                    out[1] = high;
                }
            } else {
                acc = __reduce_add_sync(0xffffffffu, acc);
                if (lane == 0) {
                    if (s_sums) s_sums[child][warp] = acc;
                    else partials[static_cast<uint64_t>(child) * static_cast<uint32_t>(p.per_row)] = acc;
                }
            }
            if (writes_table) {
                const int64_t rows = static_cast<int64_t>(p.n_trees) * p.nodes_cap, r = row0 + child;
                p.table[r] = static_cast<int32_t>(parent);
                p.table[rows + r] = i + 1;
                p.table[2 * rows + r] = forks > 0 ? p.split_step[forks - 1] : -1;
                p.table[3 * rows + r] = forks > 0 ? static_cast<int32_t>(j % p.K) : 0;
            }
        }
        parent = child;
        if (++i < p.T) {                            // go down
            st = p.step[i];
#pragma unroll
            for (int k = 0; k < VEC; ++k) m[k] = fma4(st.ca, z[k], mul4(st.cb, mu[k]));
            if (st.child0 & kForks) open_fork();
            continue;
        }
        const uint32_t K = p.K;
        while (forks > p.par && j % K == K - 1) { j /= K; --forks; }       // back to the deepest fork with a child left
        if (forks == p.par) break;
        ++j;
        i = p.split_step[forks - 1];
        st = p.step[i];
        parent = (i > 0 ? p.step[i - 1].child0 & ~kForks : 0u) + j / K;
        const int level = forks - 1 - p.par;
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            m[k] = s_stack[(level * VEC + k) * kFusedThreads + threadIdx.x];
            if (SHARED) xi0[k] = s_stack[((p.levels + level) * VEC + k) * kFusedThreads + threadIdx.x];
        }
    }
    if (!s_sums) return;
    __syncthreads();
    for (int n = threadIdx.x; n < p.nodes; n += kFusedThreads) {
        if (n == 0 || s_sums[n][0] == kNotMine) continue;
        unsigned long long s = 0;
#pragma unroll
        for (int w = 0; w < WORDS; ++w) s += s_sums[n][w];
        int step = 0;                                       // the node's depth is step + 1
        while (step + 1 < p.T && static_cast<uint32_t>(n) >= (p.step[step + 1].child0 & ~kForks)) ++step;
        p.logp[row0 + n] = logp_from_squares(s, p.half_per, p.step[step].g, p.step[step].logp_const);
    }
}

// Completes the log-probs of every non-root node: THREADS threads per node row add up its words.
template <int THREADS>
__global__ void __launch_bounds__(256)
finalize_tree_kernel(const __grid_constant__ FusedLaunch p, int32_t nodes) {
    pdl_release();
    pdl_wait();
    constexpr int kRows = 256 / THREADS;
    const int64_t w = static_cast<int64_t>(blockIdx.x) * kRows + threadIdx.x / THREADS;
    const int64_t total = static_cast<int64_t>(p.n_trees) * (nodes - 1);
    if (w >= total) return;
    const int tree = static_cast<int>(w / (nodes - 1));
    const int local = 1 + static_cast<int>(w - static_cast<int64_t>(tree) * (nodes - 1));
    int step = 0;                                       // the node's depth is step + 1
    while (step + 1 < p.T && static_cast<uint32_t>(local) >= (p.step[step + 1].child0 & ~kForks)) ++step;
    const int64_t row = static_cast<int64_t>(tree) * p.nodes_cap + local;
    if (!BGRPO_IN_BOUNDS(p.status, local < p.nodes_cap && p.per_row <= p.per_row_cap)) return;
    const uint32_t* q = p.partials + row * p.per_row;
    unsigned long long s = 0;
#pragma unroll 4
    for (int c = threadIdx.x % THREADS; c < p.per_row; c += THREADS) s += __ldcg(q + c);
    s = warp_sum_u64(s);
    if (THREADS > 32) {
        __shared__ unsigned long long s_sum[8];
        if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int i = 1; i < 8; ++i) s += s_sum[i];
    }
    if (threadIdx.x % THREADS == 0) p.logp[row] = logp_from_squares(s, p.half_per, p.step[step].g, p.step[step].logp_const);
}

constexpr int32_t kSumsInSharedNodes = 1024;

// What a launch of VEC float4 per thread needs of shared memory: the means of `levels` open forks (and their shared noise), and
// where a row is one CTA's the sums of `nodes` nodes.
constexpr size_t stack_bytes(bool shared_noise, int vec, int levels) {
    return static_cast<size_t>(levels) * kFusedThreads * vec * sizeof(float4) * (shared_noise ? 2 : 1);
}
constexpr size_t sums_bytes(bool shared_noise, int vec, int nodes) {
    return static_cast<size_t>(nodes) * fused_words_per_cta(shared_noise, vec) * sizeof(uint32_t);
}

template <bool SHARED, int VEC>
cudaError_t launch_as(const FusedLaunch& p, unsigned int grid, size_t smem, cudaStream_t s) {
    static SharedMemoryLimit limit(reinterpret_cast<const void*>(&rollout_fused_kernel<SHARED, VEC>),
                                   static_cast<int>(stack_bytes(SHARED, VEC, kFusedMaxSplits) + sums_bytes(SHARED, VEC, kSumsInSharedNodes)));
    if (smem > kSharedWithoutAsking) {
        const cudaError_t e = limit.allow();
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(rollout_fused_kernel<SHARED, VEC>, grid, kFusedThreads, smem, s, p);
}

}  // namespace

cudaError_t launch_rollout_fused(const FusedLaunch& p0, int32_t nodes, cudaStream_t s) {
    FusedLaunch p = p0;
    p.half_per = logp_half_per(p.D);
    int n_splits = 0;
    int64_t leaves = 1;
    for (int i = 0; i < p.T; ++i) {
        noise_step(static_cast<uint32_t>(i), p.keys, p.step[i].px, p.step[i].ph);
        if (!(p.step[i].child0 & kForks)) continue;
        if (n_splits == kFusedMaxSplits) return cudaErrorInvalidValue;
        p.split_step[n_splits++] = i;
        leaves *= p.K;
    }
    const int64_t D4 = p.D / 4;
    const bool shared_noise = p.shared_noise != 0;
    // Four float4 a thread are the fewest instructions per element (video tree: 355 us; two 375, one 462).  But a row that does
    // not fill a CTA of four draws noise for nothing - K = 4, six splits, 64 elements a row: 189 us with four, 98 with one, 162
    // level by level; 1 024 elements: 122 with two, 223 level by level - and a tree without forks has none to deal out: 64 steps
    // of one tree of 16 384 elements 51 us with four, 32 with one, 32 trees 98 and 79, 128 trees 160 and 197, so up to two CTAs of
    // four an SM take one (16 steps of eight image trees, 512 CTAs: equal).
    int vec = D4 <= kFusedThreads ? 1 : D4 <= 2 * kFusedThreads ? 2 : 4;
    if (leaves == 1 && p.n_trees * ((D4 + kFusedThreads * 4 - 1) / (kFusedThreads * 4)) <= 2 * 148) vec = 1;
    p.nchunks = static_cast<int32_t>((D4 + kFusedThreads * vec - 1) / (kFusedThreads * vec));
    p.per_row = p.nchunks * fused_words_per_cta(shared_noise, vec);
    if (p.per_row > p.per_row_cap) return cudaErrorInvalidValue;
    // Dealing out a fork more makes K times as many CTAs that walk a shorter subtree but compute the prefix again.  An SM works
    // at the same rate from about three CTAs on, so the time goes with the CTAs of the busiest SM (at least three) times the
    // nodes a CTA walks.  Measured, us a rollout, forks dealt out 0 / 1 / 2 / 3 (the rule's choice in brackets): four trees of
    // 129 600 elements 213 / - / [102] / 111, one video tree 255 / [249] / 268 / -; one tree of 129 600 elements 54 with none, 40
    // with four and with the rule's three.
    int64_t best = -1;
    int32_t subtrees = 1;
    for (int par = 0; par <= n_splits; ++par, subtrees *= p.K) {
        int64_t walk = 0, width = 1;
        for (int i = 0, forks = 0; i < p.T; ++i) {
            if ((p.step[i].child0 & kForks) && forks++ >= par) width *= p.K;
            walk += width;
        }
        const int64_t ctas = (static_cast<int64_t>(p.n_trees) * p.nchunks * subtrees + 147) / 148;
        const int64_t cost = (ctas < 3 ? 3 : ctas) * walk;
        if (best < 0 || cost <= best) {
            best = cost;
            p.par = par;
            p.subtrees = subtrees;
        }
    }
    p.levels = n_splits - p.par;
    const int64_t items = static_cast<int64_t>(p.n_trees) * p.nchunks * p.subtrees;
    if (items <= 0 || items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const unsigned int grid = static_cast<unsigned int>(items);
    size_t smem = stack_bytes(shared_noise, vec, p.levels);
    // Rows of one CTA keep their sums in shared memory (up to 16 KB of them, 32 with shared noise) and need no second launch,
    // which costs about 4 us of host time (toy pass, with the rewards' second launch gone as well: 27.8 -> 23.8 us).
    p.nodes = nodes;
    p.sums_at = 0;
    if (p.nchunks == 1 && nodes <= kSumsInSharedNodes) {
        p.sums_at = static_cast<int32_t>(smem / sizeof(float4)) + 1;
        smem += sums_bytes(shared_noise, vec, nodes);
    }
    const cudaError_t e = shared_noise ? (vec == 1 ? launch_as<true, 1>(p, grid, smem, s) : vec == 2 ? launch_as<true, 2>(p, grid, smem, s) : launch_as<true, 4>(p, grid, smem, s))
                                       : (vec == 1 ? launch_as<false, 1>(p, grid, smem, s) : vec == 2 ? launch_as<false, 2>(p, grid, smem, s) : launch_as<false, 4>(p, grid, smem, s));
    if (e != cudaSuccess || nodes < 2 || p.sums_at > 0) return e;
    const int64_t rows = static_cast<int64_t>(p.n_trees) * (nodes - 1);
    if (p.per_row >= 512) return launch_overlapped(finalize_tree_kernel<256>, static_cast<unsigned int>(rows), 256, 0, s, p, nodes);
    return launch_overlapped(finalize_tree_kernel<32>, static_cast<unsigned int>((rows + 7) / 8), 256, 0, s, p, nodes);
}

}  // namespace bgrpo

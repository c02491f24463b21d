// Host-side state of a batch of rollout trees and the launch interfaces of the kernels.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>
#include <mutex>
#include <utility>

#include "../../include/bgrpo.h"

namespace bgrpo {

constexpr int kStreamThreads = 256;    // threads per CTA of the root / reward kernels
constexpr int kChunkVec = 1024;        // float4 per (row, chunk) work item of the root kernel
constexpr int kRewardVec = 16;         // float4 of a row per thread of the leaf-reward kernel
constexpr int kRewardChunkVec = kStreamThreads * kRewardVec;   // float4 per (row, chunk) work item of the leaf-reward kernel
// Step kernel: 128-thread CTAs, 4 float4 per thread, four CTAs per SM so that 128 registers hold a thread's loads and noise.
// What bounds it is HBM, as far as loads are in flight while other warps draw noise.  16 steps of 32 image trees (12 B/element,
// 4.2 GB) in 1 140 us; 64 threads of 8 float4, eight CTAs per SM - the same warps, in smaller CTAs - took 1 200 us, five CTAs of
// 128 threads (96 registers) 1 170 us, eight (64 registers, spills) 1 160 us and on a video tree 622 us for 598.
// A launch of less than four such CTAs per SM has no throughput to lose: it takes as long as one thread's work, so the same
// chunk goes to 256 threads of 2 float4.
constexpr int kStepThreads = 128, kStepThreadsSmall = 256;
constexpr int kStepVec = 4;
constexpr int kStepChunkVec = kStepThreads * kStepVec;   // 512 float4 = 8 KiB per operand tile
// Three or four children with noise of their own store more than they load: a fifth CTA is worth more there than the registers
// (16 image trees, forks of three and of four: 1 168 -> 1 149 us, 2 621 -> 2 598 us).
constexpr int step_ctas_per_sm(int fan, bool shared_noise) { return fan >= 3 && !shared_noise ? 5 : 4; }
constexpr int kStepCtasPerSmSmall = 4;
constexpr int64_t kStepSmallGrid = 148 * 4;
inline int step_threads(int64_t items) { return items < kStepSmallGrid ? kStepThreadsSmall : kStepThreads; }
// Whole-tree rollout kernel: 128-thread CTAs of up to 4 float4 per thread (launch_rollout_fused chooses), four CTAs per SM (5 and
// 6: equal and 6 % slower on the video tree, 16 and 40 % slower on a single image tree), one log-prob partial per node row and
// warp; at most kFusedMaxSplits split steps (the means of the open forks wait in shared memory).
constexpr int kFusedThreads = 128;
constexpr int kFusedMostVec = 4;
constexpr int kFusedCtasPerSm = 4;
constexpr int kFusedMaxSplits = 6;
// log-prob partials of the whole-tree kernel per CTA that covers a node row: one 32-bit word per warp, two with shared noise and
// four float4 a thread (a half-warp's squares each: see the bound in tree_fused.cu)
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int fused_words_per_cta(bool shared_noise, int vec) { return kFusedThreads / 32 * (shared_noise && vec == 4 ? 2 : 1); }
// 32-bit words of log-prob partials reserved per node row: those of the step kernel, 64 bits per chunk and warp.  The whole-tree
// kernel's fit as well: per step chunk of 512 float4 at most four CTAs of one float4 a thread, four words each.  An even number,
// so that every row starts on 8 bytes.
inline int64_t partials_per_row(int64_t D) {
    return ((D / 4 + kStepChunkVec - 1) / kStepChunkVec) * (kStepThreadsSmall / 32) * 2;
}
static_assert(kStepChunkVec / kFusedThreads * (kFusedThreads / 32) <= kStepThreadsSmall / 32 * 2 && kStepChunkVec == kFusedThreads * kFusedMostVec,
              "the whole-tree kernel's partials fit the step kernel's");
constexpr int kScratchHeader = 256;    // bytes reserved at the start of scratch for the status word

constexpr uint32_t kPhiloxM0 = 0xD2511F53u;   // Philox4x32 multipliers and Weyl key increments (Salmon et al., SC'11)
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

// The ten round keys of a 64-bit seed: key r = (k0 + r*W0, k1 + r*W1).  They are the same for every thread of
// a launch, so the host computes them once and the kernels read them as launch constants.
struct PhiloxKeys {
    uint32_t k[10][2];
};

inline PhiloxKeys make_philox_keys(uint64_t seed) {
    PhiloxKeys out;
    uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        out.k[r][0] = k0;
        out.k[r][1] = k1;
        k0 += kPhiloxW0;
        k1 += kPhiloxW1;
    }
    return out;
}

// Per-step scalars of the Euler-Maruyama mean and the Gaussian transition, computed in double on the host.
//   mean = a*z + b*v                       (v given)
//        = lin_a*z + lin_b*mu              (closed-form velocity v = k z - (1 + k(1-t)) mu folded in)
struct StepCoef {
    float a, b;          // a = 1 - c, b = -(h + c (1-t)), c = sigma^2 h / (2 t)
    float lin_a, lin_b;  // valid once a linear velocity is bound
    float g;             // sigma sqrt(h)
    float inv_2g2;       // 1 / (2 g^2), 0 when g == 0
    float logp_const;    // -ln g - 0.5 ln(2 pi), 0 when g == 0
};

// Log-probs of a level whose per-(row, chunk, warp) partial sums are in scratch but not yet added up.  The sum is
// taken by the next kernel the library enqueues on the stream (the next step, beside its own work, or a small flush kernel).
struct FinalizeDesc {
    float* logp_out;       // nullptr: nothing pending
    int32_t W, off;        // rows off .. off+W-1 of every tree
    int32_t per_row;       // sums per row
    float g, logp_const;
    unsigned long long* sums;   // row r's start at sums + r * stride
    int32_t stride;        // the same for every launch of a tree: a level is summed while the next one's sums are written
    int32_t clear;         // 1: the sums were added up with atomics; whoever takes them leaves zeros for the next who adds (a
                           // replayed graph that starts after the root kernel, say)
};

struct LevelInfo {                       // layout of the tree grown so far
    int32_t width[BGRPO_MAX_T + 1];
    int32_t offset[BGRPO_MAX_T + 2];
    int32_t fanout[BGRPO_MAX_T];         // children per node produced by step i (K or 1)
};

// Runs of a finished tree: maximal stretches of depths without a fork in between.  Run r covers the depths
// first[r] .. first[r+1]-1, which all have the same width; an only child has its parent's leaves below it, hence its fused
// value, its place among the siblings at every split and its kept leaves, so the reductions do their work per run and only
// loads and stores are per depth.
struct RunInfo {
    int32_t n;
    int32_t first[BGRPO_MAX_T + 2];      // first[n] = T + 1
    int32_t chain0[BGRPO_MAX_T + 2];     // index of the run's first chain (a node and the only children below it); chain0[n] = number of chains
    int32_t of_depth[BGRPO_MAX_T + 1];
    double inv_width[BGRPO_MAX_T + 1], inv_fan;      // per run; reciprocals from the host: a double division is a few hundred cycles
};

inline RunInfo runs_of(const LevelInfo& lv, int T) {
    RunInfo r;
    r.n = 0;
    r.first[r.n++] = 0;
    for (int i = 0; i < T; ++i)
        if (lv.fanout[i] > 1) r.first[r.n++] = i + 1;
    r.first[r.n] = T + 1;
    r.chain0[0] = 0;
    r.inv_fan = 1.0;
    for (int q = 0; q < r.n; ++q) {
        r.chain0[q + 1] = r.chain0[q] + lv.width[r.first[q]];
        r.inv_width[q] = 1.0 / lv.width[r.first[q]];
        if (q > 0) r.inv_fan = 1.0 / lv.fanout[r.first[q] - 1];      // the same at every fork
        for (int d = r.first[q]; d < r.first[q + 1]; ++d) r.of_depth[d] = q;
    }
    return r;
}

}  // namespace bgrpo

struct bgrpo_tree {
    bgrpo_tree_desc desc;
    bgrpo_buffers buf;
    float t_grid[BGRPO_MAX_T + 1];
    bgrpo::StepCoef coef[BGRPO_MAX_T];
    bgrpo::LevelInfo lv;
    uint64_t ode_bits;                   // bit i set: step i is an ODE step of the hybrid schedule (sigma = 0)
    int32_t depth;                       // steps taken so far
    int64_t D;                           // elements per node
    int32_t nchunks;                     // root-kernel work items per node row (also sizes the reward partials)
    int32_t nchunks_reward;              // leaf-reward work items per node row
    int32_t nchunks_step;                // step-kernel work items per node row
    bool independent;                    // s = inf: xi_b = eta_b
    float mix_shared, mix_innov;         // xi_b = mix_shared*xi_0 + mix_innov*eta_b
    const float* mu;                     // bound linear velocity (device), or nullptr
    float s0;
    // scratch carving (device pointers inside buf.scratch)
    int32_t* status;
    unsigned long long* row_sums;        // [n_trees*nodes_cap] squares of a row's noise, where the MLP stage takes the step; zero before it and after they were taken
    double* partials;                    // [n_trees*nodes_cap][nchunks][3]   (reward reductions)
    double* node_scratch;                // [n_trees][2][nodes_cap]: per-chain state of the tree reductions when a tree
                                         // is too large for one CTA's shared memory
    void* partials_logp;                 // [n_trees*nodes_cap][partials_per_row] 32-bit words: log-prob sums, each kernel's own layout
    unsigned long long* partials_u64() const { return static_cast<unsigned long long*>(partials_logp); }
    bgrpo::FinalizeDesc pending;         // level whose log-probs still have to be summed
};

// Debug build (-DBGRPO_DEBUG_BOUNDS): every kernel tests the row, chunk and element indices it derives against the
// extents it was launched with, before the access.  A failed test sets bit 2 of the tree's status word and the access
// is skipped; nothing traps.  bgrpo_tree_sync_status reports the word.  In the normal build the tests compile to nothing.
#ifdef BGRPO_DEBUG_BOUNDS
#define BGRPO_IN_BOUNDS(status, cond) ((cond) ? true : (atomicOr((status), 2), false))
#else
#define BGRPO_IN_BOUNDS(status, cond) true
#endif
constexpr int kStatusNonFinite = 1, kStatusOutOfBounds = 2, kStatusWaitTimeout = 4;

namespace bgrpo {

// Programmatic dependent launch: a kernel launched with launch_overlapped() may be scheduled while the kernel before it
// on the stream is still draining, so the gap between two dependent launches shrinks to the set-up the new kernel can do
// on its own.  Such a kernel calls pdl_wait() before it touches anything an earlier kernel wrote or still reads, and
// pdl_release() as early as it likes to let its own successor in.
//
// Kernels the calling host thread has enqueued so far (bgrpo_launch_count): every launch goes through count_launch().
inline int64_t& launch_count() {
    thread_local int64_t n = 0;
    return n;
}
inline cudaError_t count_launch(cudaError_t e) {
    if (e == cudaSuccess) ++launch_count();
    return e;
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... Params, typename... Args>
cudaError_t launch_overlapped_clusters(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned int>(cluster);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return count_launch(cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...));
}
template <typename... Params, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    return launch_overlapped_clusters(kernel, grid, block, smem, s, 1, std::forward<Args>(args)...);
}
#endif

// The most dynamic shared memory any launch of a kernel takes, allowed once per device.  The limit belongs to the process: set
// to each launch's own size, a thread could lower it between another thread's setting and its launch.
struct SharedMemoryLimit {
    const void* kernel;
    int bytes;
    std::mutex mutex;
    uint64_t devices = 0;      // bit d: allowed on device d
    SharedMemoryLimit(const void* k, int b) : kernel(k), bytes(b) {}
    cudaError_t allow() {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        std::lock_guard<std::mutex> lock(mutex);
        const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
        if (devices & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) devices |= bit;
        return e;
    }
};
constexpr size_t kSharedWithoutAsking = 40 * 1024;      // of the 48 KB a launch may take as it is; the rest is for static arrays

// ---- streaming kernels (tree_step.cu) -------------------------------------------------------------------------
struct StepLaunch {
    float* latents;
    const float* v;            // [n_trees][W_in][D] or nullptr
    const float* mu;           // [n_trees][D] or nullptr
    float* logp;
    int32_t* table;            // SoA, stride = n_trees*nodes_cap
    int64_t D;                 // elements per row
    int32_t n_trees, nodes_cap, nchunks;   // nchunks: step-kernel chunks per row
    int32_t W_in, off_in, off_out, fan, step, is_split;
    uint32_t node_id_base;     // tree_id_base * nodes_cap
    PhiloxKeys keys;
    double half_per;           // logp_half_per(D), set by launch_step
    float ca, cb;              // mean = ca*z + cb*x, x = v or mu
    float g;
    float mix_shared, mix_innov;
    int32_t shared_noise;      // 1: finite s at a split step
    int32_t keep_v;            // step taken along by the MLP stage: 1 if the velocities are to be left in its buffer
    int32_t* status;           // the tree's status word
    int32_t per_row;           // 32-bit words reserved per node row in the partials
    unsigned long long* partials;   // by row, per_row / 2 apart: [nchunks][warps of a CTA] sums of quantized squares (philox.cuh)
    FinalizeDesc prev;         // level whose sums this launch takes (logp_out == nullptr: none)
};
cudaError_t launch_root(const bgrpo_tree* t, cudaStream_t s);
cudaError_t launch_step(const StepLaunch& p, cudaStream_t s);
cudaError_t launch_finalize(const bgrpo_tree* t, const FinalizeDesc& f, cudaStream_t s);

// ---- log-probs of all stored edges (tree_logprob.cu) ---------------------------------------------------------------
constexpr int kLogprobChunkVec = 512;      // float4 of a row per CTA; one double per (row, chunk) fits the step kernel's partials
static_assert(kLogprobChunkVec == kStepChunkVec, "two doubles per (row, chunk) take what the step kernel needs");
struct LogprobLaunch {
    const float* latents;
    const float* mu;           // [n_trees][D]
    float* logp_out;
    double* partials;          // [rows][nchunks]
    int32_t* status;
    int64_t D;
    int32_t n_trees, nodes_cap, nchunks, per_row, depth;
    int32_t families, n_runs;                          // families per tree, in all runs
    int32_t run_families[BGRPO_MAX_T + 1], run_d0[BGRPO_MAX_T + 1], run_fan[BGRPO_MAX_T + 1], run_len[BGRPO_MAX_T + 1];
    int32_t off[BGRPO_MAX_T + 2];
    float ca[BGRPO_MAX_T], cb[BGRPO_MAX_T], g[BGRPO_MAX_T], logp_const[BGRPO_MAX_T];   // by step
    double scale[BGRPO_MAX_T];
};
cudaError_t launch_logprob_tree(const LogprobLaunch& p, cudaStream_t s);      // all edges, closed form
// One step's edges.  A small parameter block of its own: with the other one's 2.4 KB the sixteen calls that score an image
// tree took 5 us longer.
struct LogprobStepLaunch {
    const float* latents;
    const float* v;            // [n_trees][W][D], or nullptr: closed-form velocity
    const float* mu;           // [n_trees][D]
    float* logp_out;
    double* partials;          // [rows][2 nchunks]: one per chunk and warp
    int32_t* status;
    int64_t D;
    int32_t n_trees, nodes_cap, nchunks, per_row;
    int32_t W, off, off_child, fan;
    float ca, cb, g, logp_const;
    double scale;              // 1 / (2 g^2 D), from the host: a double division takes longer than the rest of the sum
};
cudaError_t launch_logprob_step(const LogprobStepLaunch& p, cudaStream_t s);

struct RewardLaunch {
    const float* latents; const float* target; float* r; double* partials; int32_t* status;
    int64_t D; int32_t n_trees, nodes_cap, nchunks, nchunks_cap, leaves, off_leaf; float scale; double inv_D; int32_t mode;  // 0 mse, 1 cos; nchunks_cap: partial slots reserved per row
};
cudaError_t launch_reward(const RewardLaunch& p, cudaStream_t s);

cudaError_t launch_philox_words(uint64_t seed, uint32_t node, uint32_t step, uint32_t tag, uint32_t* out, int64_t nblk, cudaStream_t s);
cudaError_t launch_philox_normals(uint64_t seed, uint32_t node, uint32_t step, uint32_t tag, float* out, int64_t n, cudaStream_t s);

// ---- whole-tree rollout (tree_fused.cu) -------------------------------------------------------------------------
struct alignas(16) FusedStep {
    float ca, cb, g;
    uint32_t child0;           // offset of the depth the step makes, bit 31: the step forks
    uint32_t px, ph;           // what the noise counters of all nodes of the step share (noise_step in philox.cuh)
    float logp_const;
    uint32_t pad;
};
struct FusedLaunch {
    float* latents;
    const float* mu;           // [n_trees][D]
    float* logp;
    int32_t* table;
    uint32_t* partials;        // [rows][per_row]: fused_words_per_cta() words per CTA that covers a row
    int32_t* status;           // the tree's status word
    int32_t per_row_cap;       // words reserved per node row
    int64_t D;
    int32_t n_trees, nodes_cap, T, K, shared_noise;
    int32_t nchunks, per_row;  // CTAs that cover a row, words of partials they leave; set by launch_rollout_fused, like the next six
    int32_t par, subtrees, levels, nodes;              // forks dealt out to the grid, K^par, forks walked, nodes of a tree
    int32_t sums_at;           // 0, or 1 + where in shared memory (float4) the sums of a row of one CTA are
    int32_t split_step[kFusedMaxSplits];
    uint32_t node_id_base;
    PhiloxKeys keys;
    double half_per;           // logp_half_per(D), set by launch_rollout_fused
    float mix_shared, mix_innov;
    FusedStep step[BGRPO_MAX_T];                       // set by the caller but for px, ph
};
constexpr uint32_t kForks = 0x80000000u;
cudaError_t launch_rollout_fused(const FusedLaunch& p, int32_t nodes, cudaStream_t s);

// ---- tree reductions (tree_reduce.cu) -------------------------------------------------------------------------
constexpr size_t kTreeSmemLimit = 200 * 1024;   // per-chain state beyond this lives in node_scratch instead of shared memory
struct FuseLaunch {
    const float* leaf_r; const float* logp; float* rbar; float* adv; int32_t* status;
    double* node_scratch;      // [n_trees][2][nodes_cap], used when two doubles per chain exceed kTreeSmemLimit (trees of more than 12 800 chains)
    LevelInfo lv; RunInfo runs; int32_t n_trees, nodes_cap, T, nodes; double beta_scaled; float eps, clip;
};
cudaError_t launch_fuse_advantage(const FuseLaunch& p, cudaStream_t s);

struct EssLaunch {
    const float* logp; float* ess; double* node_scratch; int32_t* status;
    LevelInfo lv; RunInfo runs; int32_t n_trees, nodes_cap, T, nodes; double beta_scaled;
};
cudaError_t launch_fusion_ess(const EssLaunch& p, cudaStream_t s);

struct PruneLaunch {
    const float* rbar; uint8_t* mask; int32_t* status;
    LevelInfo lv; RunInfo runs; int32_t n_trees, nodes_cap, T, nodes, mode, k, last_split, ignore_last; uint64_t pruned_bits;
    int32_t wide_run, narrow_nodes;      // first run written chain by chain and the nodes before it; set by launch_prune
};
cudaError_t launch_prune(const PruneLaunch& p, cudaStream_t s);

struct ObjectiveLaunch {
    const float* logp_new; const float* logp_old; const float* adv; const uint8_t* mask; float* terms; float* J; int32_t* status;
    int32_t n_trees, nodes_cap, nodes; double logp_scale; float clip_eps;
};
cudaError_t launch_objective(const ObjectiveLaunch& p, cudaStream_t s);

// ---- MLP velocity (mlp_velocity.cu) -----------------------------------------------------------------------------
size_t mlp_packed_bytes(int hidden);
cudaError_t launch_mlp_pack(const uint16_t* W1, const uint16_t* W2, int hidden, void* packed, cudaStream_t s);
cudaError_t launch_debug_trip(int32_t* status, cudaStream_t s);     // debug build: fails one index test on purpose (no access involved)
// `step`: the step that follows, or nullptr.  Where the launch can take it along (launch_mlp in mlp_velocity.cu), *stepped is
// set, the squares of the noise go to row_sums, and no step kernel is needed.
cudaError_t launch_mlp(const float* latents, int64_t pool_elems, int64_t tree_stride, int64_t row_offset, int n_trees, int64_t tokens_per_tree,
                       const void* packed, int hidden, float* v_out, int32_t* status, const StepLaunch* step, unsigned long long* row_sums,
                       bool* stepped, cudaStream_t s);

}  // namespace bgrpo

// Tree reductions: reward fusion (Eq. 3) + depth-wise normalisation (Eq. 4) in one kernel, and the width / depth
// pruning masks ("Pruning Strategies") in another.  A tree usually has at most a few thousand nodes, so one CTA owns one
// tree; the kernels are latency-bound: what counts is the number of dependent steps, not the work.
//
// The work is done per run (RunInfo): between two forks every node has one child, and all nodes of such a chain share their
// fused value, their rank and their kept leaves.  State is kept per chain - doubles in shared memory, or in the caller's
// scratch for trees with more than 12 800 chains - so a tree takes as many barriers as it has forks, not depths, and the
// statistics of a depth are taken once per run.  On 32 trees of 1009 nodes (20 depths, 4 forks of 3): fusion 15.0 -> 12.4 us,
// effective sample size 26.7 -> 11.4 us, Parent-Top1 mask 16.8 -> 6.5 us, objective 8.0 -> 4.6 us (device time, cold caches).
//
// Fusion uses the bottom-up form of Eq. 3.  With a_c = beta*logp(c) the softmax weight of leaf l under node n
// factorises along the path, so  S_n = sum_c e^{a_c} S_c,  R_n = sum_c e^{a_c} R_c,  rbar(n) = R_n / S_n  with
// S_leaf = 1, R_leaf = r.  S is carried as log S (shifted by the largest term) so huge |beta*logp| cannot overflow;
// R/S is carried directly as rbar:  rbar(n) = sum_c w_c rbar(c),  w_c = e^{a_c + logS_c - m} / sum_c' e^{a_c' + logS_c' - m}.
// Along a chain a_c just adds up.
#include "internal.h"

namespace bgrpo {
namespace {

constexpr int kTreeThreads = 256;

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// s / n for a whole n, given the double nearest 1 / n: the quotient's residual corrects it to the correctly rounded one
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990) in two operations, where a
// division is a few hundred cycles.  s * (1 / n) alone misses the mean of n equal values by its last bit for n = 243 and
// 729 (K = 3): leaves with equal rewards would get an advantage that is not zero.
__device__ __forceinline__ double divide_by(double s, double n, double inv_n) {
    const double q = s * inv_n;
    return isfinite(q) ? fma(fma(-q, n, s), inv_n, q) : q;
}

// Layout tables of a tree in shared memory: per depth its offset and run, per run the index of its first chain.
struct Layout {
    int off[BGRPO_MAX_T + 2];
    int run[BGRPO_MAX_T + 1];
    int chain0[BGRPO_MAX_T + 2];        // chain0[runs.n] = number of chains
    __device__ void fill(const LevelInfo& lv, const RunInfo& runs, int T) {
        for (int d = threadIdx.x; d <= T + 1; d += kTreeThreads) off[d] = lv.offset[d];
        for (int d = threadIdx.x; d <= T; d += kTreeThreads) run[d] = runs.of_depth[d];
        for (int r = threadIdx.x; r <= runs.n; r += kTreeThreads) chain0[r] = runs.chain0[r];
    }
};

// beta * logp summed along every chain (the edge into its first node included), into out[chain]: all loads independent.
__device__ __forceinline__ void chain_sums(double* out, const float* logp, const Layout& lay, const RunInfo& runs, double beta) {
    const int chains = lay.chain0[runs.n];
    for (int m = threadIdx.x; m < chains; m += kTreeThreads) {
        int r = 0;
        while (m >= lay.chain0[r + 1]) ++r;
        const int j = m - lay.chain0[r];
        double c = 0.0;
#pragma unroll 8
        for (int d = runs.first[r + 1] - 1; d >= runs.first[r]; --d) c += beta * static_cast<double>(logp[lay.off[d] + j]);
        out[m] = c;
    }
}

__global__ void __launch_bounds__(kTreeThreads)
fuse_advantage_kernel(const __grid_constant__ FuseLaunch p) {
    pdl_release();
    extern __shared__ double sm[];
    __shared__ Layout lay;
    __shared__ int bad;
    __shared__ double s_mean[BGRPO_MAX_T + 1], s_inv[BGRPO_MAX_T + 1];
    const int tree = blockIdx.x;
    const int T = p.T, R = p.runs.n;
    lay.fill(p.lv, p.runs, T);
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    const int chains = p.runs.chain0[R];
    const bool in_smem = static_cast<size_t>(chains) * 2 * sizeof(double) <= kTreeSmemLimit;
    double* rb = in_smem ? sm : p.node_scratch + static_cast<int64_t>(tree) * 2 * p.nodes_cap;   // fused value per chain
    double* ls = rb + (in_smem ? chains : p.nodes_cap);      // log S of the chain's last node + beta * logp along the chain
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    const int leaves = p.lv.width[T];
    const double beta = p.beta_scaled;
    if (!BGRPO_IN_BOUNDS(p.status, chains <= p.nodes && p.nodes <= p.nodes_cap && tree < p.n_trees)) return;
    pdl_wait();
    if (beta != 0.0) chain_sums(ls, p.logp + row0, lay, p.runs, beta);
    for (int l = threadIdx.x; l < leaves; l += kTreeThreads) {
        const float r = p.leaf_r[static_cast<int64_t>(tree) * leaves + l];
        if (!isfinite(r)) bad = 1;
        rb[lay.chain0[R - 1] + l] = static_cast<double>(r);
    }
    __syncthreads();
    if (bad && threadIdx.x == 0) atomicOr(p.status, 1);
    for (int r = R - 2; r >= 0; --r) {       // the fork between run r and run r + 1
        const int fan = p.lv.fanout[p.runs.first[r + 1] - 1];
        const int W = lay.chain0[r + 1] - lay.chain0[r];
        for (int j = threadIdx.x; j < W; j += kTreeThreads) {
            const int me = lay.chain0[r] + j, c0 = lay.chain0[r + 1] + j * fan;
            if (!BGRPO_IN_BOUNDS(p.status, c0 + fan <= lay.chain0[r + 2])) continue;
            if (beta == 0.0) {   // uniform weights: every child of a node has the same number of leaves below it, so the
                                 // leaf mean of the parent is the plain mean of its children's leaf means
                double sum = 0.0;
#pragma unroll
                for (int b = 0; b < BGRPO_MAX_K; ++b)
                    if (b < fan) sum += rb[c0 + b];
                rb[me] = divide_by(sum, fan, p.runs.inv_fan);
                continue;
            }
            double a[BGRPO_MAX_K];
            double m = -INFINITY;
#pragma unroll
            for (int b = 0; b < BGRPO_MAX_K; ++b) {
                if (b < fan) {
                    a[b] = ls[c0 + b];
                    m = fmax(m, a[b]);
                }
            }
            double S = 0.0, Rs = 0.0;
#pragma unroll
            for (int b = 0; b < BGRPO_MAX_K; ++b) {
                if (b < fan) {
                    const double w = exp(a[b] - m);
                    S += w;
                    Rs += w * rb[c0 + b];
                }
            }
            rb[me] = Rs / S;
            ls[me] += m + log(S);
        }
        __syncthreads();
    }
    // Depth-wise statistics, the same for all depths of a run: one warp per run, two passes (mean, then centred squares),
    // fixed lane order.
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int r = warp; r < R; r += kTreeThreads / 32) {
        const double* v = rb + lay.chain0[r];
        const int W = lay.chain0[r + 1] - lay.chain0[r];
        double s = 0.0;
        for (int j = lane; j < W; j += 32) s += v[j];
        const double mean = divide_by(warp_sum_d(s), W, p.runs.inv_width[r]);
        double q = 0.0;
        for (int j = lane; j < W; j += 32) { const double c = v[j] - mean; q += c * c; }
        const double sd = sqrt(divide_by(warp_sum_d(q), W, p.runs.inv_width[r]));
        if (lane == 0) {
            s_mean[r] = mean;
            s_inv[r] = 1.0 / (sd + static_cast<double>(p.eps));
        }
    }
    __syncthreads();
    int d = 0;
    for (int n = threadIdx.x; n < p.nodes; n += kTreeThreads) {
        while (n >= lay.off[d + 1]) ++d;
        const int r = lay.run[d];
        const double v = rb[lay.chain0[r] + n - lay.off[d]];
        double A = (d == 0) ? 0.0 : (v - s_mean[r]) * s_inv[r];
        if (p.clip > 0.0f) A = fmin(fmax(A, -static_cast<double>(p.clip)), static_cast<double>(p.clip));
        p.adv[row0 + n] = static_cast<float>(A);
        p.rbar[row0 + n] = static_cast<float>(v);
    }
}

// Effective sample size of the fusion weights (appendix "Reward Fusion"): ESS(n) = (sum_l w_l)^2 / sum_l w_l^2 over the
// descendant leaves of n, w_l = exp(beta s_l).  Both sums factorise along the paths like S above:
//   log S_n = logsumexp_c(a_c + log S_c),   log Q_n = logsumexp_c(2 a_c + log Q_c),   ESS = exp(2 log S - log Q),
// and along a chain both numerator and denominator pick up the same factor - unless that factor is not finite: nodes of a
// chain above such an edge have no value.
__global__ void __launch_bounds__(kTreeThreads)
fusion_ess_kernel(const __grid_constant__ EssLaunch p) {
    pdl_release();
    extern __shared__ double sm[];
    __shared__ Layout lay;
    const int tree = blockIdx.x;
    const int T = p.T, R = p.runs.n;
    lay.fill(p.lv, p.runs, T);
    __syncthreads();
    const int chains = p.runs.chain0[R];
    const bool in_smem = static_cast<size_t>(chains) * 2 * sizeof(double) <= kTreeSmemLimit;
    double* ls = in_smem ? sm : p.node_scratch + static_cast<int64_t>(tree) * 2 * p.nodes_cap;
    double* lq = ls + (in_smem ? chains : p.nodes_cap);
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    if (!BGRPO_IN_BOUNDS(p.status, chains <= p.nodes && p.nodes <= p.nodes_cap && tree < p.n_trees)) return;
    pdl_wait();
    chain_sums(ls, p.logp + row0, lay, p.runs, p.beta_scaled);
    bool odd = false;
    for (int m = threadIdx.x; m < chains; m += kTreeThreads) {      // written by this thread
        lq[m] = 2.0 * ls[m];
        odd = odd || !isfinite(ls[m]);
    }
    for (int n = lay.off[p.runs.first[R - 1]] + threadIdx.x; n < p.nodes; n += kTreeThreads) p.ess[row0 + n] = 1.0f;
    odd = __syncthreads_or(odd) != 0;          // some edge's factor is not finite (no usual case)
    // The value of chain j of run r at all of its depths; the sums of a chain with such an edge below its first node are lost.
    auto write_chain = [&](int r, int j, float ess) {
        for (int d = p.runs.first[r + 1] - 1; d >= p.runs.first[r]; --d) {
            const int64_t n = row0 + lay.off[d] + j;
            p.ess[n] = ess;
            if (odd && d > p.runs.first[r] && !isfinite(p.beta_scaled * static_cast<double>(p.logp[n])))
                ess = ls[lay.chain0[r] + j] = lq[lay.chain0[r] + j] = NAN;
        }
    };
    if (odd) {
        for (int j = threadIdx.x; j < chains - lay.chain0[R - 1]; j += kTreeThreads) write_chain(R - 1, j, 1.0f);
        __syncthreads();
    }
    for (int r = R - 2; r >= 0; --r) {
        const int fan = p.lv.fanout[p.runs.first[r + 1] - 1];
        const int W = lay.chain0[r + 1] - lay.chain0[r];
        for (int j = threadIdx.x; j < W; j += kTreeThreads) {
            const int me = lay.chain0[r] + j, c0 = lay.chain0[r + 1] + j * fan;
            if (!BGRPO_IN_BOUNDS(p.status, c0 + fan <= lay.chain0[r + 2])) continue;
            double a1[BGRPO_MAX_K], a2[BGRPO_MAX_K];
            double m1 = -INFINITY, m2 = -INFINITY;
#pragma unroll
            for (int b = 0; b < BGRPO_MAX_K; ++b) {
                if (b < fan) {
                    a1[b] = ls[c0 + b];
                    a2[b] = lq[c0 + b];
                    m1 = fmax(m1, a1[b]);
                    m2 = fmax(m2, a2[b]);
                }
            }
            double S = 0.0, Q = 0.0;
#pragma unroll
            for (int b = 0; b < BGRPO_MAX_K; ++b) {
                if (b < fan) {
                    S += exp(a1[b] - m1);
                    Q += exp(a2[b] - m2);
                }
            }
            const double lS = m1 + log(S), lQ = m2 + log(Q);
            ls[me] += lS;
            lq[me] += lQ;
            write_chain(r, j, static_cast<float>(exp(2.0 * lS - lQ)));
        }
        __syncthreads();
    }
}

// rank of x among its siblings: number of entries that beat it (larger value, or equal value and lower index)
__device__ __forceinline__ bool beats(float v_other, int i_other, float v_me, int i_me) {
    return (v_other > v_me) || (v_other == v_me && i_other < i_me);
}

// Sort keys of the Extreme-b selection.  A float32 maps to an unsigned integer of the same order (sign bit flipped for
// non-negative values, all bits for negative ones); the leaf index goes below it, complemented, so that among equal
// values the lower index has the larger key.  "best" ranks large values first, "worst" small values first: the b
// leaves with the largest keys are the ones the ranking "value, ties to the lower leaf index" puts first.
__device__ __forceinline__ uint64_t extreme_key(float v, uint32_t leaf, bool worst) {
    uint32_t u = __float_as_uint(v);
    if ((u << 1) == 0u) u = 0u;                              // -0 and +0 compare equal
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    if (worst) u = ~u;
    return (static_cast<uint64_t>(u) << 32) | static_cast<uint64_t>(~leaf);
}

// The want-th largest key among the tree's leaves (1 <= want <= L): radix selection, eight passes of eight bits over
// the 64-bit keys; every pass histograms the keys that share the prefix fixed so far and finds the digit by a sum over
// the bins from above.  Keys are distinct (they hold the leaf index), so exactly `want` leaves have a key >= the result.
// Called by the whole CTA, one thread per bin.
struct SelectSmem {
    unsigned int hist[256], warp_sum[kTreeThreads / 32];
    uint64_t prefix;
    int want;
};
static_assert(kTreeThreads == 256, "one thread per bin");

__device__ uint64_t select_kth_largest(const float* leaf_vals, int L, int want, bool worst, SelectSmem& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) { s.prefix = 0; s.want = want; }
    for (int pass = 7; pass >= 0; --pass) {
        s.hist[threadIdx.x] = 0u;
        __syncthreads();
        const uint64_t prefix = s.prefix;
        const int left = s.want;
        const int shift = 8 * pass;
        for (int l = threadIdx.x; l < L; l += kTreeThreads) {
            const uint64_t key = extreme_key(leaf_vals[l], static_cast<uint32_t>(l), worst);
            const bool same_prefix = (pass == 7) || ((key >> (shift + 8)) == (prefix >> (shift + 8)));
            if (same_prefix) atomicAdd(&s.hist[static_cast<unsigned int>(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        const int bin = 255 - static_cast<int>(threadIdx.x);        // thread 0 holds the largest digit
        const unsigned int count = s.hist[bin];
        unsigned int upto = count;                                  // keys of this digit or a larger one
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int x = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += x;
        }
        if (lane == 31) s.warp_sum[warp] = upto;
        __syncthreads();
        for (int w = 0; w < warp; ++w) upto += s.warp_sum[w];
        if (upto >= static_cast<unsigned int>(left) && upto - count < static_cast<unsigned int>(left)) {      // one thread
            s.want = left - static_cast<int>(upto - count);
            s.prefix = prefix | (static_cast<uint64_t>(bin) << shift);
        }
        __syncthreads();
    }
    return s.prefix;
}

// Up to this many leaves Extreme-b counts, for every leaf, the leaves that beat it (L^2 comparisons, no barrier): 27
// leaves 42 -> 6.3 us for the launch.  Beyond it the radix selection's sixteen passes (about 1 us each) are cheaper.
constexpr int kRankLeaves = 512;

__global__ void __launch_bounds__(kTreeThreads)
prune_kernel(const __grid_constant__ PruneLaunch p) {
    pdl_release();
    extern __shared__ unsigned char s_kept[];      // one flag per chain, when they fit
    __shared__ Layout lay;
    __shared__ float s_leaf[kRankLeaves];
    __shared__ SelectSmem sel;
    const int tree = blockIdx.x;
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    const int T = p.T, R = p.runs.n;
    const float* rbar = p.rbar + row0;
    uint8_t* mask = p.mask + row0;
    lay.fill(p.lv, p.runs, T);
    __syncthreads();
    const int chains = p.runs.chain0[R];
    const bool in_smem = static_cast<size_t>(chains) <= kTreeSmemLimit;
    if (!BGRPO_IN_BOUNDS(p.status, chains <= p.nodes && p.nodes <= p.nodes_cap && tree < p.n_trees)) return;
    auto depth_ok = [&](int d) { return d > 0 && !((p.pruned_bits >> (d - 1)) & 1ull) && !(p.ignore_last && d == T); };
    // Top-k modes: a node is kept iff, at every ranked fork on its root path, the ancestor (or the node itself) ranks
    // among the k best of its siblings.  Chain j of run r comes from chain j / F of run r - 1.
    auto path_kept = [&](int r, int j) -> bool {
        bool kept = true;
        for (; r > 0; --r) {
            const int d = p.runs.first[r], fan = p.lv.fanout[d - 1];
            const int pj = j / fan, b = j - pj * fan;
            const bool ranked = p.mode == BGRPO_WIDTH_PER_SPLIT_TOPK || (p.mode == BGRPO_WIDTH_LAST_SPLIT_TOPK && d - 1 == p.last_split);
            if (ranked) {
                const int sib0 = lay.off[d] + pj * fan;
                if (!BGRPO_IN_BOUNDS(p.status, sib0 >= 0 && sib0 + fan <= p.nodes)) break;
                float v[BGRPO_MAX_K];
#pragma unroll
                for (int q = 0; q < BGRPO_MAX_K; ++q) v[q] = q < fan ? rbar[sib0 + q] : 0.0f;
                const float me = b == 0 ? v[0] : b == 1 ? v[1] : b == 2 ? v[2] : v[3];
                int rank = 0;
#pragma unroll
                for (int q = 0; q < BGRPO_MAX_K; ++q)
                    if (q < fan && beats(v[q], q, me, b)) ++rank;
                kept = kept && rank < p.k;
            }
            j = pj;
        }
        return kept;
    };
    const bool extreme = p.mode == BGRPO_WIDTH_EXTREME_B;
    // What does not depend on earlier kernels is cleared before the wait: flags of the chains.
    if (extreme && in_smem)
        for (int m = threadIdx.x; m < chains; m += kTreeThreads) s_kept[m] = 0;
    pdl_wait();
    if (extreme) {
        const int L = p.lv.width[T], off = p.lv.offset[T];
        const int want = p.k < L ? p.k : L;
        if (!in_smem)      // the flags are gathered in the mask itself
            for (int n = threadIdx.x; n < p.nodes; n += kTreeThreads) mask[n] = 0;
        uint64_t best_cut = 0, worst_cut = 0;
        const bool by_rank = L <= kRankLeaves;
        if (by_rank)
            for (int l = threadIdx.x; l < L; l += kTreeThreads) s_leaf[l] = rbar[off + l];
        __syncthreads();                                   // also orders the zero fill before the flags below
        if (!by_rank) {
            best_cut = select_kth_largest(rbar + off, L, want, false, sel);
            __syncthreads();
            worst_cut = select_kth_largest(rbar + off, L, want, true, sel);
        }
        for (int l = threadIdx.x; l < L; l += kTreeThreads) {
            const float v = by_rank ? s_leaf[l] : rbar[off + l];
            const uint64_t best = extreme_key(v, static_cast<uint32_t>(l), false), worst = extreme_key(v, static_cast<uint32_t>(l), true);
            bool chosen;
            if (by_rank) {
                int above = 0, below = 0;
#pragma unroll 4
                for (int o = 0; o < L; ++o) {
                    above += extreme_key(s_leaf[o], static_cast<uint32_t>(o), false) > best ? 1 : 0;
                    below += extreme_key(s_leaf[o], static_cast<uint32_t>(o), true) > worst ? 1 : 0;
                }
                chosen = above < want || below < want;
            } else {
                chosen = best >= best_cut || worst >= worst_cut;
            }
            if (!chosen) continue;
            for (int r = R - 1, j = l; r >= 0; --r) {      // root path (several threads may write the same 1)
                if (in_smem) s_kept[lay.chain0[r] + j] = 1;
                else
                    for (int d = p.runs.first[r]; d < p.runs.first[r + 1]; ++d)
                        if (depth_ok(d)) mask[lay.off[d] + j] = 1;
                if (r > 0) j /= p.lv.fanout[p.runs.first[r] - 1];
            }
        }
        if (!in_smem) return;
    } else if (in_smem) {
        for (int m = threadIdx.x; m < chains; m += kTreeThreads) {
            int r = 0;
            while (m >= lay.chain0[r + 1]) ++r;
            s_kept[m] = path_kept(r, m - lay.chain0[r]) ? 1 : 0;
        }
    }
    __syncthreads();
    // Runs narrower than the CTA (the first ones) node by node, wider ones chain by chain, which is a store per node and no search
    // for its depth: Extreme-b on 241 000 nodes (64 depths, 4 096 leaves) 212 us with the search for every node, now 68.
    int d = 0;
    for (int n = threadIdx.x; n < p.narrow_nodes; n += kTreeThreads) {
        while (n >= lay.off[d + 1]) ++d;
        const int r = lay.run[d], j = n - lay.off[d];
        const bool kept = depth_ok(d) && (in_smem ? s_kept[lay.chain0[r] + j] != 0 : path_kept(r, j));
        mask[n] = kept ? 1 : 0;
    }
    for (int r = p.wide_run; r < R; ++r) {
        const int W = lay.chain0[r + 1] - lay.chain0[r];
        for (int j = threadIdx.x; j < W; j += kTreeThreads) {
            const uint8_t kept = s_kept[lay.chain0[r] + j];
            uint8_t* m = mask + lay.off[p.runs.first[r]] + j;
#pragma unroll 4
            for (int e = p.runs.first[r]; e < p.runs.first[r + 1]; ++e, m += W) *m = depth_ok(e) ? kept : 0;
        }
    }
}

// Clipped GRPO objective (Eq. 5), forward value: one CTA per tree; per-thread strided sums, fixed-order reduction.  The loads
// of kObjBatch nodes are in flight together: the kernel waits for memory once or twice, not once per node and operand.
constexpr int kObjBatch = 4;

__global__ void __launch_bounds__(kTreeThreads)
objective_kernel(const __grid_constant__ ObjectiveLaunch p) {
    pdl_release();
    const int tree = blockIdx.x;
    const int64_t row0 = static_cast<int64_t>(tree) * p.nodes_cap;
    double sum = 0.0;
    int cnt = 0;
    if (!BGRPO_IN_BOUNDS(p.status, p.nodes <= p.nodes_cap && tree < p.n_trees)) return;
    const double lo = 1.0 - static_cast<double>(p.clip_eps), hi = 1.0 + static_cast<double>(p.clip_eps);
    pdl_wait();
    for (int n0 = threadIdx.x; n0 < p.nodes; n0 += kTreeThreads * kObjBatch) {
        float ln[kObjBatch], lold[kObjBatch], av[kObjBatch];
        bool on[kObjBatch];
#pragma unroll
        for (int i = 0; i < kObjBatch; ++i) {
            const int n = n0 + i * kTreeThreads;
            const bool in = n < p.nodes;
            ln[i] = in ? p.logp_new[row0 + n] : 0.0f;
            lold[i] = in ? p.logp_old[row0 + n] : 0.0f;
            av[i] = in ? p.adv[row0 + n] : 0.0f;
            on[i] = in && n > 0 && p.mask[row0 + n] != 0;
        }
#pragma unroll
        for (int i = 0; i < kObjBatch; ++i) {
            const int n = n0 + i * kTreeThreads;
            float term = 0.0f;
            if (on[i]) {
                const double rho = exp(p.logp_scale * (static_cast<double>(ln[i]) - static_cast<double>(lold[i])));
                const double a = static_cast<double>(av[i]);
                const double t = fmin(rho * a, fmin(fmax(rho, lo), hi) * a);
                sum += t;
                cnt += 1;
                term = static_cast<float>(t);
            }
            if (p.terms && n < p.nodes) p.terms[row0 + n] = term;
        }
    }
    __shared__ double ssum[kTreeThreads / 32];
    __shared__ int scnt[kTreeThreads / 32];
    sum = warp_sum_d(sum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0) { ssum[threadIdx.x >> 5] = sum; scnt[threadIdx.x >> 5] = cnt; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        int c = 0;
        for (int w = 0; w < kTreeThreads / 32; ++w) { s += ssum[w]; c += scnt[w]; }
        p.J[tree] = c > 0 ? static_cast<float>(s / c) : 0.0f;
    }
}

SharedMemoryLimit g_limit_ess(reinterpret_cast<const void*>(&fusion_ess_kernel), kTreeSmemLimit);
SharedMemoryLimit g_limit_fuse(reinterpret_cast<const void*>(&fuse_advantage_kernel), kTreeSmemLimit);
SharedMemoryLimit g_limit_prune(reinterpret_cast<const void*>(&prune_kernel), kTreeSmemLimit);

}  // namespace

cudaError_t launch_objective(const ObjectiveLaunch& p, cudaStream_t s) {
    return launch_overlapped(objective_kernel, p.n_trees, kTreeThreads, 0, s, p);
}

cudaError_t launch_fusion_ess(const EssLaunch& p, cudaStream_t s) {
    size_t smem = static_cast<size_t>(p.runs.chain0[p.runs.n]) * 2 * sizeof(double);
    if (smem > kTreeSmemLimit) smem = 0;          // per-chain state in the caller's scratch
    if (smem > kSharedWithoutAsking) {
        const cudaError_t e = g_limit_ess.allow();
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(fusion_ess_kernel, p.n_trees, kTreeThreads, smem, s, p);
}

cudaError_t launch_fuse_advantage(const FuseLaunch& p, cudaStream_t s) {
    size_t smem = static_cast<size_t>(p.runs.chain0[p.runs.n]) * 2 * sizeof(double);
    if (smem > kTreeSmemLimit) smem = 0;          // per-chain state in the caller's scratch
    if (smem > kSharedWithoutAsking) {
        const cudaError_t e = g_limit_fuse.allow();
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(fuse_advantage_kernel, p.n_trees, kTreeThreads, smem, s, p);
}

cudaError_t launch_prune(const PruneLaunch& p0, cudaStream_t s) {
    PruneLaunch p = p0;
    size_t smem = static_cast<size_t>(p.runs.chain0[p.runs.n]);
    p.wide_run = p.runs.n;
    if (smem > kTreeSmemLimit) smem = 0;          // the paths are walked node by node, Extreme-b flags live in the mask
    else
        while (p.wide_run > 0 && p.runs.chain0[p.wide_run] - p.runs.chain0[p.wide_run - 1] >= kTreeThreads) --p.wide_run;
    p.narrow_nodes = p.lv.offset[p.runs.first[p.wide_run]];
    if (smem > kSharedWithoutAsking) {
        const cudaError_t e = g_limit_prune.allow();
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(prune_kernel, p.n_trees, kTreeThreads, smem, s, p);
}

}  // namespace bgrpo

// Per-token MLP velocity stage on the 5th-generation tensor cores (tcgen05 + tensor memory):
//     v = GELU(bf16(z) W1) W2,   z: [tokens][64] fp32,  W1: [64][H],  W2: [H][64] bf16,  fp32 accumulation, fp32 output.
// It stands in for the denoiser mu_theta of Eq. 2 and is evaluated once per PARENT node of the frontier; the
// K children of a parent share the result (the saving the rollout tree exists for).
//
// One persistent CTA per SM walks 128-token tiles.  For each tile the hidden dimension is cut into chunks of 128:
//     GEMM1(c): D1[128 tok][128 hid]  = A[128 tok][64]      * 2 W1_c      (4 MMAs of K = 16, accumulator in TMEM)
//     GELU     : H_c = bf16(kappa E(D1 / 2)), E(x) = GELU(x) - x / 2, TMEM -> registers -> TMEM: it never leaves tensor memory
//     GEMM2(c): D2[128 tok][64]      += H_c[128 tok][128]   * W2_c        (8 MMAs of K = 16, A operand read from TMEM)
// where D2 starts as A * (kappa W1 W2 / 2), the linear half of GELU (a 64 x 64 matrix held as the sum of two bf16 ones, 8 MMAs a
// tile), and the output tile is v = D2 / kappa.  Only the even half E goes through bf16, and as |E| is a fraction of |x| / 2 its
// roundings weigh less than those of the whole activation: rms error against 64 bits 1.6e-3 of rms(v), where 2.5e-3 was reached with
// bf16(GELU), and a polynomial with one coefficient less (1 036 800 tokens, hidden 3072: 712 -> 705 us, 16 200 tokens 17.3 -> 16.5).
// Tensor memory (512 columns): three chunk buffers of 128 columns and two output accumulators of 64.  A chunk buffer
// holds D1 of its chunk and then, in place, the packed activations: a warp reads its 64 accumulator columns into
// registers and later writes its 32 packed columns over the first half of exactly those columns, so no warp ever writes
// what another still has to read.  The buffer is free again when GEMM2 of the chunk has completed.  Three buffers for two
// epilogue groups mean that GEMM1 of chunk c + 2 does not wait for the group that works on chunk c, and the group does
// not wait for GEMM2 of chunk c - 2: the roles only meet at "accumulator ready" and "activations ready".
// Warp roles:
//     warp 0       streams the packed weights with bulk asynchronous copies: lane 0 feeds a 3-stage ring of W1 chunks,
//                  lane 1 a 4-stage ring of W2 chunks;
//     warp 1       owns tensor memory and issues GEMM1 into the buffer of the chunk (chunk index mod 3);
//     warp 19      issues GEMM2 from the same buffer once the chunk's activations are in it;
//     warps 2..17  GELU epilogue in two groups of eight: group p takes the chunks of parity p, two warps per TMEM lane
//                  quarter with 64 columns each.  All sixteen warps write the output tile (D2 is double-buffered, and a
//                  tile is written out two chunks after its last GEMM2 was issued, when it has long completed);
//     warps 20..27 (where the step is taken along with whole tiles) make the children of the tile before;
//     warp 18      brings the NEXT tile's latents in with bulk asynchronous copies (one per tree the tile touches) into
//                  a float32 staging buffer and converts them to the bf16 A tile while the current tile computes.  (Plain
//                  loads from one warp kept only 4 KiB in flight and took longer per tile than the arithmetic.)  The
//                  first tile of a launch is loaded and converted by the sixteen epilogue warps, idle until then.
// Shared-memory operands are K-major tiles of 128-byte rows in the 128-byte-swizzle layout the MMA descriptors
// address; the weights are reordered once into exactly that image (bgrpo_velocity_mlp_pack), so a chunk arrives with
// one copy per matrix.  No cluster multicast is used anywhere.
//
// Small frontiers (fewer tiles than SMs) are cut along the hidden dimension as well: a cluster of S = 2 to 8 CTAs shares
// a tile, each takes 1/S of the chunks and leaves its partial output tile in its shared memory; then each adds 1/S of the
// rows over all S parts, in part order, and writes them to v.
//
// Every wait is bounded (about 2 s of SM clock): on a timeout the thread raises the abort flag, all roles drain, tensor memory is
// released and bit 2 of the status word is set.
#include <cuda_bf16.h>

#include <cstring>
#include <mutex>

#include "internal.h"
#include "philox.cuh"

namespace bgrpo {
namespace {

constexpr int kTok = 128;                 // tokens per tile = MMA M
constexpr int kCh = 64;                   // channels = K of GEMM1 = N of GEMM2
constexpr int kHc = 128;                  // hidden chunk = N of GEMM1 = K of GEMM2
constexpr int kW1Stages = 3;               // W1 slot q is free again when the GEMM1 that read it has completed
constexpr int kW2Stages = 4;               // W2 slot q is free again when the GEMM2 that read it has completed
constexpr int kMaxSplit = 8;               // CTAs of a cluster that share a tile
constexpr int kEpiWarps = 16;             // two groups of eight: two warps per TMEM lane quarter, 64 columns of a chunk each
constexpr int kLoaderWarp = 2 + kEpiWarps;
constexpr int kGemm2Warp = 3 + kEpiWarps;
constexpr int kStepWarps = 8;              // make the children of whole tiles; four: 880 us where eight take 842 (see launch_mlp), twelve 909
// What a launch does besides the velocity: nothing, or the step that follows, where tiles are split over a cluster or whole.
enum { kNoStep = 0, kStepOfSplit = 1, kStepOfWhole = 2 };
template <int MODE>
constexpr int kMlpThreads = (4 + kEpiWarps + (MODE == kStepOfWhole ? kStepWarps : 0)) * 32;
constexpr uint32_t kTileBytes = kTok * 128;              // one [128 rows][128 B] operand tile = 16 KiB
constexpr uint32_t kChunkBytes = 2 * kTileBytes;         // packed weights of a chunk: W1_c (16 KiB) then W2_c (16 KiB)
constexpr uint32_t kTmemCols = 512;       // three chunk buffers of 128 columns (index = chunk mod 3), then D2: 2 x 64 (index = tile parity)
constexpr int kBufs = 3;
constexpr uint32_t kD2Col = kBufs * kHc;
constexpr int kGroupWarps = kEpiWarps / 2; // epilogue warps that work on one chunk
constexpr long long kWaitCycles = 4000000000ll;      // about two seconds of SM clock

template <int MODE>
struct MlpSmem {
    alignas(1024) unsigned char w1[kW1Stages][kTileBytes];  // W1_c tile [128 n = hidden][128 B = 64 channels]
    alignas(1024) unsigned char w2[kW2Stages][kTileBytes];  // W2_c as two [64 n = channel][128 B = 64 hidden] tiles
    alignas(1024) unsigned char a[2][kTileBytes];           // bf16(z) tile [128 tok][128 B], double-buffered over tiles
    alignas(1024) float stage[kTok * kCh];                   // float32 latents of the next tile, as they are in global memory; split
                                                             // mode, at the end: this CTA's partial output tile
    alignas(1024) float vtile[MODE == kStepOfWhole ? kTok * kCh : 4];     // velocities of the tile whose children are being made
    unsigned long long v_full, v_free;
    unsigned long long w1_full[kW1Stages], w1_free[kW1Stages], w2_full[kW2Stages], w2_free[kW2Stages];
    unsigned long long stage_full, first_a, a_full[2], a_empty[2], d1_full[kBufs], h_full[kBufs], buf_free[kBufs], d2_full[2], d2_empty[2];
    uint32_t node_sums[MODE == kStepOfSplit ? kTok : 1][BGRPO_MAX_K][2];    // the step taken along: squares of the noise by parent in the tile and child, low 16 bits and the rest
    uint32_t tmem_base;
    int abort_flag;
};

// Position in a ring of N slots: slot index, phase parity of the slot's current use, and whether the ring has
// wrapped yet (before that, "slot is free" needs no wait).
template <int N>
struct Ring {
    int slot = 0;
    uint32_t phase = 0;
    bool wrapped = false;
    __device__ __forceinline__ void advance() {
        if (++slot == N) { slot = 0; phase ^= 1u; wrapped = true; }
    }
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bounded wait for the phase of the given parity; false once kWaitCycles have passed or another thread has raised the
// abort flag.  The loop is nothing but the hardware's own try_wait (which parks the thread until the phase completes or
// its internal time slice ends): the clock and the abort flag are looked at once every 64 polls, so a handoff between
// two roles costs the barrier's latency and not a poll of timers and flags on top.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity, volatile int* abort_flag) {
    const uint32_t addr = smem_u32(bar);
    long long t0 = 0;
    for (uint32_t polls = 1;; ++polls) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
        if ((polls & 63u) == 0u) {
            if (*abort_flag) return false;
            const long long now = clock64();
            if (t0 == 0) t0 = now;
            else if (now - t0 > kWaitCycles) { *abort_flag = 1; return false; }
        }
    }
}
// True in exactly one lane of a converged warp.  Code guarded by it is known to the compiler to run in a single
// lane, which lets the tensor-core instructions take their operands from uniform registers directly (issued under
// `lane == 0` instead, each MMA cost about twice as many issue cycles on B200).
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred P1;\n\t.reg .b32 R1;\n\telect.sync R1|P1, 0xffffffff;\n\tselp.u32 %0, 1, 0, P1;\n\t}" : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src_gmem, uint32_t bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst_smem)), "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Shared-memory operand descriptor of a K-major tile of 128-byte rows in the 128-byte-swizzle layout: start address
// >> 4 in bits 0-13, leading offset 16 B (unused with swizzle) in bits 16-29, stride between 8-row groups (1024 B) >> 4
// in bits 32-45, descriptor version 1 in bits 46-47, layout type 2 (128-byte swizzle) in bits 61-63.
// Split in words: only the low word depends on the address, and advancing by n bytes adds n >> 4.
constexpr uint32_t kDescHi = 64u | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(const void* smem_ptr) { return ((smem_u32(smem_ptr) >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint64_t desc64(uint32_t lo) { return (static_cast<uint64_t>(kDescHi) << 32) | lo; }
// kind::f16 instruction descriptor: D = f32, A = B = bf16, both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Same with the A operand in tensor memory: 128 lanes (token rows) x 8 columns, each 32-bit column holding two
// consecutive bf16 elements of K.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// The mbarrier receives one arrival when every MMA this thread has issued so far has completed.
__device__ __forceinline__ void umma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Waits for the thread's outstanding TMEM loads.  The destination registers of the load are named as read-write
// operands so that every later use of them stays behind the wait.
__device__ __forceinline__ void tmem_ld_wait16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                   "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :: "memory");
}
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                   "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]),
                   "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]),
                   "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// GELU(x) = x / 2 + E(x) with E(x) = x erf(x / sqrt 2) / 2 even.  The packed W1 is 2 W1, so the accumulator of GEMM1 is y = 2x,
// and what GEMM2 gets for an activation is kappa E(x); the linear part is a product with kappa W1 W2 / 2.
//
// kappa E in the tanh form on the hardware tanh: kappa x / 2 tanh(sqrt(2/pi) (x + 0.044715 x^3)).  The tanh form
// differs from the erf form by < 5e-4 absolute, below the bf16 rounding of the activation that follows.  One
// special-function instruction per activation: this is the slow, range-free form, used only where the packed polynomial
// below does not apply.
constexpr float kKappa = 11.144685745239258f, kInvKappa = static_cast<float>(1.0 / 11.144685745239258);
__device__ __forceinline__ float even_tanh(float y) {
    const float x = 0.5f * y, x2 = x * x;
    const float u = x * fmaf(x2, 0.0356774081f, 0.7978845608f);
    float th;
    asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(u));
    return 0.25f * kKappa * (y * th);
}
// Packed bf16 arithmetic on two activations at a time (one FMA-pipe instruction for both halves).
__device__ __forceinline__ uint32_t bf2_mul(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t bf2_fma(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// kappa E(x) for |x| < 1 without a special-function instruction: t (R0 + R1 t), t = y^2 (csrc/gelu_poly_fit.py; within 3.1e-4 of
// E, and E is rounded to bf16 at once).  kappa is what gives both coefficients short bf16 forms.  Two multiplies and one fused
// multiply-add on a packed pair, where one hardware tanh per activation (sixteen per clock and SM) bounds the whole stage at twice
// the tensor-core time.  (In float32 on pairs, fma.f32x2, three of them for a cubic: 747 us for 1 036 800 tokens.)
constexpr uint32_t kEvenR0 = 0x3f8d3f8du;   //  1.1015625
constexpr uint32_t kEvenR1 = 0xbd1bbd1bu;   // -0.037841796875
__device__ __forceinline__ uint32_t even_poly(uint32_t y) {
    const uint32_t t = bf2_mul(y, y);
    return bf2_mul(t, bf2_fma(kEvenR1, t, kEvenR0));
}
// The polynomial's range |x| < 1 is |y| < 2: the top exponent bit of both bf16 halves clear.  One bit to look at is why y
// is doubled: the check of 32 packed pairs is 16 three-operand ORs where a running maximum of magnitudes took 32
// operations (1 036 800 tokens, hidden 3072: 733 -> 719 us).  NaN and infinity have the bit set.
constexpr uint32_t kEvenOutside = 0x40004000u;
// byte offset of the 16-byte piece `c16` of row r inside a 128-byte-swizzled tile of 128-byte rows
__device__ __forceinline__ uint32_t sw128(uint32_t r, uint32_t c16) { return r * 128u + ((c16 ^ (r & 7u)) << 4); }

// Converts the float32 staging tile to the bf16 K-major swizzled A tile; one warp, two rows per
// step (16 lanes x 16 bytes cover a row).  Rows from `valid` on lie past the last token and are made zero first: left to
// what the staging buffer held before, a few NaNs sent the rows of a ragged last tile through the slow activation, and
// with one tile per CTA that CTA took twice as long as all others (16 200 tokens, hidden 3072: 31 us in place of 16).
__device__ __forceinline__ void convert_tile(float* stage, unsigned char* atile, int valid, int lane) {
    const uint32_t c4 = static_cast<uint32_t>(lane & 15);
    if (valid < kTok)         // at most once in a launch
        for (int r = lane >> 4; r < kTok; r += 2)
            if (r >= valid) *reinterpret_cast<float4*>(stage + r * kCh + c4 * 4u) = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int r0 = 0; r0 < kTok; r0 += 2) {
        const uint32_t r = static_cast<uint32_t>(r0 + (lane >> 4));
        const float4 zv = *reinterpret_cast<const float4*>(stage + r * kCh + c4 * 4u);
        uint2 packed2;
        packed2.x = pack_bf16(zv.x, zv.y);
        packed2.y = pack_bf16(zv.z, zv.w);
        *reinterpret_cast<uint2*>(atile + sw128(r, c4 >> 1) + (c4 & 1u) * 8u) = packed2;
    }
}

// Thread-block cluster: barrier over all threads of its CTAs (release / acquire), load from another CTA's shared memory.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ float4 cluster_load(uint32_t addr, uint32_t rank) {
    uint32_t remote;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote) : "memory");
    return v;
}
// 16-byte piece c4 of row r of a partial output tile; rows are staggered so that a warp's row-per-thread stores and its
// row-by-row loads both spread over the banks
__device__ __forceinline__ float4* part_piece(float* tile, uint32_t r, uint32_t c4) {
    return reinterpret_cast<float4*>(tile) + r * (kCh / 4) + (c4 ^ (r & (kCh / 4 - 1)));
}

struct MlpArgs {
    const float* latents;     // pool base
    int64_t pool_elems;       // elements in the pool
    int64_t tree_stride;      // elements between trees in the pool
    int64_t row_offset;       // elements from a tree's base to its frontier
    int64_t tokens_per_tree;  // frontier tokens of one tree (W_i * tokens)
    int64_t n_tokens;         // all frontier tokens
    const unsigned char* packed;
    float* v_out;             // nullptr: the step is taken along and the velocities are not kept
    int32_t n_chunks;         // hidden / 128
    int32_t n_tiles;
    int32_t split;            // CTAs per tile along the hidden dimension (1: none); > 1 only with one tile per cluster of that size
    int32_t* status;
    int32_t tokens;           // of a node
    unsigned long long* row_sums;
};

// One float4 of a parent of the step taken along: where it is, and the noise of its children.
struct StepPiece {
    bool live;
    int32_t row, node0;       // frontier row (tree * W + j) and first child's row in the pool
    uint32_t e;               // float4 index in the row
    float4 z, xi[BGRPO_MAX_K];
    uint32_t squares[BGRPO_MAX_K];
};
__device__ __forceinline__ void step_piece(const StepLaunch& sp, const MlpArgs& p, int64_t first, uint32_t r, uint32_t c4, StepPiece& q) {
    const uint32_t token = static_cast<uint32_t>(first) + r;          // fewer than 2^15: one tile per cluster
    q.live = r < kTok && token < p.n_tokens;
    if (!q.live) return;
    q.row = static_cast<int32_t>(token / static_cast<uint32_t>(p.tokens));
    q.e = (token - static_cast<uint32_t>(q.row) * p.tokens) * (kCh / 4) + c4;
    const int tree = q.row / sp.W_in, j = q.row - tree * sp.W_in;
    const int32_t parent = tree * sp.nodes_cap + sp.off_in + j;
    q.node0 = tree * sp.nodes_cap + sp.off_out + j * sp.fan;
    q.live = BGRPO_IN_BOUNDS(sp.status, tree < sp.n_trees && sp.off_in + j < sp.nodes_cap && sp.off_out + (j + 1) * sp.fan <= sp.nodes_cap && q.e < sp.D / 4);
    if (!q.live) return;
    q.z = __ldcs(reinterpret_cast<const float4*>(sp.latents + parent * sp.D) + q.e);
    if (q.e == 0u) {          // node-table rows of the new children
        const int64_t rows = static_cast<int64_t>(sp.n_trees) * sp.nodes_cap;
        for (int b = 0; b < sp.fan; ++b) {
            const int64_t r = q.node0 + b;
            sp.table[r] = sp.off_in + j;
            sp.table[rows + r] = sp.step + 1;
            sp.table[2 * rows + r] = sp.is_split ? sp.step : sp.table[2 * rows + parent];
            sp.table[3 * rows + r] = sp.is_split ? b : sp.table[3 * rows + parent];
        }
    }
    if (sp.g == 0.0f) return;
    float squares;
    float4 xi0;
    if (sp.shared_noise)
        xi0 = mul4(sp.mix_shared, normal4(philox_from(noise_element(q.e, BGRPO_TAG_SHARED, sp.keys), noise_node(sp.node_id_base + parent, sp.step, sp.keys), sp.keys), squares));
    const NoiseElement el = noise_element(q.e, BGRPO_TAG_INNOV, sp.keys);
#pragma unroll
    for (int b = 0; b < BGRPO_MAX_K; ++b)
        if (b < sp.fan) {
            q.xi[b] = normal4(philox_from(el, noise_node(sp.node_id_base + q.node0 + b, sp.step, sp.keys), sp.keys), squares);
            if (sp.shared_noise) {
                q.xi[b] = fma4(sp.mix_innov, q.xi[b], xi0);
                squares = squares_of(q.xi[b]);
            }
            q.squares[b] = quantized_squares(squares);
        }
}
// The children of one float4, given the velocity; adds the squares of a token (16 lanes) to the node's sums.
__device__ __forceinline__ void step_children(const StepLaunch& sp, int row0, const StepPiece& q, const float4& v, uint32_t (*node_sums)[BGRPO_MAX_K][2]) {
    const float4 m = fma4(sp.ca, q.z, mul4(sp.cb, v));
    float4* child = reinterpret_cast<float4*>(sp.latents + q.node0 * sp.D) + q.e;
    const uint32_t half = 0xffffu << (threadIdx.x & 16u);
#pragma unroll
    for (int b = 0; b < BGRPO_MAX_K; ++b)
        if (b < sp.fan) {
            child[b * (sp.D / 4)] = sp.g == 0.0f ? m : fma4(sp.g, q.xi[b], m);
            if (sp.g != 0.0f) {
                const uint32_t lo = __reduce_add_sync(half, q.squares[b] & 0xffffu), hi = __reduce_add_sync(half, q.squares[b] >> 16);
                if ((threadIdx.x & 15u) == 0u) {        // 128 tokens of 16 lanes: 27 bits.  (A 64-bit add would be a loop.)
                    atomicAdd(&node_sums[q.row - row0][b][0], lo);
                    atomicAdd(&node_sums[q.row - row0][b][1], hi);
                }
            }
        }
}

// A whole tile of the step taken along, of nodes of at least kTok tokens: it touches two nodes at most, A up to row `edge` and
// B behind it.  Addresses and element numbers are those of row 0, so that a row is one multiply-add away from its own.
struct StepTile {
    int32_t rows, edge;
    const float4 *z_a, *z_b;
    float4 *child_a, *child_b;        // first child
    uint32_t e_a, e_b;
    int32_t parent_a, parent_b, child0_a, child0_b;       // rows of the pool
};
__device__ __forceinline__ StepTile make_step_tile(const StepLaunch& sp, const MlpArgs& p, int64_t first_token, int rows) {
    StepTile q;
    const uint32_t tokens = static_cast<uint32_t>(p.tokens), first = static_cast<uint32_t>(first_token);      // a pool of 2^32 tokens is 1 TB
    const uint32_t row = first / tokens, tok = first - row * tokens;
    q.rows = rows;
    q.edge = tokens - tok < static_cast<uint32_t>(kTok) ? static_cast<int32_t>(tokens - tok) : kTok;
    auto node = [&](int32_t n, int32_t tok0, const float4*& z, float4*& child, uint32_t& e, int32_t& parent, int32_t& child0) {
        const int32_t tree = n / sp.W_in, j = n - tree * sp.W_in;
        parent = tree * sp.nodes_cap + sp.off_in + j;
        child0 = tree * sp.nodes_cap + sp.off_out + j * sp.fan;
        if (tok0 < rows && !BGRPO_IN_BOUNDS(sp.status, tree < sp.n_trees && sp.off_in + j < sp.nodes_cap && sp.off_out + (j + 1) * sp.fan <= sp.nodes_cap)) q.rows = 0;
        e = static_cast<uint32_t>(-tok0) * (kCh / 4);
        z = reinterpret_cast<const float4*>(sp.latents + parent * sp.D) - static_cast<int64_t>(tok0) * (kCh / 4);
        child = reinterpret_cast<float4*>(sp.latents + child0 * sp.D) - static_cast<int64_t>(tok0) * (kCh / 4);
    };
    node(static_cast<int32_t>(row), -static_cast<int32_t>(tok), q.z_a, q.child_a, q.e_a, q.parent_a, q.child0_a);
    node(static_cast<int32_t>(row) + 1, q.edge, q.z_b, q.child_b, q.e_b, q.parent_b, q.child0_b);
    return q;
}
// Node-table row of a child: one thread per child.
__device__ __forceinline__ void step_table(const StepLaunch& sp, int32_t parent, int32_t child0, int b) {
    const int64_t rows = static_cast<int64_t>(sp.n_trees) * sp.nodes_cap, n = child0 + b;
    sp.table[n] = parent % sp.nodes_cap;
    sp.table[rows + n] = sp.step + 1;
    sp.table[2 * rows + n] = sp.is_split ? sp.step : sp.table[2 * rows + parent];
    sp.table[3 * rows + n] = sp.is_split ? b : sp.table[3 * rows + parent];
}
template <int N>
__device__ __forceinline__ void step_load(const StepTile& q, int32_t r0, int32_t stride, uint32_t c4, float4 (&z)[N]) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int32_t r = r0 + k * stride;
        if (r < q.rows) z[k] = __ldcg((r < q.edge ? q.z_a : q.z_b) + r * (kCh / 4) + c4);
    }
}
// Adds a warp's squares of child b to the nodes' sums: 32 numbers, their 16-bit halves by themselves.
__device__ __forceinline__ void add_squares(const MlpArgs& p, const StepTile& q, int b, uint32_t sum_a, uint32_t sum_b) {
    uint32_t lo = __reduce_add_sync(0xffffffffu, sum_a & 0xffffu), hi = __reduce_add_sync(0xffffffffu, sum_a >> 16);
    if ((threadIdx.x & 31u) == 0u && (lo | hi) != 0u) atomicAdd(p.row_sums + q.child0_a + b, (static_cast<unsigned long long>(hi) << 16) + lo);
    if (q.edge < kTok) {
        lo = __reduce_add_sync(0xffffffffu, sum_b & 0xffffu);
        hi = __reduce_add_sync(0xffffffffu, sum_b >> 16);
        if ((threadIdx.x & 31u) == 0u && (lo | hi) != 0u) atomicAdd(p.row_sums + q.child0_b + b, (static_cast<unsigned long long>(hi) << 16) + lo);
    }
}
// Node-table rows of the children whose nodes start in the tile.
__device__ __forceinline__ void step_tables(const StepLaunch& sp, const StepTile& q, uint32_t t) {
    if (t < static_cast<uint32_t>(sp.fan) && q.e_a == 0u && q.rows > 0) step_table(sp, q.parent_a, q.child0_a, t);
    if (t >= 32u && t - 32u < static_cast<uint32_t>(sp.fan) && q.edge < q.rows) step_table(sp, q.parent_b, q.child0_b, t - 32);
}
// The children of one float4 of N rows, given their velocities in shared memory: N chains of noise in flight.  `z` has the
// parents; once they are used `then` may ask for the next ones.  Whole warps.
template <int N, class Then>
__device__ __forceinline__ void step_rows(const StepLaunch& sp, const MlpArgs& p, const StepTile& q, int64_t first, int32_t r0, int32_t stride, uint32_t c4,
                                          float* vtile, float4 (&z)[N], Then then) {
    float4 m[N];
    NoiseElement el[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int32_t r = r0 + k * stride;
        if (r < q.rows) {
            const float4 v = *part_piece(vtile, static_cast<uint32_t>(r), c4);
            if (p.v_out) reinterpret_cast<float4*>(p.v_out)[(first + r) * (kCh / 4) + c4] = v;
            m[k] = fma4(sp.ca, z[k], mul4(sp.cb, v));
        }
    }
    then();
    if (sp.g != 0.0f)
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int32_t r = r0 + k * stride;
            const uint32_t e = (r < q.edge ? q.e_a : q.e_b) + static_cast<uint32_t>(r) * (kCh / 4) + c4;
            el[k] = noise_element(e, BGRPO_TAG_INNOV, sp.keys);
        }
#pragma unroll 1
    for (int b = 0; b < sp.fan; ++b) {
        float4* const child_a = q.child_a + b * (sp.D / 4);
        float4* const child_b = q.child_b + b * (sp.D / 4);
        if (sp.g == 0.0f) {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const int32_t r = r0 + k * stride;
                if (r < q.rows) (r < q.edge ? child_a : child_b)[r * (kCh / 4) + c4] = m[k];
            }
            continue;
        }
        const NoiseNode node_a = noise_node(sp.node_id_base + q.child0_a + b, sp.step, sp.keys), node_b = noise_node(sp.node_id_base + q.child0_b + b, sp.step, sp.keys);
        uint32_t sum_a = 0u, sum_b = 0u;          // N numbers at most of 25 bits
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int32_t r = r0 + k * stride;
            const bool in_a = r < q.edge;
            float squares;
            const float4 xi = normal4(philox_from(el[k], {node_a.x, in_a ? node_a.z : node_b.z, in_a ? node_a.w : node_b.w}, sp.keys), squares);
            if (r < q.rows) {
                const uint32_t n = quantized_squares(squares);
                if (in_a) sum_a += n;
                else sum_b += n;
                (in_a ? child_a : child_b)[r * (kCh / 4) + c4] = fma4(sp.g, xi, m[k]);
            }
        }
        add_squares(p, q, b, sum_a, sum_b);
    }
}
// The noise of a tile's only children ahead of its velocities, to shared memory (whole warps, 128 rows by THREADS threads); then,
// with the velocities there, the children by all threads of the CTA, up to N rows each.
template <int THREADS, int N>
__device__ __forceinline__ void step_tile_noise(const StepLaunch& sp, const MlpArgs& p, const StepTile& q, uint32_t t, float* xi_tile) {
    constexpr int kStride = THREADS / (kCh / 4);
    const uint32_t c4 = t % (kCh / 4);
    const NoiseNode node_a = noise_node(sp.node_id_base + q.child0_a, sp.step, sp.keys), node_b = noise_node(sp.node_id_base + q.child0_b, sp.step, sp.keys);
    uint32_t sum_a = 0u, sum_b = 0u;          // eight numbers at most of 25 bits
    static_assert(kTok / kStride <= 8, "the sums of a thread");
#pragma unroll 1
    for (int32_t r0 = static_cast<int32_t>(t / (kCh / 4)); r0 < kTok; r0 += N * kStride) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int32_t r = r0 + k * kStride;
            const bool in_a = r < q.edge;
            const NoiseElement el = noise_element((in_a ? q.e_a : q.e_b) + static_cast<uint32_t>(r) * (kCh / 4) + c4, BGRPO_TAG_INNOV, sp.keys);
            float squares;
            *part_piece(xi_tile, static_cast<uint32_t>(r), c4) = normal4(philox_from(el, {node_a.x, in_a ? node_a.z : node_b.z, in_a ? node_a.w : node_b.w}, sp.keys), squares);
            if (r < q.rows) {
                const uint32_t n = quantized_squares(squares);
                if (in_a) sum_a += n;
                else sum_b += n;
            }
        }
    }
    add_squares(p, q, 0, sum_a, sum_b);
}
template <int THREADS>
__device__ __forceinline__ void step_tile_children(const StepLaunch& sp, const MlpArgs& p, const StepTile& q, int64_t first, uint32_t t, float* vtile, float* xi_tile) {
    constexpr int kStride = THREADS / (kCh / 4), N = (kTok + kStride - 1) / kStride;
    const uint32_t c4 = t % (kCh / 4);
    const int32_t r0 = static_cast<int32_t>(t / (kCh / 4));
    float4 z[N];
    step_load<N>(q, r0, kStride, c4, z);
    step_tables(sp, q, t);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int32_t r = r0 + k * kStride;
        if (r < q.rows) {
            const float4 v = *part_piece(vtile, static_cast<uint32_t>(r), c4);
            if (p.v_out) reinterpret_cast<float4*>(p.v_out)[(first + r) * (kCh / 4) + c4] = v;
            (r < q.edge ? q.child_a : q.child_b)[r * (kCh / 4) + c4] = fma4(sp.g, *part_piece(xi_tile, static_cast<uint32_t>(r), c4), fma4(sp.ca, z[k], mul4(sp.cb, v)));
        }
    }
}
// All rows of a tile by THREADS threads, 16 to a row, N rows of a thread at a time.  `v_ready` waits for the velocities; the
// first parents are asked for before it.  (One row at a time: 849 us for 842; four rows of four warps, which spills, 893.)
constexpr int kStepRows = 2;
template <int THREADS, int N, class Wait>
__device__ __forceinline__ bool step_tile(const StepLaunch& sp, const MlpArgs& p, const StepTile& q, int64_t first, uint32_t t, float* vtile, Wait v_ready) {
    constexpr int kStride = THREADS / (kCh / 4);
    const uint32_t c4 = t % (kCh / 4);
    int32_t r = static_cast<int32_t>(t / (kCh / 4));
    float4 z[N];
    step_load<N>(q, r, kStride, c4, z);
    step_tables(sp, q, t);
    if (!v_ready()) return false;
#pragma unroll 1
    for (int32_t done = 0; done < kTok; done += N * kStride, r += N * kStride)
        step_rows<N>(sp, p, q, first, r, kStride, c4, vtile, z, [&] {
            if (done + N * kStride < kTok) step_load<N>(q, r + N * kStride, kStride, c4, z);
        });
    return true;
}

// kStepOfWhole: see step_tile().  kStepOfSplit: the tail has the velocity of its rows in registers, so it writes
// the children next to it, and the launch and the reload of a step kernel are saved.  What does not need the velocity - the
// parent, the noise, the table - is done while the cluster's barrier is on its way.
template <int MODE>
__global__ void __launch_bounds__(kMlpThreads<MODE>, 1)
mlp_velocity_kernel(const __grid_constant__ MlpArgs p, const __grid_constant__ StepLaunch sp) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // the swizzled operand tiles need 1024-byte alignment; the launch reserves 1 KiB of slack for this round-up
    using Smem = MlpSmem<MODE>;
    constexpr int kThreads = kMlpThreads<MODE>;
    constexpr bool STEP = MODE == kStepOfSplit, WHOLE = MODE == kStepOfWhole;
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    // The shuffle tells the compiler that the warp index is the same in all lanes: roles, ring positions and tensor-memory
    // addresses then live in uniform registers (1 036 800 tokens, hidden 3072: 775 -> 744 us; 7 200 tokens: 30.9 -> 29.3 us).
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abort_flag = &sm.abort_flag;

    if (threadIdx.x == 0) {
        for (int q = 0; q < kW1Stages; ++q) {
            mbar_init(&sm.w1_full[q], 1);
            mbar_init(&sm.w1_free[q], 1);
        }
        for (int q = 0; q < kW2Stages; ++q) {
            mbar_init(&sm.w2_full[q], 1);
            mbar_init(&sm.w2_free[q], 1);
        }
        mbar_init(&sm.stage_full, 1);
        mbar_init(&sm.first_a, kEpiWarps);
        mbar_init(&sm.v_full, kEpiWarps);
        mbar_init(&sm.v_free, kStepWarps);
        for (int q = 0; q < 2; ++q) {
            mbar_init(&sm.a_full[q], 1);
            mbar_init(&sm.a_empty[q], blockIdx.x % p.split == 0 ? 2 : 1);      // GEMM1 and, where this CTA has it, the linear part
            mbar_init(&sm.d2_full[q], 1);
            mbar_init(&sm.d2_empty[q], kEpiWarps);
        }
        for (int q = 0; q < kBufs; ++q) {
            mbar_init(&sm.d1_full[q], 1);
            mbar_init(&sm.h_full[q], kGroupWarps);
            mbar_init(&sm.buf_free[q], 1);
        }
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (STEP)
        for (int i = threadIdx.x; i < kTok * BGRPO_MAX_K * 2; i += kThreads) (&sm.node_sums[0][0][0])[i] = 0u;
    if (warp == 1) {      // tensor memory: this warp allocates and, at the end, frees
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Barriers and tensor memory are set up: the next kernel on the stream may be scheduled, and this one waits here for
    // the kernels before it (they wrote the latents and the packed weights, and may still be reading the output buffer).
    pdl_release();
    pdl_wait();
    const uint32_t tmem = sm.tmem_base;
    const int S = WHOLE ? 1 : p.split;
    const int cta = static_cast<int>(blockIdx.x) / S, part = static_cast<int>(blockIdx.x) - cta * S;   // tile walker, share of the hidden dimension
    const int n_ctas = static_cast<int>(gridDim.x) / S;
    const int n_my_tiles = (p.n_tiles > cta) ? (p.n_tiles - 1 - cta) / n_ctas + 1 : 0;
    const int NC = p.n_chunks / S;            // chunks this CTA adds up per tile: part * NC .. part * NC + NC - 1
    const int n_my_chunks = n_my_tiles * NC;
    const int lin = part == 0 ? 1 : 0;        // the first of a tile's CTAs adds the linear part

    auto tile_rows = [&](int it) -> int {     // tokens of this CTA's tile number `it`
        const int64_t left = p.n_tokens - (static_cast<int64_t>(cta) + static_cast<int64_t>(it) * n_ctas) * kTok;
        return left < kTok ? static_cast<int>(left) : kTok;
    };

    // The step of whole tiles: where a node has one child the noise of a CTA's last tile is drawn before its velocities are there.
    const bool ahead = WHOLE && sp.fan == 1 && sp.g != 0.0f;
    auto last_tile = [&]() -> StepTile {
        return make_step_tile(sp, p, (static_cast<int64_t>(cta) + static_cast<int64_t>(n_my_tiles - 1) * n_ctas) * kTok, tile_rows(n_my_tiles - 1));
    };
    auto a_ready = [&](int it) -> bool {      // the bf16 latents of tile number `it`: the first has a barrier of its own
        return it == 0 ? mbar_wait(&sm.first_a, 0u, abort_flag) : mbar_wait(&sm.a_full[it & 1], static_cast<uint32_t>((it - 1) >> 1) & 1u, abort_flag);
    };

    if (warp == 0) {
        // ---------------------------------------------------------------- weight producers (lane 0: W1, lane 1: W2)
        // Every tile adds its hidden chunks in index order, whatever CTA it lands on, so a token's output does not
        // depend on how many tokens the launch holds (a shard of a batch reproduces the batch's bits as long as neither
        // launch is cut along the hidden dimension).  Starting every CTA at its own chunk instead, to spread the L2
        // requests, measured the same.
        if (lane == 0) {
            Ring<kW1Stages> r;
            int cc = 0;
            for (int g = 0; g < n_my_chunks; ++g) {
                if (r.wrapped && !mbar_wait(&sm.w1_free[r.slot], r.phase ^ 1u, abort_flag)) break;    // GEMM1 that read this slot is done
                mbar_expect_tx(&sm.w1_full[r.slot], kTileBytes);
                bulk_load(sm.w1[r.slot], p.packed + static_cast<size_t>(part * NC + cc) * kChunkBytes, kTileBytes, &sm.w1_full[r.slot]);
                r.advance();
                if (++cc == NC) cc = 0;
            }
        } else if (lane == 1) {
            Ring<kW2Stages> r;
            int cc = -lin;        // -1: the linear part
            const int64_t n = static_cast<int64_t>(n_my_tiles) * (NC + lin);
            for (int64_t g = 0; g < n; ++g) {
                if (r.wrapped && !mbar_wait(&sm.w2_free[r.slot], r.phase ^ 1u, abort_flag)) break;    // GEMM2 that read this slot is done
                mbar_expect_tx(&sm.w2_full[r.slot], kTileBytes);
                bulk_load(sm.w2[r.slot], p.packed + (cc < 0 ? static_cast<size_t>(p.n_chunks) * kChunkBytes : static_cast<size_t>(part * NC + cc) * kChunkBytes + kTileBytes),
                          kTileBytes, &sm.w2_full[r.slot]);
                r.advance();
                if (++cc == NC) cc = -lin;
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- GEMM1 issuer
        // Two warps issue MMAs, one per GEMM, so that a GEMM1 held back by the tensor pipe never delays the GEMM2 the
        // epilogue is waiting for (and vice versa); completion tracking (tcgen05.commit) is per issuing thread.  The
        // whole warp walks the loop and waits; one elected lane issues.
        constexpr uint32_t idesc1 = umma_idesc(kTok, kHc);
        constexpr uint32_t kTileUnits = kTileBytes >> 4;
        const uint32_t a_lo = desc_lo(sm.a[0]), w1_lo = desc_lo(sm.w1[0]);
        bool ok = true;
        Ring<kW1Stages> r;        // weights of the next GEMM1
        Ring<kBufs> cb;           // chunk buffer of the next GEMM1: slot = chunk mod 3, phase = parity of its use number
        for (int it = 0; it < n_my_tiles && ok; ++it) {
            const int ab = it & 1;
            ok = __all_sync(0xffffffffu, a_ready(it) ? 1 : 0) != 0;
            const uint32_t a_cur = a_lo + static_cast<uint32_t>(ab) * kTileUnits;
            for (int c = 0; c < NC && ok; ++c) {            // D1[cb] = A * W1[r]
                ok = mbar_wait(&sm.w1_full[r.slot], r.phase, abort_flag);
                if (ok && cb.wrapped)  // GEMM2 of the chunk that used this buffer three chunks ago has read its activations
                    ok = mbar_wait(&sm.buf_free[cb.slot], cb.phase ^ 1u, abort_flag);
                ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t b_lo = w1_lo + static_cast<uint32_t>(r.slot) * kTileUnits;
                const uint32_t d = tmem + static_cast<uint32_t>(cb.slot) * kHc;
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kCh / 16; ++k)      // +32 bytes (2 descriptor units) per K step inside the swizzled row
                        umma_bf16(d, desc64(a_cur + 2u * k), desc64(b_lo + 2u * k), idesc1, k > 0 ? 1u : 0u);
                    umma_commit(&sm.d1_full[cb.slot]);
                    umma_commit(&sm.w1_free[r.slot]);
                }
                __syncwarp();
                r.advance();
                cb.advance();
            }
            if (ok && elect_one()) umma_commit(&sm.a_empty[ab]);       // every GEMM1 of this tile has been issued
            __syncwarp();
        }
    } else if (warp == kGemm2Warp) {
        // ---------------------------------------------------------------- GEMM2 issuer
        constexpr uint32_t idesc2 = umma_idesc(kTok, kCh);
        constexpr uint32_t kTileUnits = kTileBytes >> 4;
        const uint32_t w2_lo = desc_lo(sm.w2[0]), a_lo = desc_lo(sm.a[0]);
        bool ok = true;
        Ring<kW2Stages> rw;       // weights of the next GEMM2
        Ring<kBufs> cb;           // chunk buffer of the next GEMM2
        for (int it = 0; it < n_my_tiles && ok; ++it) {
            const uint32_t d2 = tmem + kD2Col + static_cast<uint32_t>(it & 1) * kCh;
            if (it >= 2)      // the tile that used this D2 buffer two tiles ago has been written out
                ok = __all_sync(0xffffffffu, mbar_wait(&sm.d2_empty[it & 1], static_cast<uint32_t>((it >> 1) - 1) & 1u, abort_flag) ? 1 : 0) != 0;
            if (ok && lin) {          // D2 = A * (kappa W1 W2 / 2), the matrix as the sum of two bf16 ones
                ok = mbar_wait(&sm.w2_full[rw.slot], rw.phase, abort_flag) && a_ready(it);
                ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_cur = a_lo + static_cast<uint32_t>(it & 1) * kTileUnits;
                const uint32_t wb_lo = w2_lo + static_cast<uint32_t>(rw.slot) * kTileUnits;
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < 2 * kCh / 16; ++k)
                        umma_bf16(d2, desc64(a_cur + 2u * (k % 4)), desc64(wb_lo + (k / 4) * ((kCh * 128) >> 4) + 2u * (k % 4)), idesc2, k > 0 ? 1u : 0u);
                    umma_commit(&sm.w2_free[rw.slot]);
                    umma_commit(&sm.a_empty[it & 1]);
                }
                __syncwarp();
                rw.advance();
            }
            for (int c = 0; c < NC && ok; ++c) {            // D2 += H[cb] * W2[rw]
                ok = mbar_wait(&sm.w2_full[rw.slot], rw.phase, abort_flag);
                if (ok) ok = mbar_wait(&sm.h_full[cb.slot], cb.phase, abort_flag);
                ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t h_col = tmem + static_cast<uint32_t>(cb.slot) * kHc;
                const uint32_t wb_lo = w2_lo + static_cast<uint32_t>(rw.slot) * kTileUnits;
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kHc / 16; ++k)      // hidden 16k .. 16k+15 of the chunk: 8 packed columns, the chunk's
                                                            // first 64 hidden units at columns 0..31 of the buffer, the rest at 64..95
                        umma_bf16_ts(d2, h_col + (k / 4) * 64u + 8u * (k % 4),
                                     desc64(wb_lo + (k / 4) * ((kCh * 128) >> 4) + 2u * (k % 4)), idesc2, (lin || c > 0 || k > 0) ? 1u : 0u);
                    umma_commit(&sm.buf_free[cb.slot]);
                    umma_commit(&sm.w2_free[rw.slot]);
                    if (c == NC - 1) umma_commit(&sm.d2_full[it & 1]);
                }
                __syncwarp();
                rw.advance();
                cb.advance();
            }
        }
    } else if (warp == kLoaderWarp) {
        // ---------------------------------------------------------------- latent tile -> staging -> bf16, K-major swizzled
        // Tokens of the frontier are numbered tree by tree; the rows of one tree are contiguous in the pool, so a tile is
        // one copy per tree it touches.
        auto issue_tile_copy = [&](int it) {       // one lane
            const int64_t tok0 = (static_cast<int64_t>(cta) + static_cast<int64_t>(it) * n_ctas) * kTok;
            int64_t remaining = tile_rows(it);
            mbar_expect_tx(&sm.stage_full, static_cast<uint32_t>(remaining) * (kCh * 4u));
            int64_t q = tok0;
            float* dst = sm.stage;
            while (remaining > 0) {
                const int64_t tree = q / p.tokens_per_tree, rr = q - tree * p.tokens_per_tree;
                int64_t seg = p.tokens_per_tree - rr;
                if (seg > remaining) seg = remaining;
                const int64_t first = tree * p.tree_stride + p.row_offset + rr * kCh;
                if (!BGRPO_IN_BOUNDS(p.status, first >= 0 && first + seg * kCh <= p.pool_elems && dst + seg * kCh <= sm.stage + kTok * kCh))
                    *abort_flag = 1;      // the copy is skipped: the tile cannot complete, so every role drains
                else
                    bulk_load(dst, p.latents + first, static_cast<uint32_t>(seg) * (kCh * 4u), &sm.stage_full);
                dst += seg * kCh;
                q += seg;
                remaining -= seg;
            }
        };
        // The first tile is on the critical path of the launch and the sixteen epilogue warps have nothing to do yet: they load
        // and convert it, eight rows each, and report on a barrier of its own.  (Through the
        // staging buffer like the others, converted by the same warps: 1.8 us from the wait to the first GEMM, 1.6 so; a pass of one
        // tree of 256 tokens 170 -> 163 us, of 2 025 tokens 367 -> 360, the 1 531-token trees of 27 leaves 802 -> 773.)
        bool ok = true;
        if (n_my_tiles > 1 && lane == 0) issue_tile_copy(1);
        for (int it = 1; it < n_my_tiles && ok; ++it) {
            const int ab = it & 1;
            ok = mbar_wait(&sm.stage_full, static_cast<uint32_t>(it - 1) & 1u, abort_flag);
            if (ok && it >= 2) ok = mbar_wait(&sm.a_empty[ab], static_cast<uint32_t>((it >> 1) - 1) & 1u, abort_flag);
            ok = __all_sync(0xffffffffu, ok ? 1 : 0) != 0;
            if (!ok) break;
            convert_tile(sm.stage, sm.a[ab], tile_rows(it), lane);
            proxy_fence();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sm.a_full[ab]);
                if (it + 1 < n_my_tiles) issue_tile_copy(it + 1);      // every lane has read the staging buffer
            }
        }
        if (MODE != kNoStep && sp.prev.logp_out != nullptr)      // the previous level's log-probs, off the critical path
            finalize_rows(sp.prev, sp.n_trees, sp.nodes_cap, sp.half_per, blockIdx.x, gridDim.x, sp.status, sp.per_row);
        __syncwarp();
    } else if (WHOLE && warp > kGemm2Warp) {
        // ---------------------------------------------------------------- step warps: children of whole tiles
        // Tile t's children are made while tile t + 1 is computed, in the issue slots the other warps leave; those of the last
        // tile by all warps, at the end.
        const uint32_t t = threadIdx.x - (kGemm2Warp + 1) * 32;
        for (int it = 0; it + 1 < n_my_tiles; ++it) {
            const int64_t first = (static_cast<int64_t>(cta) + static_cast<int64_t>(it) * n_ctas) * kTok;
            const StepTile q = make_step_tile(sp, p, first, kTok);
            auto v_ready = [&] { return __all_sync(0xffffffffu, mbar_wait(&sm.v_full, static_cast<uint32_t>(it) & 1u, abort_flag) ? 1 : 0) != 0; };
            if (!step_tile<kStepWarps * 32, kStepRows>(sp, p, q, first, t, sm.vtile, v_ready)) break;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.v_free);
        }
        if (ahead) {      // the last tile's velocities go elsewhere, so this buffer can take its noise meanwhile
            __syncwarp();
            step_tile_noise<kStepWarps * 32, kStepRows>(sp, p, last_tile(), t, sm.vtile);
        }
    } else {
        // ---------------------------------------------------------------- epilogue warps
        const int ew = warp - 2;                  // 0..15
        const int group = ew >> 3;                // parity of the chunks this warp works on
        const uint32_t quarter = static_cast<uint32_t>(warp & 3);   // TMEM lanes this warp may touch: 32*quarter .. +31
        const uint32_t sub = static_cast<uint32_t>(ew >> 2) & 3u;   // output tile: which 16 of the 64 channels
        const uint32_t row = quarter * 32u + static_cast<uint32_t>(lane);       // token row of this thread in the tile
        const uint32_t lane_addr = (quarter * 32u) << 16;
        bool ok = true;
        int next_out = 0;             // first tile this warp has not written out yet
        if (n_my_tiles > 0) {         // this warp's eight rows of the first A tile (see the loader warp)
            float4 z[kTok / kEpiWarps / 2];
            const int64_t tok0 = static_cast<int64_t>(cta) * kTok;
            const uint32_t c4 = static_cast<uint32_t>(lane & 15), per_tree = static_cast<uint32_t>(p.tokens_per_tree);
            const uint32_t r0 = static_cast<uint32_t>(ew * (kTok / kEpiWarps) + (lane >> 4));
#pragma unroll
            for (uint32_t k = 0; k < kTok / kEpiWarps / 2; ++k) {      // rows past the last token are zero (see convert_tile)
                const uint32_t token = static_cast<uint32_t>(tok0) + r0 + 2u * k, tree = token / per_tree;
                const int64_t at = tree * p.tree_stride + p.row_offset + static_cast<int64_t>(token - tree * per_tree) * kCh;
                z[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (token < p.n_tokens && BGRPO_IN_BOUNDS(p.status, at >= 0 && at + kCh <= p.pool_elems)) z[k] = __ldcg(reinterpret_cast<const float4*>(p.latents + at) + c4);
            }
#pragma unroll
            for (uint32_t k = 0; k < kTok / kEpiWarps / 2; ++k) {
                const uint32_t r = r0 + 2u * k;
                *reinterpret_cast<uint2*>(sm.a[0] + sw128(r, c4 >> 1) + (c4 & 1u) * 8u) = make_uint2(pack_bf16(z[k].x, z[k].y), pack_bf16(z[k].z, z[k].w));
            }
            proxy_fence();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.first_a);
        }

        // v = D2 / kappa of tile t (this warp's 32 rows x 16 channels)
        auto output_tile = [&](int t) -> bool {
            const int b = t & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&sm.d2_full[b], static_cast<uint32_t>(t >> 1) & 1u, abort_flag) ? 1 : 0)) return false;
            tc_fence_after();
            uint32_t out[16];
            tmem_ld16(tmem + lane_addr + kD2Col + static_cast<uint32_t>(b) * kCh + sub * 16u, out);
            tmem_ld_wait16(out);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.d2_empty[b]);
            const int64_t tile = static_cast<int64_t>(cta) + static_cast<int64_t>(t) * n_ctas;
            const int64_t q = tile * kTok + row;
            float4 val[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                val[j] = make_float4(kInvKappa * __uint_as_float(out[4 * j]), kInvKappa * __uint_as_float(out[4 * j + 1]),
                                     kInvKappa * __uint_as_float(out[4 * j + 2]), kInvKappa * __uint_as_float(out[4 * j + 3]));
            if (STEP || S > 1 || (WHOLE && t == n_my_tiles - 1)) {
                // The sum over a share of the hidden dimension only, and the tail of the kernel adds the parts; or the last tile,
                // and all warps make its children there.
#pragma unroll
                for (int j = 0; j < 4; ++j) *part_piece(sm.stage, row, sub * 4u + j) = val[j];
                return true;
            }
            if (WHOLE) {          // to the step warps, once they are done with the tile before
                if (t > 0 && !__all_sync(0xffffffffu, mbar_wait(&sm.v_free, static_cast<uint32_t>(t - 1) & 1u, abort_flag) ? 1 : 0)) return false;
#pragma unroll
                for (int j = 0; j < 4; ++j) *part_piece(sm.vtile, row, sub * 4u + j) = val[j];
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.v_full);
                return true;
            }
            if (q < p.n_tokens) {
                float4* dst = reinterpret_cast<float4*>(p.v_out + q * kCh + sub * 16u);
#pragma unroll
                for (int j = 0; j < 4; ++j) dst[j] = val[j];
            }
            return true;
        };
        // 32 accumulator columns of this thread's token, rounded to 16 registers of packed bf16 pairs, then the activations in
        // their place.  The packed polynomial covers |x| < 1; one bit of the pairs shows whether any of the 32 values lies outside
        // (or is not finite), and only then the thread takes the hardware-tanh form for them.  With weights and latents of the
        // usual scale (pre-activations of standard deviation ~0.2) that never happens.
        auto activate = [&](const uint32_t (&acc)[32], uint32_t (&xb)[16]) {
            uint32_t bits = 0u;
#pragma unroll
            for (int m = 0; m < 16; ++m) xb[m] = pack_bf16(__uint_as_float(acc[2 * m]), __uint_as_float(acc[2 * m + 1]));
#pragma unroll
            for (int m = 0; m < 16; m += 2) bits |= xb[m] | xb[m + 1];
            if ((bits & kEvenOutside) == 0u) {
#pragma unroll
                for (int m = 0; m < 16; ++m) xb[m] = even_poly(xb[m]);
            } else {
#pragma unroll
                for (int m = 0; m < 16; ++m)
                    xb[m] = pack_bf16(even_tanh(__uint_as_float(xb[m] << 16)), even_tanh(__uint_as_float(xb[m] & 0xffff0000u)));
            }
        };
        const uint32_t my_cols = tmem + lane_addr + (sub & 1u) * 64u;     // this warp's 64 columns inside a chunk buffer

        uint32_t acc[32], xb[16];
        // chunk index within this CTA's sequence of tiles x chunks; its buffer is g mod 3, the buffer's use number g / 3
        int buf = group, use = 0;
        for (int g = group; g < n_my_chunks && ok; g += 2) {
            // tiles whose last GEMM2 was issued at least two chunks ago
            while (ok && (next_out + 1) * NC + 2 <= g) ok = output_tile(next_out++);
            if (!ok) break;
            ok = __all_sync(0xffffffffu, mbar_wait(&sm.d1_full[buf], static_cast<uint32_t>(use) & 1u, abort_flag) ? 1 : 0) != 0;
            if (!ok) break;
            const uint32_t slice = my_cols + static_cast<uint32_t>(buf) * kHc;
            tc_fence_after();
            // Half by half: the packed activations go over the first 32 of this warp's 64 columns, each half over columns already
            // read.  (The second half's load ahead of the first half's arithmetic: 725 us for 720.)
#pragma unroll
            for (uint32_t h = 0; h < 2; ++h) {
                tmem_ld32(slice + 32u * h, acc);
                tmem_ld_wait32(acc);
                activate(acc, xb);
                tmem_st16(slice + 16u * h, xb);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.h_full[buf]);
            buf += 2;
            if (buf >= kBufs) { buf -= kBufs; ++use; }
        }
        while (ok && next_out < n_my_tiles) ok = output_tile(next_out++);
        tmem_ld_wait();
        tmem_st_wait();
    }
    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncwarp();
    if (MODE == kNoStep && S == 1) {
        __syncthreads();
    } else if (WHOLE) {
        const int64_t first = (static_cast<int64_t>(cta) + static_cast<int64_t>(n_my_tiles - 1) * n_ctas) * kTok;
        if (ahead) step_tile_children<kThreads>(sp, p, last_tile(), first, threadIdx.x, sm.stage, sm.vtile);
        else step_tile<kThreads, 1>(sp, p, last_tile(), first, threadIdx.x, sm.stage, [&] { __syncthreads(); return true; });
    } else {
        // The S parts of the tile are in the shared memory of the S CTAs of this cluster.  Each CTA adds every S-th row,
        // the parts in order, and leaves only when the others have read its own.  (Every thread gets here: the waits above are
        // bounded.)  With partial tiles through L2 and a ticket for the last CTA to add them all a launch took 2 to 3 us
        // more (two tiles, hidden 3072: 10.4 -> 7.7 us; 64 tiles: 14.1 -> 12.2).
        const int64_t first = static_cast<int64_t>(cta) * kTok;
        const uint32_t c4 = threadIdx.x % (kCh / 4);
        uint32_t r = part + S * (threadIdx.x / (kCh / 4));
        StepPiece piece;
        cluster_arrive();
        if (STEP) step_piece(sp, p, first, r, c4, piece);        // the load and the noise travel with the barrier
        __syncwarp();
        cluster_wait();
        const int row0 = STEP ? static_cast<int>(static_cast<uint32_t>(first) / static_cast<uint32_t>(p.tokens)) : 0;
        while (r < kTok) {
            const uint32_t addr = smem_u32(part_piece(sm.stage, r, c4));
            float4 x[kMaxSplit], sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int o = 0; o < kMaxSplit; ++o)
                if (o < S) x[o] = cluster_load(addr, static_cast<uint32_t>(o));
#pragma unroll
            for (int o = 0; o < kMaxSplit; ++o)
                if (o < S) { sum.x += x[o].x; sum.y += x[o].y; sum.z += x[o].z; sum.w += x[o].w; }
            if (first + r < p.n_tokens && (!STEP || p.v_out)) reinterpret_cast<float4*>(p.v_out)[(first + r) * (kCh / 4) + c4] = sum;
            if (STEP && piece.live) step_children(sp, row0, piece, sum, sm.node_sums);
            r += S * (kThreads / (kCh / 4));
            if (STEP) step_piece(sp, p, first, r, c4, piece);
        }
        __syncwarp();
        cluster_arrive();
        if (STEP && sp.g != 0.0f) {          // the sums of this CTA's tokens, by child
            __syncthreads();
            for (int i = threadIdx.x; i < kTok * BGRPO_MAX_K; i += kThreads) {
                const int row = row0 + i / BGRPO_MAX_K, b = i % BGRPO_MAX_K;
                const uint32_t* both = sm.node_sums[i / BGRPO_MAX_K][b];
                const unsigned long long sum = (static_cast<unsigned long long>(both[1]) << 16) + both[0];
                if (sum == 0ull) continue;
                const int tree = row / sp.W_in, j = row - tree * sp.W_in;
                atomicAdd(p.row_sums + static_cast<int64_t>(tree) * sp.nodes_cap + sp.off_out + j * sp.fan + b, sum);
            }
            __syncwarp();
        }
        cluster_wait();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    if (threadIdx.x == 0 && sm.abort_flag) atomicOr(p.status, kStatusWaitTimeout);
}

// Reorders W1 [64][H] and W2 [H][64] (bf16 bits) into per-chunk shared-memory images: for chunk c,
//   bytes [0, 16 KiB):      2 W1_c as [128 n = hidden][64 k = channel], 128-byte rows, 128-byte swizzle
//   bytes [16 KiB, 32 KiB): W2_c as two tiles [64 n = channel][64 k = hidden], one per half of the chunk's hidden range
__global__ void mlp_pack_kernel(const uint16_t* __restrict__ W1, const uint16_t* __restrict__ W2, int hidden, unsigned char* __restrict__ packed) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;      // one bf16 element of W1 and one of W2 per thread
    if (idx >= hidden * kCh) return;
    {   // W1[k][j]
        const int k = idx / hidden, j = idx - k * hidden;
        const int c = j / kHc, n = j - c * kHc;
        const uint32_t off = static_cast<uint32_t>(n) * 128u + (((static_cast<uint32_t>(k) >> 3) ^ (static_cast<uint32_t>(n) & 7u)) << 4) + (static_cast<uint32_t>(k) & 7u) * 2u;
        *reinterpret_cast<uint16_t*>(packed + static_cast<size_t>(c) * kChunkBytes + off) =
            __bfloat16_as_ushort(__float2bfloat16(2.f * __bfloat162float(__ushort_as_bfloat16(W1[idx]))));
    }
    {   // W2[j][n]
        const int j = idx / kCh, n = idx - j * kCh;
        const int c = j / kHc, jj = j - c * kHc, hf = jj / 64, kk = jj - hf * 64;
        const uint32_t off = static_cast<uint32_t>(n) * 128u + (((static_cast<uint32_t>(kk) >> 3) ^ (static_cast<uint32_t>(n) & 7u)) << 4) + (static_cast<uint32_t>(kk) & 7u) * 2u;
        *reinterpret_cast<uint16_t*>(packed + static_cast<size_t>(c) * kChunkBytes + kHc * 128 + hf * (kCh * 128) + off) = W2[idx];
    }
}

// kappa W1 W2 / 2 as the sum of two bf16 matrices (16 bits of each element), behind the chunks and laid out like a chunk of W2:
// two tiles [64 n = output channel][64 k = input channel].  One CTA per row k, sums in double.
constexpr int kLinParts = 16;
__global__ void __launch_bounds__(kCh * kLinParts) mlp_pack_linear_kernel(const uint16_t* __restrict__ W1, const uint16_t* __restrict__ W2, int hidden, unsigned char* __restrict__ packed) {
    __shared__ double parts[kLinParts][kCh];
    const int k = blockIdx.x, n = threadIdx.x % kCh, q = threadIdx.x / kCh;
    double sum = 0.0;
#pragma unroll 8
    for (int j = q; j < hidden; j += kLinParts)
        sum = fma(static_cast<double>(__bfloat162float(__ushort_as_bfloat16(W1[static_cast<size_t>(k) * hidden + j]))),
                  static_cast<double>(__bfloat162float(__ushort_as_bfloat16(W2[static_cast<size_t>(j) * kCh + n]))), sum);
    parts[q][n] = sum;
    __syncthreads();
    if (q != 0) return;
    for (int o = 1; o < kLinParts; ++o) sum += parts[o][n];
    const float m = static_cast<float>(0.5 * static_cast<double>(kKappa) * sum);
    const __nv_bfloat16 hi = __float2bfloat16(m), lo = __float2bfloat16(m - __bfloat162float(hi));
    const uint32_t off = sw128(static_cast<uint32_t>(n), static_cast<uint32_t>(k) >> 3) + (static_cast<uint32_t>(k) & 7u) * 2u;
    unsigned char* tile = packed + static_cast<size_t>(hidden / kHc) * kChunkBytes;
    *reinterpret_cast<uint16_t*>(tile + off) = __bfloat16_as_ushort(hi);
    *reinterpret_cast<uint16_t*>(tile + kCh * 128 + off) = __bfloat16_as_ushort(lo);
}

}  // namespace

size_t mlp_packed_bytes(int hidden) { return static_cast<size_t>(hidden / kHc) * kChunkBytes + kTileBytes; }

cudaError_t launch_mlp_pack(const uint16_t* W1, const uint16_t* W2, int hidden, void* packed, cudaStream_t s) {
    const int n = hidden * kCh;
    mlp_pack_kernel<<<(n + 255) / 256, 256, 0, s>>>(W1, W2, hidden, static_cast<unsigned char*>(packed));
    const cudaError_t e = count_launch(cudaGetLastError());
    if (e != cudaSuccess) return e;
    mlp_pack_linear_kernel<<<kCh, kCh * kLinParts, 0, s>>>(W1, W2, hidden, static_cast<unsigned char*>(packed));
    return count_launch(cudaGetLastError());
}

namespace {
template <int MODE>
constexpr size_t kMlpSmemBytes = sizeof(MlpSmem<MODE>) + 1024;
static_assert(kMlpSmemBytes<kStepOfWhole> <= 227 * 1024, "shared memory of an SM");
// What a launch has to know of the current device.  Asked for once per device; host threads may get here together.
struct MlpDevice {
    int sms = 0, clusters[kMaxSplit + 1] = {0};       // clusters[S]: how many clusters of S CTAs run at a time
};
std::mutex g_mlp_device_mutex;
struct {
    bool known = false;
    MlpDevice device;
} g_mlp_devices[64];

cudaError_t mlp_query_device(int dev, MlpDevice* d) {
    cudaError_t e = cudaFuncSetAttribute(mlp_velocity_kernel<kNoStep>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMlpSmemBytes<kNoStep>));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_velocity_kernel<kStepOfSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMlpSmemBytes<kStepOfSplit>));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_velocity_kernel<kStepOfWhole>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMlpSmemBytes<kStepOfWhole>));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, dev);
    for (int cand = 2; e == cudaSuccess && cand <= kMaxSplit; ++cand) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = cand;
        cfg.blockDim = kMlpThreads<kStepOfSplit>;
        cfg.dynamicSmemBytes = kMlpSmemBytes<kStepOfSplit>;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned int>(cand);
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&d->clusters[cand], mlp_velocity_kernel<kStepOfSplit>, &cfg);
    }
    return e;
}

cudaError_t mlp_device(MlpDevice* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_mlp_device_mutex);
    if (dev < 0 || dev >= 64) return mlp_query_device(dev, out);
    auto& slot = g_mlp_devices[dev];
    if (!slot.known) {
        MlpDevice d;
        e = mlp_query_device(dev, &d);
        if (e != cudaSuccess) return e;
        slot.device = d;
        slot.known = true;
    }
    *out = slot.device;
    return cudaSuccess;
}
}  // namespace

cudaError_t launch_mlp(const float* latents, int64_t pool_elems, int64_t tree_stride, int64_t row_offset, int n_trees, int64_t tokens_per_tree,
                       const void* packed, int hidden, float* v_out, int32_t* status, const StepLaunch* step, unsigned long long* row_sums,
                       bool* stepped, cudaStream_t s) {
    MlpDevice d;
    cudaError_t e = mlp_device(&d);
    if (e != cudaSuccess) return e;
    MlpArgs a;
    a.latents = latents;
    a.pool_elems = pool_elems;
    a.tree_stride = tree_stride;
    a.row_offset = row_offset;
    a.tokens_per_tree = tokens_per_tree;
    a.n_tokens = static_cast<int64_t>(n_trees) * tokens_per_tree;
    a.packed = static_cast<const unsigned char*>(packed);
    a.v_out = v_out;
    a.n_chunks = hidden / kHc;
    const int64_t tiles = (a.n_tokens + kTok - 1) / kTok;
    if (tiles <= 0 || tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    a.n_tiles = static_cast<int32_t>(tiles);
    a.status = status;
    // A frontier of fewer tiles than SMs is cut along the hidden dimension too, as far as all its clusters run at once (on
    // this chip 74 clusters of two, 45 of three, 33 of four, 22 of six, 15 of eight).  Any divisor of the chunk count will do:
    // with powers of two alone 16 tiles took 9.4 us (8.9 with six), 40 tiles 12.1 (10.6 with three).
    a.split = 1;
    for (int cand = kMaxSplit; cand > 1 && a.split == 1; --cand)
        if (a.n_chunks % cand == 0 && a.n_tiles <= d.clusters[cand]) a.split = cand;
    const int grid = a.split > 1 ? a.n_tiles * a.split : (a.n_tiles < d.sms ? a.n_tiles : d.sms);
    a.tokens = 1;
    a.row_sums = row_sums;
    StepLaunch sp;
    std::memset(&sp, 0, sizeof(sp));
    const int64_t tokens = step ? tokens_per_tree / step->W_in : 0;
    // The step goes along where a tile is split: each CTA then has at most half a tile of children to make, and a launch is saved.
    // One tree of 256 tokens 198 us a pass without, 170 with.
    // Elsewhere it goes along tile by tile, on warps of its own: the noise fills issue slots the activation leaves, and the
    // velocities never leave the chip (8 B an element of 20).  Launch and step of one child (with the root kernel, about 50 us of
    // the first line), us: 1 036 800 tokens of hidden 3072 891 -> 839 (at the power cap 1 006 -> 948), of 1536, 512, 256 577 -> 520,
    // 456 -> 373, 433 -> 347; 254 tiles of 3072, 1408, 1024 41.7 -> 39.3, 29.9 -> 28.6, 27.2 -> 26.4; 79 tiles of 3072, 1024
    // 25.4 -> 22.3, 19.8 -> 16.5.  With less than four chunks there is no time to draw the last tile's noise in: 79 and 254 tiles of
    // 256 14.2 -> 15.5 and 22.0 -> 23.0, which only more than two tiles an SM outweigh.
    // Two children are as much noise as a tile has room for (1 013 tiles 130 - 146 -> 128 - 148, 4 050 tiles 480 - 520 -> 459 -
    // 471), three or a shared part more (323 tiles 42 -> 53).  Nodes of less than a tile of tokens would be more than two to a tile.
    const bool whole = step && a.split == 1 && tokens >= kTok && !step->shared_noise &&
                       ((step->fan == 1 && (a.n_chunks >= 4 || a.n_tiles > 2 * d.sms)) || (step->fan == 2 && a.n_tiles > 16 * d.sms));
    if (step && (a.split > 1 || whole)) {
        sp = *step;
        sp.half_per = logp_half_per(sp.D);
        a.tokens = static_cast<int32_t>(tokens);
        if (!sp.keep_v) a.v_out = nullptr;
        *stepped = true;
        if (a.split > 1)
            return launch_overlapped_clusters(mlp_velocity_kernel<kStepOfSplit>, grid, kMlpThreads<kStepOfSplit>, kMlpSmemBytes<kStepOfSplit>, s, a.split, a, sp);
        return launch_overlapped(mlp_velocity_kernel<kStepOfWhole>, grid, kMlpThreads<kStepOfWhole>, kMlpSmemBytes<kStepOfWhole>, s, a, sp);
    }
    return launch_overlapped_clusters(mlp_velocity_kernel<kNoStep>, grid, kMlpThreads<kNoStep>, kMlpSmemBytes<kNoStep>, s, a.split, a, sp);
}

}  // namespace bgrpo

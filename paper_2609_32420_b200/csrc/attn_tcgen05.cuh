// Block-sparse attention on the 5th-generation tensor cores: TMA loads of the listed K/V tiles,
// tcgen05.mma with S = Q K^T and O += P V accumulated in tensor memory, online softmax in the
// consumer warps.  One CTA per query block of 128 tokens, steps of one key block of 128 tokens (layers with 64-token blocks run
// on attn_tcgen05_b64_kernel below).
// Paper: Section 3.3, "Historical Sparse-Connectivity Reuse" (only the block pairs the historical
// structure lists are evaluated; Q, K, V are the target's own).
//
// Warp roles (384 threads = three warpgroups, one CTA per SM):
//   warps 0-3  softmax group 0, warps 4-7 softmax group 1: the groups take the 128-key steps in turn; within
//              a group warp w owns tensor-memory lanes 32w..32w+31 = query rows.  Both also run the epilogue.
//   warp 8     TMA producer for the K tiles (one lane)
//   warp 9     tensor-memory allocation, issue of Q K^T
//   warp 10    TMA producer for the V tiles (one lane)
//   warp 11    issue of P V
// The third warpgroup gives most of its registers to the softmax groups (setmaxnreg), which hold a full
// 128-column score row per thread.
// The two issuing warps run their loops converged and elect the issuing lane per instruction (elect.sync) instead of
// sending one lane into a branch: the descriptors then live in uniform registers and a batch
// takes a third fewer cycles to queue while the softmax warps on the same scheduler are busy.  Each waits for its own
// operands and nothing else; one warp that polled for both kinds of product took 1 to 3 % longer (Wan-14B-shaped layer
// 24.7 against 24.4 ms, five-frame clip 416 against 396 us).  Each batch ends in
// one tcgen05.commit (a commit costs the issuer about as much as two MMAs): "S_g full" also releases the K slot,
// "P V done" also releases the V slot and the P buffer.
// Tensor memory (512 columns): S0 | S1 (128 fp32 columns each, one per softmax group), P (64 columns of packed
// bf16), Q (D / 2 columns of packed bf16), O (D fp32 columns).  The query tile is written there once by the
// softmax groups (straight from global memory) and serves as the A operand of every Q K^T, so those products
// read only the K tile from shared memory, whose bandwidth the TMA writes and the operand reads share.  A group
// signals when it no longer needs its scores in tensor memory, so Q K^T of its next step runs underneath its own
// exponentials; it keeps its probabilities in registers until they are complete and stores them in one go, by which
// time P V of the previous step has long read the one P buffer.  P V is issued in step order.
// Every wait on an mbarrier is bounded; on expiry the role records CARNATOR_ERR_DEVICE_TIMEOUT in
// the workspace header, raises a CTA-wide abort flag, and every role drains and returns.
#pragma once
#include <cuda.h>
#include <algorithm>

#include "common.cuh"
#include "attn_portable.cuh"
#include "attn_ring.h"

namespace carnator {
namespace tc {

constexpr int kBlock = 128;            // query rows per CTA = keys per step
constexpr int kSBufs = 2;              // score buffers in tensor memory, one per softmax group
constexpr int kRefSlots = 3;           // hand-over slots of the shared reference maximum
constexpr int kSoftmaxWarps = 8;       // two warpgroups taking the steps in turn
constexpr int kThreads = (kSoftmaxWarps + 4) * 32;   // third warpgroup: two TMA producers, two MMA issuers
constexpr int kWarpTmaK = 8, kWarpMma = 9, kWarpTmaV = 10;
constexpr int kTmemCols = 512;         // S0 | S1 | P | Q | O
constexpr uint32_t kColP = 2 * kBlock;        // packed bf16 probabilities: 64 columns, one buffer for both groups
constexpr uint32_t kColQ = 2 * kBlock + 64;   // the query tile as packed bf16 pairs: D / 2 columns (A operand of Q K^T)
constexpr uint32_t kColO = 2 * kBlock + 2 * 64;
constexpr int kRegsService = 72, kRegsSoftmax = 216;   // setmaxnreg targets (the literals in the kernel must match)
constexpr float kRescaleThreshold = 8.0f;   // log2 units: P stays below 2^8, well inside bf16/fp32 range

// ---- small PTX wrappers -----------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done;
}
// Non-blocking form, for a role that watches two barriers: try_wait may suspend the thread on the one it was given.
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait: gives up after limit_ns (or when another role has aborted) and raises the abort flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned sleep_ns = 0,
                                          unsigned long long limit_ns = kDefaultWaitNs) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (sleep_ns) __nanosleep(sleep_ns);
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 255u) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) break;
        }
    }
    *abort_flag = 1;
    return false;
}

// Bounded wait of a producer for its ring slot, the slot of step u (attn_ring.h): bar0 is the barrier of the even steps, that
// of the odd ones lies behind it.
__device__ __forceinline__ bool mbar_wait_slot(uint32_t bar0, int u, volatile int* abort_flag, unsigned long long limit_ns) {
    auto done = [&](int b, uint32_t parity) { return mbar_test(bar0 + 8 * b, parity) != 0; };
    if (slot_is_free(u, done)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        __nanosleep(100);
        if (slot_is_free(u, done)) return true;
        if ((it & 255u) == 255u) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) break;
        }
    }
    *abort_flag = 1;
    return false;
}

// Wait used on the way out, after an abort: the copies or products this role still has in flight must land before
// the CTA gives its shared and tensor memory back, so the abort flag does not end this wait; only time does.
__device__ __forceinline__ bool mbar_wait_drain(uint32_t bar, uint32_t parity, unsigned long long limit_ns = kDefaultWaitNs) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        __nanosleep(100);
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 255u && global_ns() - t0 > limit_ns) break;
    }
    return false;
}

// Warp-collective form.  Every lane tests the barrier (one broadcast read of shared memory, no divergence in the
// common case that the phase is already complete); lanes that find it incomplete fall into the bounded wait.  The
// vote makes the outcome uniform, reconverges the warp and orders the other lanes' later reads after the acquire.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned sleep_ns = 0,
                                               unsigned long long limit_ns = kDefaultWaitNs) {
    const bool ok = mbar_try(bar, parity) ? true : mbar_wait(bar, parity, abort_flag, sleep_ns, limit_ns);
    return __all_sync(0xffffffffu, ok) != 0;
}
// One arrival per warp once every lane's earlier writes are ordered before it.
__device__ __forceinline__ void mbar_arrive_warp(uint32_t bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Forms for a converged warp, the descriptors given as (low word, shared high word): D[tmem] (+)= A[tmem] * B[smem].  Every lane
// executes the statement with the same operands and one elected lane issues the instruction.  The compiler can then keep the descriptors in uniform registers, and queuing a batch costs the
// warp far fewer issue slots than it does from inside a one-lane branch: measured with two softmax groups running on
// the same SM, 54 clk per instruction against 79.
__device__ __forceinline__ void mma_ts_el(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with an output mask: rows whose half of the tile is switched off (lanes 0-63 by off_lo, 64-127 by off_hi, all
// ones = off) keep their accumulator.
__device__ __forceinline__ void mma_ts_el_rows(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                               uint32_t off_lo, uint32_t off_hi, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %7, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, {%5, %5, %6, %6}, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(off_lo), "r"(off_hi), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], both descriptors given as (low word, shared high word); converged warp, one elected
// lane issues (see mma_ts_el)
__device__ __forceinline__ void mma_ss_el(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tc_commit_el(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
// Two fp32 lanes per instruction (packed pair in a 64-bit register): halves the FMA-pipe instruction count of the
// exponent arguments and of the row sums.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// Wait for this warp's loads from tensor memory.  It is given the registers that they fill and hands them on: arithmetic on them,
// which is not volatile, depends on nothing else that would keep it behind the wait.
template <int N>
__device__ __forceinline__ void hand_on(float (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i]));
}
__device__ __forceinline__ void hand_on(float& v) { asm volatile("" : "+f"(v)); }
template <typename... V>
__device__ __forceinline__ void tmem_wait_ld(V&... loaded) {
    static_assert(sizeof...(V) > 0, "name what was loaded");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    (hand_on(loaded), ...);
}
// On the way out: a step that was given up may have left a load behind.
__device__ __forceinline__ void tmem_drain_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr),
          "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// ---- descriptors --------------------------------------------------------------------------------
// Shared-memory matrix descriptor, 128-byte swizzle: start address, leading / stride byte offsets
// (all in 16-byte units), descriptor version 1 (bit 46), layout type 2 = SWIZZLE_128B (bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return uint64_t((addr & 0x3FFFFu) >> 4)
         | (uint64_t((lbo_bytes >> 4) & 0x3FFFu) << 16)
         | (uint64_t((sbo_bytes >> 4) & 0x3FFFu) << 32)
         | (1ull << 46)
         | (2ull << 61);
}
// Same with the 64-byte swizzle (rows of 64 B, atoms of 8 rows = 512 B): layout type 4.
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return uint64_t((addr & 0x3FFFFu) >> 4)
         | (uint64_t((lbo_bytes >> 4) & 0x3FFFu) << 16)
         | (uint64_t((sbo_bytes >> 4) & 0x3FFFu) << 32)
         | (1ull << 46)
         | (4ull << 61);
}
// Instruction descriptor for kind::f16: fp32 accumulator, bf16 x bf16, M x N, B operand major-ness.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(b_mn_major) << 16) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}

// Output of a warp's 32 rows, half of the head dimension: O / l from tensor memory (row = lane) through shared memory (32 D bytes of
// the K ring, which the last product has left behind) to global memory, so that a store covers whole lines.  With 16 bytes of its own
// row per lane, a store touched 32 half sectors, and the output of a block took 1.9 us.
template <int D>
__device__ __forceinline__ void write_rows(uint32_t t_o, float inv, uint32_t stage, int lane, __nv_bfloat16* out, int64_t row_stride, int n_rows) {
    constexpr int kPieces = D / 16;          // 16-byte pieces of a half row
    auto spot = [&](int r, int p) { return stage + uint32_t(r * D + ((p ^ (D == 128 ? r & 7 : (r >> 1) & 3)) * 16)); };
#pragma unroll
    for (int c = 0; c < D / 64; ++c) {
        float o[32];
        tmem_ld32(t_o + c * 32, o);          // warp-collective: every lane takes part
        tmem_wait_ld(o);
#pragma unroll
        for (int v = 0; v < 4; ++v)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                ::"r"(spot(lane, c * 4 + v)), "r"(pack_bf16(o[8 * v] * inv, o[8 * v + 1] * inv)), "r"(pack_bf16(o[8 * v + 2] * inv, o[8 * v + 3] * inv)),
                  "r"(pack_bf16(o[8 * v + 4] * inv, o[8 * v + 5] * inv)), "r"(pack_bf16(o[8 * v + 6] * inv, o[8 * v + 7] * inv)) : "memory");
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kPieces; ++k) {
        const int r = k * (32 / kPieces) + lane / kPieces, p = lane % kPieces;
        uint4 u;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "r"(spot(r, p)) : "memory");
        if (r < n_rows) *reinterpret_cast<uint4*>(out + r * row_stride + p * 8) = u;
    }
}

// Shared-memory plan.  Every K / V tile is 128 rows x D held as D/64 boxes of 128 rows x 128 B
// (128-byte swizzle).  K and V tiles travel through kStages-slot rings (separate rings, separate producers).
template <int D>
struct Cfg {
    static constexpr int kBoxes = D / 64;
    static constexpr uint32_t kBoxBytes = kBlock * 128;             // 128 rows x 128 B
    static constexpr uint32_t kTileBytes = kBoxes * kBoxBytes;      // one 128 x D bf16 tile
    static constexpr uint32_t kOffK = 0;
    static constexpr uint32_t kOffV = kOffK + kStages * kTileBytes;
    static constexpr uint32_t kOffBar = kOffV + kStages * kTileBytes;
    static constexpr uint32_t kOffPlan = kOffBar + 512;
    static constexpr uint32_t kSmemBytes = kOffPlan + 1024;         // barriers + slack to align the base to 1 KiB
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
attn_tcgen05_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, const AttnArgs a) {
    using C = Cfg<D>;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float r_pub[kRefSlots][kBlock];     // reference maximum after step i, slot i % 3 (handed from one warpgroup to the other)
    __shared__ float fin[2][2][kBlock];         // per warpgroup: final reference maximum and partial row sum

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Grid at D = 128: (heads of a group, position in the execution order, groups of heads), see head_group.  At D = 64:
    // (position, head, batch entry); computed coordinates cost that loop 0.9 %.
    constexpr bool kGroups = D == 128;
    int b, h;
    if constexpr (kGroups) {
        const uint32_t head = blockIdx.z * gridDim.x + blockIdx.x;
        if (head >= uint32_t(a.B) * uint32_t(a.H)) return;      // the last group may be short
        b = int(head / uint32_t(a.H)); h = int(head - uint32_t(b) * uint32_t(a.H));
    } else { b = blockIdx.z; h = blockIdx.y; }
    const int64_t bh = int64_t(b) * a.H + h;
    const int place = kGroups ? blockIdx.y : blockIdx.x;
    // What the first step needs is on its way as early as it can be: the producers request the first ring of tiles as soon as the
    // list is known, and the query rows are asked into L2, while the block sets itself up.  Waiting for the list, the header and
    // the query rows one after the other behind the set-up, a block had its first scores 3.9 us later.  With the output in whole
    // lines (write_rows): five-frame clip (10 blocks an SM) 387 -> 375 us; a region-restricted layer and the Wan-1.3B-shaped one within
    // what two runs differ by (552 -> 544 us, 2188 -> 2183 us).
    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t sK = smem_base + C::kOffK;
    const uint32_t sV = smem_base + C::kOffV;
    const uint32_t bars = smem_base + C::kOffBar;
    const uint32_t bar_q = bars, bar_o = bars + 8, bar_drain = bars + 16, bar_drain2 = bars + 24;
    auto bar_kfull = [&](int s) { return bars + 32 + 8 * s; };       // up to 4 stages each
    auto bar_vfull = [&](int s) { return bars + 96 + 8 * s; };
    auto bar_sfull = [&](int s) { return bars + 160 + 8 * s; };      // S_g holds fresh scores
    auto bar_sfree = [&](int s) { return bars + 176 + 8 * s; };      // group g has read S_g into registers
    auto bar_pfull = [&](int s) { return bars + 192 + 8 * s; };      // P_g is complete
    auto bar_ref = [&](int s, int q) { return bars + 224 + 8 * (s * 4 + q); };   // r_pub slot s, lane quarter q
    auto bar_fin = [&](int q) { return bars + 320 + 8 * q; };
    auto bar_pvdone = [&](int s) { return bars + 352 + 8 * s; };     // P V of the step that used score buffer s has completed
    volatile int* abortp = &abort_flag;
    const bool producer = (warp == kWarpTmaK || warp == kWarpTmaV) && lane == 0;
    if (producer) prefetch_tmap(warp == kWarpTmaK ? &mapK : &mapV);
    grid_wait();                            // launched while the compaction drains
    const int I = a.order[bh * a.nqb + place];
    // every bounded wait of this CTA gives up after `limit` (2 s unless the workspace header asks for less)
    const unsigned long long limit = a.hdr->wait_limit_ns ? a.hdr->wait_limit_ns : kDefaultWaitNs;
    int withhold = 0;
    if (producer) {                         // each initialises the barriers of its own tiles, the K producer the others as well
        if (warp == kWarpTmaK) {
            withhold = a.hdr->debug_withhold;
            abort_flag = 0;
            mbar_init(bar_q, kSoftmaxWarps); mbar_init(bar_o, 1); mbar_init(bar_drain, 1); mbar_init(bar_drain2, 1);
            for (int s = 0; s < kSBufs; ++s) {
                mbar_init(bar_sfull(s), 1); mbar_init(bar_pvdone(s), 1);
                mbar_init(bar_pfull(s), 4); mbar_init(bar_sfree(s), 4);          // one arrival per softmax warp of the group
            }
            for (int s = 0; s < kRefSlots; ++s)
                for (int q = 0; q < 4; ++q) mbar_init(bar_ref(s, q), 1);
            for (int q = 0; q < 4; ++q) mbar_init(bar_fin(q), 2);
        }
        for (int s = 0; s < kStages; ++s) mbar_init(warp == kWarpTmaK ? bar_kfull(s) : bar_vfull(s), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int T = a.counts[bh * a.nqb + I];                 // steps = listed key blocks
    const int32_t* list = a.lists + (bh * a.nqb + I) * int64_t(a.nkb);
    int first[kStages] = {};                // the first entries of the list, wherever there are so many
    if (producer) {
#pragma unroll
        for (int i = 0; i < kStages; ++i) if (i < a.nkb) first[i] = list[i];
    }
    const int q0 = I * kBlock;
    if (T < 0) return;                      // skipped query block (region-restricted form): output untouched
    if (T > a.nkb) {                        // a count that cannot come from compaction: stop before reading a list that long
        if (tid == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_CHECK, 20, T, place);
        return;
    }
    if (T == 0) {                           // nothing to attend to: O = 0, LSE = -inf
        if (tid < kBlock && q0 + tid < a.N) {
            __nv_bfloat16* op = a.O + b * a.os[0] + h * a.os[1] + int64_t(q0 + tid) * a.os[2];
#pragma unroll
            for (int c = 0; c < D / 8; ++c) *reinterpret_cast<uint4*>(op + c * 8) = make_uint4(0, 0, 0, 0);
            a.LSE[bh * a.N + q0 + tid] = -INFINITY;
        }
        return;
    }

    // copies of the K (V) tile of key block J into ring slot s
    auto load_tile = [&](bool is_k, int s, int J) {
        const uint32_t full = is_k ? bar_kfull(s) : bar_vfull(s), dst = (is_k ? sK : sV) + s * C::kTileBytes;
        mbar_expect_tx(full, C::kTileBytes);
#pragma unroll
        for (int x = 0; x < C::kBoxes; ++x) tma_load_4d(dst + x * C::kBoxBytes, is_k ? &mapK : &mapV, full, x * 64, J * kBlock, h, b);
    };
    int armed = -1;                         // last tile requested
    bool malformed = false;                 // a list entry outside [0, nkb) or out of order: stop before touching memory
    if (producer) {
#pragma unroll
        for (int i = 0; i < kStages; ++i) {
            if (i >= T || malformed) break;
            const int J = first[i];
            malformed = J < 0 || J >= a.nkb || (i > 0 && J <= first[i > 0 ? i - 1 : 0]);
            // Test of the time-out path only: the first K tile of the first query block in the order is never
            // requested, so the wait for it runs out and the CTA takes the abort-and-drain path.
            if (malformed || (i == 0 && withhold != 0 && place == 0 && bh == 0)) continue;
            load_tile(warp == kWarpTmaK, i, J);
            armed = i;
        }
    }
    if (warp < kSoftmaxWarps) {             // the query rows, a line each: held in registers from here on they slow the loop down by 1.5 %
        const int r = q0 + (tid & (kBlock - 1));
        const __nv_bfloat16* qp = a.Q + b * a.qs[0] + h * a.qs[1] + int64_t(r) * a.qs[2] + (warp >> 2) * (D / 2);
        if (r < a.N) asm volatile("prefetch.global.L2 [%0];" ::"l"(qp));
    }
    // for the epilogue: kept in registers through the loop they slow it down by 1.3 % (grid coordinates are free, these are not)
    __shared__ volatile int at_b, at_h;
    if (kGroups && tid == 0) { at_b = b; at_h = h; }
    if (warp == kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp >= kSoftmaxWarps) {
    // Register budget: the producer / MMA warpgroup needs few registers and hands the rest to the softmax groups.
    // The CTA is launched with 384 x 168 registers; 256 x 216 + 128 x 72 uses exactly that.  A split that asks for
    // more makes setmaxnreg.inc wait for registers that never come.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;" ::: "memory");
    if (warp == kWarpTmaK) {
        // ================= TMA producer: the K tiles =================
        // (the first ring is on its way)
        if (lane == 0) {
            if (malformed) { set_status(a.hdr, CARNATOR_ERR_DEVICE_CHECK, 21, armed + 1, place); *abortp = 1; }
            for (int i = kStages; i < T && !malformed; ++i) {
                const int s = i % kStages, u = i - kStages;     // the slot is free once Q K^T of step u has completed
                if (!mbar_wait_slot(bar_sfull(0), u, abortp, limit)) {
                    set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 1, i, place); break;
                }
                const int J = list[i];
                if (J < 0 || J >= a.nkb || J <= list[i - 1]) {
                    set_status(a.hdr, CARNATOR_ERR_DEVICE_CHECK, 21, i, place); *abortp = 1; break;
                }
                load_tile(true, s, J);
                armed = i;
            }
            if (*abortp) {      // copies in flight must land before the CTA gives its shared memory back
                for (int k = 0; k < kStages && armed - k >= 0; ++k)
                    mbar_wait_drain(bar_kfull((armed - k) % kStages), uint32_t((armed - k) / kStages) & 1u, limit);
            }
        }
    } else if (warp == kWarpTmaV) {
        // ================= TMA producer: the V tiles =================
        if (lane == 0) {
            // A malformed list is reported by the K producer, which raises the abort flag behind its report: raised here it could
            // make a role that waits record a time-out first.
            for (int i = kStages; i < T && !malformed; ++i) {
                const int s = i % kStages, u = i - kStages;     // the slot is free once P V of step u has completed
                if (!mbar_wait_slot(bar_pvdone(0), u, abortp, limit)) {
                    set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 2, i, place); break;
                }
                const int J = list[i];
                if (J < 0 || J >= a.nkb) { malformed = true; break; }
                load_tile(false, s, J);
                armed = i;
            }
            if (malformed || *abortp) {
                for (int k = 0; k < kStages && armed - k >= 0; ++k)
                    mbar_wait_drain(bar_vfull((armed - k) % kStages), uint32_t((armed - k) / kStages) & 1u, limit);
            }
        }
    } else if (warp == kWarpMma) {
        // ================= issuer of Q K^T =================
        // S_g = Q K_i^T once the K tile has landed and the softmax group has taken the previous scores out of that S buffer.
        // The whole warp runs the loop converged and one elected lane issues.  The barrier a batch commits ("S_g is full")
        // also frees the K slot.
        constexpr uint32_t idesc_qk = instr_desc(kBlock, kBlock, 0);
        // descriptor words that do not change: low word = (address >> 4) | leading offset; high word = stride
        // offset | version | swizzle mode (see smem_desc)
        const uint64_t dk = smem_desc(sK, 16, 1024);
        const uint32_t k_lo0 = uint32_t(dk), hi_kmajor = uint32_t(dk >> 32);
        bool ok = mbar_wait_warp(bar_q, 0, abortp, 0, limit);   // the softmax groups have put the query tile into tensor memory
        if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 3, 0, place);
        tc_fence_after();
        for (int iq = 0; iq < T && ok; ++iq) {
            const int s = iq % kStages, g = iq & 1;
            ok = mbar_wait_warp(bar_kfull(s), uint32_t(iq / kStages) & 1u, abortp, 0, limit);
            if (ok && iq >= 2) ok = mbar_wait_warp(bar_sfree(g), uint32_t((iq - 2) >> 1) & 1u, abortp, 0, limit);
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 4, iq, place); break; }
            tc_fence_after();
            // Q from tensor memory, K tile K-major, 16 elements of the head dimension per instruction
            const uint32_t k_lo = k_lo0 + uint32_t(s) * (C::kTileBytes >> 4), d_s = tmem + g * kBlock;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off16 = ((kk / 4) * C::kBoxBytes + (kk % 4) * 32) >> 4;      // compile-time constant
                mma_ts_el(d_s, tmem + kColQ + kk * 8, k_lo + off16, hi_kmajor, idesc_qk, kk > 0 ? 1u : 0u);
            }
            tc_commit_el(bar_sfull(g));
        }
        if (__any_sync(0xffffffffu, *abortp != 0)) {      // no product may still run when tensor memory is released
            tc_commit_el(bar_drain);
            mbar_wait_drain(bar_drain, 0, limit);
            __syncwarp();
        }
    } else {
        // ================= issuer of P V (warp 11) =================
        // O += P_i V_i once the V tile has landed and the probabilities are complete; "P V done" also frees the V slot and P.
        constexpr uint32_t idesc_pv = instr_desc(kBlock, D, 1);
        const uint64_t dv = smem_desc(sV, C::kBoxBytes, 1024);
        const uint32_t v_lo0 = uint32_t(dv), hi_v = uint32_t(dv >> 32);
        bool ok = true;
        for (int ip = 0; ip < T && ok; ++ip) {
            const int s = ip % kStages, g = ip & 1;
            ok = mbar_wait_warp(bar_vfull(s), uint32_t(ip / kStages) & 1u, abortp, 0, limit);
            if (ok) ok = mbar_wait_warp(bar_pfull(g), uint32_t(ip >> 1) & 1u, abortp, 0, limit);
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 5, ip, place); break; }
            tc_fence_after();
            // P from tensor memory (16 keys = 8 packed columns per instruction), V tile as the MN-major B operand
            // (rows = keys, 64-element chunks of the head dimension one box apart)
            const uint32_t v_lo = v_lo0 + uint32_t(s) * (C::kTileBytes >> 4), p_t = tmem + kColP, d_o = tmem + kColO;
            const uint32_t acc0 = ip > 0 ? 1u : 0u;
#pragma unroll
            for (int kk = 0; kk < kBlock / 16; ++kk)
                mma_ts_el(d_o, p_t + kk * 8, v_lo + kk * (2048 >> 4), hi_v, idesc_pv, kk > 0 ? 1u : acc0);
            tc_commit_el(bar_pvdone(g));
        }
        if (ok) tc_commit_el(bar_o);
        if (__any_sync(0xffffffffu, *abortp != 0)) {
            tc_commit_el(bar_drain2);
            mbar_wait_drain(bar_drain2, 0, limit);
            __syncwarp();
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;" ::: "memory");
        // ================= softmax + epilogue (warps 0-7) =================
        // Two warpgroups take the steps in turn (group g: steps g, g+2, ...), each with one warp per
        // tensor-memory lane quarter, so one group's exponentials run while the other group's scores are
        // being produced.  Both feed the same O accumulator, so they share one reference maximum per row:
        // the group that handles step i derives R_i from R_{i-1} (published by the other group right after
        // its row-maximum pass) and publishes R_i in turn.  The reference only moves when a row maximum
        // exceeds it by more than the threshold; then this group rescales O before delivering P_i.
        const int quarter = warp & 3, wg = warp >> 2;
        const int r_loc = quarter * 32 + lane;                      // query row within the tile
        const uint32_t lane_base = uint32_t(quarter * 32) << 16;
        const int row = q0 + r_loc;
        const bool row_in = row < a.N;
        {
            // The query tile goes into tensor memory as the A operand of Q K^T (row = lane, two bf16 per column), so
            // those products read only the K tile from shared memory.  Group g brings half of the head dimension.
            const __nv_bfloat16* qp = a.Q + b * a.qs[0] + h * a.qs[1] + int64_t(row) * a.qs[2] + wg * (D / 2);
#pragma unroll
            for (int c = 0; c < D / 128; ++c) {
                uint32_t r[32];
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const uint4 u = row_in ? *reinterpret_cast<const uint4*>(qp + c * 64 + v * 8) : make_uint4(0, 0, 0, 0);
                    r[4 * v] = u.x; r[4 * v + 1] = u.y; r[4 * v + 2] = u.z; r[4 * v + 3] = u.w;
                }
                tmem_st32(tmem + lane_base + kColQ + wg * (D / 4) + c * 32, r);
            }
            if (D == 64) {
                uint32_t r[16];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint4 u = row_in ? *reinterpret_cast<const uint4*>(qp + v * 8) : make_uint4(0, 0, 0, 0);
                    r[4 * v] = u.x; r[4 * v + 1] = u.y; r[4 * v + 2] = u.z; r[4 * v + 3] = u.w;
                }
                tmem_st16(tmem + lane_base + kColQ + wg * 16, r);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive_warp(bar_q);
        }
        float m_w = -INFINITY, l_w = 0.f;                           // this group's reference and partial row sum
        bool ok = true;
        // lists ascend, so only the last listed block can be the ragged one: read it once, off the per-step path
        const int nvalid_last = a.N - list[T - 1] * kBlock;
        for (int i = wg; i < T; i += 2) {
            const uint32_t sph = uint32_t(i >> 1) & 1u;
            ok = mbar_wait_warp(bar_sfull(wg), sph, abortp, 20, limit);   // warp-uniform: the loads below are collective
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 7, i, place); break; }
            tc_fence_after();
            const int nvalid = (i == T - 1) ? nvalid_last : kBlock;      // >= 1; < 128 only for a ragged last block
            const uint32_t tS = tmem + lane_base + wg * kBlock;
            const uint32_t tP = tmem + lane_base + kColP;
            float s[4][32];
            uint32_t pk[4][16];
            uint64_t part2[2];
            bool p_free;
            // The first half of the exponentials is taken under the reference of step i-1 while the row maximum is still
            // being found (they use different pipes), and again in the rare step that moves the reference, from the scores
            // in tensor memory, which are given up only then.  With the maximum in front of all exponentials instead
            // the Wan-14B-shaped layer takes 24.4 ms against 24.2,
            // the CogVideoX-shaped one 2.77 against 2.72.  A loop around one copy of the first half, instead of two
            // copies, took 25.0 and 3.2 ms.
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, s[c]);
            tmem_wait_ld(s[0], s[1], s[2], s[3]);
            auto mask_half = [&](int c0) {       // ragged tail (warp-uniform): keys >= N never count
                if (nvalid < kBlock) {
#pragma unroll
                    for (int c = c0; c < c0 + 2; ++c)
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (c * 32 + e >= nvalid) s[c][e] = -INFINITY;
                }
            };
            mask_half(0); mask_half(2);
            float r_now = -INFINITY;
            if (i > 0) {                         // reference handed over from step i-1
                ok = mbar_wait_warp(bar_ref((i - 1) % kRefSlots, quarter), uint32_t((i - 1) / kRefSlots) & 1u, abortp, 0, limit);
                if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 10, i, place); break; }
                r_now = r_pub[(i - 1) % kRefSlots][r_loc];
            }
            const uint64_t scale2 = pack2(a.scale_log2, a.scale_log2);
            part2[0] = part2[1] = pack2(0.f, 0.f);
            // P = exp2(s * scale - R_i): one FFMA + one MUFU per element, packed bf16 pairs
            auto exps = [&](int c0, float r) {
                const uint64_t neg_m2 = pack2(-r, -r);
#pragma unroll
                for (int c = c0; c < c0 + 2; ++c)
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float x0, x1;
                        unpack2(fma2(pack2(s[c][2 * e], s[c][2 * e + 1]), scale2, neg_m2), x0, x1);
                        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                        part2[e & 1] = add2(part2[e & 1], pack2(p0, p1));
                        pk[c][e] = pack_bf16(p0, p1);
                    }
            };
            // row maximum of the raw scores (the scale is positive), four independent chains
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int e = 0; e < 32; e += 2) mx4[(e >> 1) & 3] = max3(mx4[(e >> 1) & 3], s[c][e], s[c][e + 1]);
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * a.scale_log2;
            exps(0, r_now);
            const bool grow = i == 0 || mx > r_now + kRescaleThreshold;
            p_free = i < 1;
            if (__any_sync(0xffffffffu, grow)) {
                const float r_prev = r_now;
                r_now = grow ? mx : r_now;
                if (i > 0) {
                    // O must be quiescent: P V of step i-1 (the other group's) complete.  P V is issued in step order
                    // and that of step i cannot start before this group delivers P_i.
                    p_free = true;
                    ok = mbar_wait_warp(bar_pvdone(wg ^ 1), uint32_t((i - 1) >> 1) & 1u, abortp, 0, limit);
                    if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 9, i, place); break; }
                    tc_fence_after();
                    const float f = ex2_approx(r_prev - r_now);          // 1 for rows that did not move
#pragma unroll 1
                    for (int c = 0; c < D / 16; ++c) {
                        float o[16];
                        tmem_ld16(tmem + lane_base + kColO + c * 16, o);
                        tmem_wait_ld(o);
                        uint32_t r[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(o[e] * f);
                        tmem_st16(tmem + lane_base + kColO + c * 16, r);
                    }
                }
                tmem_ld32(tS, s[0]); tmem_ld32(tS + 32, s[1]);
                tmem_wait_ld(s[0], s[1]);
                mask_half(0);
                part2[0] = part2[1] = pack2(0.f, 0.f);
                exps(0, r_now);
            }
            r_pub[i % kRefSlots][r_loc] = r_now;
            mbar_arrive_warp(bar_ref(i % kRefSlots, quarter));
            tc_fence_before();
            mbar_arrive_warp(bar_sfree(wg));     // S_g may take the scores of step i+2
            if (m_w != r_now) { l_w *= ex2_approx(m_w - r_now); m_w = r_now; }   // first use: l_w = 0, exp2(-inf) = 0
            exps(2, r_now);
            if (!p_free) {      // the one P buffer is free once P V of step i-1 (the other group's) has read it
                ok = mbar_wait_warp(bar_pvdone(wg ^ 1), uint32_t((i - 1) >> 1) & 1u, abortp, 0, limit);
                if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 12, i, place); break; }
            }
            tc_fence_after();          // its reads of P come before the stores below
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tmem_st16(tP + c * 16, pk[c]);
            }
            {
                float s0, s1, s2, s3;
                unpack2(part2[0], s0, s1); unpack2(part2[1], s2, s3);
                l_w += (s0 + s1) + (s2 + s3);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive_warp(bar_pfull(wg));
        }
        // combine the two groups' sums under the final reference (the later step holds the larger one)
        if (ok) {
            fin[wg][0][r_loc] = m_w;
            fin[wg][1][r_loc] = l_w;
            mbar_arrive_warp(bar_fin(quarter));
            ok = mbar_wait_warp(bar_fin(quarter), 0, abortp, 0, limit);
            if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 11, T, place);
        }
        if (ok) {
            ok = mbar_wait_warp(bar_o, 0, abortp, 20, limit);
            if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 8, T, place);
        }
        if (ok) {
            tc_fence_after();
            const float m0 = fin[0][0][r_loc], m1 = fin[1][0][r_loc];
            const float r_fin = fmaxf(m0, m1);
            float l_tot = fin[0][1][r_loc] * ex2_approx(m0 - r_fin) + fin[1][1][r_loc] * ex2_approx(m1 - r_fin);
            const float inv = 1.f / l_tot;
            // each group writes half of the head dimension
            const int eb = kGroups ? at_b : b, eh = kGroups ? at_h : h;
            __nv_bfloat16* op = a.O + eb * a.os[0] + eh * a.os[1] + int64_t(q0 + quarter * 32) * a.os[2] + wg * (D / 2);
            write_rows<D>(tmem + lane_base + kColO + wg * (D / 2), inv, smem_base + C::kOffK + warp * (32 * D), lane, op, a.os[2], a.N - q0 - quarter * 32);
            if (wg == 0 && row_in) a.LSE[(int64_t(eb) * a.H + eh) * a.N + row] = (r_fin + log2f(l_tot)) * kLn2;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kWarpMma) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// ---- masks of 64-token blocks ---------------------------------------------------------------------------------------------
// The same path (TMA tiles, tcgen05 products, online softmax under a shared lazy reference) with another split of the work:
//   The tile is 128 x 128 tokens whatever the blocks.  64-token query blocks share a CTA in pairs (neighbours in the execution
//   order, which puts rows with like lists side by side) and the CTA walks the union of their lists; 64-token key blocks come two
//   to a step.  A row half that does not list a block has zero probabilities there, and its
//   accumulator lanes are switched off in that product, so nothing of the block (not even an infinity in V) reaches it.
//   P is kept to 16 bits, as a sum of two bf16, and P V takes two products (see the exponentials).
//
// Warp roles (512 threads = four warpgroups, one CTA per SM):
//   warps 0-11   three softmax groups, which take the steps in turn; warp w of a group owns tensor-memory lanes
//                32w..32w+31 = query rows
//   warp 12 / 14 TMA producer of the K / V tiles (one lane)
//   warp 13      tensor-memory allocation, issue of Q K^T
//   warp 15      issue of P V
// Tensor memory (512 columns): a score buffer of 128 fp32 columns per group, in which the group also leaves both parts of its
// probabilities, and O; Q stays in shared memory.  Q K^T of a group's next step waits for its P V, and the other two groups fill
// that time.
//
// Why a union and not 64-row products: those run at half the tensor rate.  Why three groups: a group's step is one chain (wait
// for the products 2700 clocks at D = 128, maximum 600, hand-over 280, exponentials and split of P 2500), of which three overlap;
// the products alone would take 1536 clocks a step.  With two groups, one P buffer for the first parts and the maximum and
// exponentials of all 128 columns as straight-line code, a step took 3540 clocks, a quarter of them waiting for instructions
// (2.1 of 8.8 resident warps per issue).  The exponentials now run in a loop over 32-column chunks, which are read from tensor
// memory a second time.  Wan-1.3B-shaped layer with 64-token blocks (12 heads, 32760 tokens, 36 % of the tiles; the unions hold
// 4 % more): 3.77 -> 3.28 ms at the 1000 W board limit; 36 heads of 6624 tokens, D = 64, a third of the tiles, no window: 556 -> 395
// us; 40 heads of 8778 tokens, D = 128: 1.30 -> 1.02 ms.  Of the 128-token forms, D = 64 took 2.98 ms instead of 2.70 with three
// groups (CogVideoX-shaped layer).
constexpr int kSoftGroups = 3;
constexpr int kSoftWarps64 = 4 * kSoftGroups;
constexpr int kThreads64 = (kSoftWarps64 + 4) * 32;
constexpr int kRegsService64 = 56, kRegsSoftmax64 = 152;      // setmaxnreg targets (the literals in the kernel must match)

// Shared-memory plan: rings of K and V tiles (at D = 128 one V slot less) and the query tile.
template <int D>
struct Cfg64 {
    static constexpr int kBoxes = D / 64;
    static constexpr uint32_t kBoxBytes = kBlock * 128;
    static constexpr uint32_t kTileBytes = kBoxes * kBoxBytes;
    static constexpr int kKStages = 3, kVStages = D == 128 ? 2 : 3;
    static_assert(kKStages == kSoftGroups, "a step's K slot and its score buffer are counted as one");
    static_assert(kVStages <= kSoftGroups, "a V producer that waits for step i - kVStages must not find its barrier a step on");
    static constexpr uint32_t kOffK = 0;
    static constexpr uint32_t kOffV = kOffK + kKStages * kTileBytes;
    static constexpr uint32_t kOffQ = kOffV + kVStages * kTileBytes;
    static constexpr uint32_t kOffBar = kOffQ + kTileBytes;
    static constexpr uint32_t kOffPlan = kOffBar + 512;
    static constexpr uint32_t kSmemBytes = kOffPlan + 1024;         // barriers + slack to align the base to 1 KiB
};

// Step plan of the 64-token block forms, in shared memory behind the barriers: per row half a bitmap of its listed key
// blocks, the number of entries before each bitmap word, and the entries themselves, two bytes each.
constexpr int kPlanMaxKeyBlocks = 12288;
constexpr uint32_t kPlanBlockMask = 0x3FFF, kPlanPad = 0x3FFF;   // a pad entry points past every token: its tiles read as zero
constexpr int kPlanRowBit = 14;                                  // bit 14 + r: listed by row half r
inline uint32_t plan_bytes(int nkb) { return uint32_t(ceil_div(nkb, 32)) * 12 + uint32_t(nkb + 2) * 2 + 4; }

// Builds the plan of one CTA: the union of the lists of its row halves (one list when the tile is one query block).
// Returns the number of entries, or -1 when a list is malformed (an index outside [0, nkb) or not ascending).
template <bool kPairs>
__device__ __forceinline__ int build_plan(const AttnArgs& a, const int32_t* list0, int n0, const int32_t* list1, int n1,
                                          uint32_t* words, uint16_t* plan, int* total) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int bad = 0;
    if (!kPairs) {
        for (int i = tid; i < n0; i += kThreads64) {
            const int J = list0[i];
            if (J < 0 || J >= a.nkb || (i > 0 && J <= list0[i - 1])) bad = 1;
            plan[i] = uint16_t((uint32_t(J) & kPlanBlockMask) | (1u << kPlanRowBit));
        }
        if (tid == 0) plan[n0] = uint16_t(kPlanPad);
        return __syncthreads_or(bad) ? -1 : n0;
    }
    const int nw = (a.nkb + 31) >> 5;
    uint32_t *map0 = words, *map1 = words + nw, *before = words + 2 * nw;
    for (int i = tid; i < 2 * nw; i += kThreads64) words[i] = 0u;
    __syncthreads();
    for (int i = tid; i < n0 + n1; i += kThreads64) {
        const bool second = i >= n0;
        const int32_t* l = second ? list1 : list0;
        const int k = second ? i - n0 : i;
        const int J = l[k];
        if (J < 0 || J >= a.nkb || (k > 0 && J <= l[k - 1])) bad = 1;
        else atomicOr((second ? map1 : map0) + (J >> 5), 1u << (J & 31));
    }
    if (__syncthreads_or(bad)) return -1;
    if (warp == 0) {
        int base = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int n = w0 + lane < nw ? __popc(map0[w0 + lane] | map1[w0 + lane]) : 0;
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += up;
            }
            if (w0 + lane < nw) before[w0 + lane] = base + incl - n;
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) { *total = base; plan[base] = uint16_t(kPlanPad); }
    }
    __syncthreads();
    for (int w = warp; w < nw; w += kThreads64 / 32) {
        const uint32_t m0 = map0[w], m1 = map1[w], both = m0 | m1;
        if ((both >> lane) & 1u)
            plan[before[w] + __popc(both & ((1u << lane) - 1u))] =
                uint16_t(uint32_t(w * 32 + lane) | (((m0 >> lane) & 1u) << kPlanRowBit) | (((m1 >> lane) & 1u) << (kPlanRowBit + 1)));
    }
    __syncthreads();
    return *total;
}

template <int D, int BQ, int BK>
__global__ void __launch_bounds__(kThreads64, 1)
attn_tcgen05_b64_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV, const AttnArgs a) {
    using C = Cfg64<D>;
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float r_pub[kSoftGroups][kBlock];           // reference maximum after step i, slot i % 3 (handed from group to group)
    __shared__ float fin[kSoftGroups][2][kBlock];          // per group: final reference maximum and partial row sum

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Grid at D = 128: (heads of a group, position in the execution order, groups of heads), see head_group.  At D = 64:
    // (position, head, batch entry).
    constexpr bool kHeadGroups = D == 128;
    int b, h;
    if constexpr (kHeadGroups) {
        const uint32_t head = blockIdx.z * gridDim.x + blockIdx.x;
        if (head >= uint32_t(a.B) * uint32_t(a.H)) return;      // the last group may be short
        b = int(head / uint32_t(a.H)); h = int(head - uint32_t(b) * uint32_t(a.H));
    } else { b = blockIdx.z; h = blockIdx.y; }
    const int64_t bh = int64_t(b) * a.H + h;
    grid_wait();                            // launched while the compaction drains
    static_assert(BQ == 64 || BK == 64, "128-token blocks run on attn_tcgen05_kernel");
    constexpr bool kPairs = BQ == 64;
    constexpr int kPerStep = kBlock / BK;             // listed key blocks in a step
    constexpr uint32_t kO = kSoftGroups * kBlock;         // tensor-memory column of O, behind the score buffers
    const int place = kHeadGroups ? blockIdx.y : blockIdx.x;
    const int x0 = kPairs ? 2 * place : place;
    const int I = a.order[bh * a.nqb + x0];
    const int T1 = a.counts[bh * a.nqb + I];          // listed key blocks of the (first) query block
    const int32_t* list = a.lists + (bh * a.nqb + I) * int64_t(a.nkb);
    const int q0 = I * BQ;
    // rows 64..127 of a paired tile: the next query block in the order (none: as if skipped)
    const int I2 = kPairs && x0 + 1 < a.nqb ? a.order[bh * a.nqb + x0 + 1] : -1;
    const int T2 = I2 >= 0 ? a.counts[bh * a.nqb + I2] : -1;
    const int q0_2 = I2 * BQ;
    if (T1 > a.nkb || T2 > a.nkb) {                   // counts that cannot come from compaction
        if (tid == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_CHECK, 20, max(T1, T2), place);
        return;
    }
    if (T1 <= 0 && T2 <= 0) {                         // nothing to attend to: O = 0, LSE = -inf where a block is listed empty
        const bool second = kPairs && tid >= BQ;
        const int row = second ? q0_2 + tid - BQ : q0 + tid;
        if (tid < kBlock && (second ? T2 : T1) == 0 && row < a.N) {
            __nv_bfloat16* op = a.O + b * a.os[0] + h * a.os[1] + int64_t(row) * a.os[2];
#pragma unroll
            for (int c = 0; c < D / 8; ++c) *reinterpret_cast<uint4*>(op + c * 8) = make_uint4(0, 0, 0, 0);
            a.LSE[bh * a.N + row] = -INFINITY;
        }
        return;
    }
    uint4 q_rows[D / 16];                             // half of a query row, by the first two softmax groups, fetched under the plan
    if (warp < 8) {
        const int r = tid & (kBlock - 1);
        const bool second = kPairs && r >= BQ, in = (second ? T2 : T1) >= 0;
        const int row = second ? q0_2 + r - BQ : q0 + r;
        const __nv_bfloat16* qp = a.Q + b * a.qs[0] + h * a.qs[1] + int64_t(row) * a.qs[2] + (warp >> 2) * (D / 2);
#pragma unroll
        for (int v = 0; v < D / 16; ++v) q_rows[v] = in && row < a.N ? *reinterpret_cast<const uint4*>(qp + v * 8) : make_uint4(0, 0, 0, 0);
    }
    __shared__ int plan_total;
    unsigned char* area = smem_dyn + (((smem_u32(smem_dyn) + 1023u) & ~1023u) - smem_u32(smem_dyn)) + C::kOffPlan;
    uint16_t* plan = reinterpret_cast<uint16_t*>(area + (kPairs ? ((a.nkb + 31) >> 5) * 12 : 0));
    const int n_listed = build_plan<kPairs>(a, list, max(T1, 0), a.lists + (bh * a.nqb + max(I2, 0)) * int64_t(a.nkb), max(T2, 0),
                                            reinterpret_cast<uint32_t*>(area), plan, &plan_total);
    if (n_listed < 0) {
        if (tid == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_CHECK, 21, I, place);
        return;
    }
    const int T = (n_listed + kPerStep - 1) / kPerStep;       // steps

    const uint32_t smem_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t sK = smem_base + C::kOffK, sV = smem_base + C::kOffV, sQ = smem_base + C::kOffQ;
    const uint32_t bars = smem_base + C::kOffBar;
    const uint32_t bar_q = bars, bar_o = bars + 8, bar_drain = bars + 16, bar_drain2 = bars + 24;
    auto bar_kfull = [&](int s) { return bars + 32 + 8 * s; };
    auto bar_vfull = [&](int s) { return bars + 64 + 8 * s; };
    auto bar_sfull = [&](int g) { return bars + 96 + 8 * g; };       // S_g holds fresh scores; also frees the K slot of the step
    auto bar_pfull = [&](int g) { return bars + 128 + 8 * g; };      // P_g is complete
    auto bar_pvdone = [&](int g) { return bars + 160 + 8 * g; };     // P V of the step in S_g has completed: S_g and the V slot are free
    auto bar_ref = [&](int s, int q) { return bars + 192 + 8 * (s * 4 + q); };   // r_pub slot s, lane quarter q
    auto bar_fin = [&](int q) { return bars + 288 + 8 * q; };
    volatile int* abortp = &abort_flag;
    // every bounded wait of this CTA gives up after `limit` (2 s unless the workspace header asks for less)
    const unsigned long long limit = a.hdr->wait_limit_ns ? a.hdr->wait_limit_ns : kDefaultWaitNs;

    if (tid == 0) {
        abort_flag = 0;
        mbar_init(bar_q, 8); mbar_init(bar_o, 1); mbar_init(bar_drain, 1); mbar_init(bar_drain2, 1);
        for (int s = 0; s < 3; ++s) {
            mbar_init(bar_kfull(s), 1); mbar_init(bar_vfull(s), 1);
            mbar_init(bar_sfull(s), 1); mbar_init(bar_pvdone(s), 1);
            mbar_init(bar_pfull(s), 4);                              // one arrival per softmax warp of the group
            for (int q = 0; q < 4; ++q) mbar_init(bar_ref(s, q), 1);
        }
        for (int q = 0; q < 4; ++q) mbar_init(bar_fin(q), kSoftGroups);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kSoftWarps64 && lane == 0) prefetch_tmap(&mapK);
    if (warp == kSoftWarps64 + 2 && lane == 0) prefetch_tmap(&mapV);
    if (warp == kSoftWarps64 + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp >= kSoftWarps64) {
    // The CTA is launched with 512 x 128 registers; 384 x 152 + 128 x 56 uses exactly that.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;" ::: "memory");
    if (warp == kSoftWarps64 || warp == kSoftWarps64 + 2) {
        // ================= TMA producers: the K tiles, the V tiles =================
        // A slot is free once Q K^T (or P V) of the step that last used it has completed.  The producer waits for each of those
        // phases in turn, and the next one on the same barrier needs the tile it is about to fetch.
        if (lane == 0) {
            const bool is_k = warp == kSoftWarps64;
            const int stages = is_k ? C::kKStages : C::kVStages;
            const uint32_t tiles = is_k ? sK : sV, full0 = is_k ? bar_kfull(0) : bar_vfull(0), done0 = is_k ? bar_sfull(0) : bar_pvdone(0);
            const CUtensorMap* map = is_k ? &mapK : &mapV;
            int armed = -1, s = 0;
            Ring<kSoftGroups> u;                              // step that last used the slot
            for (int i = 0; i < T; ++i) {
                if (i >= stages) {
                    if (!mbar_wait(done0 + 8 * u.slot, u.phase, abortp, 100, limit)) {
                        set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, is_k ? 1 : 2, i, place); break;
                    }
                    u.next();
                }
                // Test of the time-out path only: the first K tile of the first query block in the order is never
                // requested, so the wait for it runs out and the CTA takes the abort-and-drain path.
                if (is_k && i == 0 && a.hdr->debug_withhold != 0 && place == 0 && bh == 0) { s = 1; continue; }
                mbar_expect_tx(full0 + 8 * s, C::kTileBytes);
#pragma unroll
                for (int kh = 0; kh < kPerStep; ++kh) {
                    const int key0 = int(plan[i * kPerStep + kh] & kPlanBlockMask) * BK;
#pragma unroll
                    for (int x = 0; x < C::kBoxes; ++x)
                        tma_load_4d(tiles + s * C::kTileBytes + x * C::kBoxBytes + kh * BK * 128, map, full0 + 8 * s, x * 64, key0, h, b);
                }
                armed = i;
                if (++s == stages) s = 0;
            }
            if (*abortp) {      // copies in flight must land before the CTA gives its shared memory back
                for (int k = 0; k < stages && armed - k >= 0; ++k)
                    mbar_wait_drain(full0 + 8 * ((armed - k) % stages), uint32_t((armed - k) / stages) & 1u, limit);
            }
        }
    } else if (warp == kSoftWarps64 + 1) {
        // ================= issuer of Q K^T (converged warp, one elected lane issues) =================
        constexpr uint32_t idesc_qk = instr_desc(kBlock, kBlock, 0);
        const uint64_t dk = smem_desc(sK, 16, 1024), dq = smem_desc(sQ, 16, 1024);
        const uint32_t k_lo0 = uint32_t(dk), q_lo0 = uint32_t(dq), hi_kmajor = uint32_t(dk >> 32);
        bool ok = mbar_wait_warp(bar_q, 0, abortp, 0, limit);   // the query tile is in place
        if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 3, 0, place);
        Ring<kSoftGroups> r;
        for (int iq = 0; iq < T && ok; ++iq) {
            ok = mbar_wait_warp(bar_kfull(r.slot), r.phase, abortp, 0, limit);
            if (ok && iq >= kSoftGroups) ok = mbar_wait_warp(bar_pvdone(r.slot), r.phase ^ 1u, abortp, 0, limit);
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 4, iq, place); break; }
            tc_fence_after();
            const uint32_t k_lo = k_lo0 + uint32_t(r.slot) * (C::kTileBytes >> 4), d_s = tmem + r.slot * kBlock;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off16 = ((kk / 4) * C::kBoxBytes + (kk % 4) * 32) >> 4;      // compile-time constant
                mma_ss_el(d_s, q_lo0 + off16, k_lo + off16, hi_kmajor, idesc_qk, kk > 0 ? 1u : 0u);
            }
            tc_commit_el(bar_sfull(r.slot));
            r.next();
        }
        if (__any_sync(0xffffffffu, *abortp != 0)) {      // no product may still run when tensor memory is released
            tc_commit_el(bar_drain);
            mbar_wait_drain(bar_drain, 0, limit);
            __syncwarp();
        }
    } else {
        // ================= issuer of P V =================
        constexpr uint32_t idesc_pv = instr_desc(kBlock, D, 1);
        const uint64_t dv = smem_desc(sV, C::kBoxBytes, 1024);
        const uint32_t v_lo0 = uint32_t(dv), hi_v = uint32_t(dv >> 32);
        bool ok = true;
        Ring<kSoftGroups> r;
        Ring<C::kVStages> rv;
        for (int ip = 0; ip < T && ok; ++ip) {
            // Which rows list the step's key blocks.  Taken before the waits, with one choice between two batches.
            uint32_t e_step = 0u;
            if (kPairs) {
#pragma unroll
                for (int kh = 0; kh < kPerStep; ++kh) e_step |= uint32_t(plan[ip * kPerStep + kh] >> kPlanRowBit) << (2 * kh);
                e_step = __reduce_or_sync(0xffffffffu, e_step);
            }
            ok = mbar_wait_warp(bar_vfull(rv.slot), rv.phase, abortp, 0, limit);
            if (ok) ok = mbar_wait_warp(bar_pfull(r.slot), r.phase, abortp, 0, limit);
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 5, ip, place); break; }
            tc_fence_after();
            // P from tensor memory (16 keys = 8 packed columns per instruction; a chunk of 32 keys every 32 columns, its second
            // part 16 columns on), V tile as the MN-major B operand (rows = keys, 64-element chunks of the head dimension one box apart)
            const uint32_t v_lo = v_lo0 + uint32_t(rv.slot) * (C::kTileBytes >> 4), p_t = tmem + r.slot * kBlock, d_o = tmem + kO;
            const uint32_t acc0 = ip > 0 ? 1u : 0u;
            if (kPairs && e_step != (kPerStep == 2 ? 15u : 3u)) {      // rows that do not list a block keep what they have
#pragma unroll
                for (int kh = 0; kh < kPerStep; ++kh) {
                    const uint32_t off_lo = ((e_step >> (2 * kh)) & 1u) - 1u, off_hi = ((e_step >> (2 * kh + 1)) & 1u) - 1u;
#pragma unroll
                    for (int kk = kh * (BK / 16); kk < (kh + 1) * (BK / 16); ++kk) {
                        const uint32_t p_k = p_t + (kk >> 1) * 32 + (kk & 1) * 8;
                        mma_ts_el_rows(d_o, p_k, v_lo + kk * (2048 >> 4), hi_v, idesc_pv, off_lo, off_hi, 1u);
                        mma_ts_el_rows(d_o, p_k + 16, v_lo + kk * (2048 >> 4), hi_v, idesc_pv, off_lo, off_hi, 1u);
                    }
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < kBlock / 16; ++kk) {
                    const uint32_t p_k = p_t + (kk >> 1) * 32 + (kk & 1) * 8;
                    mma_ts_el(d_o, p_k, v_lo + kk * (2048 >> 4), hi_v, idesc_pv, kPairs || kk > 0 ? 1u : acc0);      // kPairs: O starts at zero
                    mma_ts_el(d_o, p_k + 16, v_lo + kk * (2048 >> 4), hi_v, idesc_pv, 1u);
                }
            }
            tc_commit_el(bar_pvdone(r.slot));
            r.next(); rv.next();
        }
        if (ok) tc_commit_el(bar_o);
        if (__any_sync(0xffffffffu, *abortp != 0)) {
            tc_commit_el(bar_drain2);
            mbar_wait_drain(bar_drain2, 0, limit);
            __syncwarp();
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;" ::: "memory");
        // ================= softmax + epilogue (warps 0-11) =================
        // All groups feed the same O accumulator, so they share one reference maximum per row: the group that handles step i
        // derives R_i from R_{i-1} (published by the group before it right after its row-maximum pass) and publishes R_i in turn.
        // The reference only moves when a row maximum exceeds it by more than the threshold; then this group rescales O before
        // delivering P_i.
        const int quarter = warp & 3, wg = warp >> 2;
        const int r_loc = quarter * 32 + lane;                      // query row within the tile
        const uint32_t lane_base = uint32_t(quarter * 32) << 16;
        const bool second = kPairs && quarter >= 2;                 // warp-uniform: rows of the pair's second query block
        const int row = second ? q0_2 + r_loc - BQ : q0 + r_loc;
        const bool row_in = row < a.N && (!kPairs || (second ? T2 : T1) >= 0);   // rows of a skipped query block are left alone
        // the last entry of the plan is the only one that can be ragged
        const int nvalid_last = ((n_listed - 1) % kPerStep) * BK + min(BK, a.N - int(plan[n_listed - 1] & kPlanBlockMask) * BK);
        const uint32_t tS = tmem + lane_base + wg * kBlock;
        const int prev = wg == 0 ? kSoftGroups - 1 : wg - 1;            // group of the step before, and the slot of its reference
        const uint64_t scale2 = pack2(a.scale_log2, a.scale_log2), minus1 = pack2(-1.f, -1.f);
        if (wg < 2) {
            // The query tile goes into shared memory as the K tiles lie there (rows of 128 bytes, 16-byte pieces exchanged by
            // row); each of the first two groups brings half of the head dimension.
            const uint32_t dst = sQ + (D == 128 ? wg * C::kBoxBytes : 0u) + r_loc * 128;
#pragma unroll
            for (int v = 0; v < D / 16; ++v) {
                const uint4 u = q_rows[v];
                const int piece = D == 128 ? v : wg * 4 + v;
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + uint32_t((piece ^ (r_loc & 7)) * 16)), "r"(u.x), "r"(u.y), "r"(u.z), "r"(u.w) : "memory");
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (kPairs) {       // products into O may be masked by rows, so none of them can be the one that starts it
                const uint32_t zero[32] = {};
#pragma unroll
                for (int c = 0; c < D / 64; ++c) tmem_st32(tmem + lane_base + kO + wg * (D / 2) + c * 32, zero);
                tmem_wait_st();
                tc_fence_before();
            }
            mbar_arrive_warp(bar_q);
        }
        float m_w = -INFINITY, l_w = 0.f;                           // this group's reference and partial row sum
        bool ok = true;
        uint32_t ph = 0;
        for (int i = wg; i < T; i += kSoftGroups, ph ^= 1u) {
            const uint32_t ph_prev = wg == 0 ? ph ^ 1u : ph;
            ok = mbar_wait_warp(bar_sfull(wg), ph, abortp, 20, limit);   // warp-uniform: the loads below are collective
            if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 7, i, place); break; }
            tc_fence_after();
            const int nvalid = (i == T - 1) ? nvalid_last : kBlock;      // >= 1; < 128 only for a ragged last block
            // the halves of the step that this warp's rows list (a pad entry is listed by nobody)
            const int bit = kPlanRowBit + (second ? 1 : 0);
            const bool on0 = (plan[i * kPerStep] >> bit) & 1, on1 = (plan[i * kPerStep + kPerStep - 1] >> bit) & 1;
            // columns of chunk c that count: its rows list the block, and the key is a token (warp-uniform)
            auto columns = [&](int c) { return (c < 2 ? on0 : on1) ? min(32, max(0, nvalid - c * 32)) : 0; };
            // row maximum of the raw scores (the scale is positive), four independent chains
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            auto max_of = [&](const float (&s)[32]) {
#pragma unroll
                for (int e = 0; e < 32; e += 2) mx4[(e >> 1) & 3] = max3(mx4[(e >> 1) & 3], s[e], s[e + 1]);
            };
            if (on0 && on1 && nvalid == kBlock) {
                float s0[32], s1[32], s2[32], s3[32];
                tmem_ld32(tS, s0); tmem_ld32(tS + 32, s1);
                tmem_wait_ld(s0, s1);
                tmem_ld32(tS + 64, s2); tmem_ld32(tS + 96, s3);
                max_of(s0); max_of(s1);
                tmem_wait_ld(s2, s3);
                max_of(s2); max_of(s3);
            } else {
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    const int n = columns(c);
                    if (n == 0) continue;
                    float v[32];
                    tmem_ld32(tS + c * 32, v);
                    tmem_wait_ld(v);
                    if (n < 32) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) if (e >= n) v[e] = -INFINITY;
                    }
                    max_of(v);
                }
            }
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * a.scale_log2;
            float v[32];
            tmem_ld32(tS, v);                    // first chunk for the exponentials, while the reference is on its way
            // reference handed over from step i-1
            float r_prev = -INFINITY, r_now = mx;
            bool grow = false;
            if (i > 0) {
                ok = mbar_wait_warp(bar_ref(prev, quarter), ph_prev, abortp, 0, limit);
                if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 10, i, place); break; }
                r_prev = r_pub[prev][r_loc];
                grow = mx > r_prev + kRescaleThreshold;
                r_now = grow ? mx : r_prev;
            }
            r_pub[wg][r_loc] = r_now;
            mbar_arrive_warp(bar_ref(wg, quarter));
            if (i > 0 && __any_sync(0xffffffffu, grow)) {
                // O must be quiescent: P V of step i-1 complete.  P V is issued in step order and that of step i cannot start
                // before this group delivers P_i.  (Q K^T of step i waited for P V of step i-3, so the phase is exact.)
                ok = mbar_wait_warp(bar_pvdone(prev), ph_prev, abortp, 0, limit);
                if (!ok) { if (lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 9, i, place); break; }
                tc_fence_after();
                // 1 for rows that did not move (rows of a pair may both times be at -inf: nothing listed so far)
                const float f = !kPairs || grow ? ex2_approx(r_prev - r_now) : 1.f;
#pragma unroll 1
                for (int c = 0; c < D / 16; ++c) {
                    float o[16];
                    tmem_ld16(tmem + lane_base + kO + c * 16, o);
                    tmem_wait_ld(o);
                    uint32_t r[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(o[e] * f);
                    tmem_st16(tmem + lane_base + kO + c * 16, r);
                }
            }
            if (m_w != r_now) { l_w *= ex2_approx(m_w - r_now); m_w = r_now; }   // first use: l_w = 0, exp2(-inf) = 0
            // P = exp2(s * scale - R_i), as two bf16: the upper half of the word and what that leaves.  The portable kernel has one
            // bf16, but its reference is the running maximum, so that the largest weight of a row is 1 and exact.  Under a
            // reference that lags the largest weight is rounded as well, and O comes out further from the fp64 result: relative
            // error 1.713e-3 against 1.698e-3 on a 1024-token layer of D = 64, where the rounding of O alone is 1.654e-3; with
            // scores three times as large the error of P is 2.4 times as large.  As two bf16 it is 1.654e-3.
            // A chunk goes back to the columns it came from, the first parts of its 32 probabilities in front of the second.  The
            // loop is not unrolled: with four copies the instruction cache misses (Wan-1.3B-shaped layer 3.08 -> 3.74 ms).
            const uint64_t neg_m2 = pack2(-r_now, -r_now);
            uint64_t part2[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                const int n = columns(c);
                tmem_wait_ld(v);
                uint32_t hi[16], lo[16];
                if (n == 0) {                    // nothing of the chunk belongs to these rows (their reference may be -inf)
                    if (c < 3) tmem_ld32(tS + c * 32 + 32, v);
#pragma unroll
                    for (int e = 0; e < 16; ++e) hi[e] = lo[e] = 0u;
                } else {
                    if (n < 32) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) if (e >= n) v[e] = -INFINITY;
                    }
                    float x[32];
#pragma unroll
                    for (int e = 0; e < 16; ++e) unpack2(fma2(pack2(v[2 * e], v[2 * e + 1]), scale2, neg_m2), x[2 * e], x[2 * e + 1]);
                    if (c < 3) tmem_ld32(tS + c * 32 + 32, v);
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float p0 = ex2_approx(x[2 * e]), p1 = ex2_approx(x[2 * e + 1]);
                        const uint64_t p = pack2(p0, p1);
                        part2[e & 1] = add2(part2[e & 1], p);
                        const uint32_t b0 = __float_as_uint(p0), b1 = __float_as_uint(p1);
                        hi[e] = __byte_perm(b0, b1, 0x7632);
                        float d0, d1;            // p less its upper half, exact
                        unpack2(fma2(pack2(__uint_as_float(b0 & 0xFFFF0000u), __uint_as_float(b1 & 0xFFFF0000u)), minus1, p), d0, d1);
                        lo[e] = pack_bf16(d0, d1);
                    }
                }
                tmem_st16(tS + c * 32, hi);      // this warp has read these rows' scores, and nobody else does
                tmem_st16(tS + c * 32 + 16, lo);
            }
            {
                float s0, s1, s2, s3;
                unpack2(part2[0], s0, s1); unpack2(part2[1], s2, s3);
                l_w += (s0 + s1) + (s2 + s3);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive_warp(bar_pfull(wg));
        }
        tmem_drain_ld();
        // combine the groups' sums under the final reference (the later step holds the larger one)
        if (ok) {
            fin[wg][0][r_loc] = m_w;
            fin[wg][1][r_loc] = l_w;
            mbar_arrive_warp(bar_fin(quarter));
            ok = mbar_wait_warp(bar_fin(quarter), 0, abortp, 0, limit);
            if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 11, T, place);
        }
        if (ok && wg < 2) {
            ok = mbar_wait_warp(bar_o, 0, abortp, 20, limit);
            if (!ok && lane == 0) set_status(a.hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 8, T, place);
        }
        if (ok && wg < 2) {                 // the first two groups write half of the head dimension each
            tc_fence_after();
            float r_fin = fin[0][0][r_loc];
#pragma unroll
            for (int g = 1; g < kSoftGroups; ++g) r_fin = fmaxf(r_fin, fin[g][0][r_loc]);
            float l_tot = 0.f;
#pragma unroll
            for (int g = 0; g < kSoftGroups; ++g) l_tot += fin[g][1][r_loc] * ex2_approx(fin[g][0][r_loc] - r_fin);
            if (kPairs && (second ? T2 : T1) <= 0) l_tot = 0.f;
            // rows of a pair that list nothing, and rows whose sum is NaN: LSE = -inf, as the portable kernel has it
            const float inv = l_tot > 0.f ? 1.f / l_tot : 0.f;
            // this warp's rows are consecutive tokens of one query block
            const int row0 = row - lane;
            __nv_bfloat16* op = a.O + b * a.os[0] + h * a.os[1] + int64_t(row0) * a.os[2] + wg * (D / 2);
            write_rows<D>(tmem + lane_base + kO + wg * (D / 2), inv, sK + warp * (32 * D), lane, op, a.os[2], (kPairs && (second ? T2 : T1) < 0) ? 0 : a.N - row0);
            if (wg == 0 && row_in) a.LSE[bh * a.N + row] = l_tot > 0.f ? (r_fin + log2f(l_tot)) * kLn2 : -INFINITY;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kSoftWarps64 + 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Self-test of the bounded wait: one warp waits on a barrier that nothing ever arms, with the limit the caller gives,
// and must come back with CARNATOR_ERR_DEVICE_TIMEOUT in the header (same helpers as the kernels above).
__global__ void wait_timeout_selftest_kernel(WsHeader* hdr, unsigned long long limit_ns) {
    __shared__ __align__(8) unsigned long long bar_mem;
    __shared__ int abort_flag;
    const uint32_t bar = smem_u32(&bar_mem);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait_warp(bar, 0, &abort_flag, 50, limit_ns);
    if (!ok && threadIdx.x == 0) set_status(hdr, CARNATOR_ERR_DEVICE_TIMEOUT, 90, 0, 0);
}

// ---- host side ------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = [] {       // a call that comes during the first one's look-up waits for it
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        cudaGetLastError();
        return EncodeTiledFn(nullptr);
    }();
    return fn;
}

// 4-D map over a [B,H,N,D] bf16 tensor with arbitrary (16-byte multiple) strides: box = 64 x box_rows x 1 x 1,
// 128-byte swizzle, rows >= N read as zero.
inline bool make_map(CUtensorMap* map, const void* base, int B, int H, int N, int D, const int64_t st[3], int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {cuuint64_t(D), cuuint64_t(N), cuuint64_t(H), cuuint64_t(B)};
    // the stride of a size-1 axis is never used for addressing but must still be a valid value; a zero stride on a
    // longer axis cannot be expressed (callers check tma_strides_ok before they get here)
    const cuuint64_t row = cuuint64_t(st[2]) * 2;
    if ((H > 1 && st[1] <= 0) || (B > 1 && st[0] <= 0)) return false;
    const cuuint64_t s_h = st[1] > 0 ? cuuint64_t(st[1]) * 2 : row * N;
    const cuuint64_t s_b = st[0] > 0 ? cuuint64_t(st[0]) * 2 : s_h * H;
    cuuint64_t strides[3] = {row, s_h, s_b};
    cuuint32_t box[4] = {64, cuuint32_t(box_rows), 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// The same tensor with the head dimension split into its 64-element halves as a dimension of its own, behind the
// tokens: one box = D/64 halves x box_rows tokens x 64 elements lands in shared memory as [half][token][64] (each
// half a 128-byte-swizzled slab), so one copy fetches what make_map's boxes fetch in D/64.
inline bool make_map_halves(CUtensorMap* map, const void* base, int B, int H, int N, int D, const int64_t st[3], int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[5] = {64, cuuint64_t(N), cuuint64_t(D / 64), cuuint64_t(H), cuuint64_t(B)};
    const cuuint64_t row = cuuint64_t(st[2]) * 2;
    if ((H > 1 && st[1] <= 0) || (B > 1 && st[0] <= 0)) return false;
    const cuuint64_t s_h = st[1] > 0 ? cuuint64_t(st[1]) * 2 : row * N;
    const cuuint64_t s_b = st[0] > 0 ? cuuint64_t(st[0]) * 2 : s_h * H;
    cuuint64_t strides[4] = {row, 128, s_h, s_b};
    cuuint32_t box[5] = {64, cuuint32_t(box_rows), cuuint32_t(D / 64), 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// 2-D map over a row-major [rows, D] bf16 array: box = box_cols x box_rows (64 columns: 128-byte swizzle, 32 columns:
// 64-byte swizzle), rows past the end read as zero.
inline bool make_map_2d(CUtensorMap* map, const void* base, int64_t rows, int D, int box_rows, int box_cols = 64) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {cuuint64_t(D), cuuint64_t(rows)};
    cuuint64_t strides[1] = {cuuint64_t(D) * 2};
    cuuint32_t box[2] = {cuuint32_t(box_cols), cuuint32_t(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace tc

// A tensor map cannot express a zero stride, so a tensor that is shared over heads or batch entries (stride 0 on an
// axis longer than 1) is not read through TMA: such shapes run on the portable kernel.
inline bool tma_strides_ok(const carnator_shape* s, const int64_t st[3]) {
    return (s->B == 1 || st[0] > 0) && (s->H == 1 || st[1] > 0);
}

// Shapes for which the caller may ask for this kernel by name: 128-token blocks.
inline bool tcgen05_supported(const carnator_shape* s) {
    return s->block_q == tc::kBlock && s->block_k == tc::kBlock && (s->D == 64 || s->D == 128) &&
           tma_strides_ok(s, s->k_stride) && tma_strides_ok(s, s->v_stride);
}

// Heads that run side by side, the longest rows of all of them first.  One head after the other, the full rows of the last
// head start when nearly everything else is done, and most SMs wait for them: five-frame clip (24 heads, 10 tiles per SM)
// 406 -> 390 us.  Only for layers of up to 16 tiles per SM: on longer ones that wait is no longer seen.  At most as many heads as
// keep K and V within 24 MB, so that they stay in either half of L2 (64 MB took 399 us), in groups of equal size: a short last
// group leaves SMs idle at the end (15 heads of 3.1 MB in groups of 7, 7 and 1: 215 us, in three of 5: 198 us; on 38 layers of 7 to 25
// heads of 3000 to 12000 tokens groups of unequal size took 1.4 % longer in the middle, at most 14 % longer and once 3 % less).
constexpr int64_t kHeadGroupBytes = int64_t(24) << 20;
constexpr int64_t kHeadGroupTiles = 16 * 148;
inline int64_t head_group(const AttnArgs& a, int D, int tiles_per_head) {
    const int64_t heads = int64_t(a.B) * a.H, per_head = int64_t(a.N) * D * 4;
    if (heads * tiles_per_head > kHeadGroupTiles && heads <= 65535) return 1;
    const int64_t most = std::max<int64_t>(1, std::min(heads, kHeadGroupBytes / per_head)), groups = (heads + most - 1) / most;
    return (heads + groups - 1) / groups;
}

template <int D>
inline carnator_status launch_tc(const AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv,
                                 cudaStream_t stream, char* err, size_t errlen) {
    const uint32_t smem = tc::Cfg<D>::kSmemBytes;
    auto kern = tc::attn_tcgen05_kernel<D>;
    static SmemAllowed allowed;
    cudaError_t e;
    const unsigned long long ctx = context_id();
    if (!allowed.has(ctx)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(tcgen05)", err, errlen);
        // The register hand-over inside the kernel only completes if the CTA owns enough registers: check what the
        // compiler allocated instead of finding out on the device.
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, kern);
        if (e != cudaSuccess) return cuda_error(e, "cudaFuncGetAttributes(tcgen05)", err, errlen);
        if (fa.numRegs * tc::kThreads < tc::kSoftmaxWarps * 32 * tc::kRegsSoftmax + 128 * tc::kRegsService) {
            snprintf(err, errlen, "attn_tcgen05_kernel was built with %d registers per thread: too few for its setmaxnreg split", fa.numRegs);
            return CARNATOR_ERR_UNSUPPORTED;
        }
        allowed.add(ctx);
    }
    dim3 grid(a.nqb, a.H, a.B);
    if (D == 128) {
        const int64_t heads = int64_t(a.B) * a.H, group = head_group(a, D, a.nqb);
        grid = dim3(unsigned(group), unsigned(a.nqb), unsigned((heads + group - 1) / group));
    }
    e = launch_dependent(kern, grid, dim3(tc::kThreads), smem, stream, mk, mv, a);
    if (e != cudaSuccess) return cuda_error(e, "attn_tcgen05_kernel", err, errlen);
    return CARNATOR_OK;
}

// Shapes that run on the tensor cores when the library chooses.  The kernel for 64-token blocks keeps a plan of the listed key
// blocks in shared memory, 2.4 bytes a block beside 194 KB of tiles at D = 128; beyond 12288 key blocks the portable kernel stays.
inline bool tcgen05_takes(const carnator_shape* s) {
    if (s->block_q == tc::kBlock && s->block_k == tc::kBlock) return tcgen05_supported(s);
    return (s->D == 64 || s->D == 128) && ceil_div(s->N, s->block_k) <= tc::kPlanMaxKeyBlocks &&
           tma_strides_ok(s, s->k_stride) && tma_strides_ok(s, s->v_stride);
}

template <int D, int BQ, int BK>
inline carnator_status launch_b64(const AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv,
                                    cudaStream_t stream, char* err, size_t errlen) {
    const uint32_t smem = tc::Cfg64<D>::kSmemBytes + tc::plan_bytes(a.nkb);
    auto kern = tc::attn_tcgen05_b64_kernel<D, BQ, BK>;
    static SmemAllowed allowed;
    cudaError_t e;
    const unsigned long long ctx = context_id();
    if (!allowed.has(ctx)) {             // once: with room for the longest plan
        const uint32_t most = tc::Cfg64<D>::kSmemBytes + tc::plan_bytes(tc::kPlanMaxKeyBlocks);
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most));
        if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(tcgen05_b64)", err, errlen);
        // The register hand-over inside the kernel only completes if the CTA owns enough registers: check what the
        // compiler allocated instead of finding out on the device.
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, kern);
        if (e != cudaSuccess) return cuda_error(e, "cudaFuncGetAttributes(tcgen05_b64)", err, errlen);
        if (fa.numRegs * tc::kThreads64 < tc::kSoftWarps64 * 32 * tc::kRegsSoftmax64 + 128 * tc::kRegsService64) {
            snprintf(err, errlen, "attn_tcgen05_b64_kernel was built with %d registers per thread: too few for its setmaxnreg split", fa.numRegs);
            return CARNATOR_ERR_UNSUPPORTED;
        }
        allowed.add(ctx);
    }
    const unsigned tiles = unsigned(BQ == 64 ? ceil_div(a.nqb, 2) : a.nqb);      // of a head
    dim3 grid(tiles, a.H, a.B);
    if (D == 128) {
        const int64_t heads = int64_t(a.B) * a.H, group = head_group(a, D, int(tiles));
        grid = dim3(unsigned(group), tiles, unsigned((heads + group - 1) / group));
    }
    e = launch_dependent(kern, grid, dim3(tc::kThreads64), smem, stream, mk, mv, a);
    if (e != cudaSuccess) return cuda_error(e, "attn_tcgen05_b64_kernel", err, errlen);
    return CARNATOR_OK;
}

template <int D>
inline carnator_status launch_tc_blocks(const AttnArgs& a, const CUtensorMap& mk, const CUtensorMap& mv,
                                        cudaStream_t stream, char* err, size_t errlen) {
    if (a.block_q == 128) return a.block_k == 128 ? launch_tc<D>(a, mk, mv, stream, err, errlen)
                                                  : launch_b64<D, 128, 64>(a, mk, mv, stream, err, errlen);
    return a.block_k == 128 ? launch_b64<D, 64, 128>(a, mk, mv, stream, err, errlen)
                            : launch_b64<D, 64, 64>(a, mk, mv, stream, err, errlen);
}

inline carnator_status launch_tcgen05(const AttnArgs& a, const carnator_shape* s, cudaStream_t stream,
                                      char* err, size_t errlen, long long* launches) {
    CUtensorMap mk, mv;      // Q is read with plain loads (once per CTA, into tensor memory)
    if (!tc::make_map(&mk, a.K, a.B, a.H, a.N, s->D, a.ks, a.block_k) ||
        !tc::make_map(&mv, a.V, a.B, a.H, a.N, s->D, a.vs, a.block_k)) {
        snprintf(err, errlen, "cuTensorMapEncodeTiled failed or is unavailable");
        return CARNATOR_ERR_CUDA;
    }
    carnator_status st = (s->D == 128) ? launch_tc_blocks<128>(a, mk, mv, stream, err, errlen)
                                       : launch_tc_blocks<64>(a, mk, mv, stream, err, errlen);
    if (st == CARNATOR_OK) *launches = 1;
    return st;
}

}  // namespace carnator

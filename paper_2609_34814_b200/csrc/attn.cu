// Block-sparse FlashAttention-style forward for sm_100a, scheduled by a row order.
//
// What it computes (Sections 2.1-2.3 of the WaveAlign paper): for query block i of head h,
//   O_i = softmax(scale * Q_i K_sel^T) V_sel  over the tokens of the K/V blocks listed for
// (h, i), visited in the listed order, with the online-softmax state and the partial output
// kept on chip and written once.  The order in which query blocks are started is the
// head-major concatenation of row_order (Algorithm 2's output): persistent CTAs, one per
// SM, take tickets from a global counter, so a freed SM starts the next row of the list at
// once - the streaming "wave" behaviour of Section 2.3 that the schedule is built for.
//
// Structure of one CTA (640 threads; calls of many 64-row blocks have k_bsattn_fwd_rows64 as their first launch):
//   warp 0      producer: takes tickets, publishes tasks, issues TMA loads of the Q tile and of the K
//               tiles (128-byte-swizzled slabs) into shared-memory rings, as far ahead as the rings allow
//   warp 19     requests the V tiles (a box costs the warp that requests it ~150 clk)
//   warp 18     MMA issuer 1: S_j = Q K_j^T (operands in shared memory) into one of three S
//               buffers in tensor memory, up to three blocks ahead of the softmax
//   warp 1      MMA issuer 2: O += P_j V_j (P read from tensor memory, where it lies over the
//               columns S_j came from), fp32 accumulator in tensor memory.  Two issuing warps:
//               the waits and ring arithmetic of one run while the other's MMAs execute
//   warps 2-17  softmax, two teams of eight warps that share the KV tiles of a task (by turns, but for the first two
//               in one kernel);
//               inside a team a row of S has two owners, one per half of its columns (row max
//               in the tiles that take one, then exponentials and P in a second read of S,
//               32 columns at a time).  On every scheduler two warps of each
//               team are resident, the teams half a block apart, so one team's waits and loads
//               hide behind the other's arithmetic.  Both teams have the reference max of a row
//               from shared memory, in the first launch once a task, in the second from tile to
//               tile; every thread keeps the row sum of its own columns; O in tensor memory is rescaled only in the second launch, when the
//               max grew by more than 2^8; the epilogue adds the four partial sums of a row, normalises
//               and stores O at the ORIGINAL row (no inverse permutation; 128-row blocks through shared memory)
// Two launches per call: in the first the row max is taken in the first tile of a task only
// and the reference stays fixed afterwards (softmax does not depend on it short of
// overflow: P in bf16, the sums and O in fp32 have the same exponent range); a task in which a
// tile's sum of exponentials reaches 2^60 or a result is not finite is listed in the workspace and computed
// again by the second launch, which takes the max of every tile.
// Every wait on an mbarrier is bounded; when one runs out the CTA records
// {WAVEAL_ERR_TIMEOUT, site} and all roles leave through the common teardown.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cmath>
#include <type_traits>
#include "host_common.h"

namespace {

// 20 warps: producer, two MMA issuers, sixteen softmax warps, V tile loader
constexpr int kThreads = 640;
constexpr int kProducerWarp = 0, kPvWarp = 1, kSoftmaxWarp0 = 2, kQkWarp = 18, kVLoadWarp = 19;
constexpr long long kTimeoutCycles = 4000000000ll;   // ~2 s at boost clock
constexpr long long kSelfTestCycles = 4000000ll;     // ~2 ms: wait limit under WAVEAL_ATTN_SELFTEST_LOST_TILE
// 1 pair of elements in n takes 2^x from the FMA pipe, the others from the transcendental unit (dense 128-row
// tiles, clk per tile: n = 3: 1,449, 4: 1,439, 5: 1,431)
constexpr int kPolyEvery = 5;

// ------------------------------------------------------------------ PTX wrappers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One lane of a converged warp gets true.  tcgen05.mma / tcgen05.commit are issued under
// this predicate, one instruction at a time, with their operands computed by the whole warp:
// the operands then stay in uniform registers (a branch on the lane index instead makes the
// compiler move every operand from vector registers, which halves the MMA issue rate).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t pred = 0;
  asm volatile(
      "{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\t"
      "elect.sync rx|px, 0xFFFFFFFF;\n\t"
      "@px mov.s32 %0, 1;\n\t}"
      : "+r"(pred));
  return pred;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
// one bulk group per store; the coordinates of elements beyond the tensor are left out by the copy engine
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* tm, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {   // whole warp calls; one lane issues
  if (elect_one())
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem], bf16 inputs, fp32 accumulate, one CTA: four of them along K, 32 bytes of A and B further each.
// ONE: one election for the four instead of one each.  128-row blocks: 0.6 to 1.2 % of the cycles less (488 k -> 484 k on 5 heads of
// 256 rows, 2,059 k -> 2,035 k on 3 dense heads); 64-row blocks, head_dim 128: 1 to 2 % more (300.3 k -> 306.7 k on 300 rows of 150 blocks,
// 91.4 k -> 93.0 k on 200 of 60; at head_dim 64 the same), so those elect each time.  For the products with A in tensor memory,
// below, it lost 3 %.
template <bool ONE>
__device__ __forceinline__ void umma4_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  if constexpr (!ONE) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (elect_one())
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc + 2 * k), "l"(b_desc + 2 * k), "r"(idesc), "r"(k ? 1u : accumulate)
            : "memory");
    return;
  }
  asm volatile(
      "{\n\t.reg .b32 rx;\n\t.reg .pred e, p, t;\n\t.reg .b64 a, b;\n\t"
      "elect.sync rx|e, 0xFFFFFFFF;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, %3, %3;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]: A is 128 lanes x K bf16, two K elements per 32-bit column
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  if (elect_one())
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[smem] * B[smem] for 64 rows of A: row m of D lies in lanes m and 64 + m, the first half of the N columns in the
// lower lanes, the second half in the upper ones
// N (4 or 8) of them along K, then the commit of all that this thread has issued.  A and B are a step further each time, and a
// jump further from the fifth on.  One election for all: with one for each, the issuing warp's own instructions took
// longer than the products.
template <int N, int A_STEP, int A_JUMP, int B_STEP, int B_JUMP>
__device__ __forceinline__ void umma_ws_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate, uint32_t bar) {
  static_assert(N == 4 || N == 8, "four products or eight");
#define WAVEAL_WS(a, b, p) "@e tcgen05.mma.ws.cta_group::1.kind::f16 [%0], " a ", " b ", %3, " p ";\n\t"
  if constexpr (N == 8)
    asm volatile(
        "{\n\t.reg .b32 rx;\n\t.reg .pred e, p, t;\n\t.reg .b64 a, b;\n\t"
        "elect.sync rx|e, 0xFFFFFFFF;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, %3, %3;\n\t"
        WAVEAL_WS("%1", "%2", "p")
        "add.s64 a, %1, %6;\n\tadd.s64 b, %2, %8;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, 2 * %6;\n\tadd.s64 b, %2, 2 * %8;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, 3 * %6;\n\tadd.s64 b, %2, 3 * %8;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, %7;\n\tadd.s64 b, %2, %9;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, %7 + %6;\n\tadd.s64 b, %2, %9 + %8;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, %7 + 2 * %6;\n\tadd.s64 b, %2, %9 + 2 * %8;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, %7 + 3 * %6;\n\tadd.s64 b, %2, %9 + 3 * %8;\n\t" WAVEAL_WS("a", "b", "t")
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(bar), "n"(A_STEP >> 4), "n"(A_JUMP >> 4), "n"(B_STEP >> 4), "n"(B_JUMP >> 4)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .b32 rx;\n\t.reg .pred e, p, t;\n\t.reg .b64 a, b;\n\t"
        "elect.sync rx|e, 0xFFFFFFFF;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, %3, %3;\n\t"
        WAVEAL_WS("%1", "%2", "p")
        "add.s64 a, %1, %6;\n\tadd.s64 b, %2, %7;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, 2 * %6;\n\tadd.s64 b, %2, 2 * %7;\n\t" WAVEAL_WS("a", "b", "t")
        "add.s64 a, %1, 3 * %6;\n\tadd.s64 b, %2, 3 * %7;\n\t" WAVEAL_WS("a", "b", "t")
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(bar), "n"(A_STEP >> 4), "n"(B_STEP >> 4)
        : "memory");
#undef WAVEAL_WS
}

// two fp32 operations per instruction (register pairs)
__device__ __forceinline__ void ffma2(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2,%3};\n\tmov.b64 rb, {%4,%5};\n\tmov.b64 rc, {%6,%7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0,%1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void fadd2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2,%3};\n\tmov.b64 rb, {%4,%5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0,%1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// 2^(x) for two values on the FMA and integer pipes (for a share of the elements, to take load
// off the transcendental unit: at 16 results per clock and SM it is as busy as the tensor
// cores).  The caller passes s and the pair (a, b) of x = a*s + b.  The argument is first
// confined to the window [kPolyLo, kPolyLo + 128] by a saturating multiply-add
// (y = sat(x/128 - kPolyLo/128) in [0, 1]; x is taken back from y with an absolute error
// below 2^-17), so that the exponent arithmetic below can neither wrap into the sign bit
// (x >= 128.5 would) nor underflow: an x above the window comes out as 2^(kPolyLo+128) = 2^64,
// far above the limit at which the fixed-reference pass hands a task to the second launch; an x
// below it (a key that does not exist, -inf) as 2^-64.  x is then rounded to the nearest integer
// n with the 1.5*2^23 trick, a degree-3 polynomial gives 2^(x-n) on [-0.5, 0.5] (relative error
// 7.5e-5, far below the bf16 cut of P), and n is added to the exponent field.
constexpr float kPolyLo = -64.0f;
constexpr float kRedoLimit = 1152921504606846976.0f;     // 2^60: tile sums at or above it (or NaN) list the task
constexpr float kCheckSum = 16777216.0f;                 // 2^24: results of rows with a sum at or above it are checked for being finite
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float d;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ void ex2_fma2(float& e0, float& e1, float s0, float s1, float a128, float b128) {
  // a128 = a/128, b128 = (b - kPolyLo)/128
  const float y0 = fma_sat(s0, a128, b128), y1 = fma_sat(s1, a128, b128);
  constexpr float kMagic = 12582912.0f;                 // 1.5 * 2^23
  float xi0, xi1, n0, n1, f0, f1, q0, q1;
  ffma2(xi0, xi1, y0, y1, 128.0f, 128.0f, kMagic + kPolyLo, kMagic + kPolyLo);   // bits: 0x4B400000 + n
  fadd2(n0, n1, xi0, xi1, -(kMagic + kPolyLo), -(kMagic + kPolyLo));             // n - kPolyLo = round(128 y)
  ffma2(f0, f1, y0, y1, 128.0f, 128.0f, -n0, -n1);                               // x - n
  ffma2(q0, q1, f0, f1, 0.05517137423157692f, 0.05517137423157692f, 0.2426110953092575f, 0.2426110953092575f);
  ffma2(q0, q1, q0, q1, f0, f1, 0.6932610273361206f, 0.6932610273361206f);
  ffma2(q0, q1, q0, q1, f0, f1, 0.9999280571937561f, 0.9999280571937561f);
  e0 = __int_as_float(__float_as_int(q0) + (__float_as_int(xi0) << 23));
  e1 = __int_as_float(__float_as_int(q1) + (__float_as_int(xi1) << 23));
}

#define WAVEAL_R32(v, o) \
  "=r"(v[o+0]), "=r"(v[o+1]), "=r"(v[o+2]), "=r"(v[o+3]), "=r"(v[o+4]), "=r"(v[o+5]), "=r"(v[o+6]), "=r"(v[o+7]), \
  "=r"(v[o+8]), "=r"(v[o+9]), "=r"(v[o+10]), "=r"(v[o+11]), "=r"(v[o+12]), "=r"(v[o+13]), "=r"(v[o+14]), "=r"(v[o+15]), \
  "=r"(v[o+16]), "=r"(v[o+17]), "=r"(v[o+18]), "=r"(v[o+19]), "=r"(v[o+20]), "=r"(v[o+21]), "=r"(v[o+22]), "=r"(v[o+23]), \
  "=r"(v[o+24]), "=r"(v[o+25]), "=r"(v[o+26]), "=r"(v[o+27]), "=r"(v[o+28]), "=r"(v[o+29]), "=r"(v[o+30]), "=r"(v[o+31])
#define WAVEAL_RW32(v, o) \
  "+r"(v[o+0]), "+r"(v[o+1]), "+r"(v[o+2]), "+r"(v[o+3]), "+r"(v[o+4]), "+r"(v[o+5]), "+r"(v[o+6]), "+r"(v[o+7]), \
  "+r"(v[o+8]), "+r"(v[o+9]), "+r"(v[o+10]), "+r"(v[o+11]), "+r"(v[o+12]), "+r"(v[o+13]), "+r"(v[o+14]), "+r"(v[o+15]), \
  "+r"(v[o+16]), "+r"(v[o+17]), "+r"(v[o+18]), "+r"(v[o+19]), "+r"(v[o+20]), "+r"(v[o+21]), "+r"(v[o+22]), "+r"(v[o+23]), \
  "+r"(v[o+24]), "+r"(v[o+25]), "+r"(v[o+26]), "+r"(v[o+27]), "+r"(v[o+28]), "+r"(v[o+29]), "+r"(v[o+30]), "+r"(v[o+31])
#define WAVEAL_IN32(v, o) \
  "r"(v[o+0]), "r"(v[o+1]), "r"(v[o+2]), "r"(v[o+3]), "r"(v[o+4]), "r"(v[o+5]), "r"(v[o+6]), "r"(v[o+7]), \
  "r"(v[o+8]), "r"(v[o+9]), "r"(v[o+10]), "r"(v[o+11]), "r"(v[o+12]), "r"(v[o+13]), "r"(v[o+14]), "r"(v[o+15]), \
  "r"(v[o+16]), "r"(v[o+17]), "r"(v[o+18]), "r"(v[o+19]), "r"(v[o+20]), "r"(v[o+21]), "r"(v[o+22]), "r"(v[o+23]), \
  "r"(v[o+24]), "r"(v[o+25]), "r"(v[o+26]), "r"(v[o+27]), "r"(v[o+28]), "r"(v[o+29]), "r"(v[o+30]), "r"(v[o+31])

// 32 consecutive fp32 columns of this thread's tensor-memory lane -> registers v[o..o+31]
#define WAVEAL_TMEM_LD32(taddr, v, o)                                                            \
  asm volatile(                                                                                  \
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "                  \
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"  \
      : WAVEAL_R32(v, o)                                                                         \
      : "r"(taddr)                                                                               \
      : "memory")
// wait for outstanding tensor-memory loads; the registers are operands so that no use of
// them can be moved above the wait
#define WAVEAL_TMEM_WAIT_LD32(v, o) asm volatile("tcgen05.wait::ld.sync.aligned;" : WAVEAL_RW32(v, o)::"memory")
#define WAVEAL_TMEM_ST32(taddr, v, o)                                                            \
  asm volatile(                                                                                  \
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "                                           \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "                  \
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"         \
      ::WAVEAL_IN32(v, o), "r"(taddr)                                                            \
      : "memory")

// 16 consecutive fp32 columns
#define WAVEAL_TMEM_LD16(taddr, v, o)                                                            \
  asm volatile(                                                                                  \
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"           \
      : "=r"(v[o+0]), "=r"(v[o+1]), "=r"(v[o+2]), "=r"(v[o+3]), "=r"(v[o+4]), "=r"(v[o+5]), "=r"(v[o+6]), "=r"(v[o+7]), \
        "=r"(v[o+8]), "=r"(v[o+9]), "=r"(v[o+10]), "=r"(v[o+11]), "=r"(v[o+12]), "=r"(v[o+13]), "=r"(v[o+14]), "=r"(v[o+15]) \
      : "r"(taddr)                                                                               \
      : "memory")
#define WAVEAL_TMEM_WAIT_LD16(v, o)                                                              \
  asm volatile("tcgen05.wait::ld.sync.aligned;"                                                  \
      : "+r"(v[o+0]), "+r"(v[o+1]), "+r"(v[o+2]), "+r"(v[o+3]), "+r"(v[o+4]), "+r"(v[o+5]), "+r"(v[o+6]), "+r"(v[o+7]), \
        "+r"(v[o+8]), "+r"(v[o+9]), "+r"(v[o+10]), "+r"(v[o+11]), "+r"(v[o+12]), "+r"(v[o+13]), "+r"(v[o+14]), "+r"(v[o+15]) \
      ::"memory")
#define WAVEAL_TMEM_ST16(taddr, v, o)                                                            \
  asm volatile(                                                                                  \
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "                                           \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"                  \
      ::"r"(v[o+0]), "r"(v[o+1]), "r"(v[o+2]), "r"(v[o+3]), "r"(v[o+4]), "r"(v[o+5]), "r"(v[o+6]), "r"(v[o+7]), \
        "r"(v[o+8]), "r"(v[o+9]), "r"(v[o+10]), "r"(v[o+11]), "r"(v[o+12]), "r"(v[o+13]), "r"(v[o+14]), "r"(v[o+15]), \
        "r"(taddr)                                                                               \
      : "memory")

// one 32-byte store (the address must be 32-byte aligned)
__device__ __forceinline__ void st_global_v8(void* ptr, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(ptr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// largest of 32 scores
__device__ __forceinline__ float row_max32(const uint32_t (&sv)[32]) {
  float mx4[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) mx4[i] = __uint_as_float(sv[i]);
#pragma unroll
  for (int c = 4; c < 28; c += 8) {
#pragma unroll
    for (int i = 0; i < 4; ++i) mx4[i] = fmax3(mx4[i], __uint_as_float(sv[c + 2 * i]), __uint_as_float(sv[c + 2 * i + 1]));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) mx4[i] = fmaxf(mx4[i], __uint_as_float(sv[28 + i]));
  return fmaxf(fmax3(mx4[0], mx4[1], mx4[2]), mx4[3]);
}

// shared-memory matrix descriptor, 128-byte swizzle, Blackwell version field
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version
  d |= (uint64_t)2 << 61;   // SWIZZLE_128B
  return d;
}

// instruction descriptor: bf16 x bf16 -> fp32, A K-major, B K-major or MN-major
// (A and B must have the same 16-bit format: an f16 A with a bf16 B is an illegal instruction)
__host__ __device__ constexpr uint32_t make_idesc(int m, int n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

// ------------------------------------------------------------------ kernel

// n: KV tiles of the task (a tile = 128 keys = 128/block consecutive entries of the row's list),
// len: entries of the list, tail_valid: keys of the last tile that exist.
// row2 (64-row query blocks only): a second query block with the very same list, or -1; its rows
// fill the other half of a 128-row product, so the pair costs what one block costs there.  The
// ticket of the second block of a pair carries n = kAbsorbed and is skipped by whoever draws it.
// pick: large calls of 64-row blocks, in the table's first entry: 1 if the call runs in products of 128 rows, 0: of 64 (k_sort_tail).
// Every other entry's is not read.
struct Task { int h, row, lo, n, tail_valid, len, row2, pick; };
constexpr int kAbsorbed = -2;

// tiles, list length and valid keys of the last tile from a list of `len` blocks of `block` keys
// whose last entry is `last`
__host__ __device__ inline void fill_tiles(Task& tk, int len, int block, int last, int n_b, int seq_kv) {
  const int kb = 128 / block;
  tk.len = len;
  tk.n = (len + kb - 1) / kb;
  tk.tail_valid = 128;
  if (len > 0) {
    tk.tail_valid = (len - (tk.n - 1) * kb) * block;
    if ((seq_kv % block) != 0 && last == n_b - 1) tk.tail_valid -= block - seq_kv % block;
  }
}

// (a kernel's parameters travel with every launch: 8 bytes more than these 160 and the tensor maps took the smallest step 0.5 us of host time)
struct AttnParams {
  __nv_bfloat16* O;
  float* lse;
  const int* row_ptr;
  const int* kv_idx;
  const int* row_order;
  int* ws;            // [0] ticket counter, [1] abort flag, [2] number of tasks to redo, [3] ticket counter of
                      // the redo pass, [8 + 2i], [9 + 2i] = (head, query block) of redo entry i
  int redo_pass;      // 0: all tasks by ticket; 1: only the tasks the first pass listed
  int choose;         // first launch of large calls of 64-row blocks: `pick` of the table's first entry says whose they are
  const Task* table;         // task of every ticket of the first pass (k_task_table)
  int direct;         // CTAs that take the ticket of their own number before the table is there (0: none, else the grid)
  long long first_tail;      // tickets before this one are in the caller's order, the rest longest first
  int* dev_status;
  long long o_stride_h, o_stride_t;
  int heads, m_b, n_b, seq_q, seq_kv, interleaved;
  long long total_tasks;
  long long wait_limit;   // cycles a bounded wait may take (kTimeoutCycles; far shorter under the self-test flag)
  int drop_tile;          // self-test: the producer never loads the first K tile of ticket 0
  int no_pairing;         // 64-row blocks: never put two blocks with identical lists into one tile
  float sl2;          // scale * log2(e)
};
static_assert(sizeof(AttnParams) == 160, "parameters of the attention kernels");


// Task of every ticket (head-major or position-major over the planned order), so that the
// persistent CTAs need one load behind a ticket instead of a chain through row_order, the row
// pointers and the index list.
// The inputs are checked on the way (a thread per task, so it costs nothing): an entry of
// row_order outside [0, M_B), a row-pointer pair that is negative, decreasing or beyond the end
// of the index list, or a last index outside [0, N_B) is reported as
// {WAVEAL_ERR_BAD_MASK, site, head, offending value} and the task is given an empty list
// (its output rows become 0) instead of reading out of range.
__device__ __forceinline__ Task make_task(const AttnParams& p, int block_k, int h, int pos) {
  auto report = [&](int site, int value) {
    if (p.dev_status && atomicCAS(p.dev_status, 0, WAVEAL_ERR_BAD_MASK) == 0) {
      p.dev_status[1] = site; p.dev_status[2] = h; p.dev_status[3] = value;
    }
  };
  int row = p.row_order ? p.row_order[(size_t)h * p.m_b + pos] : pos;
  bool bad = false;
  if (row < 0 || row >= p.m_b) { report(31, row); row = pos; bad = true; }
  const long long nnz = p.row_ptr[p.total_tasks];
  const int lo = p.row_ptr[(size_t)h * p.m_b + row], hi = p.row_ptr[(size_t)h * p.m_b + row + 1];
  if (lo < 0 || hi < lo || (long long)hi > nnz) { report(32, lo < 0 ? lo : hi); bad = true; }
  Task tk{};
  tk.h = h; tk.row = row; tk.lo = bad ? 0 : lo; tk.row2 = -1;
  int len = bad ? 0 : hi - lo, last = 0;
  if (len > 0) {
    last = p.kv_idx[hi - 1];
    if (last < 0 || last >= p.n_b) { report(33, last); len = 0; }
  }
  fill_tiles(tk, len, block_k, last, p.n_b, p.seq_kv);
  if (bad) tk.pick = 1;                             // (on its way into the table: takes no part in pairing)
  return tk;
}

__device__ __forceinline__ Task task_of_ticket(const AttnParams& p, int block_k, long long t) {
  const int h = p.interleaved ? (int)(t % p.heads) : (int)(t / p.m_b), pos = p.interleaved ? (int)(t / p.heads) : (int)(t % p.m_b);
  Task tk = make_task(p, block_k, h, pos);
  tk.pick = 0;
  return tk;
}

template <int BLOCK, int D>
struct Geo {
  // A KV tile is always 128 keys wide: one 128-key block, or two 64-key blocks that follow each
  // other in the row's list (their rows land one after the other in the tile, so the MMAs, the
  // softmax and the rings see the same shapes for both block sizes; a list of odd length ends
  // in a half tile whose missing keys are treated like keys beyond the sequence end)
  static constexpr int BQ = BLOCK, BK = 128, KB = 128 / BLOCK;
  static constexpr int SLABS = D / 64;               // 128-byte column slabs of a Q/K/V tile
  static constexpr int Q_BYTES = SLABS * 128 * 128;  // smem reserved for the 128 MMA rows
  static constexpr int TILE_BYTES = SLABS * BK * 128;
  static constexpr int KV_SLAB_BYTES = BK * 128;
  // Q tiles: with two, the next task's is requested while this one's is in use, for a K ring of two stages
  // instead of three (128-row tiles of 8 tiles a task: 16.0k against 16.4k clk; 64-row tiles: 18.5 M against
  // 18.2 M cycles on 8 heads of 1536 rows, their tasks are longer and their rings do the work)
  static constexpr int NQ = KB == 1 ? 2 : 1;
  // O leaves through shared memory: staged in the task's own Q tile, which nobody reads any more, and stored by the copy
  // engine.  64-row blocks have one Q tile, which the next task's Q is loaded into meanwhile; they store from registers.
  static constexpr bool STAGED = NQ == 2;
  static constexpr int NSTAGE_RAW = (200 * 1024 - NQ * Q_BYTES) / TILE_BYTES;
  static constexpr int NSTAGE = NSTAGE_RAW > 8 ? 8 : NSTAGE_RAW;
  static constexpr int NKS = (NSTAGE + 1) / 2;       // K tile ring
  static constexpr int NVS = NSTAGE / 2;             // V tile ring
  static constexpr int NSBUF = 3;                    // S/P buffers in tensor memory
  static constexpr int HC = BK / 2;                  // S columns of a row one softmax thread owns (a row has two owners)
  static constexpr int CH = 32;                      // S columns a softmax thread holds at a time
  static constexpr int NCH = HC / CH;                // such chunks per thread and block
  // chunks of the exponential loop in line: both at head_dim 64 (128x64 blocks 1,229 -> 1,212 clk a tile), one at head_dim 128
  // (both: 1,346 -> 1,368).  In line the kernels spill a few words at the 96 registers there are (28 to 48 bytes stored, 32 to
  // 56 loaded; rolled none), in these figures too; the second launch's, 4 heads of 256 dense rows, rolled and in line: 128x64
  // 2,606 k and 2,508 k cycles, 64x64 1,324 k and 1,294 k
  static constexpr int UNROLL = D == 64 ? NCH : 1;
  static constexpr int LAG = KB == 1 && D == 64 ? 0 : 4;   // pairs of exponentials under way before the first is used
  static constexpr int CO = D / 2;                   // O columns per epilogue thread
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + NQ * Q_BYTES;
  static constexpr int OFF_V = OFF_K + NKS * TILE_BYTES;
  static constexpr int OFF_BAR = OFF_V + NVS * TILE_BYTES;
  static constexpr int N_BAR = 4 + 4 + 2 * NKS + 2 * NVS + 4 * NSBUF + 2 + 2 + 16 + 16 + 8;
  static constexpr int OFF_TASK = OFF_BAR + ((N_BAR * 8 + 15) / 16) * 16;
  static constexpr int OFF_MX = OFF_TASK + 2 * (int)sizeof(Task);
  static constexpr int OFF_MISC = OFF_MX + 4 * 128 * 4 + 2 * 2 * 2 * 128 * 4 + 4 * 4 * 128 * 8;
  static constexpr int SMEM_BYTES = OFF_MISC + 48 + 1024;   // + slack for 1024-byte alignment
  // tensor memory: three S/P buffers of 128 columns, then the output accumulator
  static constexpr uint32_t S_STRIDE = 128, O_COL = 384, TMEM_COLS = 512;
};

struct Ctx {
  uint32_t bar_base;
  volatile int* abort_smem;
  int* ws;
  int* dev_status;
  long long limit;      // cycles a wait may take before the CTA gives up
};

__device__ __noinline__ void signal_abort(const Ctx& c, int site) {
  *c.abort_smem = 1;
  waveal::wait_for_previous_kernel();      // (which clears the flag)
  atomicExch(&c.ws[1], 1);
  if (c.dev_status && atomicCAS(c.dev_status, 0, WAVEAL_ERR_TIMEOUT) == 0) {
    c.dev_status[1] = site;
    c.dev_status[2] = blockIdx.x;
    c.dev_status[3] = threadIdx.x;
  }
}

// bounded wait; false = gave up (this CTA is aborting).  The polling loop is one function for all the
// waits of the kernel: inlined twenty times it cost 3 % of the cycles in instruction fetches (the softmax
// loop and the waits around it have to stay in the schedulers' instruction caches).
__device__ __noinline__ bool mbar_wait_slow(const Ctx& c, uint32_t bar, uint32_t parity, int site) {
  long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*c.abort_smem) return false;
    if (clock64() - t0 > c.limit) { signal_abort(c, site); return false; }
  }
}

__device__ __forceinline__ bool mbar_wait(const Ctx& c, uint32_t bar, uint32_t parity, int site) {
  return mbar_try_wait(bar, parity) || mbar_wait_slow(c, bar, parity, site);
}

// same, with one answer for the whole warp (the roles use warp-collective instructions).  All
// lanes wait: a warp suspended as a whole in try_wait takes no issue slots, which measured
// better than polling and far better than one waiting lane with the rest at the vote.
__device__ __forceinline__ bool warp_wait(const Ctx& c, uint32_t bar, uint32_t parity, int site) {
  return __all_sync(0xffffffffu, mbar_wait(c, bar, parity, site));
}

// One K or V tile of a task into its ring stage (called by a whole warp).  Tile j covers entries
// KB*j .. of the row's list (the last tile of an odd list of 64-key blocks has one block).
// State of the caller: it (tiles loaded so far), armed / parity (per stage: a load is in flight,
// and the parity its barrier completes with), chunk_base / my_idx (32 list entries at a time,
// one per lane).  dropped: self-test of the abort path, the tile is never requested.
template <class G, int BLOCK, bool IS_K>
__device__ __forceinline__ bool load_kv_tile(const Ctx& ctx, const AttnParams& p, const Task& tk, bool dropped, int j,
                                             int lane, uint32_t sbase, uint32_t bar_full0, uint32_t bar_empty0,
                                             const CUtensorMap* tm, const CUtensorMap* tm2, uint32_t& it,
                                             uint32_t& armed, uint32_t& parity, int& chunk_base, int& my_idx) {
  constexpr uint32_t NST = IS_K ? G::NKS : G::NVS;
  auto entry = [&](int q) -> int {
    if (q < chunk_base || q >= chunk_base + 32) {
      chunk_base = q & ~31;
      const int e = chunk_base + lane;
      my_idx = e < tk.len ? p.kv_idx[tk.lo + e] : 0;
    }
    int blk = __shfl_sync(0xffffffffu, my_idx, q - chunk_base);
    if (blk < 0 || blk >= p.n_b) {                   // malformed list: report it and stay in range
      if (lane == 0 && p.dev_status && atomicCAS(p.dev_status, 0, WAVEAL_ERR_BAD_MASK) == 0) {
        p.dev_status[1] = 30; p.dev_status[2] = tk.h; p.dev_status[3] = blk;
      }
      blk = 0;
    }
    return blk;
  };
  const int nblk = G::KB == 1 ? 1 : min(G::KB, tk.len - G::KB * j);
  int blk[G::KB];
#pragma unroll
  for (int e = 0; e < G::KB; ++e) blk[e] = e < nblk ? entry(G::KB * j + e) : 0;
  const uint32_t st = it % NST, sph = (it / NST) & 1;
  const uint32_t b_full = bar_full0 + 8u * st, b_empty = bar_empty0 + 8u * st;
  if (!warp_wait(ctx, b_empty, sph ^ 1, IS_K ? 3 : 4)) return false;
  ++it;
  if (dropped) return true;
  // one lane per box: lane e*SLABS + s requests slab s of block e
  if (lane == 0) mbar_expect_tx(b_full, (uint32_t)nblk * G::SLABS * BLOCK * 128);
  __syncwarp();
  const uint32_t dst = sbase + (IS_K ? G::OFF_K : G::OFF_V) + st * G::TILE_BYTES;
  const int e = lane / G::SLABS, sl = lane % G::SLABS;
  // two 64-key blocks that follow each other in memory come as one box of 128 rows per slab
  const bool joined = G::KB == 2 && nblk == 2 && blk[G::KB - 1] == blk[0] + 1;
  if (joined) {
    if (e == 0) tma_load_3d(dst + sl * G::KV_SLAB_BYTES, tm2, sl * 64, blk[0] * BLOCK, tk.h, b_full);
  } else {
    int my_blk = blk[0];
#pragma unroll
    for (int i = 1; i < G::KB; ++i) if (e == i) my_blk = blk[i];
    if (e < nblk) tma_load_3d(dst + sl * G::KV_SLAB_BYTES + e * BLOCK * 128, tm, sl * 64, my_blk * BLOCK, tk.h, b_full);
  }
  armed |= 1u << st;
  parity = (parity & ~(1u << st)) | (sph << st);
  return true;
}

// scores of a thread's own columns of a tile from column `valid` on become -inf (in tensor memory and out of
// line, so that the two loops over the scores carry no code for the rare ragged tile)
template <int NCH>
__device__ __noinline__ void mask_scores(uint32_t s_addr, int valid) {
#pragma unroll 1
  for (int ch = 0; ch < NCH; ++ch) {
    uint32_t sv[32];
    WAVEAL_TMEM_LD32(s_addr + ch * 32, sv, 0);
    WAVEAL_TMEM_WAIT_LD32(sv, 0);
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (ch * 32 + c >= valid) sv[c] = __float_as_uint(-INFINITY);
    WAVEAL_TMEM_ST32(s_addr + ch * 32, sv, 0);
  }
  tc_wait_st();
}

// a task for the second launch, unless another warp has listed it already; the blocks of a pair are computed again one by one
// (in line for 128-row blocks: 521 k -> 506 k cycles on 5 heads of 256 rows, a call there makes the compiler spill; out of line
// for 64-row blocks in products of 128 rows, 18.75 M -> 18.35 M on 8 heads of 1536 rows)
__device__ __forceinline__ void list_task(int* ws, int* listed, int task_no, int h, int row, int row2) {
  if (atomicExch(listed, task_no) == task_no) return;
  waveal::wait_for_previous_kernel();      // (which clears the count: a first task may end before it)
  const int e = atomicAdd(&ws[2], row2 >= 0 ? 2 : 1);
  ws[8 + 2 * e] = h;
  ws[9 + 2 * e] = row;
  if (row2 >= 0) { ws[10 + 2 * e] = h; ws[11 + 2 * e] = row2; }
}
__device__ __noinline__ void list_task_call(int* ws, int* listed, int task_no, int h, int row, int row2) {
  list_task(ws, listed, task_no, h, row, row2);
}

// First launch of 64-row blocks: this kernel does small calls and, where k_sort_tail picks it, large ones, all others are
// k_bsattn_fwd_rows64's.  It sums the rows by tile mod 4 as that one does, so that a head has the same bits in every call.
template <int BLOCK, int D, bool FAST>
__global__ void __launch_bounds__(kThreads, 1)
k_bsattn_fwd(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
             const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmK2,
             const __grid_constant__ CUtensorMap tmV2, const __grid_constant__ CUtensorMap tmO, const AttnParams p) {
  // tmK2 / tmV2: the same K and V with boxes of 128 rows, used by the 64-key-block kernels when the
  // two blocks of a tile lie next to each other in memory (for 128-key blocks they equal tmK / tmV).
  // tmO: O in boxes of 32 rows and half of head_dim, what a warp stores (128-row blocks only)
  using G = Geo<BLOCK, D>;
  constexpr bool MOD4 = FAST && BLOCK == 64;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // provably warp-uniform role index
  waveal::let_next_kernel_start();
  if (p.redo_pass) waveal::wait_for_previous_kernel();

  // second pass with nothing listed (or after an abort): leave before anything is set up
  if (p.redo_pass && (p.ws[2] == 0 || p.ws[1] != 0)) return;
  // a call that k_bsattn_fwd_rows64 has done
  if (MOD4 && p.choose) {
    waveal::wait_for_previous_kernel();
    if (p.table->pick == 0 || p.ws[1] != 0) return;
  }

  const uint32_t bar0 = sbase + G::OFF_BAR;
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  constexpr int B_TASK_FULL = 0, B_TASK_EMPTY = 2, B_Q_FULL = 4, B_Q_EMPTY = 6, B_K_FULL = 8,
                B_K_EMPTY = B_K_FULL + G::NKS, B_V_FULL = B_K_EMPTY + G::NKS, B_V_EMPTY = B_V_FULL + G::NVS,
                B_S_FULL = B_V_EMPTY + G::NVS, B_P_FULL = B_S_FULL + G::NSBUF, B_S_FREE = B_P_FULL + 2 * G::NSBUF,
                B_O_FULL = B_S_FREE + G::NSBUF, B_O_FREE = B_O_FULL + 1, B_FINAL = B_O_FREE + 1, B_MX = B_FINAL + 2,
                B_EX = B_MX + 16, B_HX = B_EX + 16;
  static_assert(B_HX + 8 <= G::N_BAR, "barrier count");
  Task* tasks = reinterpret_cast<Task*>(smem + G::OFF_TASK);
  volatile float* mpub = reinterpret_cast<volatile float*>(smem + G::OFF_MX);   // [tile count mod 4][128] reference max after a tile; FAST: [tile count mod 4][column half][128], over mhalf too
  volatile float* mhalf = reinterpret_cast<volatile float*>(smem + G::OFF_MX + 4 * 128 * 4);   // [use parity][team][column half][128] max of a half row
  float2* ex = reinterpret_cast<float2*>(smem + G::OFF_MX + 4 * 128 * 4 + 2 * 2 * 2 * 128 * 4);    // [task mod 4][role*2+half][128] (reference, sum); role 0: the team of the task's first tile
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + G::OFF_MISC);
  volatile int* abort_smem = reinterpret_cast<volatile int*>(smem + G::OFF_MISC + 4);
  // by task mod 4: number (from 1) of the last task that a tile wants computed again, and of the last one listed for it
  volatile int* redo_flag = reinterpret_cast<volatile int*>(smem + G::OFF_MISC + 8);
  int* redo_listed = reinterpret_cast<int*>(smem + G::OFF_MISC + 24);
  Ctx ctx{bar0, abort_smem, p.ws, p.dev_status, p.wait_limit};

  if (tid == 0) {
    // a task is read by the V loader, the two MMA issuers and the sixteen softmax warps
    for (int i = 0; i < 2; ++i) { mbar_init(BAR(B_TASK_FULL + i), 1); mbar_init(BAR(B_TASK_EMPTY + i), 19); }
    // a Q tile is free when the last Q K^T has read it and, where O is staged in it, its eight warps' stores have
    for (int i = 0; i < 2; ++i) { mbar_init(BAR(B_Q_FULL + i), 1); mbar_init(BAR(B_Q_EMPTY + i), G::STAGED ? 9 : 1); }
    for (int i = 0; i < G::NKS; ++i) { mbar_init(BAR(B_K_FULL + i), 1); mbar_init(BAR(B_K_EMPTY + i), 1); }
    for (int i = 0; i < G::NVS; ++i) { mbar_init(BAR(B_V_FULL + i), 1); mbar_init(BAR(B_V_EMPTY + i), 1); }
    for (int i = 0; i < G::NSBUF; ++i) {
      mbar_init(BAR(B_S_FULL + i), 1);
      mbar_init(BAR(B_P_FULL + 2 * i), 4);      // one per half of P (the four warps that own that half in the block's team)
      mbar_init(BAR(B_P_FULL + 2 * i + 1), 4);
      mbar_init(BAR(B_S_FREE + i), 1);
    }
    mbar_init(BAR(B_O_FULL), 1);
    mbar_init(BAR(B_O_FREE), 8);              // the team that runs the epilogue
    mbar_init(BAR(B_FINAL), 1);
    mbar_init(BAR(B_FINAL + 1), 1);
    for (int i = 0; i < 16; ++i) mbar_init(BAR(B_MX + i), FAST ? 2 : 1);   // (lane quadrant, tile count mod 4)
    for (int i = 0; i < 16; ++i) mbar_init(BAR(B_EX + i), 4);   // (task mod 4, lane quadrant): its four warps, once per task
    for (int i = 0; i < 8; ++i) mbar_init(BAR(B_HX + i), 2);    // the two owners of a row (team, quadrant), once per max
    *abort_smem = 0;
    for (int i = 0; i < 4; ++i) { redo_flag[i] = 0; redo_listed[i] = 0; }
    fence_mbar_init();
    fence_proxy_async();
  }
  // the MMA reads all 128 rows of the Q region even when a query block has 64 rows: clear it once
  for (int i = tid; i < G::NQ * G::Q_BYTES / 16; i += kThreads) reinterpret_cast<uint4*>(smem + G::OFF_Q)[i] = make_uint4(0, 0, 0, 0);
  fence_proxy_async();
  if (warp == kPvWarp) {
    tmem_alloc(smem_u32(tmem_holder), G::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_holder, 0);
  // Tickets, table and counters are the work of the kernel before this one.  It was launched the ordinary way, so all that
  // came before it (the lists, Q, K, V) is there by now: a CTA with a first task of its own (p.direct) begins, and whoever
  // touches the counters or the table waits there.
  if (!p.direct) waveal::wait_for_previous_kernel();
  // (without a first task of its own that kernel's time is not this launch's; with one the count starts here, and what the
  // CTA still waits for that kernel is in it)
  const long long t_start = clock64();

  // Every role walks the same sequence of tasks (query blocks) and, inside a task, of KV blocks;
  // block number g (counted over the CTA's whole life) uses S buffer g mod 3, K stage g mod NKS
  // and V stage g mod NVS, so no role needs to be told where a tile or a buffer is.
  if (warp == kProducerWarp) {
    // ============================================================== producer
    if (lane == 0) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmK2); prefetch_tmap(&tmV2); if (G::STAGED) prefetch_tmap(&tmO); }
    uint32_t task_it = 0, q_it = 0, k_it = 0;
    int n_tiles = 0, n_pairs = 0;        // words 7 and 6 of the workspace: KV tiles (128 rows x 128 keys) and shared tiles this call ran
    bool ok = true;
    uint32_t k_armed = 0, k_parity = 0;   // per stage: parity of the last load armed on it
    uint32_t q_armed = 0, q_parity = 0;
    // the next task: a ticket from the global counter and the task it stands for (n = -1: none left)
    auto draw = [&](long long& t_out) -> Task {
      if (p.direct) waveal::wait_for_previous_kernel();
      for (;;) {
        long long t = 0, n_tasks = p.total_tasks;
        if (lane == 0) {
          if (p.redo_pass) n_tasks = min((long long)p.ws[2], p.total_tasks);   // written by the first pass
          // (volatile: another SM raises the flag while this kernel runs; a cached copy would hide it)
          t = (*reinterpret_cast<volatile int*>(&p.ws[1]) != 0) ? n_tasks
                                                               : (long long)(unsigned)atomicAdd(&p.ws[p.redo_pass ? 3 : 0], 1);
        }
        t = __shfl_sync(0xffffffffu, t, 0);
        n_tasks = __shfl_sync(0xffffffffu, n_tasks, 0);
        t_out = t;
        Task tk{};
        if (t >= n_tasks) {
          tk.n = -1;
        } else if (!p.redo_pass) {
          // one 32-byte load behind the ticket instead of a chain through three lists
          const uint4* e = reinterpret_cast<const uint4*>(p.table + t);
          const uint4 a = e[0], b = e[1];
          tk.h = (int)a.x; tk.row = (int)a.y; tk.lo = (int)a.z; tk.n = (int)a.w; tk.tail_valid = (int)b.x; tk.len = (int)b.y;
          tk.row2 = (int)b.z;
          if (tk.n == kAbsorbed) continue;          // second block of a pair: computed with its partner
        } else {
          int h = p.ws[8 + 2 * t], row = p.ws[9 + 2 * t];
          if (h < 0 || h >= p.heads) h = 0;
          if (row < 0 || row >= p.m_b) row = 0;
          int lo = p.row_ptr[(size_t)h * p.m_b + row], hi = p.row_ptr[(size_t)h * p.m_b + row + 1];
          tk.h = h; tk.row = row; tk.lo = lo; tk.row2 = -1;
          fill_tiles(tk, max(hi - lo, 0), BLOCK, hi > lo ? p.kv_idx[hi - 1] : 0, p.n_b, p.seq_kv);
        }
        return tk;
      }
    };
    // The ticket of the next task is drawn a few tiles before the current task's last loads are
    // requested, while this warp would wait for a ring stage anyway: the round trips of the
    // counter and of the table entry (~2,000 cycles) then no longer stand between the end of a
    // task and the request for the next Q tile.
    constexpr int kDrawAhead = 3;
    long long t = 0, t_next = blockIdx.x;
    Task tk_next;
    if (FAST && G::KB == 1 && p.direct) tk_next = task_of_ticket(p, BLOCK, t_next);
    else tk_next = draw(t_next);
    while (ok) {
      Task tk = tk_next;
      t = t_next;
      bool drawn = false;
      const uint32_t slot = task_it & 1, ph = (task_it >> 1) & 1;
      ok = warp_wait(ctx, BAR(B_TASK_EMPTY + slot), ph ^ 1, 1);
      if (!ok) break;
      if (lane == 0) {
        tasks[slot] = tk;
        mbar_arrive(BAR(B_TASK_FULL + slot));
      }
      ++task_it;
      if (tk.n < 0) break;
      if (tk.n <= kDrawAhead) { tk_next = draw(t_next); drawn = true; }
      if (tk.n == 0) continue;
      n_tiles += tk.n;
      n_pairs += G::KB == 2 && tk.row2 >= 0;
      // Q tile
      const uint32_t qb = G::NQ == 2 ? q_it & 1 : 0, q_ph = (G::NQ == 2 ? q_it >> 1 : q_it) & 1, q_smem = sbase + G::OFF_Q + qb * G::Q_BYTES;
      ok = warp_wait(ctx, BAR(B_Q_EMPTY + qb), q_ph ^ 1, 2);
      if (!ok) break;
      if (lane == 0) {
        const bool two = G::KB == 2 && tk.row2 >= 0;
        mbar_expect_tx(BAR(B_Q_FULL + qb), (two ? 2 : 1) * G::SLABS * G::BQ * 128);
#pragma unroll
        for (int s = 0; s < G::SLABS; ++s)
          tma_load_3d(q_smem + s * 128 * 128, &tmQ, s * 64, tk.row * G::BQ, tk.h, BAR(B_Q_FULL + qb));
        if (two) {
          // the partner's 64 rows go to rows 64..127 of the tile
#pragma unroll
          for (int s = 0; s < G::SLABS; ++s)
            tma_load_3d(q_smem + s * 128 * 128 + 64 * 128, &tmQ, s * 64, tk.row2 * G::BQ, tk.h, BAR(B_Q_FULL + qb));
        }
      }
      q_armed |= 1u << qb; q_parity = (q_parity & ~(1u << qb)) | q_ph << qb;
      ++q_it;
      int chunk_base = -64, my_idx = 0;
      // all K tiles of the task, as fast as the ring takes them
      for (int j = 0; j < tk.n && ok; ++j) {
        if (!drawn && j >= tk.n - kDrawAhead) { tk_next = draw(t_next); drawn = true; }
        ok = load_kv_tile<G, BLOCK, true>(ctx, p, tk, p.drop_tile && t == 0 && j == 0, j, lane, sbase, BAR(B_K_FULL),
                                          BAR(B_K_EMPTY), &tmK, &tmK2, k_it, k_armed, k_parity, chunk_base, my_idx);
      }
    }
    if (p.direct) waveal::wait_for_previous_kernel();       // (after an abort: the counters below are cleared by it)
    if (lane == 0 && !p.redo_pass) {
      if (n_tiles) atomicAdd(&p.ws[7], n_tiles);
      if (n_pairs) atomicAdd(&p.ws[6], n_pairs);
    }
    if (*abort_smem) {
      // leave no bulk copy in flight into this CTA's shared memory (bounded)
      for (int st = 0; st < G::NKS; ++st)
        if (k_armed & (1u << st)) {
          long long t0 = clock64();
          while (!mbar_try_wait(BAR(B_K_FULL + st), (k_parity >> st) & 1) && clock64() - t0 < p.wait_limit / 4) {}
        }
      for (int st = 0; st < G::NQ; ++st)
        if (q_armed & (1u << st)) {
          long long t0 = clock64();
          while (!mbar_try_wait(BAR(B_Q_FULL + st), (q_parity >> st) & 1) && clock64() - t0 < p.wait_limit / 4) {}
        }
    }
  } else if (warp == kVLoadWarp) {
    // ============================================================== V tile loader
    uint32_t task_slot = 0, task_ph = 0, v_it = 0, v_armed = 0, v_parity = 0;
    bool ok = true;
    while (ok) {
      ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
      if (!ok) break;
      const Task tk = tasks[task_slot];
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
      task_slot ^= 1;
      task_ph ^= (task_slot == 0);
      if (tk.n < 0) break;
      int chunk_base = -64, my_idx = 0;
      for (int j = 0; j < tk.n && ok; ++j)
        ok = load_kv_tile<G, BLOCK, false>(ctx, p, tk, false, j, lane, sbase, BAR(B_V_FULL), BAR(B_V_EMPTY), &tmV, &tmV2,
                                           v_it, v_armed, v_parity, chunk_base, my_idx);
    }
    if (*abort_smem) {
      // leave no bulk copy in flight into this CTA's shared memory (bounded)
      for (int st = 0; st < G::NVS; ++st)
        if (v_armed & (1u << st)) {
          long long t0 = clock64();
          while (!mbar_try_wait(BAR(B_V_FULL + st), (v_parity >> st) & 1) && clock64() - t0 < p.wait_limit / 4) {}
        }
    }
  } else if (warp == kQkWarp) {
    // ============================================================== MMA issuer 1: S = Q K^T
    // Two warps issue the MMAs, one per product: the bookkeeping of each (barrier waits, ring
    // arithmetic, descriptor set-up: a few hundred cycles of dependent scalar work per block)
    // then runs while the other's MMAs execute, and the tensor pipe is not left waiting for
    // it.  MMAs of different threads are ordered through completion barriers only.
    // Every operand of a tcgen05 instruction stays warp-uniform in the compiler's eyes
    // (shuffle-broadcast values, compare-and-reset ring positions).
    constexpr uint32_t IDESC_QK = make_idesc(128, G::BK, false);
    uint32_t task_slot = 0, task_ph = 0, q_it = 0, k_st = 0, k_ph = 0, sb = 0, free_bits = 0, first_uses = G::NSBUF;
    const uint64_t qdesc0 = make_desc(sbase + G::OFF_Q, 16, 1024);
    const uint64_t kdesc0 = make_desc(sbase + G::OFF_K, 16, 1024);
    bool ok = true;
    while (ok) {
      ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
      if (!ok) break;
      const int n = __shfl_sync(0xffffffffu, tasks[task_slot].n, 0);
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
      task_slot ^= 1;
      task_ph ^= (task_slot == 0);
      if (n < 0) break;
      if (n == 0) continue;
      const uint32_t qb = G::NQ == 2 ? q_it & 1 : 0;
      ok = warp_wait(ctx, BAR(B_Q_FULL + qb), (G::NQ == 2 ? q_it >> 1 : q_it) & 1, 11);
      if (!ok) break;
      ++q_it;
      const uint64_t qdesc = qdesc0 + (uint64_t)(qb * (uint32_t)(G::Q_BYTES >> 4));
      for (int j = 0; j < n && ok; ++j) {
        ok = warp_wait(ctx, BAR(B_K_FULL + k_st), k_ph, 12);
        if (!ok) break;
        // S[sb] also holds the P tile of the block that used it last: wait until that block's
        // P V has completed (its commit is phase number uses-1 of the buffer's barrier)
        if (first_uses > 0) {
          --first_uses;
        } else {
          ok = warp_wait(ctx, BAR(B_S_FREE + sb), ((free_bits >> sb) & 1u) ^ 1u, 13);
          if (!ok) break;
        }
        free_bits ^= 1u << sb;
        tc_fence_after();
        {
          // descriptors differ from the per-kernel bases only in the 14-bit address field
          const uint64_t kd = kdesc0 + (uint64_t)(k_st * (uint32_t)(G::TILE_BYTES >> 4));
          const uint32_t d_s = tmem_base + sb * G::S_STRIDE;
#pragma unroll
          for (int s = 0; s < G::SLABS; ++s)
            umma4_bf16<BLOCK == 128>(d_s, qdesc + (uint64_t)((s * 128 * 128) >> 4), kd + (uint64_t)((s * G::KV_SLAB_BYTES) >> 4), IDESC_QK, s);
          tc_commit(BAR(B_K_EMPTY + k_st));
          tc_commit(BAR(B_S_FULL + sb));
          if (j == n - 1) tc_commit(BAR(B_Q_EMPTY + qb));
        }
        if (++k_st == (uint32_t)G::NKS) { k_st = 0; k_ph ^= 1; }
        if (++sb == (uint32_t)G::NSBUF) sb = 0;
      }
    }
    // none of this thread's MMAs is still running when tensor memory is released (in a regular
    // run the last P V already depends on all of them; after an abort nothing else orders them)
    tc_commit(BAR(B_FINAL + 1));
    __syncwarp();
    {
      long long t0 = clock64();
      while (!mbar_try_wait(BAR(B_FINAL + 1), 0) && clock64() - t0 < p.wait_limit / 4) {}
    }
  } else if (warp == kPvWarp) {
    // ============================================================== MMA issuer 2: O += P V
    constexpr uint32_t IDESC_PV = make_idesc(128, D, true);
    uint32_t task_slot = 0, task_ph = 0, o_ph = 1, v_st = 0, v_ph = 0, sb = 0, p_phase = 0;
    const uint64_t vdesc0 = make_desc(sbase + G::OFF_V, G::KV_SLAB_BYTES, 1024);
    bool ok = true;
    while (ok) {
      ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
      if (!ok) break;
      const int n = __shfl_sync(0xffffffffu, tasks[task_slot].n, 0);
      const bool half_tail = __shfl_sync(0xffffffffu, tasks[task_slot].tail_valid, 0) <= 64;
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
      task_slot ^= 1;
      task_ph ^= (task_slot == 0);
      if (n < 0) break;
      if (n == 0) continue;
      // the output accumulator of the previous task has been read by the epilogue
      ok = warp_wait(ctx, BAR(B_O_FREE), o_ph, 16);
      if (!ok) break;
      o_ph ^= 1;
      for (int j = 0; j < n && ok; ++j) {
        // P_j arrives in two halves (the first and the second half of the block's keys), each
        // with its own barrier: the MMAs on the first half run while the softmax team is still
        // computing the second
        const uint64_t vd = vdesc0 + (uint64_t)(v_st * (uint32_t)(G::TILE_BYTES >> 4));
        const uint32_t pbase = tmem_base + sb * G::S_STRIDE;
        const uint32_t d_o = tmem_base + G::O_COL;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t pb = sb * 2 + h;
          ok = warp_wait(ctx, BAR(B_P_FULL + pb), (p_phase >> pb) & 1u, 14);
          if (!ok) break;
          p_phase ^= 1u << pb;
          if (h == 0) {
            ok = warp_wait(ctx, BAR(B_V_FULL + v_st), v_ph, 15);
            if (!ok) break;
          }
          tc_fence_after();
          // (the second half of a half tile has no keys: its V rows were never loaded)
          if (G::KB == 2 && h == 1 && j == n - 1 && half_tail) continue;
          // V tile as the N x K operand with N (head_dim) contiguous: 8 keys per 1024-byte
          // group along K (16 keys = 2048 bytes per MMA), next 64 columns of head_dim one slab further
#pragma unroll
          for (int kk = 0; kk < G::BK / 32; ++kk) {
            const int k = h * (G::BK / 32) + kk;
            // P of key half h lies over the first columns of that half's own S columns
            umma_bf16_ts(d_o, pbase + h * G::HC + kk * 8, vd + (uint64_t)((k * 16 * 128) >> 4), IDESC_PV, (j > 0 || k > 0) ? 1u : 0u);
          }
        }
        if (!ok) break;
        {
          tc_commit(BAR(B_V_EMPTY + v_st));
          tc_commit(BAR(B_S_FREE + sb));
          if (j == n - 1) tc_commit(BAR(B_O_FULL));
        }
        if (++v_st == (uint32_t)G::NVS) { v_st = 0; v_ph ^= 1; }
        if (++sb == (uint32_t)G::NSBUF) sb = 0;
      }
    }
    // every MMA has completed before tensor memory is released: the last P V depends on all
    // the Q K^T products through the softmax warps
    tc_commit(BAR(B_FINAL));
    __syncwarp();
    {
      long long t0 = clock64();
      while (!mbar_try_wait(BAR(B_FINAL), 0) && clock64() - t0 < p.wait_limit / 4) {}
    }
  } else {
    // ============================================================== softmax / epilogue
    // Sixteen warps: two teams share the KV tiles of a task (which tile is whose: below), and
    // inside a team a row of S has two owners, one per half of its columns (a warp can reach
    // only the 32 tensor-memory lanes of its quadrant, so the two owners of a row sit in warps
    // four apart).  Four softmax warps per scheduler instead of two: the loop is bound by
    // instruction issue and latency, and twice the warps hide twice the latency.  Each owner
    // keeps the sum of its own columns; P of a column half is written over the first columns of
    // that half's own S columns and released with its own barrier.  Both teams accumulate into the
    // same O, so they need the same reference max of a row.  First launch: the two owners of the row in
    // the task's first tile leave the maxima of their halves in shared memory, and they and the
    // other team, at its first tile, wait at one mbarrier (a lane quadrant's, four slots).  Second launch:
    // the two owners of a row exchange their maxima in every tile, and the team of a tile leaves the
    // running reference for that of the next (an mbarrier per lane quadrant and tile count mod 4).
    // The epilogue adds the four partial sums of a row.
    const int sw = warp - kSoftmaxWarp0;       // 0..15
    const int quad = warp & 3;                 // tensor-memory lane quadrant this warp may access
    const int team = (sw >> 2) & 1;            // owns every second tile (by the tile's number over the CTA's life, or as kTwoFirst says)
    const int half = sw >> 3;                  // column half of S; epilogue: the same half of the O columns
    const int r = quad * 32 + lane;            // row of the 128-row MMA tile
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t o_row = tmem_base + lane_addr + G::O_COL;
    // Tiles alternate between the teams across the boundary of two tasks: the team of a task's last tile
    // runs its epilogue (waits for the last P V, reads O, stores it) while the other one is already at the
    // next task's first tile, whose max pass, exponentials and P would otherwise come after all of that.
    // (With both teams in the epilogue a task cost ~6,000 clk beyond its tiles.)  What a team leaves for
    // the other (running reference, partial sums, redo flag) therefore lies in four slots each: three S
    // buffers let a team run ahead of the other's epilogue by two of its own tiles, hence two tasks.
    uint32_t task_it = 0, o_it = 0, mx_phase = 0, hx_it = 0;
    // kTwoFirst: the team that is not in the epilogue of the task before takes the first two tiles, then they alternate: 0 1 3 5 ...
    // and 2 4 6 ...  By turns from the first tile on, the second one's P waits for the end of that epilogue, and the P V of
    // the third, long ready, for it.  First launch of 128-row blocks at head_dim 64: tasks of 16 / 24 / 256 tiles 1,292 -> 1,266 /
    // 1,246 -> 1,228 / 1,160 -> 1,151 clk a tile.  (At head_dim 128 tasks of 17 tiles gained 2 %, but every form of it made the
    // compiler's code for the loop over the tiles slower, 1,366 -> 1,404 clk a tile of long tasks.  The second launch hands a
    // reference on from tile to tile.)
    constexpr bool kTwoFirst = FAST && D == 64 && G::KB == 1;
    uint32_t g0 = 0;                           // tiles before this task
    int first_team = 0;                        // kTwoFirst: the team of the task's first tile
    uint32_t sb = (uint32_t)team, s_ph = 0;    // S buffer of this team's next tile and the parity of that use
    auto next_buffer = [&](int j) { sb += kTwoFirst && j == 0 ? 1 : 2; if (sb >= (uint32_t)G::NSBUF) { sb -= (uint32_t)G::NSBUF; s_ph ^= 1; } };
    bool ok = true, storing = false;           // storing: the stores of this warp's last epilogue may still read the Q tile
    while (ok) {
      const uint32_t slot = task_it & 1, ph = (task_it >> 1) & 1;
      ok = warp_wait(ctx, BAR(B_TASK_FULL + slot), ph, 20);
      if (!ok) break;
      const Task tk = tasks[slot];
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + slot));
      // (here and not behind the stores: what came after them, the second launch's list, does not wait for the copy engine.  The
      // next task is mostly published by then, so lane 0 waits for the rest of its reads.  It is published before the
      // one whose Q needs this tile, so nobody waits for this in a circle)
      if (G::STAGED && storing) {
        if (lane == 0) { bulk_wait_read(); mbar_arrive(BAR(B_Q_EMPTY + ((o_it - 1) & 1))); }
        storing = false;
      }
      float2* exb = ex + (o_it & 3) * 512;
      const int task_no = (int)o_it + 1;
      const uint32_t rslot = o_it & 3, ex_bar = B_EX + quad + 4 * (o_it & 3), ex_ph = (o_it >> 2) & 1;
      ++task_it;
      if (tk.n < 0) break;
      // rows 64..127 of the tile belong to the partner block of a pair (64-row blocks only)
      const bool second = G::KB == 2 && r >= G::BQ;
      const long long q_tok = second ? (long long)tk.row2 * G::BQ + (r - G::BQ) : (long long)tk.row * G::BQ + r;
      const bool row_live = (second ? tk.row2 >= 0 : r < G::BQ) && q_tok < p.seq_q;
      // rows 64..127 of a tile that no second block shares hold nothing: their warps only keep
      // the barriers of the tile going (each output row of an MMA depends on its own row of S / P alone)
      const bool idle = G::KB == 2 && quad >= 2 && tk.row2 < 0;
      __nv_bfloat16* o_ptr = p.O + (size_t)tk.h * p.o_stride_h + (size_t)q_tok * p.o_stride_t + half * G::CO;
      if (tk.n == 0) {
        if (row_live && team == 0) {
#pragma unroll
          for (int c = 0; c < G::CO / 8; ++c) reinterpret_cast<uint4*>(o_ptr)[c] = make_uint4(0, 0, 0, 0);
          if (p.lse && half == 0) p.lse[(size_t)tk.h * p.seq_q + q_tok] = -INFINITY;
        }
        continue;
      }
      // l_run: sum over this thread's columns of this team's blocks, relative to the reference m_ref
      // (MOD4: l_other that of the tiles two further or before)
      float m_ref = -INFINITY, l_run = 0.f, l_other = 0.f;
      const int last = tk.n - 1;
      const int role = kTwoFirst ? (team == first_team ? 0 : 1) : (int)((g0 ^ (uint32_t)team) & 1u);       // 0: has the first tile
      const int j0 = kTwoFirst ? 2 * role : role;
      if (kTwoFirst) { sb = (g0 + (uint32_t)j0) % G::NSBUF; s_ph = ((g0 + (uint32_t)j0) / G::NSBUF) & 1u; }
      for (int j = j0; j < tk.n; j += kTwoFirst && j == 0 ? 1 : 2) {
        const uint32_t g = g0 + (uint32_t)j;
        ok = warp_wait(ctx, BAR(B_S_FULL + sb), s_ph, 21);
        if (!ok) break;
        if (idle) {
          if (lane == 0) mbar_arrive(BAR(B_P_FULL + sb * 2 + half));
          next_buffer(j);
          continue;
        }
        {
          tc_fence_after();
          const uint32_t s_addr = tmem_base + lane_addr + sb * G::S_STRIDE + half * G::HC;
          const bool ragged = j == last && tk.tail_valid < G::BK;
          if (ragged) mask_scores<G::NCH>(s_addr, tk.tail_valid - half * G::HC);   // keys beyond seq_kv (ragged last block) do not exist
          // ---- pass 1: row max (the values are loaded again for the exponentials: a second
          // tensor-memory load is cheaper than keeping them in registers)
          // In the first pass over the tasks (FAST) only the first tile of a task takes a max; both teams keep it as
          // their reference.  Any reference gives the same softmax as long as nothing overflows, so all tiles watch the
          // sum of the exponentials they produce: if it ever reaches 2^60 the task is put on a list and computed again
          // by the second launch, which takes the max of every tile (the rule of the paper's online softmax).
          // One tile and one meeting of all who need its max, and nothing of the rule for a max that grows in this kernel
          // (no rescale of O, no hand-over from tile to tile): against the code with both in it 128x128 tasks of 38 / 256
          // tiles 1,520 -> 1,492 / 1,385 -> 1,363 clk a tile, 128x64 1,311 -> 1,272.  A max over 32 keys only
          // would save another 1-4 %, but scores that spread by 40 nats inside a tile then need the second launch.
          float m_new;
          if constexpr (FAST) {
            // The two owners of the row in the first tile leave the largest of their own scores; they and, at its first tile,
            // the other team take the larger of the two.  (Slot and barrier by tile count mod 4: a later task's first tile
            // that uses the slot again waits for its S buffer, hence for the P V of this task's second tile.  kTwoFirst, where the other
            // team comes to it in the task's third tile: by task count mod 4, so that the first tile that uses the slot again lies
            // six tiles or more behind this one, four if the task has no third tile; it waits for the P V of the tile
            // three before it.)
            if (kTwoFirst ? j == j0 : j <= 1) {
              const uint32_t mx = kTwoFirst ? o_it & 3 : (g - (uint32_t)j) & 3;
              volatile float* mh = mpub + mx * 256;
              if (j == 0) {
                float mloc = -INFINITY;
#pragma unroll 1
                for (int ch = 0; ch < G::NCH; ++ch) {
                  uint32_t sv[G::CH];
                  WAVEAL_TMEM_LD32(s_addr + ch * G::CH, sv, 0);
                  WAVEAL_TMEM_WAIT_LD32(sv, 0);
                  mloc = fmaxf(mloc, row_max32(sv));
                }
                mh[half * 128 + r] = mloc;
                __syncwarp();
                if (lane == 0) mbar_arrive(BAR(B_MX + quad * 4 + mx));
              }
              ok = warp_wait(ctx, BAR(B_MX + quad * 4 + mx), (mx_phase >> mx) & 1u, 24);
              if (!ok) break;
              mx_phase ^= 1u << mx;
              m_ref = fmaxf(mh[r], mh[128 + r]) * p.sl2;
            }
            m_new = m_ref;
          } else {
          float mloc = -INFINITY;
          {
#pragma unroll 1
            for (int ch = 0; ch < G::NCH; ++ch) {
              uint32_t sv[G::CH];
              WAVEAL_TMEM_LD32(s_addr + ch * G::CH, sv, 0);
              WAVEAL_TMEM_WAIT_LD32(sv, 0);
              mloc = fmaxf(mloc, row_max32(sv));
            }
            // the other owner of the row (same team and quadrant, other column half)
            // (two buffers by use parity: the partner's next value cannot land on one not yet read)
            volatile float* mh = mhalf + (hx_it & 1u) * 512;
            mh[(team * 2 + half) * 128 + r] = mloc;
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR(B_HX + team * 4 + quad));
            ok = warp_wait(ctx, BAR(B_HX + team * 4 + quad), hx_it & 1u, 26);
            if (!ok) break;
            ++hx_it;
            mloc = fmaxf(mloc, mh[(team * 2 + (half ^ 1)) * 128 + r]);
          }
          // ---- the row's reference after block j-1, from the other team
          float m_prev = m_ref;
          if (j > 0) {
            mx_phase ^= 1u << ((g - 1) & 3);                   // the other team's arrival for tile g-1
            // that team's arrival for tile g-1 is phase number (arrivals of that slot so far) - 1
            const uint32_t mx = (g - 1) & 3;
            ok = warp_wait(ctx, BAR(B_MX + quad * 4 + mx), ((mx_phase >> mx) & 1u) ^ 1u, 24);
            if (!ok) break;
            m_prev = mpub[((g - 1) & 3) * 128 + r];
          }
          const float m_cand = fmaxf(m_prev, mloc * p.sl2);
          // keep the stale reference unless it is exceeded by more than 2^8 (exact: the final
          // normalisation divides by a sum taken with the same reference); both owners of a row
          // see the same values and take the same decision
          const bool grow = __any_sync(0xffffffffu, m_cand > m_prev + 8.0f);
          m_new = grow ? m_cand : m_prev;
          if (half == 0) {
            // (slot and barrier g mod 4: the owner of tile g+4 cannot get there before both owners of
            // tile g+1 have read this one, which its S buffer waits for)
            mpub[(g & 3) * 128 + r] = m_new;
            __syncwarp();
            if (lane == 0) mbar_arrive(BAR(B_MX + quad * 4 + (g & 3)));
          }
          if (m_new != m_ref) {
            l_run *= (m_ref == -INFINITY) ? 0.f : ex2(m_ref - m_new);
            m_ref = m_new;
          }
          // rare: the reference grew, so O (blocks 0..j-1) is rescaled; its last MMA (block j-1)
          // must be complete: that is the latest phase of the barrier of the S buffer before
          // this one (the next P V on that buffer needs a P this team has not produced yet).
          // The owner of the first half of P does it for all columns of O before it releases that half: the P V
          // warp starts on the first half as soon as it has arrived, its MMAs add to all columns, and those on the
          // second half come behind.  (Split between the two owners, each would have to wait for the other.)
          if (grow && j > 0 && half == 0) {
            const uint32_t sbp = sb == 0 ? (uint32_t)G::NSBUF - 1u : sb - 1u;
            ok = warp_wait(ctx, BAR(B_S_FREE + sbp), sb == 0 ? s_ph ^ 1u : s_ph, 22);
            if (!ok) break;
            tc_fence_after();
            const float alpha = ex2(m_prev - m_new);
#pragma unroll 1
            for (int c0 = 0; c0 < D; c0 += 32) {
              uint32_t ov[32];
              WAVEAL_TMEM_LD32(o_row + c0, ov, 0);
              WAVEAL_TMEM_WAIT_LD32(ov, 0);
#pragma unroll
              for (int c = 0; c < 32; ++c) ov[c] = __float_as_uint(__uint_as_float(ov[c]) * alpha);
              WAVEAL_TMEM_ST32(o_row + c0, ov, 0);
            }
          }
          }
          // p' = 2^(s*scale*log2e - m + log2(1 + 2^-9)); P is p' cut to its top 16 bits (one byte
          // permute per pair instead of a conversion).  The extra factor centres the cut's error
          // around zero, like a rounding; the row sum adds the uncut p' and the epilogue takes
          // the factor out again.  Multiply-adds and sums work on register pairs (f32x2).
          const float neg_m = ((m_new == -INFINITY) ? 0.f : -m_new) + 0.0028150156f;
          const float a128 = p.sl2 * 0.0078125f, b128 = (neg_m - kPolyLo) * 0.0078125f;   // polynomial share
          float ls4[4] = {0.f, 0.f, 0.f, 0.f};
          // ---- pass 2: exponentials; P (bf16 pairs) goes over the first half of the thread's own
          // S columns, each chunk after its S values have been read.  A loop over
          // 32-column chunks, rolled at head_dim 128.
#pragma unroll G::UNROLL
          for (int ch = 0; ch < G::NCH; ++ch) {
            uint32_t sv[G::CH];
            WAVEAL_TMEM_LD32(s_addr + ch * G::CH, sv, 0);
            WAVEAL_TMEM_WAIT_LD32(sv, 0);
            uint32_t pk[G::CH / 2];
            // a pair's results are used LAG pairs later (written so, the compiler keeps more exponentials under way: 1,366 -> 1,347
            // clk a tile of 128x128 tasks of 256 tiles; 128x64 blocks lost 0.6 % and use them at once, and so
            // does the second launch: four pairs later 64x128 and 64x64 blocks took 0.6 % longer there)
            float x[G::CH];
            constexpr int kLag = FAST ? G::LAG : 0;
            auto use = [&](int c, float e0, float e1) {
              fadd2(ls4[c & 2], ls4[(c & 2) + 1], ls4[c & 2], ls4[(c & 2) + 1], e0, e1);
              pk[c / 2] = __byte_perm(__float_as_uint(e0), __float_as_uint(e1), 0x7632);
            };
#pragma unroll
            for (int c = 0; c < G::CH; c += 2) {
              if ((c >> 1) % kPolyEvery == kPolyEvery - 1) {
                ex2_fma2(x[c], x[c + 1], __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]), a128, b128);
              } else {
                ffma2(x[c], x[c + 1], __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]), p.sl2, p.sl2, neg_m, neg_m);
                x[c] = ex2(x[c]); x[c + 1] = ex2(x[c + 1]);
              }
              if (c >= 2 * kLag) use(c - 2 * kLag, x[c - 2 * kLag], x[c + 1 - 2 * kLag]);
            }
#pragma unroll
            for (int c = G::CH - 2 * kLag; c < G::CH; c += 2) use(c, x[c], x[c + 1]);
            WAVEAL_TMEM_ST16(s_addr + ch * 16, pk, 0);
          }
          const float l_blk = (ls4[0] + ls4[1]) + (ls4[2] + ls4[3]);
          l_run += l_blk;
          if (MOD4) { const float t = l_run; l_run = l_other; l_other = t; }
          // all terms are positive (the transcendental unit returns +inf on overflow, the
          // polynomial share saturates at 2^64), so a sum below 2^60 bounds every exponent it
          // covers; at or above it (or not a number) the fixed reference is too far off:
          // redo the task
          if (FAST && __any_sync(0xffffffffu, !(l_blk < kRedoLimit))) redo_flag[rslot] = task_no;
          tc_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(BAR(B_P_FULL + sb * 2 + half));
        }
        // one flip per arrival on that slot's barrier (before the exponentials it cost 64x128 blocks 2-3 % of the cycles)
        if (!FAST) mx_phase ^= 1u << (g & 3);
        next_buffer(j);
      }
      if (!ok) break;
      // ---- epilogue: O / l at the original row position; l = the four partial sums of the row (by whether
      // the team had the task's first tile, so that the result does not depend on which team had which) brought to
      // the final reference (the larger of the two teams', references never shrink)
      // (a thread's partial sum is final once its last tile is done)
      if (MOD4 && (((tk.n - role + 1) >> 1) & 1)) { const float t = l_run; l_run = l_other; l_other = t; }
      exb[(role * 2 + half) * 128 + r] = MOD4 ? make_float2(l_run, l_other) : make_float2(m_ref, l_run);
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(ex_bar));
      // (the team of the last tile; at least one of the first two is the first team's)
      const bool mine = kTwoFirst ? (role == 0) == (last == 0 || (last & 1)) : (int)((g0 + (uint32_t)last) & 1u) == team;
      if (kTwoFirst) {
        if (j0 >= tk.n && !idle) mx_phase ^= 1u << (o_it & 3);
        first_team = mine ? team ^ 1 : team;
      } else if (!mine && !idle && !(FAST && last > 0)) {
        mx_phase ^= 1u << ((g0 + (uint32_t)last) & 3);
      }
      g0 += (uint32_t)tk.n;
      const uint32_t o_ph = o_it & 1;
      ++o_it;
      if (!mine) continue;
      // All four warps of this lane quadrant have left their sums; the other team's are there long
      // before.  (This wait stands before the one for O: a team that has run ahead could otherwise
      // take the completion of the task before the previous one for that of its own.)  Bounded
      // like every other wait, so that a warp whose partners gave up does not stay behind.
      ok = warp_wait(ctx, BAR(ex_bar), ex_ph, 25);
      if (!ok) break;
      const float2 e00 = exb[0 * 128 + r], e01 = exb[1 * 128 + r], e10 = exb[2 * 128 + r], e11 = exb[3 * 128 + r];
      float m_all, l_tot;
      if constexpr (MOD4) {
        m_all = m_ref;                                                     // (the same for all; no reference: for the second launch)
        l_tot = m_ref == -INFINITY ? 0.f : ((e00.x + e01.x) + (e10.x + e11.x)) + ((e00.y + e01.y) + (e10.y + e11.y));
      } else {
        const float m0 = fmaxf(e00.x, e01.x), m1 = fmaxf(e10.x, e11.x);   // the two owners of a team's rows agree; a team
        m_all = fmaxf(m0, m1);                                             // without tiles (n == 1) has -inf
        const float a0 = (m0 == -INFINITY) ? 0.f : ex2(m0 - m_all);
        const float a1 = (m1 == -INFINITY) ? 0.f : ex2(m1 - m_all);
        l_tot = a0 * (e00.y + e01.y) + a1 * (e10.y + e11.y);
      }
      const float inv_l = 1.0019531f / l_tot;    // the sums carry the centring factor 1 + 2^-9
      ok = warp_wait(ctx, BAR(B_O_FULL), o_ph, 23);
      if (!ok) break;
      tc_fence_after();
      uint32_t ov[G::CO];
      static_assert(G::CO == 64 || G::CO == 32, "half of head_dim 128 or 64");
      WAVEAL_TMEM_LD32(o_row + half * G::CO, ov, 0);
      if constexpr (G::CO == 64) WAVEAL_TMEM_LD32(o_row + half * G::CO + 32, ov, 32);
      WAVEAL_TMEM_WAIT_LD32(ov, 0);
      if constexpr (G::CO == 64) WAVEAL_TMEM_WAIT_LD32(ov, 32);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_O_FREE));
      bool bad = false;
      // From registers a store instruction touches 32 rows and the memory pipe takes 2 clk for each: 2,300 clk a task for the
      // 1,024 row pieces of 32 bytes, in which the team could have been at its next tile.
      // Staged: 128x64 tasks of 24 tiles 1,272 -> 1,247 clk a tile, 128x128 tasks of 17 tiles 1,698 -> 1,664, of 32 tiles
      // 1,501 -> 1,489; tasks of 256 tiles pay 1 % for it (1,364 -> 1,380).
      const uint32_t stage = sbase + G::OFF_Q + (G::NQ == 2 ? ((uint32_t)o_it - 1u) & 1u : 0u) * G::Q_BYTES + (uint32_t)(quad * 2 + half) * (32 * G::CO * 2);
      if (row_live) {
        uint32_t w[G::CO / 2];
#pragma unroll
        for (int c = 0; c < G::CO; c += 2) {
          __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(ov[c]) * inv_l, __uint_as_float(ov[c + 1]) * inv_l);
          w[c / 2] = *reinterpret_cast<uint32_t*>(&b2);
        }
        // |O| <= l_tot max|V|: only a large sum (or none) can have led out of fp32's range
        if (FAST && !(l_tot > 0.f && l_tot < kCheckSum)) {
          uint32_t top = 0;                // an exponent field of ones in either half of a pair carries into its top bit
#pragma unroll
          for (int c = 0; c < G::CO / 2; ++c) top |= (w[c] & 0x7F807F80u) + 0x00800080u;
          bad = (top & 0x80008000u) != 0;
        }
        if constexpr (G::STAGED) {
          // the box's rows of 128 (64) bytes, 16-byte pieces swizzled as the tensor map says: eight (four) lanes a wavefront
          const uint32_t row0 = stage + (uint32_t)lane * (G::CO * 2), sw = G::CO == 64 ? lane & 7 : (lane >> 1) & 3;
#pragma unroll
          for (int c = 0; c < G::CO / 8; ++c) st_shared_v4(row0 + (((uint32_t)c ^ sw) << 4), w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
        } else if ((reinterpret_cast<uintptr_t>(o_ptr) & 31) == 0) {
          // a thread holds a piece of one row, so a store instruction of a warp touches 32 rows:
          // its cost in the memory pipe is per row, not per byte.  32-byte stores halve the number
          // of instructions where the row piece is 32-byte aligned (else 16-byte stores)
#pragma unroll
          for (int c = 0; c < G::CO / 2; c += 8) st_global_v8(o_ptr + 2 * c, w + c);
        } else {
#pragma unroll
          for (int c = 0; c < G::CO / 2; c += 4)
            *reinterpret_cast<uint4*>(o_ptr + 2 * c) = make_uint4(w[c], w[c + 1], w[c + 2], w[c + 3]);
        }
        if (p.lse && half == 0) p.lse[(size_t)tk.h * p.seq_q + q_tok] = (m_all + log2f(l_tot) - 0.0028150156f) * 0.6931471805599453f;
      }
      if constexpr (G::STAGED) {
        fence_proxy_async();
        __syncwarp();
        const int tok0 = tk.row * G::BQ + quad * 32;         // (rows beyond seq_q are left out)
        if (lane == 0 && tok0 < p.seq_q) { tma_store_3d(&tmO, stage, half * G::CO, tok0, tk.h); bulk_commit(); }
        storing = true;
      }
      // The task goes to the second launch if the sum of a tile left the range (every warp's tiles of this task lie
      // before O_FULL) or if a result is not finite: with sums of up to 2^60 O overflows from |V| = 2^67 on, and a
      // first tile whose scores are all -inf leaves no reference.  (Where V itself holds an inf or NaN the second
      // launch finds the same again.)  Whichever of the epilogue's warps sees it first writes the entry.
      if (FAST && (__any_sync(0xffffffffu, bad) || redo_flag[rslot] == task_no) && lane == 0) {
        if constexpr (G::KB == 2) list_task_call(p.ws, &redo_listed[rslot], task_no, tk.h, tk.row, tk.row2);
        else list_task(p.ws, &redo_listed[rslot], task_no, tk.h, tk.row, -1);
      }
    }
  }

  // (stores still under way read this CTA's shared memory)
  if (G::STAGED && warp >= kSoftmaxWarp0 && warp < kQkWarp && lane == 0) bulk_wait_all();
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kPvWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, G::TMEM_COLS);
  }
  // SM cycles since the CTA's first task could start (t_start): the largest over the grid is the launch's length in
  // cycles, a figure that does not depend on the clock the GPU happened to run at
  if (tid == 0) {
    const long long dt = clock64() - t_start;
    atomicMax(&p.ws[p.redo_pass ? 5 : 4], (int)(dt > 0x7fffffffll ? 0x7fffffffll : dt));
  }
}

// ------------------------------------------------------------------ 64-row query blocks, first launch
//
// A lone 64-row block leaves half of a 128-row product empty, and an ordinary product of 64 rows takes as long as one of 128
// (64 clk for N = 128, K = 16).  tcgen05.mma.ws with M = 64 takes 48.7 clk: it lays row m of the result over lanes m and 64 + m,
// half of the columns in each, so that all of tensor memory's lanes work and the softmax has 64 columns a lane.  What bounds
// it is shared memory: A and B are read anew for every product, 6 KB at 128 bytes a clock (N = 256 takes 80).  One item, a block of
// 64 rows against a tile of 128 keys, is 8 + 8 products = 779 clk at head_dim 128 and 4 + 8 = 484 at 64; P goes through
// shared memory too (as an operand in tensor memory it would have to lie in both halves of the lanes).  64 KB of K and V an item are
// 850 clk at the 77 bytes per clock and SM that all SMs draw from L2 together at the full clock.
// Against the 128-row products (which a lone block half filled) with the same softmax: 8 heads of 1,536 rows of the LTX recipe, head_dim 128,
// 1,319 -> 1,110 clk a tile (907 an item; two blocks that share the tiles of one list take two items each), 11.2 -> 9.4 ms;
// 8 heads of 768 rows, head_dim 64, 1,165 -> 930, 2.17 -> 1.70 ms; 8 heads of 317 rows of 9 or 10 tiles 1,773 -> 1,330, 185 -> 144 us.
// Pairs as ordinary products of 128 rows (the same bits): 1,170, the code for both slows a lone block's softmax.
//
// At this pace the issuing warps' and the loaders' own instructions count (~10 clk each beside four softmax warps a scheduler):
//  - an item has ONE barrier on which its product waits (the tile's bytes and the softmax group's arrivals together) and ONE that it
//    completes, by item number mod 8; loaders and softmax look at the same ones.  With barriers by ring stage and by buffer (two
//    waits and two commits a product) an item took 1,020 clk instead of 919;
//  - the products of an item are one block of instructions under one election (one for each: 1,286 -> 1,076);
//  - four loaders, every second K and every second V tile each: a box of 64 rows costs its warp ~150 clk to request, a
//    tile of two blocks is four (two loaders: 1,076, four: 1,020).
//
// Softmax: four groups of four warps; item q (counted over the CTA's life) belongs to group and S buffer q mod 4 and P buffer
// q mod 3.  A lane has 64 columns of one row, lanes m and 64 + m the two halves of a tile.  The S buffer is free as soon as its scores are
// in registers.  The accumulator has two copies, by task, so that the next task's products do not wait for this one's epilogue,
// which the group of a block's last item runs while the others go on.
// Which kernel a call takes: two blocks that share their tiles (a pair) fill a product of 128 rows, which takes 1,327 clk a tile
// (1,140 at head_dim 64) against their two items' 1,770 (1,370), a lone block's tile as long against its item's 886
// (735): products of 64 rows are quicker until pairs have 47 % (64 %) of the tiles, or the longest pair outlasts an SM's share of the
// work.  k_sort_tail, which has the counts, picks; the kernel not picked leaves at once (with the counts 4 to 6 us where products of 128
// rows run, 1 to 2 where the others do).  (8 heads of the LTX recipe, a quarter: 11.2 -> 9.3 ms; 2 dense heads of 512 rows, all: 892 us
// with the one, 1,100 with the other.)  Calls of no more tasks than SMs last as long as their longest task and stay with products of 128
// rows, and so do small ones (launch()).
// Pairs: two blocks with the very same list are items 2 i and 2 i + 1 of tile i, each with an accumulator of its own.  Everything a row
// sees is as it would be alone: the products in the same order, a reference from the same first 128 keys, and the same
// sums, which a lone block has by tile mod 4 (its groups) and a pair's groups keep two of.
constexpr long long kRows64Tiles = 320;              // tiles an SM that the lists of a call may have, from which this kernel is launched
constexpr int kThreads64 = 704, kLoadWarps64 = 20;   // 22 warps: those of the kernel above and two more loaders

// clk a tile of 128 keys in products of 128 rows, and in products of 64 of a block on its own, of a pair, and of a long pair that
// starts with the call
struct Pace { int rows128, lone, pair, first_pair; };

template <int D>
struct Geo64 {
  static constexpr int BQ = 64, BK = 128;            // a KV tile is 128 keys: two consecutive entries of the row's list
  static constexpr int SLABS = D / 64;               // 128-byte column slabs of a Q/K/V tile
  static constexpr int Q_BYTES = SLABS * BQ * 128;   // one query block
  static constexpr int KV_SLAB_BYTES = BK * 128;
  static constexpr int TILE_BYTES = SLABS * KV_SLAB_BYTES;     // K tile
  static constexpr int P_PANEL_BYTES = BQ * 128;     // P of 64 rows and 64 keys
  static constexpr int P_BYTES = 2 * P_PANEL_BYTES;
  static constexpr int NQ = 2;                       // query blocks: two of a pair, or this task's and the next one's
  static constexpr int NP = 3;                       // P buffers
  static constexpr int NKS = D == 128 ? 2 : 4;       // K tiles
  static constexpr int NVS = NKS;                    // V tiles
  static constexpr int NG = 4;                       // softmax groups of four warps, each with its own S buffer
  static constexpr int CO = D / 2;                   // O columns per epilogue thread
  static constexpr int NSL = 3;                      // slots by task for what the groups leave each other
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_P = OFF_Q + NQ * Q_BYTES;
  static constexpr int OFF_K = OFF_P + NP * P_BYTES;
  static constexpr int OFF_V = OFF_K + NKS * TILE_BYTES;
  static constexpr int OFF_BAR = OFF_V + NVS * TILE_BYTES;
  static constexpr int N_BAR = 4 + 2 * NQ + 4 * 8 + 4 + 4 + 2 + NSL * 4 + NSL * 2;
  static constexpr int OFF_TASK = OFF_BAR + ((N_BAR * 8 + 15) / 16) * 16;
  static constexpr int OFF_MX = OFF_TASK + 4 * (int)sizeof(Task);             // [slot][block][128] largest score of a half row
  static constexpr int OFF_EX = OFF_MX + NSL * 2 * 128 * 4;                   // [slot][block][tile mod 4][128] sums
  static constexpr int OFF_MISC = OFF_EX + NSL * 2 * 4 * 128 * 4;
  static constexpr int SMEM_BYTES = OFF_MISC + 48 + 1024;   // + slack for 1024-byte alignment
  static_assert(SMEM_BYTES <= 232448, "shared memory of a CTA");
  // tensor memory: an S buffer of 64 columns per softmax group, then two sets of output accumulators (by task) for two blocks
  static constexpr uint32_t S_STRIDE = 64, O_COL = NG * 64, O_STRIDE = 64, TMEM_COLS = 512;
  // As measured on the kernels as they are: to be measured again when the pace of either changes (dense heads; 8 heads of the LTX
  // recipe without pairs; rows that are all in pairs; a pair of 350 or 750 tiles among the first rows, the others 10 to 30 tiles).
  // Over 300 mixes of both (long rows none to a third, first, last or spread; none, half or all of the others in pairs; 1 to 16
  // heads) the kernel picked takes 0.15 % longer than the quicker one on average, 7.6 % at most
  // (products of 64 rows always 20 %, of 128 always 47 % at most).
  static constexpr Pace PACE = D == 128 ? Pace{1327, 886, 1772, 1615} : Pace{1140, 735, 1372, 1372};
};

// One K or V tile of a task into its ring stage (called by a whole warp); see load_kv_tile.  done: the product that read the
// stage's tile before this one (an item, or -1); item: the first that reads this one, of `blocks`.
template <class G, bool IS_K>
__device__ __forceinline__ bool load_tile64(const Ctx& ctx, const AttnParams& p, const Task& tk, bool dropped, int j, int lane,
                                            uint32_t sbase, uint32_t stage, uint32_t bar_ready0, uint32_t bar_done0, int done,
                                            int item, int blocks, const CUtensorMap* tm, const CUtensorMap* tm2, int& chunk_base,
                                            int& my_idx) {
  if (2 * j >= chunk_base + 32) {
    chunk_base = (2 * j) & ~31;
    my_idx = chunk_base + lane < tk.len ? p.kv_idx[tk.lo + chunk_base + lane] : 0;
    if (my_idx < 0 || my_idx >= p.n_b) {             // malformed list: report it and stay in range
      if (IS_K && p.dev_status && atomicCAS(p.dev_status, 0, WAVEAL_ERR_BAD_MASK) == 0) {
        p.dev_status[1] = 30; p.dev_status[2] = tk.h; p.dev_status[3] = my_idx;
      }
      my_idx = 0;
    }
  }
  const int sl = lane % G::SLABS, e = lane / G::SLABS, nblk = min(2, tk.len - 2 * j);
  const int blk0 = __shfl_sync(0xffffffffu, my_idx, 2 * j - chunk_base), blk1 = __shfl_sync(0xffffffffu, my_idx, 2 * j + 1 - chunk_base);
  if (done >= 0 && !warp_wait(ctx, bar_done0 + 8u * (done & 7), (done >> 3) & 1, IS_K ? 3 : 4)) return false;
  if (dropped) return true;
  const uint32_t b_ready = bar_ready0 + 8u * (item & 7);
  if (lane == 0) {
    mbar_expect_tx(b_ready, (uint32_t)nblk * G::SLABS * 64 * 128);
    if (blocks == 2) mbar_arrive(bar_ready0 + 8u * ((item + 1) & 7));      // (of a pair; its two products are issued in order)
  }
  __syncwarp();
  // one lane per box: lane e*SLABS + s requests slab s of block e; two blocks that follow each other in memory come as one box
  const uint32_t dst = sbase + (IS_K ? G::OFF_K : G::OFF_V) + stage * G::TILE_BYTES + sl * G::KV_SLAB_BYTES;
  if (nblk == 2 && blk1 == blk0 + 1) {
    if (e == 0) tma_load_3d(dst, tm2, sl * 64, blk0 * 64, tk.h, b_ready);
  } else if (e < nblk) {
    tma_load_3d(dst + e * 64 * 128, tm, sl * 64, (e ? blk1 : blk0) * 64, tk.h, b_ready);
  }
  return true;
}

// Every second tile of all tasks, by the tile's number over the CTA's life
template <class G, bool IS_K>
struct TileLoader {
  static constexpr int NST = IS_K ? G::NKS : G::NVS, NOWN = NST / 2;       // stages in all, and of this warp
  uint32_t odd, base = 0;                            // tiles before this task
  int q0 = 0;                                        // items before this task
  int item[NOWN], done[NOWN];                        // of the tiles in this warp's stages, oldest first: first and last item
  __device__ __forceinline__ explicit TileLoader(uint32_t o) : odd(o) {
#pragma unroll
    for (int i = 0; i < NOWN; ++i) item[i] = done[i] = -1;
  }
  template <class F>
  __device__ __forceinline__ bool task(const Ctx& ctx, const AttnParams& p, const Task& tk, int lane, uint32_t sbase, uint32_t bar_ready0,
                                       uint32_t bar_done0, const CUtensorMap* tm, const CUtensorMap* tm2, bool drop_first, F before) {
    const int blocks = tk.row2 >= 0 ? 2 : 1;
    int chunk_base = -64, my_idx = 0;
#pragma unroll 1
    for (int j = (int)((base ^ odd) & 1); j < tk.n; j += 2) {
      before(j);
      const int it = q0 + j * blocks;
      if (!load_tile64<G, IS_K>(ctx, p, tk, drop_first && j == 0, j, lane, sbase, (base + (uint32_t)j) % NST, bar_ready0, bar_done0,
                                done[0], it, blocks, tm, tm2, chunk_base, my_idx))
        return false;
#pragma unroll
      for (int i = 0; i + 1 < NOWN; ++i) { item[i] = item[i + 1]; done[i] = done[i + 1]; }
      item[NOWN - 1] = it;
      done[NOWN - 1] = it + blocks - 1;
    }
    if (tk.n > 0) { base += (uint32_t)tk.n; q0 += tk.n * blocks; }
    return true;
  }
  // leave no bulk copy in flight into this CTA's shared memory (bounded)
  __device__ __forceinline__ void drain(const AttnParams& p, uint32_t bar_ready0) const {
#pragma unroll
    for (int i = 0; i < NOWN; ++i)
      if (item[i] >= 0) {
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_ready0 + 8u * (item[i] & 7), (item[i] >> 3) & 1) && clock64() - t0 < p.wait_limit / 4) {}
      }
  }
};

template <int D>
__global__ void __launch_bounds__(kThreads64, 1)
k_bsattn_fwd_rows64(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmK2,
                    const __grid_constant__ CUtensorMap tmV2, const AttnParams p) {
  // tmK2 / tmV2: K and V in boxes of 128 rows, for two blocks of a tile that lie next to each other in memory
  using G = Geo64<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // provably warp-uniform role index
  waveal::let_next_kernel_start();

  const uint32_t bar0 = sbase + G::OFF_BAR;
  auto BAR = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  constexpr int B_TASK_FULL = 0, B_TASK_EMPTY = 2, B_Q_FULL = 4, B_Q_EMPTY = B_Q_FULL + G::NQ, B_QK_READY = B_Q_EMPTY + G::NQ,
                B_QK_DONE = B_QK_READY + 8, B_PV_READY = B_QK_DONE + 8, B_PV_DONE = B_PV_READY + 8, B_O_FULL = B_PV_DONE + 8,
                B_O_FREE = B_O_FULL + 4, B_FINAL = B_O_FREE + 4,
                B_MX = B_FINAL + 2, B_EX = B_MX + G::NSL * 4;
  static_assert(B_EX + G::NSL * 2 <= G::N_BAR, "barrier count");
  Task* tasks = reinterpret_cast<Task*>(smem + G::OFF_TASK);
  volatile float* mx = reinterpret_cast<volatile float*>(smem + G::OFF_MX);
  float* ex = reinterpret_cast<float*>(smem + G::OFF_EX);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + G::OFF_MISC);
  volatile int* abort_smem = reinterpret_cast<volatile int*>(smem + G::OFF_MISC + 4);
  // [slot]: number (from 1) of the last task that a tile wants computed again, and of the last one listed for it
  volatile int* redo_flag = reinterpret_cast<volatile int*>(smem + G::OFF_MISC + 8);
  int* redo_listed = reinterpret_cast<int*>(smem + G::OFF_MISC + 8 + G::NSL * 4);
  Ctx ctx{bar0, abort_smem, p.ws, p.dev_status, p.wait_limit};

  if (tid == 0) {
    // a task is read by the three other loaders, the two MMA issuers and the sixteen softmax warps
    for (int i = 0; i < 2; ++i) { mbar_init(BAR(B_TASK_FULL + i), 1); mbar_init(BAR(B_TASK_EMPTY + i), 21); }
    for (int i = B_Q_FULL; i < B_QK_READY; ++i) mbar_init(BAR(i), 1);       // one load, one commit
    for (int i = 0; i < 8; ++i) {
      mbar_init(BAR(B_QK_READY + i), 5);                                    // the K tile, and the group's four warps have read their S buffer
      mbar_init(BAR(B_PV_READY + i), 5);                                    // the V tile, and P by the group's four warps
      mbar_init(BAR(B_QK_DONE + i), 1);
      mbar_init(BAR(B_PV_DONE + i), 1);
    }
    for (int i = 0; i < 4; ++i) { mbar_init(BAR(B_O_FULL + i), 1); mbar_init(BAR(B_O_FREE + i), 4); }
    for (int i = 0; i < 2; ++i) mbar_init(BAR(B_FINAL + i), 1);
    for (int i = 0; i < G::NSL * 4; ++i) mbar_init(BAR(B_MX + i), 2);       // the two warps that have a row's first tile
    for (int i = 0; i < G::NSL * 2; ++i) mbar_init(BAR(B_EX + i), 8);       // all warps that have sums of a row
    *abort_smem = 0;
    for (int i = 0; i < G::NSL; ++i) { redo_flag[i] = 0; redo_listed[i] = 0; }
    fence_mbar_init();
    fence_proxy_async();
  }
  if (warp == kPvWarp) {
    tmem_alloc(smem_u32(tmem_holder), G::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_holder, 0);
  waveal::wait_for_previous_kernel();
  const long long t_start = clock64();

  // every role walks the same sequence of tasks and, inside a task, of items
  const bool mine = p.table->pick == 0;
  if (!mine) {
    // (the other kernel's call)
  } else if (warp == kProducerWarp) {
    // ============================================================== producer: tickets, Q, every second K tile
    if (lane == 0) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmK2); prefetch_tmap(&tmV2); }
    uint32_t task_it = 0, q_it = 0, q_armed = 0, q_parity = 0;
    TileLoader<G, true> k_tiles{0};
    int n_tiles = 0, n_pairs = 0;        // words 7 and 6 of the workspace
    bool ok = true;
    auto draw = [&](long long& t_out) -> Task {
      for (;;) {
        long long t = 0;
        if (lane == 0)                   // (volatile: another SM raises the flag while this kernel runs)
          t = *reinterpret_cast<volatile int*>(&p.ws[1]) != 0 ? p.total_tasks : (long long)(unsigned)atomicAdd(&p.ws[0], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        t_out = t;
        Task tk{};
        if (t >= p.total_tasks) { tk.n = -1; return tk; }
        const uint4* e = reinterpret_cast<const uint4*>(p.table + t);
        const uint4 a = e[0], b = e[1];
        tk.h = (int)a.x; tk.row = (int)a.y; tk.lo = (int)a.z; tk.n = (int)a.w; tk.tail_valid = (int)b.x; tk.len = (int)b.y;
        tk.row2 = (int)b.z;
        if (tk.n != kAbsorbed) return tk;             // (else the second block of a pair: computed with its partner)
      }
    };
    constexpr int kDrawAhead = 3;        // tiles before the task's last K loads: the round trips of the ticket hide behind the ring
    long long t = 0, t_next = 0;
    Task tk_next = draw(t_next);
    while (ok) {
      const Task tk = tk_next;
      t = t_next;
      bool drawn = false;
      const uint32_t slot = task_it & 1, ph = (task_it >> 1) & 1;
      ok = warp_wait(ctx, BAR(B_TASK_EMPTY + slot), ph ^ 1, 1);
      if (!ok) break;
      if (lane == 0) {
        tasks[task_it & 3] = tk;           // (four places: an epilogue looks a task up when the next two may be there)
        mbar_arrive(BAR(B_TASK_FULL + slot));
      }
      ++task_it;
      if (tk.n < 0) break;
      if (tk.n <= kDrawAhead) { tk_next = draw(t_next); drawn = true; }
      if (tk.n == 0) continue;
      const int blocks = tk.row2 >= 0 ? 2 : 1;
      n_tiles += tk.n;
      n_pairs += blocks - 1;
      for (int b = 0; b < blocks && ok; ++b, ++q_it) {
        const uint32_t qb = q_it % G::NQ, q_ph = (q_it / G::NQ) & 1;
        ok = warp_wait(ctx, BAR(B_Q_EMPTY + qb), q_ph ^ 1, 2);
        if (!ok) break;
        if (lane == 0) {
          mbar_expect_tx(BAR(B_Q_FULL + qb), G::Q_BYTES);
#pragma unroll
          for (int s = 0; s < G::SLABS; ++s)
            tma_load_3d(sbase + G::OFF_Q + qb * G::Q_BYTES + s * G::BQ * 128, &tmQ, s * 64, (b ? tk.row2 : tk.row) * G::BQ, tk.h, BAR(B_Q_FULL + qb));
        }
        q_armed |= 1u << qb; q_parity = (q_parity & ~(1u << qb)) | q_ph << qb;
      }
      ok = ok && k_tiles.task(ctx, p, tk, lane, sbase, BAR(B_QK_READY), BAR(B_QK_DONE), &tmK, &tmK2, p.drop_tile && t == 0, [&](int j) {
        if (!drawn && j >= tk.n - kDrawAhead) { tk_next = draw(t_next); drawn = true; }
      });
    }
    if (lane == 0) {
      if (n_tiles) atomicAdd(&p.ws[7], n_tiles);
      if (n_pairs) atomicAdd(&p.ws[6], n_pairs);
    }
    if (*abort_smem) {
      // leave no bulk copy in flight into this CTA's shared memory (bounded)
      k_tiles.drain(p, BAR(B_QK_READY));
      for (int st = 0; st < G::NQ; ++st)
        if (q_armed & (1u << st)) {
          long long t0 = clock64();
          while (!mbar_try_wait(BAR(B_Q_FULL + st), (q_parity >> st) & 1) && clock64() - t0 < p.wait_limit / 4) {}
        }
    }
  } else if (warp == kVLoadWarp || warp >= kLoadWarps64) {
    // ============================================================== loaders of V and of the other K tiles
    auto load_tiles = [&](auto tiles, uint32_t bar_ready0, uint32_t bar_done0, const CUtensorMap* tm, const CUtensorMap* tm2) {
      uint32_t task_slot = 0, task_ph = 0;
      bool ok = true;
      while (ok) {
        ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
        if (!ok) break;
        const Task tk = tasks[task_slot + 2 * task_ph];
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
        task_slot ^= 1;
        task_ph ^= (task_slot == 0);
        if (tk.n < 0) break;
        ok = tiles.task(ctx, p, tk, lane, sbase, bar_ready0, bar_done0, tm, tm2, false, [](int) {});
      }
      if (*abort_smem) tiles.drain(p, bar_ready0);
    };
    if (warp == kLoadWarps64) load_tiles(TileLoader<G, true>{1}, BAR(B_QK_READY), BAR(B_QK_DONE), &tmK, &tmK2);
    else load_tiles(TileLoader<G, false>{warp == kVLoadWarp ? 0u : 1u}, BAR(B_PV_READY), BAR(B_PV_DONE), &tmV, &tmV2);
  } else if (warp == kQkWarp) {
    // ============================================================== MMA issuer 1: S = Q K^T
    constexpr uint32_t IDESC_QK = make_idesc(64, G::BK, false);
    uint32_t task_slot = 0, task_ph = 0, q_it = 0, k_st = 0, it = 0;
    const uint64_t qdesc0 = make_desc(sbase + G::OFF_Q, 16, 1024);
    const uint64_t kdesc0 = make_desc(sbase + G::OFF_K, 16, 1024);
    bool ok = true;
    while (ok) {
      ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
      if (!ok) break;
      const int n = __shfl_sync(0xffffffffu, tasks[task_slot + 2 * task_ph].n, 0);
      const int blocks = __shfl_sync(0xffffffffu, tasks[task_slot + 2 * task_ph].row2, 0) >= 0 ? 2 : 1;
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
      task_slot ^= 1;
      task_ph ^= (task_slot == 0);
      if (n < 0) break;
      if (n == 0) continue;
      for (int b = 0; b < blocks && ok; ++b)
        ok = warp_wait(ctx, BAR(B_Q_FULL + ((q_it + b) % G::NQ)), ((q_it + b) / G::NQ) & 1, 11);
      for (int j = 0; j < n && ok; ++j) {
        const uint64_t kd = kdesc0 + (uint64_t)(k_st * (uint32_t)(G::TILE_BYTES >> 4));
#pragma unroll 1
        for (int b = 0; b < blocks; ++b) {
          const uint32_t qb = (q_it + b) % G::NQ;
          const uint64_t qd = qdesc0 + (uint64_t)(qb * (uint32_t)(G::Q_BYTES >> 4));
          const uint32_t d_s = tmem_base + (it % G::NG) * G::S_STRIDE;
          // the K tile is there, and the group has read the scores of its item before this one
          ok = warp_wait(ctx, BAR(B_QK_READY + (it & 7)), (it >> 3) & 1, 12);
          if (!ok) break;
          tc_fence_after();
          umma_ws_bf16<D / 16, 32, G::BQ * 128, 32, G::KV_SLAB_BYTES>(d_s, qd, kd, IDESC_QK, 0, BAR(B_QK_DONE + (it & 7)));
          if (j == n - 1) tc_commit(BAR(B_Q_EMPTY + qb));
          ++it;
        }
        if (++k_st == (uint32_t)G::NKS) k_st = 0;
      }
      q_it += (uint32_t)blocks;
    }
    // none of this thread's MMAs is still running when tensor memory is released
    tc_commit(BAR(B_FINAL + 1));
    __syncwarp();
    {
      long long t0 = clock64();
      while (!mbar_try_wait(BAR(B_FINAL + 1), 0) && clock64() - t0 < p.wait_limit / 4) {}
    }
  } else if (warp == kPvWarp) {
    // ============================================================== MMA issuer 2: O += P V
    constexpr uint32_t IDESC_PV = make_idesc(64, D, true);
    uint32_t task_slot = 0, task_ph = 0, o_it = 0, o_free = 0xFu, v_st = 0, pb = 0, it = 0;
    const uint64_t pdesc0 = make_desc(sbase + G::OFF_P, 16, 1024);
    const uint64_t vdesc0 = make_desc(sbase + G::OFF_V, G::KV_SLAB_BYTES, 1024);
    bool ok = true;
    while (ok) {
      ok = warp_wait(ctx, BAR(B_TASK_FULL + task_slot), task_ph, 10);
      if (!ok) break;
      const int n = __shfl_sync(0xffffffffu, tasks[task_slot + 2 * task_ph].n, 0);
      const int blocks = __shfl_sync(0xffffffffu, tasks[task_slot + 2 * task_ph].row2, 0) >= 0 ? 2 : 1;
      const bool half_tail = __shfl_sync(0xffffffffu, tasks[task_slot + 2 * task_ph].tail_valid, 0) <= 64;
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + task_slot));
      task_slot ^= 1;
      task_ph ^= (task_slot == 0);
      if (n < 0) break;
      if (n == 0) continue;
      // the accumulators of the task before the previous one have been read by the epilogue
      const uint32_t ob = (o_it & 1) * 2;
      ++o_it;
      for (int b = 0; b < blocks && ok; ++b) {
        ok = warp_wait(ctx, BAR(B_O_FREE + ob + b), (o_free >> (ob + b)) & 1u, 16);
        o_free ^= 1u << (ob + b);
      }
      for (int j = 0; j < n && ok; ++j) {
        const bool half = j == n - 1 && half_tail;     // (the second half of a half tile has no keys: nothing was loaded for it)
        const uint64_t vd = vdesc0 + (uint64_t)(v_st * (uint32_t)(G::TILE_BYTES >> 4));
#pragma unroll 1
        for (int b = 0; b < blocks; ++b) {
          const uint64_t pd = pdesc0 + (uint64_t)(pb * (uint32_t)(G::P_BYTES >> 4));
          const uint32_t d_o = tmem_base + G::O_COL + (ob + b) * G::O_STRIDE;
          ok = warp_wait(ctx, BAR(B_PV_READY + (it & 7)), (it >> 3) & 1, 14);
          if (!ok) break;
          tc_fence_after();
          // V tile as the N x K operand with N (head_dim) contiguous: 16 keys = 2048 bytes per MMA, the next 64 columns
          // of head_dim one slab further
          if (half) umma_ws_bf16<4, 32, 0, 16 * 128, 0>(d_o, pd, vd, IDESC_PV, j > 0, BAR(B_PV_DONE + (it & 7)));
          else umma_ws_bf16<8, 32, G::P_PANEL_BYTES, 16 * 128, 64 * 128>(d_o, pd, vd, IDESC_PV, j > 0, BAR(B_PV_DONE + (it & 7)));
          if (j == n - 1) tc_commit(BAR(B_O_FULL + ob + b));
          ++it;
          if (++pb == (uint32_t)G::NP) pb = 0;
        }
        if (++v_st == (uint32_t)G::NVS) v_st = 0;
      }
    }
    tc_commit(BAR(B_FINAL));
    __syncwarp();
    {
      long long t0 = clock64();
      while (!mbar_try_wait(BAR(B_FINAL), 0) && clock64() - t0 < p.wait_limit / 4) {}
    }
  } else {
    // ============================================================== softmax / epilogue (see the kernel above for what is the same)
    const int quad = warp & 3;                          // tensor-memory lane quadrant this warp may access
    const uint32_t group = (uint32_t)(warp - kSoftmaxWarp0) >> 2;
    const int half = quad >> 1;                         // keys 64 half .. of a tile; epilogue: half of O's columns
    const int rp = quad & 1, r = rp * 32 + lane;        // row of the query block
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t s_addr = tmem_base + lane_addr + group * G::S_STRIDE;
    uint32_t task_it = 0, o_it = 0, slot3 = 0, slot3_ph = 0, q0 = 0, mx1_bits = 0, of_bits = 0;
    if (lane == 0) mbar_arrive(BAR(B_QK_READY + group));        // (the buffers are free)
    bool ok = true;
    while (ok) {
      const uint32_t slot = task_it & 1, ph = (task_it >> 1) & 1;
      ok = warp_wait(ctx, BAR(B_TASK_FULL + slot), ph, 20);
      if (!ok) break;
      const volatile Task* tk = tasks + (task_it & 3);  // (what the epilogue needs of it is not kept in registers meanwhile)
      const int n = tk->n, tail_valid = tk->tail_valid;
      const bool pair = tk->row2 >= 0;
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR(B_TASK_EMPTY + slot));
      ++task_it;
      if (n < 0) break;
      if (n == 0) {
        const long long q_tok = (long long)tk->row * G::BQ + r;
        if (group == 0 && q_tok < p.seq_q) {
          uint4* o = reinterpret_cast<uint4*>(p.O + (size_t)tk->h * p.o_stride_h + (size_t)q_tok * p.o_stride_t + half * G::CO);
#pragma unroll 1
          for (int c = 0; c < G::CO / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
          if (p.lse && half == 0) p.lse[(size_t)tk->h * p.seq_q + q_tok] = -INFINITY;
        }
        continue;
      }
      const int n_items = pair ? 2 * n : n, i0 = (int)((group - q0) & 3u);      // this group's first item of the task
      const int blk = pair ? i0 & 1 : 0;                // its query block (the same in all its items: four items are two tiles further)
      const int task_no = (int)o_it + 1;
      const uint32_t mslot = slot3 * 2 + blk, mx_bar = BAR(B_MX + (slot3 * 2 + blk) * 2 + rp);
      // sums of this thread's columns of its tiles; of a pair, two tiles apart, l_run and l_other take turns: one sum for the tiles of
      // equal number mod 4, as the group of a block on its own has it
      float m_ref = -INFINITY, l_run = 0.f, l_other = 0.f;
      for (int i = i0; i < n_items; i += 4) {
        const uint32_t q = q0 + (uint32_t)i;
        const int tile = pair ? i >> 1 : i;
        ok = warp_wait(ctx, BAR(B_QK_DONE + (q & 7)), (q >> 3) & 1, 21);
        if (!ok) break;
        tc_fence_after();
        const int valid = tile == n - 1 ? tail_valid - half * 64 : 64;
        if (valid < 64 && valid > 0) mask_scores<2>(s_addr, valid);      // keys beyond seq_kv (ragged last block) do not exist
        if (i == i0) {
          if (tile == 0) {
            float mloc = -INFINITY;
            if (valid > 0) {
#pragma unroll 1
              for (int ch = 0; ch < 2; ++ch) {
                uint32_t sv[32];
                WAVEAL_TMEM_LD32(s_addr + ch * 32, sv, 0);
                WAVEAL_TMEM_WAIT_LD32(sv, 0);
                mloc = fmaxf(mloc, row_max32(sv));
              }
            }
            mx[mslot * 128 + half * 64 + r] = mloc;
            __syncwarp();
            if (lane == 0) mbar_arrive(mx_bar);
          }
          ok = warp_wait(ctx, mx_bar, blk ? (mx1_bits >> slot3) & 1u : slot3_ph, 24);
          if (!ok) break;
          m_ref = fmaxf(mx[mslot * 128 + r], mx[mslot * 128 + 64 + r]) * p.sl2;
        }
        if (valid > 0) {
          const float neg_m = ((m_ref == -INFINITY) ? 0.f : -m_ref) + 0.0028150156f;
          const float a128 = p.sl2 * 0.0078125f, b128 = (neg_m - kPolyLo) * 0.0078125f;   // polynomial share
          float ls4[4] = {0.f, 0.f, 0.f, 0.f};
          const uint32_t p_row = sbase + G::OFF_P + (q % G::NP) * G::P_BYTES + half * G::P_PANEL_BYTES + (uint32_t)r * 128;
          // (both chunks in line: 1,141 -> 1,113 clk a tile, 1,055 -> 930 at head_dim 64; a pair's results used four pairs later, as in the
          // kernel above: +0.4 .. +0.7 %)
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            uint32_t sv[32], pk[16];
            WAVEAL_TMEM_LD32(s_addr + ch * 32, sv, 0);
            WAVEAL_TMEM_WAIT_LD32(sv, 0);
            if (ch == 1) {                              // the scores are read: the group's next product may begin
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(BAR(B_QK_READY + ((q + 4) & 7)));
            }
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              float e0, e1;
              if ((c >> 1) % kPolyEvery == kPolyEvery - 1) {
                ex2_fma2(e0, e1, __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]), a128, b128);
              } else {
                ffma2(e0, e1, __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]), p.sl2, p.sl2, neg_m, neg_m);
                e0 = ex2(e0); e1 = ex2(e1);
              }
              fadd2(ls4[c & 2], ls4[(c & 2) + 1], ls4[c & 2], ls4[(c & 2) + 1], e0, e1);
              pk[c / 2] = __byte_perm(__float_as_uint(e0), __float_as_uint(e1), 0x7632);
            }
            if (ch == 0) {
              // the product of the buffer's item before this one has completed
              ok = q < G::NP || warp_wait(ctx, BAR(B_PV_DONE + ((q - G::NP) & 7)), ((q - G::NP) >> 3) & 1, 22);
              if (!ok) break;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
              st_shared_v4(p_row + ((((uint32_t)(ch * 4 + c)) ^ (uint32_t)(r & 7)) << 4), pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
          }
          if (!ok) break;
          const float l_blk = (ls4[0] + ls4[1]) + (ls4[2] + ls4[3]);
          l_run += l_blk;
          // all terms are positive, so a sum below 2^60 bounds every exponent it covers; at or above it (or not a number) the
          // fixed reference is too far off: redo the task
          if (__any_sync(0xffffffffu, !(l_blk < kRedoLimit))) redo_flag[slot3] = task_no;
          fence_proxy_async();
        } else {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(BAR(B_QK_READY + ((q + 4) & 7)));
          ok = q < G::NP || warp_wait(ctx, BAR(B_PV_DONE + ((q - G::NP) & 7)), ((q - G::NP) >> 3) & 1, 22);
          if (!ok) break;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_PV_READY + (q & 7)));
        if (pair) { const float t = l_run; l_run = l_other; l_other = t; }
      }
      if (!ok) break;
      // ---- epilogue: the four sums of a row and its two halves of every tile, in an order that does not depend on which group had which
      {
        const int steps = i0 < n_items ? (n_items - i0 + 3) >> 2 : 0;       // this group's items
        if (pair && (steps & 1)) { const float t = l_run; l_run = l_other; l_other = t; }
        const int role = pair ? i0 >> 1 : i0;
        float* e = ex + (mslot * 4 + role) * 128 + half * 64 + r;
        e[0] = l_run;
        if (pair) e[2 * 128] = l_other;
        __syncwarp();
        if (lane == 0) mbar_arrive(BAR(B_EX + slot3 * 2 + rp));
      }
      // the group of a block's last item has its epilogue
      const uint32_t last_group = (q0 + (uint32_t)n_items - 1u) & 3u;
      const bool mine = group == last_group || (pair && group == ((last_group - 1u) & 3u));
      const int my_blk = pair && group == last_group ? 1 : 0;
      const uint32_t ob = (o_it & 1) * 2 + my_blk, of_ph = (of_bits >> ob) & 1u, ex_ph = slot3_ph;
      const uint32_t tslot = slot3, es = slot3 * 2 + my_blk, ex_bar = BAR(B_EX + slot3 * 2 + rp);
      of_bits ^= (pair ? 3u : 1u) << ((o_it & 1) * 2);
      if (pair) mx1_bits ^= 1u << slot3;
      if (++slot3 == (uint32_t)G::NSL) { slot3 = 0; slot3_ph ^= 1; }
      q0 += (uint32_t)n_items;
      ++o_it;
      if (!mine) continue;
      ok = warp_wait(ctx, ex_bar, ex_ph, 25);
      if (!ok) break;
      float l_tot;
      {
        const float* e = ex + es * 512 + r;
        l_tot = ((e[0] + e[64]) + (e[128] + e[192])) + ((e[256] + e[320]) + (e[384] + e[448]));
      }
      const float m_all = fmaxf(mx[es * 128 + r], mx[es * 128 + 64 + r]) * p.sl2;
      if (m_all == -INFINITY) l_tot = 0.f;       // no reference: a result that is not finite, for the second launch
      const float inv_l = 1.0019531f / l_tot;    // the sums carry the centring factor 1 + 2^-9
      const int h = tk->h;
      const long long q_tok = (long long)(my_blk ? tk->row2 : tk->row) * G::BQ + r;
      __nv_bfloat16* o_ptr = p.O + (size_t)h * p.o_stride_h + (size_t)q_tok * p.o_stride_t + half * G::CO;
      ok = warp_wait(ctx, BAR(B_O_FULL + ob), of_ph, 23);
      if (!ok) break;
      tc_fence_after();
      const uint32_t o_addr = tmem_base + lane_addr + G::O_COL + ob * G::O_STRIDE;
      bool bad = false;
      // (all 64 columns at once do not fit the 80 registers that six warps a scheduler leave: with them, and the task held in registers,
      // 930 -> 994 clk a tile at head_dim 64, 1,333 -> 1,409 for the short rows)
#pragma unroll 1
      for (int c0 = 0; c0 < G::CO; c0 += 32) {
        uint32_t ov[32];
        WAVEAL_TMEM_LD32(o_addr + c0, ov, 0);
        WAVEAL_TMEM_WAIT_LD32(ov, 0);
        if (c0 == G::CO - 32) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(BAR(B_O_FREE + ob));
        }
        if (q_tok < p.seq_q) {
          uint32_t w[16];
#pragma unroll
          for (int c = 0; c < 32; c += 2) {
            __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(ov[c]) * inv_l, __uint_as_float(ov[c + 1]) * inv_l);
            w[c / 2] = *reinterpret_cast<uint32_t*>(&b2);
          }
          // |O| <= l_tot max|V|: only a large sum (or none) can have led out of fp32's range
          if (!(l_tot > 0.f && l_tot < kCheckSum)) {
            uint32_t top = 0;              // an exponent field of ones in either half of a pair carries into its top bit
#pragma unroll
            for (int c = 0; c < 16; ++c) top |= (w[c] & 0x7F807F80u) + 0x00800080u;
            bad |= (top & 0x80008000u) != 0;
          }
          if ((reinterpret_cast<uintptr_t>(o_ptr) & 31) == 0) {
            // (a store instruction of a warp touches 32 rows and costs the memory pipe per row, not per byte)
#pragma unroll
            for (int c = 0; c < 16; c += 8) st_global_v8(o_ptr + c0 + 2 * c, w + c);
          } else {
#pragma unroll
            for (int c = 0; c < 16; c += 4)
              *reinterpret_cast<uint4*>(o_ptr + c0 + 2 * c) = make_uint4(w[c], w[c + 1], w[c + 2], w[c + 3]);
          }
        }
      }
      if (p.lse && half == 0 && q_tok < p.seq_q) p.lse[(size_t)h * p.seq_q + q_tok] = (m_all + log2f(l_tot) - 0.0028150156f) * 0.6931471805599453f;
      // to the second launch if the sum of a tile left the range (all items' flags were set before B_EX) or a result is not finite
      if ((__any_sync(0xffffffffu, bad) || redo_flag[tslot] == task_no) && lane == 0)
        list_task(p.ws, &redo_listed[tslot], task_no, h, tk->row, tk->row2);
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kPvWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, G::TMEM_COLS);
  }
  if (tid == 0 && mine) {
    const long long dt = clock64() - t_start;
    atomicMax(&p.ws[4], (int)(dt > 0x7fffffffll ? 0x7fffffffll : dt));
  }
}

// The kernel that makes the table also clears the call's counters (the launch before it on the stream has ended);
// tickets are counted from behind those that the CTAs have without asking.
__device__ __forceinline__ void clear_counters(const AttnParams& p) {
  if (blockIdx.x == 0 && threadIdx.x < 8) p.ws[threadIdx.x] = threadIdx.x == 0 ? p.direct : 0;
}

// The last kTailTasks tickets of a call are handed out longest first (1,024 = 7 per SM).  In the planned
// or natural order a long row may start last and leave the other SMs waiting for it: the row lengths of
// the masks in use spread over a factor of ten.  Calls of a few tasks per SM gain most (5 heads of 256
// rows: 655k -> 494k cycles), the largest lose nothing: before the last 1,024 tickets the order is the
// caller's, and no result depends on it.  The tail reads K and V more often than the planned order would (8 heads of 591
// rows: 0.88 GB against 0.58 GB), which costs less than the balance brings also where a head's K+V exceed L2: 1 / 2 / 5
// heads of 2,841 planned rows 2.38 / 5.25 / 13.25 ms, without the tail 3.18 / 5.74 / 13.63 ms.  A histogram of 1,024 lengths is enough (which of two tasks of
// about the same length goes first makes no difference).
constexpr int kTailTasks = 1024;
__device__ __forceinline__ int tail_place(int n, bool live) {            // called by a block of kTailTasks threads
  __shared__ int bins[kTailTasks], warp_sum[kTailTasks / 32], longest;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bins[tid] = 0;
  if (tid == 0) longest = 1;
  __syncthreads();
  const int w = __reduce_max_sync(0xffffffffu, live ? n : 0);
  if (lane == 0) atomicMax(&longest, w);
  __syncthreads();
  // absorbed and empty tasks last.  One atomic per warp and length (rows of one length are common)
  const int bin = kTailTasks - 1 - (n <= 0 ? 0 : (int)((long long)n * (kTailTasks - 1) / longest));
  const unsigned same = __match_any_sync(0xffffffffu, live ? bin : -1 - lane);
  int at = 0;
  if (live && lane == __ffs(same) - 1) at = atomicAdd(&bins[bin], __popc(same));
  at = __shfl_sync(0xffffffffu, at, __ffs(same) - 1) + __popc(same & ((1u << lane) - 1u));
  __syncthreads();
  const int c = bins[tid];
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  const int before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum[lane] : 0);
  bins[tid] = before + incl - c;
  __syncthreads();
  return bins[bin] + at;
}

__global__ void __launch_bounds__(kTailTasks) k_task_table(AttnParams p, int block_k, Task* table) {
  waveal::let_next_kernel_start();
  clear_counters(p);
  // block 0: the last kTailTasks tickets (or all of them); the others the rest in order
  const long long t = blockIdx.x == 0 ? p.first_tail + threadIdx.x : (long long)(blockIdx.x - 1) * kTailTasks + threadIdx.x;
  const bool live = blockIdx.x == 0 ? t < p.total_tasks : t < p.first_tail;
  Task tk{};
  if (live) tk = task_of_ticket(p, block_k, t);
  if (blockIdx.x == 0) {
    const int at = tail_place(tk.n, live);
    if (live) table[p.first_tail + at] = tk;
  } else if (live) {
    table[t] = tk;
  }
}

// 64-row blocks: what k_task_table_pairs<true> leaves k_sort_tail<true> for every 32 positions of a head: [0] tiles in all and of pairs,
// [1] tiles of the longest block on its own and of the longest pair (a single position has no room for it: its [0] says the same).  It
// lies where the list of tasks to compute again (8 bytes a task) has its entries for those positions: that list is empty until the
// first launch.
__device__ __forceinline__ int head_parts(const AttnParams& p) { return (p.m_b + 31) / 32; }
__device__ __forceinline__ int2* part_counts(const AttnParams& p, int h, int pos) {
  return reinterpret_cast<int2*>(p.ws + 8) + (size_t)h * p.m_b + pos;
}

// the same for a table that is there already (64-row blocks: pairs are formed first)
template <bool PICK>
__global__ void __launch_bounds__(kTailTasks) k_sort_tail(AttnParams p, Task* table, Pace pace, int sms) {
  waveal::let_next_kernel_start();
  waveal::wait_for_previous_kernel();
  const long long t = p.first_tail + threadIdx.x;
  const bool live = t < p.total_tasks;
  Task tk{};
  tk.row2 = -1;
  if (live) tk = table[t];
  int n = tk.n;
  bool rows128 = false;
  if constexpr (PICK) {
    // Which kernel: see k_bsattn_fwd_rows64.  Either takes as long as its share of the work an SM, or its longest task.  In products
    // of 64 rows a long pair that starts with the call runs faster than one that the last 1,024 tickets begin with (pace.first_pair;
    // of those 1,024 alone, 2 heads of 700 rows with a long pair among the first took 365 us there instead of 310 in products of 128).
    // (This stands in front of every large call: sums by warp and floats instead of atomics and 64-bit division, and a kernel not picked
    // that leaves from where it waited: 0.8 to 2 us less.)
    __shared__ int sums[5][kTailTasks / 32];          // by warp: tiles in all, of pairs; of the longest block on its own, pair, and pair in the tail
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int all = 0, paired = 0, lone_n = 0, pair_n = 0;
    const int per_head = head_parts(p);
    for (int i = threadIdx.x; i < p.heads * per_head; i += kTailTasks) {
      const int pos = i % per_head * 32;
      const int2* part = part_counts(p, i / per_head, pos);
      const int2 c = part[0], most = pos + 1 < p.m_b ? part[1] : make_int2(c.x - c.y, c.y);
      all += c.x; paired += c.y;
      lone_n = max(lone_n, most.x); pair_n = max(pair_n, most.y);
    }
    all = __reduce_add_sync(0xffffffffu, all);
    paired = __reduce_add_sync(0xffffffffu, paired);
    lone_n = __reduce_max_sync(0xffffffffu, lone_n);
    pair_n = __reduce_max_sync(0xffffffffu, pair_n);
    const int tail_pair_n = __reduce_max_sync(0xffffffffu, tk.row2 >= 0 ? tk.n : 0);
    if (lane == 0) {
      sums[0][warp] = all; sums[1][warp] = paired;
      sums[2][warp] = lone_n; sums[3][warp] = pair_n; sums[4][warp] = tail_pair_n;
    }
    __syncthreads();
    const float share = 1.f / (float)sms;
    const float total = (float)__reduce_add_sync(0xffffffffu, sums[0][lane]) * share, pairs = (float)__reduce_add_sync(0xffffffffu, sums[1][lane]) * share;
    const float lone_most = (float)__reduce_max_sync(0xffffffffu, sums[2][lane]), pair_most = (float)__reduce_max_sync(0xffffffffu, sums[3][lane]);
    const float tail_most = (float)__reduce_max_sync(0xffffffffu, sums[4][lane]);
    const float t128 = pace.rows128 * fmaxf(total, fmaxf(lone_most, pair_most));
    const float t64 = fmaxf(fmaxf(pace.lone * (total - pairs) + pace.pair * pairs, pace.lone * lone_most), fmaxf(pace.first_pair * pair_most, pace.pair * tail_most));
    rows128 = t128 < t64;
    if (tk.row2 >= 0 && !rows128) n *= 2;                     // (a pair: two items a tile)
  }
  const int at = tail_place(n, live);
  if (live) table[p.first_tail + at] = tk;
  if constexpr (PICK) {
    __syncthreads();
    if (threadIdx.x == 0) table[0].pick = rows128;
  }
}

// The same for 64-row query blocks, where two blocks with the very same list share their tiles.
// Candidates:
//  - rows that select every KV block (list length = N_B: rows that attend to everything), wherever
//    they stand: the 1st and 2nd, the 3rd and 4th, ... such row of the head's order form pairs,
//    run at the position of the first of the two;
//  - any other two rows at positions 2i and 2i+1 of the order (Stage 2 of the plan puts rows of
//    equal count side by side).
// A pair is formed only if the two lists are equal entry by entry; the first row keeps the task, the
// second one's ticket is absorbed.
// A block takes 64 consecutive positions of a head.  Its warps compare the lists 32 entries at a time;
// rows that select everything know their number in the head's order from a count over the positions
// before the block's own (a thread each, so the block reads the row lengths of its head once).  One thread
// per row that counted and compared alone took 488 us on 32 heads of 1536 rows, a tenth of them full.
constexpr int kPairRows = 64, kPairThreads = 256;
// COUNT: also what k_sort_tail picks the kernel by (a test in the kernel instead took calls of 80 short rows from 18.6 to 19.7 us)
template <bool COUNT>
__global__ void __launch_bounds__(kPairThreads) k_task_table_pairs(AttnParams p, Task* table, int chunks) {
  __shared__ int s_row[kPairRows], s_lo[kPairRows], s_len[kPairRows];      // (len -1: takes no part)
  __shared__ int s_mate[kPairRows];                 // list start of the candidate partner, -1: none
  __shared__ int s_mate_row[kPairRows], s_mate_pos[kPairRows], s_same[kPairRows];   // its row; its position here, -1: elsewhere
  __shared__ int s_full[kPairRows];                 // positions of the full rows of this block, in order
  __shared__ int s_before, s_prev, s_next, s_n_full;
  waveal::let_next_kernel_start();
  clear_counters(p);
  const int h = blockIdx.x / chunks, c0 = (blockIdx.x - h * chunks) * kPairRows, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const size_t hb = (size_t)h * p.m_b;
  const long long nnz = p.row_ptr[p.total_tasks];
  Task tk{};
  const int pos = c0 + tid;
  const bool live = tid < kPairRows && pos < p.m_b;
  if (tid == 0) { s_before = 0; s_prev = -1; s_next = p.m_b; s_n_full = 0; }
  if (live) tk = make_task(p, 64, h, pos);
  const bool open = live && !tk.pick && tk.len > 0 && !p.no_pairing;
  auto full_at = [&](int ps) {                      // the row at position ps if it selects everything by its length, else -1
    const int r = p.row_order ? p.row_order[hb + ps] : ps;
    return (r < 0 || r >= p.m_b || p.row_ptr[hb + r + 1] - p.row_ptr[hb + r] != p.n_b) ? -1 : r;
  };
  __syncthreads();
  if (tid < kPairRows) {
    s_row[tid] = tk.row; s_lo[tid] = tk.lo; s_len[tid] = open ? tk.len : -1;
    s_mate[tid] = -1; s_mate_pos[tid] = -1; s_same[tid] = 0;
  }
  __syncthreads();
  // ---- full rows of this block in order, and those of the head around it.  All of them count, also
  // malformed ones (every block must number them alike); those form no pair.
  const bool full = open && tk.len == p.n_b;
  if (warp == 0) {
    const bool any = !p.no_pairing;
    const unsigned a = __ballot_sync(0xffffffffu, any && c0 + lane < p.m_b && full_at(c0 + lane) >= 0);
    const unsigned b = __ballot_sync(0xffffffffu, any && c0 + lane + 32 < p.m_b && full_at(c0 + lane + 32) >= 0);
    const unsigned below = (1u << lane) - 1u;
    if (a >> lane & 1u) s_full[__popc(a & below)] = lane;
    if (b >> lane & 1u) s_full[__popc(a) + __popc(b & below)] = lane + 32;
    if (lane == 0) s_n_full = __popc(a) + __popc(b);
  }
  __syncthreads();
  const int n_full = s_n_full;
  if (n_full > 0) {
    int before = 0, prev = -1, next = p.m_b;
#pragma unroll 4
    for (int ps = tid; ps < p.m_b; ps += kPairThreads) {
      if (ps >= c0 && ps < c0 + kPairRows) continue;
      if (full_at(ps) < 0) continue;
      if (ps < c0) { ++before; prev = max(prev, ps); } else { next = min(next, ps); }
    }
    before = __reduce_add_sync(0xffffffffu, before);
    prev = __reduce_max_sync(0xffffffffu, prev);
    next = __reduce_min_sync(0xffffffffu, next);
    if (lane == 0) { atomicAdd(&s_before, before); atomicMax(&s_prev, prev); atomicMin(&s_next, next); }
    __syncthreads();
    if (tid < n_full) {
      const int e = s_full[tid], k = ((s_before + tid) ^ 1) - s_before;      // the partner's number here
      int mrow = -1, mpos = -1;
      if (k >= 0 && k < n_full) { mpos = s_full[k]; mrow = s_len[mpos] == p.n_b ? s_row[mpos] : -1; }
      else if (k < 0 && s_prev >= 0) mrow = full_at(s_prev);
      else if (k >= n_full && s_next < p.m_b) mrow = full_at(s_next);
      if (mrow >= 0 && s_len[e] == p.n_b) { s_mate[e] = p.row_ptr[hb + mrow]; s_mate_row[e] = mrow; s_mate_pos[e] = mpos; }
    }
  }
  if (open && !full && pos + 1 - 2 * (pos & 1) < p.m_b && s_len[tid ^ 1] == tk.len) {
    s_mate[tid] = s_lo[tid ^ 1]; s_mate_row[tid] = s_row[tid ^ 1]; s_mate_pos[tid] = tid ^ 1;
  }
  __syncthreads();
  // ---- comparisons: a warp per pair, by the first of the two where both are here
  for (int e = warp; e < kPairRows; e += kPairThreads / 32) {
    const int lo2 = s_mate[e], mpos = s_mate_pos[e], len = s_len[e], lo = s_lo[e];
    if (lo2 < 0 || mpos >= 0 && mpos < e || s_mate_row[e] == s_row[e] || (long long)lo2 + len > nnz) continue;
    // the first 32 entries tell most pairs apart; behind them 256 at a time
    bool same = __all_sync(0xffffffffu, lane >= len || p.kv_idx[lo + lane] == p.kv_idx[lo2 + lane]);
    for (int i0 = 32; i0 < len && same; i0 += 256) {
      bool eq = true;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int i = i0 + k * 32 + lane;
        eq &= i >= len || p.kv_idx[lo + i] == p.kv_idx[lo2 + i];
      }
      same = __all_sync(0xffffffffu, eq);
    }
    if (lane == 0) { s_same[e] = same; if (mpos >= 0) s_same[mpos] = same; }
  }
  __syncthreads();
  if (live && s_same[tid]) {
    const int mpos = s_mate_pos[tid];
    // the first of the two in the order: partners elsewhere stand before (odd number) or behind (even)
    bool first = mpos > tid;
    if (mpos < 0) {
      int k = 0;
      while (s_full[k] != tid) ++k;
      first = ((s_before + k) & 1) == 0;
    }
    if (first) tk.row2 = s_mate_row[tid];
    else tk.n = kAbsorbed;
  }
  tk.pick = 0;
  if (live) table[p.interleaved ? (long long)pos * p.heads + h : (long long)hb + pos] = tk;
  if (COUNT && tid < kPairRows) {
    const int n = live ? max(tk.n, 0) : 0, pair_n = live && tk.row2 >= 0 ? n : 0, lone_n = n - pair_n;
    const int2 sum = make_int2(__reduce_add_sync(0xffffffffu, n), __reduce_add_sync(0xffffffffu, pair_n));
    const int2 most = make_int2(__reduce_max_sync(0xffffffffu, lone_n), __reduce_max_sync(0xffffffffu, pair_n));
    if (lane == 0 && live) {
      part_counts(p, h, pos)[0] = sum;
      if (pos + 1 < p.m_b) part_counts(p, h, pos)[1] = most;
    }
  }
}

// ------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// bf16 tensor [heads][seq][head_dim] with element strides {head, token}; box = 64 (or 32) columns x rows
waveal_status make_map(CUtensorMap* tm, const void* base, int head_dim, int seq, int heads, long long stride_h,
                       long long stride_t, int box_rows, const char* what, int box_cols = 64) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return waveal::fail(WAVEAL_ERR_CUDA, "cuTensorMapEncodeTiled entry point not available");
  cuuint64_t dims[3] = {(cuuint64_t)head_dim, (cuuint64_t)seq, (cuuint64_t)heads};
  cuuint64_t strides[2] = {(cuuint64_t)stride_t * 2, (cuuint64_t)stride_h * 2};
  cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return waveal::fail(WAVEAL_ERR_CUDA, "tensor map for %s rejected (CUresult %d)", what, (int)r);
  return WAVEAL_OK;
}

waveal_status check_desc(const waveal_attn_desc* d) {
  if (!d) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "desc is NULL");
  if (d->heads <= 0 || d->seq_q <= 0 || d->seq_kv <= 0)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "heads, seq_q and seq_kv must be positive");
  if (d->head_dim != 64 && d->head_dim != 128)
    return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "head_dim %d (supported: 64, 128)", d->head_dim);
  if (d->block_q != d->block_kv || (d->block_q != 64 && d->block_q != 128))
    return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "block %dx%d (supported: 64x64, 128x128)", d->block_q, d->block_kv);
  const int64_t* strides[4] = {d->q_stride, d->k_stride, d->v_stride, d->o_stride};
  for (int i = 0; i < 4; ++i) {
    if (strides[i][1] < d->head_dim || strides[i][0] < 0)
      return waveal::fail(WAVEAL_ERR_INVALID_ARG, "token stride must be >= head_dim and head stride >= 0");
    if (strides[i][0] % 8 || strides[i][1] % 8)
      return waveal::fail(WAVEAL_ERR_INVALID_ARG, "strides must be multiples of 8 elements (16 bytes)");
  }
  return WAVEAL_OK;
}

// byte offset of the ticket table in the workspace (32-byte aligned, behind header and redo list)
long long table_offset(long long tasks) { return (32 + 8 * tasks + 31) / 32 * 32; }

template <int BLOCK, int D>
waveal_status launch(const waveal_attn_desc* d, const void* Q, const void* K, const void* V, AttnParams& p,
                     int sms, cudaStream_t st) {
  using G = Geo<BLOCK, D>;
  CUtensorMap tq, tk, tv, tk2, tv2, to;
  waveal_status s;
  if ((s = make_map(&tq, Q, D, d->seq_q, d->heads, d->q_stride[0], d->q_stride[1], BLOCK, "Q")) != WAVEAL_OK) return s;
  if ((s = make_map(&tk, K, D, d->seq_kv, d->heads, d->k_stride[0], d->k_stride[1], BLOCK, "K")) != WAVEAL_OK) return s;
  if ((s = make_map(&tv, V, D, d->seq_kv, d->heads, d->v_stride[0], d->v_stride[1], BLOCK, "V")) != WAVEAL_OK) return s;
  if (BLOCK == 128) {                     // (each kernel reads the maps of its own block size)
    tk2 = tk; tv2 = tv;
    if ((s = make_map(&to, p.O, D, d->seq_q, d->heads, d->o_stride[0], d->o_stride[1], 32, "O", D / 2)) != WAVEAL_OK) return s;
  } else {
    if ((s = make_map(&tk2, K, D, d->seq_kv, d->heads, d->k_stride[0], d->k_stride[1], 128, "K (128-row boxes)")) != WAVEAL_OK) return s;
    if ((s = make_map(&tv2, V, D, d->seq_kv, d->heads, d->v_stride[0], d->v_stride[1], 128, "V (128-row boxes)")) != WAVEAL_OK) return s;
    to = tq;
  }
  WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_bsattn_fwd<BLOCK, D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES));
  WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_bsattn_fwd<BLOCK, D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM_BYTES));
  long long grid = p.total_tasks < sms ? p.total_tasks : sms;
  Task* table = reinterpret_cast<Task*>(reinterpret_cast<char*>(p.ws) + table_offset(p.total_tasks));
  p.table = table;
  bool pick = false;
  p.redo_pass = 0;
  p.wait_limit = kTimeoutCycles;
  p.drop_tile = 0;
  if (d->flags & WAVEAL_ATTN_SELFTEST_LOST_TILE) { p.wait_limit = kSelfTestCycles; p.drop_tile = 1; }
  p.no_pairing = (d->flags & WAVEAL_ATTN_NO_ROW_PAIRING) ? 1 : 0;
  // From two tasks an SM on, the first task of every CTA is the ticket of its own number: it runs while the table is made
  // (10 us: 1,320 tasks of 17 tiles 196.7 -> 187.2 us a call, 1,280 of 38 386 -> 373, 3,816 of 24 at head_dim 64 501 -> 494).  Those tickets stay out of the sorted tail.  (64-row blocks: which blocks share a tile is known from the table only.)
  p.first_tail = p.total_tasks > kTailTasks ? p.total_tasks - kTailTasks : 0;
  p.direct = 0;
  if (BLOCK == 128 && p.total_tasks >= 2 * sms && !(d->flags & WAVEAL_ATTN_ONLINE_MAX_ONLY)) {
    p.direct = (int)grid;
    if (p.first_tail < grid) p.first_tail = grid;
  }
  int launches = 1;
  if (BLOCK == 64) {
    const int chunks = (p.m_b + kPairRows - 1) / kPairRows;
    // The choice costs a launch and its counts, of which the host knows only the most that a mask can select.  us a call with products of
    // 128 rows alone / with the choice, lists of 3 / 12 / 40 % of the blocks, none in pairs, and of all blocks (all in pairs: the choice falls
    // on products of 128), by the tiles an SM that the lists may have, head_dim 128:
    //    68 (2 heads of 100 rows): 24.7 / 24.7   30.9 / 30.9   50.9 / 45.6    62.5 / 67.7
    //   135 (1 head of 200):       26.7 / 26.8   39.1 / 37.0   78.9 / 65.8   102.6 / 107.5
    //   219 (2 heads of 180):      30.9 / 30.9   49.5 / 44.5   101.7 / 83.5  160.2 / 165.6
    //   304 (1 head of 300):       35.0 / 32.9   62.2 / 53.7   150.1 / 114.8 253.1 / 258.0
    // (head_dim 64: 56.8 -> 48.5 at 132 and 40 %, 102.6 -> 80.1 at 298; all in pairs + 4.5 .. 5).  The line lies where the 5 us are 2 to 4 %
    // of a dense call; below it a call of lone blocks gives away up to a quarter.  From the line on the sparsest lists repay the choice
    // (3 heads of 180 rows, 328: rows of 2 blocks 30.8 / 30.9, of 6 37.0 / 36.4, of 12 46.4 / 43.0; head_dim 64 28.6 / 29.8, 32.9 / 32.9, 41.0 / 39.0),
    // short pairs do not (8 heads of 200 rows of 10 blocks, all in pairs, head_dim 64: 56.9 / 60.7).
    const bool many = p.total_tasks > sms;            // (else all tasks start at once)
    pick = many && !(d->flags & WAVEAL_ATTN_ONLINE_MAX_ONLY) && p.total_tasks * ((p.n_b + 1) / 2) >= kRows64Tiles * sms;
    (pick ? k_task_table_pairs<true> : k_task_table_pairs<false>)<<<(unsigned)((long long)p.heads * chunks), kPairThreads, 0, st>>>(p, table, chunks);
    if (many) {
      WAVEAL_CUDA_OK(cudaGetLastError());
      WAVEAL_CUDA_OK(waveal::launch_chained(pick ? k_sort_tail<true> : k_sort_tail<false>, dim3(1), kTailTasks, 0, st, p, table, Geo64<D>::PACE, sms));
      ++launches;
    }
  } else {
    k_task_table<<<(unsigned)(1 + (p.first_tail + kTailTasks - 1) / kTailTasks), kTailTasks, 0, st>>>(p, BLOCK, table);
  }
  WAVEAL_CUDA_OK(cudaGetLastError());
  if (d->flags & WAVEAL_ATTN_ONLINE_MAX_ONLY) {
    p.redo_pass = 0;
    WAVEAL_CUDA_OK(waveal::launch_chained(k_bsattn_fwd<BLOCK, D, false>, dim3((unsigned)grid), kThreads, G::SMEM_BYTES, st, tq, tk, tv, tk2, tv2, to, p));
    waveal::launch_counter() = launches + 1;
    return WAVEAL_OK;
  }
  // first pass: reference fixed after the first tile of a task; second pass: the tasks the
  // first one listed (normally none: its CTAs leave at once), max of every block
  p.redo_pass = 0;
  if constexpr (BLOCK == 64) {
    // k_sort_tail says which kernel is quicker; the other one leaves at once
    if (pick) {
      p.choose = 1;
      WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_bsattn_fwd_rows64<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, Geo64<D>::SMEM_BYTES));
      WAVEAL_CUDA_OK(waveal::launch_chained(k_bsattn_fwd_rows64<D>, dim3((unsigned)grid), kThreads64, Geo64<D>::SMEM_BYTES, st, tq, tk, tv, tk2, tv2, p));
      ++launches;
    }
  }
  WAVEAL_CUDA_OK(waveal::launch_chained(k_bsattn_fwd<BLOCK, D, true>, dim3((unsigned)grid), kThreads, G::SMEM_BYTES, st, tq, tk, tv, tk2, tv2, to, p));
  p.redo_pass = 1;
  p.direct = 0;
  WAVEAL_CUDA_OK(waveal::launch_chained(k_bsattn_fwd<BLOCK, D, false>, dim3((unsigned)grid), kThreads, G::SMEM_BYTES, st, tq, tk, tv, tk2, tv2, to, p));
  waveal::launch_counter() = launches + 2;
  return WAVEAL_OK;
}

}  // namespace

extern "C" waveal_status waveal_bsattn_workspace_bytes(const waveal_attn_desc* desc, size_t* bytes) {
  waveal_status s = check_desc(desc);
  if (s != WAVEAL_OK) return s;
  if (!bytes) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "bytes is NULL");
  // 32 bytes of counters and flags, one (head, query block) pair per task for the redo list,
  // then the 32-byte task of every ticket
  const long long tasks = (long long)desc->heads * ((desc->seq_q + desc->block_q - 1) / desc->block_q);
  *bytes = (size_t)((table_offset(tasks) + 32 * tasks + 255) / 256 * 256);
  return WAVEAL_OK;
}

extern "C" waveal_status waveal_bsattn_fwd(const waveal_attn_desc* d, const void* Q, const void* K, const void* V,
                                           void* O, float* lse, const int32_t* kv_row_ptr,
                                           const int32_t* kv_block_indices, const int32_t* row_order, float scale,
                                           void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream) {
  waveal_status s = check_desc(d);
  if (s != WAVEAL_OK) return s;
  if (!Q || !K || !V || !O) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "Q, K, V and O are required");
  if (!kv_row_ptr || !kv_block_indices) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "index lists are required");
  if (!waveal::aligned(Q, 16) || !waveal::aligned(K, 16) || !waveal::aligned(V, 16) || !waveal::aligned(O, 16))
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "Q, K, V and O must be 16-byte aligned");
  size_t ws_need = 0;
  if ((s = waveal_bsattn_workspace_bytes(d, &ws_need)) != WAVEAL_OK) return s;
  if (!ws || ws_bytes < ws_need) return waveal::fail(WAVEAL_ERR_WORKSPACE, "workspace of %zu bytes needed", ws_need);
  if (!waveal::aligned(ws, 16)) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "workspace must be 16-byte aligned");
  if (!(scale == scale) || std::isinf(scale)) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "scale is not finite");
  int dev = 0, sms = 0, major = 0;
  WAVEAL_CUDA_OK(cudaGetDevice(&dev));
  WAVEAL_CUDA_OK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
  if (major != 10) return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "device compute capability %d.x; sm_100a is required", major);
  WAVEAL_CUDA_OK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  AttnParams p{};
  p.O = static_cast<__nv_bfloat16*>(O);
  p.lse = lse;
  p.row_ptr = kv_row_ptr; p.kv_idx = kv_block_indices; p.row_order = row_order;
  p.ws = static_cast<int*>(ws); p.dev_status = dev_status;
  p.o_stride_h = d->o_stride[0]; p.o_stride_t = d->o_stride[1];
  p.heads = d->heads;
  p.m_b = (d->seq_q + d->block_q - 1) / d->block_q;
  p.n_b = (d->seq_kv + d->block_kv - 1) / d->block_kv;
  p.seq_q = d->seq_q; p.seq_kv = d->seq_kv;
  p.interleaved = d->order_heads_interleaved ? 1 : 0;
  p.total_tasks = (long long)d->heads * p.m_b;
  const float sc = scale > 0.f ? scale : 1.0f / sqrtf((float)d->head_dim);
  p.sl2 = sc * 1.4426950408889634f;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (d->block_q == 128 && d->head_dim == 128) return launch<128, 128>(d, Q, K, V, p, sms, st);
  if (d->block_q == 64 && d->head_dim == 128) return launch<64, 128>(d, Q, K, V, p, sms, st);
  if (d->block_q == 64 && d->head_dim == 64) return launch<64, 64>(d, Q, K, V, p, sms, st);
  if (d->block_q == 128 && d->head_dim == 64) return launch<128, 64>(d, Q, K, V, p, sms, st);
  return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "no kernel for block %d, head_dim %d", d->block_q, d->head_dim);
}

// Window-score kernel for bf16 inputs on the sm_100a tensor cores: one persistent
// launch per layer runs both passes over the keys.
//
//   pass A (rows)   D[row][key]  = Q K^T : one thread owns one window row and keeps
//                   its running max / sum (softmax denominator, Eq. 2) and
//                   sum e*log2(e) (row entropy, Eq. 4).
//   pass B (cols)   D[key][row]  = K Q^T : one thread owns one key and reduces its
//                   normalised column over the window rows: group-mean attention,
//                   Mean + gamma Var (Eq. 11) and the per-head Var (Eq. 5).
//
// K tiles of 128 keys stream through shared memory with TMA (no multicast), are
// multiplied against the resident window queries with tcgen05.mma (bf16 operands,
// fp32 accumulators in tensor memory) and reduced on chip; the S_w x N score matrix
// never reaches HBM.
//
// Schedule.  The (request, KV head) pairs of a layer are grouped into waves of at
// most kWaveBytes of K.  Every CTA owns the same slice of a wave in both passes and runs
//     A(wave 0), A(wave 1), B(wave 0), A(wave 2), B(wave 1), ... , B(last wave)
// so pass B re-reads a wave's K from L2 shortly after pass A brought it in, and DRAM
// sees K once.  Pass B of a pair needs the pair's softmax denominators, i.e. every
// CTA's pass-A partial rows.  The merge is spread over the grid by rows: the merger warp
// of CTA (pair * rows + r) % grid waits for row r's partials, merges them and hands the row to all
// CTAs.  The pass A of the next wave sits between a pair's pass A and its pass B, so the
// denominators are normally there in time.
//
// Exchange.  Rows that go from CTA to CTA carry the mark of their launch beside the data, in one 16- or 8-byte
// access: the reader polls the data itself.  With counters (fence, count, poll, load, and the same again for
// the merged rows) the denominators came 7 to 12 us after the last CTA's pass A; they come after 4.
//
// Bound.  A key tile of 128 keys and 128 rows is 16 384 exponentials per pass: 1024 cycles of the special-function
// unit.  A statistics warp takes 3400 to 3700 cycles for its share of three tiles (3072 at the unit's rate) with the
// next TMEM columns on their way during the arithmetic; with a load, a wait and a check per 32 columns it
// took 3800 (pass B) and 4600 (pass A).  128K layer, 128 CTAs: 206 k cycles per launch before, 198 k now.  Long
// prompts run into the device's power limit (1.75 instead of 1.965 GHz).
//
// Warp roles in a CTA of 512 threads: warps 0..11 are "statistics" warps in three groups of
// four (a group takes every third accumulator tile, a warp owns 32 of its TMEM lanes and writes
// its own partial results; warps meet only where partial rows are exchanged, see xrow_slot), warp 12 issues TMA loads, warp 13 owns the
// tensor-memory allocation and issues the MMAs (both as converged warps with an elected lane),
// warp 14 merges rows, warp 15 stages the denominators of the next pass-B op in shared memory.  Every wait
// (mbarrier or exchanged row) is bounded; a timed-out wait raises CAKE_ERR_TIMEOUT and the CTA
// drains and exits.
#include "cake_internal.cuh"

#include <cuda.h>
#include <math_constants.h>

#include <algorithm>
#include <cstring>
#include <vector>

namespace cake {
namespace {

constexpr int TILE = 128;            // keys per tile
constexpr int STAGES = 4;            // K tiles in flight
constexpr int NBUF = 4;              // accumulator buffers of 128 columns, all of tensor memory: one more than there are
                                     // groups, so that a group's next tile is multiplied while it holds this one
constexpr int NWG = kScoreGroups;    // statistics warp groups
static_assert((NBUF & (NBUF - 1)) == 0, "a tile's buffer and phase are bit fields of its number");
constexpr int STAT_THREADS = NWG * 128;
constexpr int TC_THREADS = STAT_THREADS + 128;  // + TMA, MMA, row-merger and denominator warps
constexpr int WARP_TMA = NWG * 4, WARP_MMA = NWG * 4 + 1, WARP_MERGE = NWG * 4 + 2,
              WARP_LSE = NWG * 4 + 3;
constexpr int NSTATW = NWG * 4;      // statistics warps
constexpr int SLAB_BYTES = TILE * 128;   // one 64-element slab of a 128-row tile
constexpr long long kSpinLimit = 4000000000ll;   // default cycles (~2 s) before a wait gives up
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kTileSumMax = 1.2676506e30f;    // pass A: a tile whose sum is beyond 2^100 is taken again from its maxima,
constexpr float kShiftSum = 256.f;              // one beyond this moves the row's reference up afterwards
constexpr int64_t kWaveBytes = 32ll << 20;
constexpr int kLseStride = 16;        // merged rows lie a line of L2 (128 bytes) apart, see lse2
constexpr int kDirectSegs = 40;       // segments of a pair up to which every CTA merges its rows for itself

struct TcParams {
  const ScoreOp* ops;
  const int32_t* cta_op;        // [n_cta + 1]
  const int32_t* group_begin;   // [n_groups + 1] first pair of every merge group; null: every merge_ways pairs
  int n_groups;
  const int32_t* pair_aseg;     // [pairs + 1] pass-A segment ranges per pair
  int both;                     // 0: pass B alone
  uint32_t tag, want;           // mark of this launch's exchanged rows, and the one that readers wait for
  uint2* lse2;                  // [pair][128] in tile row order r' = i*G + h, kLseStride apart: base-2 log-sum-exp, tag.  A
                                // line that several CTAs write while others poll it costs a round trip per write
  const float* lse_ext;         // caller's natural-log LSE [req][H_q][S_w], or null
  float4* rowpart;              // pass A out: [A-segment][group][128], see pack_part
  float* raw;                   // pass B out: [H_kv][T]
  float* colpart;               // pass B out: [B-segment][statistics warp][G][2]
  float* hrow;                  // [pair][128] sum_j p log2 p of every window row
  int32_t* status;
  long long spin_limit;         // cycles after which a wait gives up and raises CAKE_ERR_TIMEOUT
  int n_pairs;
  int Hkv, Hq, Sw, rows, d;
  float scale2, inv_scale2, gamma, bessel;
  int ind_mode;                 // CAKE_IND_*
  int merge_ways;               // rows the merger warp merges side by side: 1, or 2 to 32 when pairs are short
  int reps;                     // copies of the window rows in a pass-A tile: 128 / rows for 32 and 64 rows, else 1
};

// ------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
               "@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.b32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait of a whole warp: false (and the sticky status set) if the phase never completes.  Its lanes agree: what
// follows (TMEM loads, votes, elected issue) is the whole warp's, and a phase may complete just as the limit is reached.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int32_t* status,
                                          long long limit) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
    if (__any_sync(0xffffffffu, clock64() - t0 > limit)) {
      atomicCAS(status, 0, CAKE_ERR_TIMEOUT);
      return false;
    }
  }
  return true;
}
// 3-D tiled TMA load with an L2 eviction-priority hint: a whole key tile (both 64-element slabs)
// in one copy.
__device__ __forceinline__ void tma_load_3d_hint(void* dst, const CUtensorMap* map, uint64_t* bar,
                                                 int c0, int c1, int c2, uint64_t policy) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5}], [%2], %6;\n}"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int c0, int c1, int c2) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];\n}"
      ::"l"(map), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0,
                                            int c1, int c2, int c3) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];\n}"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// The MMA and TMA warps run converged, all 32 lanes executing the same loop, and one elected lane
// issues each asynchronous instruction.  Issued from inside a one-lane branch the operands of
// every tcgen05.mma are moved to uniform registers one by one and an M128 x N128 x K16 MMA costs
// about 70 cycles to issue, more than the 64 cycles it takes to execute; from a converged warp
// the descriptor arithmetic stays in the uniform datapath and the tensor pipe sets the pace.
// Descriptors differ only in the 14-bit address field of their low word, the high word (stride,
// version, swizzle) is a constant, and the accumulate flag is an immediate.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);   // SBO, version 1, SWIZZLE_128B
template <int kAcc>
__device__ __forceinline__ void umma_ss(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p, e;\n.reg .b64 da, db;\nsetp.ne.b32 p, %4, 0;\nelect.sync _|e, 0xffffffff;\n"
      "mov.b64 da, {%1, %5};\nmov.b64 db, {%2, %5};\n"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}"
      ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(idesc), "n"(kAcc), "r"(kDescHi)
      : "memory");
}
// The same with an explicit high descriptor word: operands that are not in the 128-byte swizzle.
template <int kAcc>
__device__ __forceinline__ void umma_ss_hi(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc,
                                           uint32_t hi) {
  asm volatile(
      "{\n.reg .pred p, e;\n.reg .b64 da, db;\nsetp.ne.b32 p, %4, 0;\nelect.sync _|e, 0xffffffff;\n"
      "mov.b64 da, {%1, %5};\nmov.b64 db, {%2, %5};\n"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}"
      ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(idesc), "n"(kAcc), "r"(hi)
      : "memory");
}
// Pass B folds the rows' log-sum-exps into the contraction: one more K = 16 step whose key-side
// operand holds 1 in its first three columns and whose row-side operand holds -lse / scale split
// into three bf16 terms, so the accumulator is (q.k - lse/scale) and the statistics warps neither
// load nor subtract anything per logit.  These two operands are 128 rows x 16 bf16 in the
// K-major layout without swizzle: 8-row x 16-byte core matrices, the two core matrices of a row
// group 128 bytes apart (leading-dimension offset), row groups 256 bytes apart (stride offset).
constexpr uint32_t kExtBytes = 128 * 32;
constexpr uint32_t kExtDescHi = (256u >> 4) | (1u << 14);            // SBO, version 1, no swizzle
constexpr uint32_t kExtDescLoLbo = (128u >> 4) << 16;                // LBO field of the low word
__device__ __forceinline__ uint32_t ext_row_offset(int r) { return (uint32_t)((r >> 3) * 256 + (r & 7) * 16); }

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
               "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}"
               ::"r"(smem_u32(bar)) : "memory");
}
// Starts the load of 16 consecutive fp32 columns of this thread's TMEM lane; the registers
// are valid only after tmem_ld_wait on the same array.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// Waits for the thread's outstanding TMEM loads.  The registers pass through the statement so
// that no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
// Columns [lo, hi) of this thread's TMEM lane, 16 at a time: f(chunk) while the next chunk is on its way, so
// that a warp has exponentials to issue all the time; `loaded` is called once all columns are in registers.
template <typename F, typename L>
__device__ __forceinline__ void for_columns(uint32_t taddr, int lo, int hi, F f, L loaded) {
  uint32_t r0[16], r1[16];
  tmem_ld16_issue(taddr + lo, r0);
#pragma unroll 1
  for (int c = lo; c < hi; c += 32) {
    tmem_ld_wait(r0);
    if (c + 16 < hi) tmem_ld16_issue(taddr + c + 16, r1);
    else loaded();
    f(r0);
    if (c + 16 >= hi) break;
    tmem_ld_wait(r1);
    if (c + 32 < hi) tmem_ld16_issue(taddr + c + 32, r0);
    else loaded();
    f(r1);
  }
}
__device__ __forceinline__ float max_or_nan(float a, float b) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Two fp32 values in one 64-bit register and the packed fp32x2 arithmetic on them: one
// instruction issue for two FMAs or adds.  The statistics loops are bound by issue slots, not by
// the FMA pipe, so halving their FFMA/FADD count matters although the pipe rate is the same.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__device__ __forceinline__ uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Rows that CTAs exchange carry the mark of the launch that wrote them, in the same 16 (or 8) bytes as the
// data: they are written and read as one access each, so a reader that sees the mark has the data, and
// neither side needs a fence, a counter or a second trip.
__device__ __forceinline__ void st_row16(float4* p, float4 v) {
  asm volatile("{\n.reg .b128 t;\n.reg .b64 lo, hi;\nmov.b64 lo, {%1, %2};\nmov.b64 hi, {%3, %4};\nmov.b128 t, {lo, hi};\n"
               "st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ float4 ld_row16(const void* p) {
  float4 v;
  asm volatile("{\n.reg .b128 t;\n.reg .b64 lo, hi;\nld.relaxed.gpu.global.b128 t, [%4];\nmov.b128 {lo, hi}, t;\n"
               "mov.b64 {%0, %1}, lo;\nmov.b64 {%2, %3}, hi;\n}" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint2 ld_row8(const uint2* p) {
  uint2 v;
  asm volatile("{\n.reg .b64 t;\nld.relaxed.gpu.global.b64 t, [%2];\nmov.b64 {%0, %1}, t;\n}" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_row8(uint2* p, uint32_t a, uint32_t b) {
  asm volatile("{\n.reg .b64 t;\nmov.b64 t, {%1, %2};\nst.relaxed.gpu.global.b64 [%0], t;\n}" ::"l"(p), "r"(a), "r"(b) : "memory");
}

struct Smem {
  uint8_t* q;          // 2 buffers x (2 slabs x 128 rows x 128 B)
  uint8_t* k;          // STAGES x (2 slabs x 128 rows x 128 B)
  uint64_t* full;      // [STAGES]
  uint64_t* empty;     // [STAGES]
  uint64_t* acc_full;  // [NBUF]
  uint64_t* acc_empty; // [NBUF]
  uint64_t* q_full;    // [2]
  uint64_t* q_empty;   // [2]
  uint64_t* lse_full;  // [2]
  uint64_t* lse_free;  // [2]
  uint32_t* tmem_holder;
  uint8_t* ext_a;      // the constant key-side operand of the extra K step of pass B
  uint8_t* ext_b;      // [2] its row-side operand: -lse/scale of the current / next pass-B op
  float4* xrow;        // [2][NWG][128] partial rows of a group: copies of a row in pass A, then (direct merge) the
                       //   group's share of a pair's partials of a pass-B op; slots by xrow_slot
  ScoreOp* ops;        // [kSmemOps] the first ops of this CTA's program
};

constexpr size_t kQBytes = 2 * SLAB_BYTES;
constexpr int kSmemOps = 128;        // ops of a CTA's program kept in shared memory
constexpr size_t kSmemBytes = 1024 /*align*/ + 2 * kQBytes + (size_t)STAGES * 2 * SLAB_BYTES + 320 +
                              128 + 3 * kExtBytes + 2 * NWG * 128 * sizeof(float4) + kSmemOps * sizeof(ScoreOp) + 64;
static_assert(kSmemBytes <= 227 * 1024, "a CTA has 227 KB of shared memory");

__device__ __forceinline__ Smem carve(uint8_t* base) {
  Smem s;
  uint8_t* p = (uint8_t*)(((uintptr_t)base + 1023) & ~(uintptr_t)1023);
  s.q = p;                    p += 2 * kQBytes;
  s.k = p;                    p += (size_t)STAGES * 2 * SLAB_BYTES;
  s.full = (uint64_t*)p;      p += 8 * STAGES;
  s.empty = (uint64_t*)p;     p += 8 * STAGES;
  s.acc_full = (uint64_t*)p;  p += 8 * NBUF;
  s.acc_empty = (uint64_t*)p; p += 8 * NBUF;
  s.q_full = (uint64_t*)p;    p += 16;
  s.q_empty = (uint64_t*)p;   p += 16;
  s.lse_full = (uint64_t*)p;  p += 16;
  s.lse_free = (uint64_t*)p;  p += 16;
  s.tmem_holder = (uint32_t*)p; p += 8;
  p = (uint8_t*)(((uintptr_t)p + 15) & ~(uintptr_t)15);
  p = (uint8_t*)(((uintptr_t)p + 127) & ~(uintptr_t)127);
  s.ext_a = p;                p += kExtBytes;
  s.ext_b = p;                p += 2 * kExtBytes;
  s.xrow = (float4*)p;        p += 2 * NWG * 128 * sizeof(float4);
  s.ops = (ScoreOp*)p;
  return s;
}

// A partial softmax row (m, z_all, z_win, w) with base-2 exponents: sums of e = 2^(logit2 - m) over all keys of the
// segment and over those of the window, and w = sum over the observed keys of e * (logit2 - m).  m is any reference: on
// its way to other CTAs a row has the one that puts z_all into [1, 2) (a scaling by a power of two), and the
// launch's mark takes the place of z_all's exponent.  No keys: m = -inf and z_all = 0.  A sum that is not finite
// (whatever m): m = inf, which makes the merged row NaN.
__device__ __forceinline__ float4 pack_part(float m, float z, float zwin, float w, uint32_t tag) {
  const uint32_t zb = __float_as_uint(z);
  const int k = (int)(zb >> 23) - 127;
  const float f = __uint_as_float((uint32_t)(127 - k) << 23);
  float4 o = make_float4(m + (float)k, __uint_as_float((zb & 0x7FFFFFu) | (tag << 23)), zwin * f, fmaf(-(float)k, z - zwin, w) * f);
  if (!(z <= 1e38f)) o.x = CUDART_INF_F;
  else if (m == -CUDART_INF_F) o = make_float4(m, __uint_as_float(tag << 23), 0.f, 0.f);
  else if (k < -120) o.x = CUDART_INF_F;
  return o;
}
__device__ __forceinline__ bool part_tagged(const float4& v, uint32_t want) { return (__float_as_uint(v.y) >> 23) == want; }
__device__ __forceinline__ float4 unpack_part(float4 v) {
  v.y = v.x == -CUDART_INF_F ? 0.f : __uint_as_float((__float_as_uint(v.y) & 0x7FFFFFu) | 0x3F800000u);
  return v;
}

// Merge of two partial rows.
__device__ __forceinline__ float4 merge_rows(float4 a, float4 b) {
  if (b.x == -CUDART_INF_F && b.y == 0.f) return a;
  if (a.x == -CUDART_INF_F && a.y == 0.f) return b;
  const float mn = fmaxf(a.x, b.x);
  const float fa = exp2f(a.x - mn), fb = exp2f(b.x - mn);
  float4 o;
  o.x = mn;
  o.y = a.y * fa + b.y * fb;
  o.z = a.z * fa + b.z * fb;
  o.w = fa * fmaf(a.x - mn, a.y - a.z, a.w) + fb * fmaf(b.x - mn, b.y - b.z, b.w);
  return o;
}

// The same for a batch at once: the largest reference first, then independent terms.
template <int K>
__device__ __forceinline__ float4 merge_batch(float4 acc, const float4 (&v)[K]) {
  float m = acc.x;
#pragma unroll
  for (int u = 0; u < K; ++u) m = fmaxf(m, v[u].x);
  if (m == -CUDART_INF_F) return acc;
  auto term = [&](const float4& t, float4& o) {
    const float d = t.x == -CUDART_INF_F ? 0.f : t.x - m, f = t.x == -CUDART_INF_F ? 0.f : exp2f(d);
    o.y = fmaf(t.y, f, o.y);
    o.z = fmaf(t.z, f, o.z);
    o.w = fmaf(f, fmaf(d, t.y - t.z, t.w), o.w);
  };
  float4 o = make_float4(m, 0.f, 0.f, 0.f);
  term(acc, o);
#pragma unroll
  for (int u = 0; u < K; ++u) term(v[u], o);
  return o;
}

// Loads up to K partial rows per lane, at `stride` from one another, `count` of them in this lane (0 or less: none),
// and waits until all have come, by the whole warp.  The first of every lane's is waited for alone, so that a
// long wait costs the memory system little.  False (and the status set) if they do not come.
template <int K>
__device__ __forceinline__ bool wait_parts(const float4* p, int64_t stride, int count, uint32_t want, float4 (&v)[K],
                                           int32_t* status, long long limit) {
  const long long t0 = clock64();
  uint32_t missing = 0;
#pragma unroll
  for (int u = 0; u < K; ++u) {
    v[u] = make_float4(-CUDART_INF_F, 0.f, 0.f, 0.f);
    missing |= u < count ? 1u << u : 0u;
  }
  for (bool first = true;; ) {
    const uint32_t get = first ? missing & 1u : missing;
#pragma unroll
    for (int u = 0; u < K; ++u)
      if (get >> u & 1u) v[u] = ld_row16(p + u * stride);
#pragma unroll
    for (int u = 0; u < K; ++u)
      if ((get >> u & 1u) && part_tagged(v[u], want)) { v[u] = unpack_part(v[u]); missing &= ~(1u << u); }
    const bool open = first ? (missing & 1u) != 0 : missing != 0;
    if (!__any_sync(0xffffffffu, open)) {
      if (!first) return true;
      first = false;
      continue;
    }
    if (__any_sync(0xffffffffu, clock64() - t0 > limit)) {
      atomicCAS(status, 0, CAKE_ERR_TIMEOUT);
      return false;
    }
    if (first) __nanosleep(40);
  }
}

// -lse / scale as three bf16 terms (24 bits) in columns 0..2 of the rows' operand of the extra K step.
__device__ __forceinline__ void put_ext_row(uint8_t* ext, int r, int rows, float lse2, float inv_scale2) {
  const float t = -lse2 * inv_scale2;
  const __nv_bfloat16 hi = __float2bfloat16_rn(t);
  const float r1 = t - __bfloat162float(hi);
  const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
  const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
  const uint32_t w0 = (uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(mid) << 16);
  const uint32_t w1 = (uint32_t)__bfloat16_as_ushort(lo);
  *reinterpret_cast<uint2*>(ext + ext_row_offset(r)) = r < rows ? make_uint2(w0, w1) : make_uint2(0u, 0u);
}

// Slot of the exchange rows (Smem::xrow) that a statistics warp uses after n_a pass-A ops and n_b pass-B
// ops.  A use writes its slot, meets a barrier and reads: the group's barrier in pass A (the warps of the
// first copy read their group's rows), the barrier of all statistics warps in a direct merge (group 0 reads
// every group's).  The next use may therefore not write the same slot, since slower warps still read it, but
// the one after that may: its writers have met the readers at the barrier between.  So the slots
// alternate over the whole program, from the last pass-A op into the first pass-B op too, and pass A may
// not follow a direct merge, whose readers a group's barrier does not meet (one wave: it never does).
__host__ __device__ constexpr int xrow_slot(uint32_t n_a, uint32_t n_b) { return (int)((n_a + n_b) & 1u); }

// ------------------------------------------------------------------ kernel
// kCopies: the window has 32 or 64 rows and a pass-A tile holds them 4 or 2 times, so that every
// statistics warp has rows to work on: copy c sums the c-th part of a key tile's columns.
// kDirect: one wave; every CTA merges the partial rows of its own pass-B ops (see tc_build_plan).
template <int G, bool kEntropyB, bool kCopies, bool kDirect>
__global__ void __launch_bounds__(TC_THREADS, 1)
score_fused_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                   const TcParams P) {
  extern __shared__ uint8_t smem_raw[];
  const Smem S = carve(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_slab = P.d / 64;
  const uint32_t stage_bytes = (uint32_t)(TILE * P.d * 2);
  const int rows_pad = (P.rows + 15) & ~15;
  const int op_lo = P.cta_op[blockIdx.x], op_hi = P.cta_op[blockIdx.x + 1];

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&S.full[i], 1); mbar_init(&S.empty[i], 1); }
    for (int i = 0; i < NBUF; ++i) { mbar_init(&S.acc_full[i], 1); mbar_init(&S.acc_empty[i], 4); }
    for (int i = 0; i < 2; ++i) { mbar_init(&S.q_full[i], 1); mbar_init(&S.q_empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&S.lse_full[i], kDirect ? 4 : 1); mbar_init(&S.lse_free[i], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the program of this CTA: a global read per op would put an L2 round trip on every op
  for (int i = threadIdx.x; i < min(op_hi - op_lo, kSmemOps); i += TC_THREADS) S.ops[i] = P.ops[op_lo + i];
  auto get_op = [&](int oi) -> ScoreOp {
    return oi - op_lo < kSmemOps ? S.ops[oi - op_lo] : P.ops[oi];
  };
  // rows of the query tiles that TMA never writes must read as zero
  for (int i = threadIdx.x; i < (int)(2 * kQBytes / 16); i += TC_THREADS)
    reinterpret_cast<uint4*>(S.q)[i] = make_uint4(0, 0, 0, 0);
  // operands of the extra K step: zero, then ones in the first three columns of the key side
  for (int i = threadIdx.x; i < (int)(3 * kExtBytes / 16); i += TC_THREADS)
    reinterpret_cast<uint4*>(S.ext_a)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if (threadIdx.x < 128)
    *reinterpret_cast<uint2*>(S.ext_a + ext_row_offset(threadIdx.x)) = make_uint2(0x3F803F80u, 0x00003F80u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == WARP_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(S.tmem_holder)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *S.tmem_holder;
  if (warp == WARP_TMA && op_lo < op_hi) {
    // The first key tiles start on their way to L2 while the kernel before this one ends.  (A prefetch reads nothing: if
    // that kernel still writes K, its stores go to the same L2 lines.)
    const ScoreOp op = get_op(op_lo);
    const int n = min(STAGES, (op.nkeys + TILE - 1) / TILE);
    for (int it = 0; it < n; ++it) tma_prefetch_3d(&k_map, 0, (int)(op.base + op.key0) + it * TILE, 0);
  }
  // Up to here nothing was read that the kernel before this one in the stream may write (the op tables
  // come with the batch): a CTA starts as soon as an SM is free, while that kernel's last CTAs still run.
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == WARP_TMA) {
    // ------------------------------------------------ TMA producer (converged warp, elected lane issues)
    {
      if (lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&q_map) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&k_map) : "memory");
      }
      __syncwarp();
      // pass A's tiles are read again by pass B: keep them in L2; pass B's read is the last
      const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
      uint32_t t = 0, qn = 0;
      bool ok = true;
      for (int oi = op_lo; oi < op_hi && ok; ++oi) {
        const ScoreOp op = get_op(oi);
        const uint64_t pol = (op.phase || !P.both) ? drop : keep;
        const int qb = qn & 1;
        // the MMAs of the op that used this query buffer two ops ago must be done
        ok = mbar_wait(&S.q_empty[qb], ((qn >> 1) & 1) ^ 1, P.status, P.spin_limit);
        ++qn;
        if (!ok) break;
        const int reps = kCopies && !op.phase ? P.reps : 1;
        mbar_expect_tx(&S.q_full[qb], (uint32_t)(reps * P.rows * P.d * 2));
        for (int rp = 0; rp < reps; ++rp)
          for (int sl = 0; sl < n_slab; ++sl)
            tma_load_4d(S.q + qb * kQBytes + sl * SLAB_BYTES + rp * P.rows * 128, &q_map, &S.q_full[qb], sl * 64, op.g * G,
                        0, op.req);
        const int64_t row0 = op.base + op.key0;
        const int ntiles = (op.nkeys + TILE - 1) / TILE;
        for (int it = 0; it < ntiles; ++it, ++t) {
          const int s = t % STAGES;
          ok = mbar_wait(&S.empty[s], ((t / STAGES) & 1) ^ 1, P.status, P.spin_limit);
          if (!ok) break;
          mbar_expect_tx(&S.full[s], stage_bytes);
          uint8_t* dst = S.k + (size_t)s * 2 * SLAB_BYTES;
          // the map's dimensions are (64 elements, key rows, slabs): the box lands slab by slab
          tma_load_3d_hint(dst, &k_map, &S.full[s], 0, (int)(row0 + it * TILE), 0, pol);
        }
      }
      // The next kernel of the stream may start once every CTA has issued its last loads; in shorter
      // launches (one wave, column pass alone) once it is done with its statistics.  Earlier the next kernel's CTAs take
      // the SMs that are left to the cascade's.  (Measured when an eviction still had a launch of its own there: a start with
      // this kernel made layers of the 4K MHA and 32K GQA prompts 10 % slower, one with the last op 8 %, and this one
      // 1 to 7 % faster than none.)
      if constexpr (!kDirect && !kEntropyB) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      // do not leave the CTA while a bulk copy may still be writing its shared memory
      const uint32_t issued = t;
      for (uint32_t u = issued > STAGES ? issued - STAGES : 0; u < issued; ++u)
        mbar_wait(&S.full[u % STAGES], (u / STAGES) & 1, P.status, P.spin_limit);
      for (uint32_t u = qn > 2 ? qn - 2 : 0; u < qn; ++u)
        mbar_wait(&S.q_full[u & 1], (u >> 1) & 1, P.status, P.spin_limit);
    }
  } else if (warp == WARP_MMA) {
    // ------------------------------------------------ MMA issuer (converged warp, elected lane issues)
    {
      uint32_t t = 0, qn = 0, kbm = 0;
      const uint32_t k_lo0 = (smem_u32(S.k) & 0x3FFFFu) >> 4;
      const uint32_t ext_a_lo = ((smem_u32(S.ext_a) & 0x3FFFFu) >> 4) | kExtDescLoLbo;
      bool ok = true;
      for (int oi = op_lo; oi < op_hi && ok; ++oi) {
        const ScoreOp op = get_op(oi);
        const uint32_t idesc = op.phase ? instr_desc(128, rows_pad) : instr_desc(128, TILE);
        const int eslot = kbm & 1;
        const uint32_t ext_b_lo = ((smem_u32(S.ext_b + eslot * kExtBytes) & 0x3FFFFu) >> 4) | kExtDescLoLbo;
        const int qb = qn & 1;
        ok = mbar_wait(&S.q_full[qb], (qn >> 1) & 1, P.status, P.spin_limit);
        ++qn;
        if (!ok) break;
        const uint32_t qaddr = smem_u32(S.q + qb * kQBytes);
        const uint32_t q_lo = (qaddr & 0x3FFFFu) >> 4;      // address field of the descriptors
        if (op.phase) {
          // the rows' -lse/scale operand of this op (written by the denominator warp)
          ok = mbar_wait(&S.lse_full[eslot], (kbm >> 1) & 1, P.status, P.spin_limit);
          if (!ok) break;
        }
        const int ntiles = (op.nkeys + TILE - 1) / TILE;
        for (int it = 0; it < ntiles; ++it, ++t) {
          const int s = t % STAGES, b = t % NBUF;
          ok = mbar_wait(&S.acc_empty[b], ((t / NBUF) & 1) ^ 1, P.status, P.spin_limit);
          if (!ok) break;
          ok = mbar_wait(&S.full[s], (t / STAGES) & 1, P.status, P.spin_limit);
          if (!ok) break;
          tc_fence_after();
          const uint32_t k_lo = k_lo0 + (uint32_t)s * (uint32_t)((2 * SLAB_BYTES) >> 4);
          const uint32_t tmem_d = tmem_base + (uint32_t)(b * 128);
          if (op.phase) {
            // D[key][row] = K Q^T
            umma_ss<0>(tmem_d, k_lo, q_lo, idesc);
            umma_ss<1>(tmem_d, k_lo + 2, q_lo + 2, idesc);
            umma_ss<1>(tmem_d, k_lo + 4, q_lo + 4, idesc);
            umma_ss<1>(tmem_d, k_lo + 6, q_lo + 6, idesc);
            if (n_slab == 2) {
              constexpr uint32_t o = SLAB_BYTES >> 4;
              umma_ss<1>(tmem_d, k_lo + o, q_lo + o, idesc);
              umma_ss<1>(tmem_d, k_lo + o + 2, q_lo + o + 2, idesc);
              umma_ss<1>(tmem_d, k_lo + o + 4, q_lo + o + 4, idesc);
              umma_ss<1>(tmem_d, k_lo + o + 6, q_lo + o + 6, idesc);
            }
            umma_ss_hi<1>(tmem_d, ext_a_lo, ext_b_lo, idesc, kExtDescHi);      // ... - lse/scale
          } else {
            // D[row][key] = Q K^T
            umma_ss<0>(tmem_d, q_lo, k_lo, idesc);
            umma_ss<1>(tmem_d, q_lo + 2, k_lo + 2, idesc);
            umma_ss<1>(tmem_d, q_lo + 4, k_lo + 4, idesc);
            umma_ss<1>(tmem_d, q_lo + 6, k_lo + 6, idesc);
            if (n_slab == 2) {
              constexpr uint32_t o = SLAB_BYTES >> 4;
              umma_ss<1>(tmem_d, q_lo + o, k_lo + o, idesc);
              umma_ss<1>(tmem_d, q_lo + o + 2, k_lo + o + 2, idesc);
              umma_ss<1>(tmem_d, q_lo + o + 4, k_lo + o + 4, idesc);
              umma_ss<1>(tmem_d, q_lo + o + 6, k_lo + o + 6, idesc);
            }
          }
          umma_commit(&S.empty[s]);
          umma_commit(&S.acc_full[b]);
        }
        umma_commit(&S.q_empty[qb]);     // query buffer free once every MMA of the op has run
        if (op.phase) {
          umma_commit(&S.lse_free[eslot]);   // and so is the op's -lse/scale operand
          ++kbm;
        }
      }
    }
  } else if (warp == WARP_MERGE) {
    // ------------------------------------------------ row merger
    // Every (pair, row) is merged by one CTA of the grid: row r of pair p by CTA (p * rows + r) % grid, so that with
    // many short pairs every CTA gets a few rows.  The warp waits for the row's partials, merges them in a
    // fixed order and publishes the row's base-2 log-sum-exp and entropy term.  Short pairs (a ragged batch,
    // MHA) have few partials per row: the rows of `ways` consecutive pairs are merged side by side, by
    // 32 / ways lanes each.
    if (P.both && !kDirect) {
      constexpr int kBatch = 12;                     // loads per lane in flight: the 384 partials of a row at 128 CTAs
      const int ways = P.merge_ways, lpr = 32 / ways;         // lanes per row
      const int sub = lane / lpr, l8 = lane % lpr;
      bool ok = true;
      for (int gi = 0; gi < P.n_groups && ok; ++gi) {
        const int pair = (P.group_begin ? P.group_begin[gi] : gi * ways) + sub;
        const bool have = pair < (P.group_begin ? P.group_begin[gi + 1] : P.n_pairs);
        const int s_lo = have ? P.pair_aseg[pair] * NWG : 0, s_hi = have ? P.pair_aseg[pair + 1] * NWG : 0;
        const int r0 = have ? (int)((blockIdx.x + gridDim.x - (unsigned)(((long long)pair * P.rows) % gridDim.x)) % gridDim.x)
                            : P.rows;
        for (int r = r0; ok; r += gridDim.x) {
          const bool active = have && r < P.rows;
          if (!__any_sync(0xffffffffu, active)) break;
          float4 acc = make_float4(-CUDART_INF_F, 0.f, 0.f, 0.f);
          for (int base = s_lo;; base += kBatch * lpr) {
            if (!__any_sync(0xffffffffu, active && base < s_hi)) break;
            const int left = s_hi - base - l8;         // partials base + l8, base + l8 + lpr, ...
            float4 pv[kBatch];
            ok = wait_parts(&P.rowpart[(size_t)(base + l8) * 128 + (active ? r : 0)], (int64_t)lpr * 128,
                            active ? (left + lpr - 1) / lpr : 0, P.want, pv, P.status, P.spin_limit);
            if (!ok) break;
            acc = merge_batch(acc, pv);
          }
          if (!ok) break;
          // over the lanes of a row: the largest reference, then the sums
          float mx = acc.x;
          for (int o = lpr >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          const float d = acc.x == -CUDART_INF_F ? 0.f : acc.x - mx, f = acc.x == -CUDART_INF_F ? 0.f : exp2f(d);
          float w = f * fmaf(d, acc.y - acc.z, acc.w), z = acc.y * f, zwin = acc.z * f;
          for (int o = lpr >> 1; o > 0; o >>= 1) {
            z += __shfl_xor_sync(0xffffffffu, z, o);
            zwin += __shfl_xor_sync(0xffffffffu, zwin, o);
            w += __shfl_xor_sync(0xffffffffu, w, o);
          }
          if (active && l8 == 0) {
            const float lz = log2f(z);
            st_row8(&P.lse2[((size_t)pair * 128 + r) * kLseStride], __float_as_uint(mx + lz), P.tag);
            // sum_j p log2 p over the observed keys = (w - log2(z) * z_obs) / z
            __stcg(&P.hrow[(size_t)pair * 128 + r], (w - lz * (z - zwin)) / z);
          }
        }
      }
    }
  } else if (warp == WARP_LSE) {
    // ------------------------------------------------ denominator fetcher
    // For every pass-B op of this CTA, in program order: wait until all rows of the op's pair are
    // merged, write the pair's -lse/scale operand into a two-slot shared-memory ring.
    uint32_t kb = 0;
    bool ok = true;
    for (int oi = op_lo; oi < op_hi && ok && !kDirect; ++oi) {
      const ScoreOp op = get_op(oi);
      if (!op.phase) continue;
      const int slot = kb & 1;
      const int pair = op.req * P.Hkv + op.g;
      ok = mbar_wait(&S.lse_free[slot], ((kb >> 1) & 1) ^ 1, P.status, P.spin_limit);
      if (!ok) break;
      float4 v;
      if (P.lse_ext) {
        // the caller's natural-log values [req][H_q][S_w]: tile row r' = i*G + h, base 2
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int r = 4 * lane + e, i = r / G, h = r - i * G;
          x[e] = r < P.rows ? __ldg(&P.lse_ext[((size_t)op.req * P.Hq + op.g * G + h) * P.Sw + i]) * kLog2e : 0.f;
        }
        v = make_float4(x[0], x[1], x[2], x[3]);
      } else {
        const uint2* at = P.lse2 + ((size_t)pair * 128 + 4 * lane) * kLseStride;      // rows 4 * lane ..
        const bool mine = 4 * lane < P.rows;           // (rows is a multiple of 32)
        const long long t0 = clock64();
        // A CTA waits for one row, another one than its neighbours, before it asks for all: 128 CTAs that poll the
        // same lines delay the stores they wait for.
        const int probe = (int)(blockIdx.x % (unsigned)P.rows);
        uint2 x[4];
        for (bool all = false;;) {
          if (!all) {
            uint2 p = make_uint2(0u, 0u);
            if (lane == 0) p = ld_row8(P.lse2 + ((size_t)pair * 128 + probe) * kLseStride);
            all = __any_sync(0xffffffffu, p.y == P.want);
          }
          bool got = all;
          if (all) {
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = mine ? ld_row8(at + e * kLseStride) : make_uint2(0u, P.want);
#pragma unroll
            for (int e = 0; e < 4; ++e) got = got && x[e].y == P.want;
          }
          if (__all_sync(0xffffffffu, got)) break;
          if (__any_sync(0xffffffffu, clock64() - t0 > P.spin_limit)) { atomicCAS(P.status, 0, CAKE_ERR_TIMEOUT); ok = false; break; }
          __nanosleep(32);
        }
        if (!ok) break;
        v = make_float4(__uint_as_float(x[0].x), __uint_as_float(x[1].x), __uint_as_float(x[2].x), __uint_as_float(x[3].x));
      }
      {
        const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) put_ext_row(S.ext_b + slot * kExtBytes, 4 * lane + e, P.rows, vv[e], P.inv_scale2);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.lse_full[slot]);
      ++kb;
    }
  } else {
    // ------------------------------------------------ statistics warps
    // Every warp owns TMEM lanes 32*quad.. of the tiles its group takes and writes its own partial
    // results.  It waits for other statistics warps only where rows are exchanged: with kCopies for its
    // group at the end of a pass-A op, with kDirect for all of them at the start of a pass-B op.
    // Group wg takes the tiles t with t % NWG == wg, from buffer t % NBUF.
    const int wg = warp >> 2;
    const int quad = warp & 3;                      // TMEM lane quadrant this warp may read
    const int lane_row = quad * 32 + lane;          // accumulator lane (row in pass A, key in pass B)
    const uint32_t taddr0 = tmem_base + ((uint32_t)(quad * 32) << 16);
    uint32_t t = wg, t_op = 0;                      // the group's next tile, the first tile of the op
    uint32_t n_a_done = 0;                          // pass-A ops this warp has delivered
    uint32_t kbs = 0;                               // pass-B ops so far
    // pass A: the window row of this lane, and the columns its copy of the rows sums
    const int copy = kCopies ? (quad * P.reps) >> 2 : 0;
    const int i_row = (kCopies ? lane_row - copy * P.rows : lane_row) / G;
    const int c_lo = kCopies ? copy * (TILE / P.reps) : 0, c_hi = kCopies ? c_lo + TILE / P.reps : TILE;
    bool ok = true;
    const float inv_sw = 1.f / (float)P.Sw, inv_g = 1.f / (float)G;
    for (int oi = op_lo; oi < op_hi; ++oi) {
      const ScoreOp op = get_op(oi);
      const int ntiles = (op.nkeys + TILE - 1) / TILE;
      const int it0 = (int)(t - t_op);                           // the group's first tile of the op
      t_op += (uint32_t)ntiles;
      if (kEntropyB || op.phase) {
        // ---------------- pass B: thread = key, columns = rows r' = i*G + h
        if constexpr (kDirect) {
          // One thread per row and group; every CTA adds in the same order.
          const int slot = kbs & 1, xslot = xrow_slot(n_a_done, kbs), pair = op.req * P.Hkv + op.g;
          const int s_lo = P.pair_aseg[pair], s_hi = P.pair_aseg[pair + 1];
          const uint32_t free_par = ((kbs >> 1) & 1) ^ 1;
          ++kbs;
          float4 acc = make_float4(-CUDART_INF_F, 0.f, 0.f, 0.f);
          for (int sg = s_lo; sg < s_hi && ok; sg += 8) {
            float4 pv[8];
            ok = wait_parts(&P.rowpart[((size_t)sg * NWG + wg) * 128 + lane_row], (int64_t)NWG * 128,
                            lane_row < P.rows ? s_hi - sg : 0, P.want, pv, P.status, P.spin_limit);
            if (ok) acc = merge_batch(acc, pv);
          }
          S.xrow[(xslot * NWG + wg) * 128 + lane_row] = acc;
          asm volatile("bar.sync 1, %0;" ::"n"(STAT_THREADS) : "memory");
          if (wg == 0) {
            acc = make_float4(-CUDART_INF_F, 0.f, 0.f, 0.f);
            if (lane_row < P.rows) {
              float4 pv[NWG];
#pragma unroll
              for (int q = 0; q < NWG; ++q) pv[q] = S.xrow[(xslot * NWG + q) * 128 + lane_row];
              acc = merge_batch(acc, pv);
            }
            // the MMAs of the op that used this slot two ops ago must be done
            if (ok) ok = mbar_wait(&S.lse_free[slot], free_par, P.status, P.spin_limit);
            const float lz = log2f(acc.y);
            put_ext_row(S.ext_b + slot * kExtBytes, lane_row, P.rows, acc.x + lz, P.inv_scale2);
            if (op.key0 == 0 && lane_row < P.rows)
              P.hrow[(size_t)pair * 128 + lane_row] = (acc.w - lz * (acc.y - acc.z)) / acc.y;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.lse_full[slot]);
          }
        }
        float vacc[G], hs[G];
#pragma unroll
        for (int h = 0; h < G; ++h) { vacc[h] = 0.f; hs[h] = 0.f; }
        for (int it = it0; it < ntiles; it += NWG, t += NWG) {
          if (ok) ok = mbar_wait(&S.acc_full[t % NBUF], (t / NBUF) & 1, P.status, P.spin_limit);
          if (!ok) continue;
          uint64_t* const my_empty = &S.acc_empty[t % NBUF];
          const uint32_t taddr = taddr0 + (t % NBUF) * 128u;
          tc_fence_after();
          float s1[G], s2[G], hk[G], a2 = 0.f;
#pragma unroll
          for (int h = 0; h < G; ++h) { s1[h] = 0.f; s2[h] = 0.f; hk[h] = 0.f; }
          f32x2 s1p[(G + 1) / 2], s2p[(G + 1) / 2], hkp[(G + 1) / 2];   // the same, two heads per register
#pragma unroll
          for (int hp = 0; hp < (G + 1) / 2; ++hp) { s1p[hp] = 0ull; s2p[hp] = 0ull; hkp[hp] = 0ull; }
          auto release = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(my_empty);
          };
          for_columns(taddr, 0, P.rows, [&](const uint32_t (&r)[16]) {
            // 16 columns = 16/G window rows x G heads; the accumulator is q.k - lse/scale
            if constexpr (G % 2 == 0) {
              // two heads per instruction
              const f32x2 sc2 = pack2(P.scale2, P.scale2);
#pragma unroll
              for (int ii = 0; ii < 16 / G; ++ii) {
                f32x2 asum = 0ull;
#pragma unroll
                for (int hp = 0; hp < G / 2; ++hp) {
                  const int c = ii * G + 2 * hp;
                  const f32x2 tt2 = mul2(pack2(__uint_as_float(r[c]), __uint_as_float(r[c + 1])), sc2);
                  float t0, t1;
                  unpack2(tt2, t0, t1);
                  const f32x2 p2 = pack2(ex2(t0), ex2(t1));
                  s1p[hp] = add2(s1p[hp], p2);
                  s2p[hp] = fma2(p2, p2, s2p[hp]);
                  if (kEntropyB) hkp[hp] = fma2(p2, tt2, hkp[hp]);
                  asum = hp == 0 ? p2 : add2(asum, p2);
                }
                float a0, a1;
                unpack2(asum, a0, a1);
                const float a = a0 + a1;
                a2 = fmaf(a, a, a2);
              }
            } else {
#pragma unroll
              for (int ii = 0; ii < 16 / G; ++ii) {
                float a = 0.f;
#pragma unroll
                for (int h = 0; h < G; ++h) {
                  const float tt = __uint_as_float(r[ii * G + h]) * P.scale2;
                  const float p = ex2(tt);
                  s1[h] += p;
                  s2[h] = fmaf(p, p, s2[h]);
                  if (kEntropyB) hk[h] = fmaf(p, tt, hk[h]);
                  a += p;
                }
                a2 = fmaf(a, a, a2);
              }
            }
          }, release);
          if constexpr (G % 2 == 0) {
#pragma unroll
            for (int hp = 0; hp < G / 2; ++hp) {
              unpack2(s1p[hp], s1[2 * hp], s1[2 * hp + 1]);
              unpack2(s2p[hp], s2[2 * hp], s2[2 * hp + 1]);
              if (kEntropyB) unpack2(hkp[hp], hk[2 * hp], hk[2 * hp + 1]);
            }
          }
          const int j = op.key0 + it * TILE + lane_row;          // key index inside the request
          if (j < op.n && it * TILE + lane_row < op.nkeys) {
            float a1 = 0.f;
#pragma unroll
            for (int h = 0; h < G; ++h) {
              a1 += s1[h];
              const float mh = s1[h] * inv_sw;
              vacc[h] += fmaxf(s2[h] * inv_sw - mh * mh, 0.f) * P.bessel;
              if (kEntropyB) hs[h] += hk[h];
            }
            const float mean = a1 * inv_g * inv_sw;
            const float var = fmaxf(a2 * inv_g * inv_g * inv_sw - mean * mean, 0.f) * P.bessel;
            P.raw[op.base + j] = combine_indicator(P.ind_mode, P.gamma, mean, var, (float)P.Sw);
          }
        }
        // fixed-order reduction over the warp's keys
#pragma unroll
        for (int h = 0; h < G; ++h) {
          float x = vacc[h], y = hs[h];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            if (kEntropyB) y += __shfl_xor_sync(0xffffffffu, y, o);
          }
          if (lane == h) {
            float* dst = P.colpart + (((size_t)op.seg * NSTATW + warp) * G + h) * 2;
            dst[0] = y;
            dst[1] = x;
          }
        }
      } else {
        // ---------------- pass A: thread = window row r' = i*G + h, columns = keys
        float m = -CUDART_INF_F, z = 0.f, zwin = 0.f, w = 0.f;
        for (int it = it0; it < ntiles; it += NWG, t += NWG) {
          if (ok) ok = mbar_wait(&S.acc_full[t % NBUF], (t / NBUF) & 1, P.status, P.spin_limit);
          if (!ok) continue;
          uint64_t* const my_empty = &S.acc_empty[t % NBUF];
          const uint32_t taddr = taddr0 + (t % NBUF) * 128u;
          tc_fence_after();
          // columns of observed keys (every row sees them), and of keys at all
          const int c_key = op.nkeys - it * TILE, c_obs = min(op.n - op.key0 - it * TILE, c_key);
          const int c_fast = c_obs >= c_hi ? c_hi : max(c_lo, c_obs & ~15);
          if (!kCopies && quad * 32 >= P.rows) {       // these TMEM lanes hold padding rows
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(my_empty);
            continue;
          }
          bool again = false;
          if (c_fast > c_lo) {
            // Whole chunks of observed keys.  The exponentials are taken against the row's running reference m
            // without looking for the tile's maximum first (an op's first tile: that of its first chunk).
            // Afterwards the reference moves up by the binary exponent of a sum that is far above 1; only where the
            // sum nears the end of fp32's range is the tile taken again, from its maxima.
            // (All rows of the warp at once: the load is a collective.  A row whose first keys all have logits of -inf takes
            // a finite reference, so that the -inf reach its entropy term as 0 * -inf and its other logits are summed.)
            if (it == it0) {
              uint32_t r[16];
              tmem_ld16_issue(taddr + c_lo, r);
              tmem_ld_wait(r);
              float cm = __uint_as_float(r[0]);
#pragma unroll
              for (int e = 1; e < 16; ++e) cm = fmaxf(cm, __uint_as_float(r[e]));
              m = cm > -CUDART_INF_F ? cm * P.scale2 : 0.f;
            }
            // two keys per instruction: four partial sums in two packed accumulators
            const f32x2 sc2 = pack2(P.scale2, P.scale2), nm2 = pack2(-m, -m);
            f32x2 zc[2] = {0ull, 0ull}, wc[2] = {0ull, 0ull};
            for_columns(taddr, c_lo, c_fast, [&](const uint32_t (&r)[16]) {
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                const f32x2 tt2 = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sc2, nm2);
                float t0, t1;
                unpack2(tt2, t0, t1);
                const f32x2 ee2 = pack2(ex2(t0), ex2(t1));
                zc[(e >> 1) & 1] = add2(zc[(e >> 1) & 1], ee2);
                wc[(e >> 1) & 1] = fma2(ee2, tt2, wc[(e >> 1) & 1]);
              }
            }, []() {});
            float z0, z1, w0, w1;
            unpack2(add2(zc[0], zc[1]), z0, z1);
            unpack2(add2(wc[0], wc[1]), w0, w1);
            const float zs = z0 + z1;
            again = zs > kTileSumMax;                  // (a NaN is added and stays)
            if (!again) {
              z += zs;
              w += w0 + w1;
              if (zs > kShiftSum) {
                const int k = (int)(__float_as_uint(z) >> 23) - 127;
                const float f = __uint_as_float((uint32_t)(127 - k) << 23);
                m += (float)k;
                w = fmaf(-(float)k, z - zwin, w) * f;
                z *= f; zwin *= f;
              }
            }
          }
          // The chunks at the end of the prompt (window keys, which a row sees up to its own and which are not
          // observed) and those of a tile taken again, from the chunk's maximum.
          const int c_slow = __any_sync(0xffffffffu, again) ? c_lo : c_fast;
#pragma unroll 1
          for (int c0 = c_slow; c0 < c_hi && c0 < c_key; c0 += 16) {
            uint32_t r[16];
            tmem_ld16_issue(taddr + c0, r);
            tmem_ld_wait(r);
            const int n_obs = c_obs - c0;                                        // observed keys of the chunk
            const int n_vis = c0 < c_fast && !again ? 0 : min(c_key - c0, n_obs + i_row + 1);   // visible ones
            float cm = -CUDART_INF_F;
#pragma unroll
            for (int e = 0; e < 16; ++e) cm = e < n_vis ? max_or_nan(cm, __uint_as_float(r[e])) : cm;
            if (cm != -CUDART_INF_F) {                        // (a NaN goes into z, where it stays)
              cm *= P.scale2;
              if (cm > m) {
                const float mn = cm;
                const float f = ex2(m - mn);                  // 0 while m = -inf
                const float dm = (m == -CUDART_INF_F) ? 0.f : (m - mn);
                w = f * fmaf(dm, z - zwin, w);
                z *= f; zwin *= f;
                m = mn;
              }
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const float tt = fmaf(__uint_as_float(r[e]), P.scale2, -m);
                const float ee = e < n_vis ? ex2(tt) : 0.f;
                z += ee;
                zwin += e < n_obs ? 0.f : ee;
                w = e < n_obs && e < n_vis ? fmaf(ee, tt, w) : w;
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(my_empty);
        }
        // Deliver this warp's 32 partial rows of the segment.
        float4 part = make_float4(m, z, zwin, w);
        if constexpr (kCopies) {
          // the group's copies of a row become one partial
          float4* x = S.xrow + (xrow_slot(n_a_done, kbs) * NWG + wg) * 128;
          x[lane_row] = part;
          asm volatile("bar.sync %0, 128;" ::"r"(2 + wg) : "memory");
          if (copy == 0)
            for (int c = 1; c < P.reps; ++c) part = merge_rows(part, x[c * P.rows + lane_row]);
        }
        if (!kCopies || copy == 0)
          st_row16(&P.rowpart[((size_t)op.seg * NWG + wg) * 128 + lane_row], pack_part(part.x, part.y, part.z, part.w, P.tag));
        ++n_a_done;
      }
    }
  }
  // ------------------------------------------------ teardown
  if ((kDirect || kEntropyB) && warp == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  if (warp == WARP_MMA) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512)
                 : "memory");
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}


template <int G>
cudaError_t launch_g(int device, bool entropy_b, bool copies, bool direct, bool early, int n_cta, cudaStream_t st, const CUtensorMap& qmap,
                     const CUtensorMap& kmap, const TcParams& P) {
  typedef void (*Kernel)(const CUtensorMap, const CUtensorMap, const TcParams);
  static const Kernel kernels[5] = {score_fused_kernel<G, false, false, false>, score_fused_kernel<G, false, false, true>,
                                    score_fused_kernel<G, false, true, false>, score_fused_kernel<G, false, true, true>,
                                    score_fused_kernel<G, true, false, false>};
  static PerDeviceOnce attr;
  if (attr.need(device)) {
    for (Kernel k : kernels) {
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
      if (e != cudaSuccess) return e;
    }
    attr.mark(device);
  }
  const Kernel k = kernels[entropy_b ? 4 : (copies ? 2 : 0) + (direct ? 1 : 0)];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta, 1, 1);
  cfg.blockDim = dim3(TC_THREADS, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, qmap, kmap, P);
}

// Copies of the window rows in a pass-A tile.
int tc_reps(int rows) { return rows == 32 ? 4 : rows == 64 ? 2 : 1; }

// Cuts the `tiles` tiles of one (request, head) pair, which start at flat tile index `flat`
// of a wave of `W` tiles shared by `n_cta` CTAs (slot c owns flat tiles
// [c*W/n_cta, (c+1)*W/n_cta)), into per-slot segments; slot c belongs to CTA (c+rot) of all, modulo their number.
void cut_pair(std::vector<std::vector<ScoreOp>>& per_cta, int rot, int n_cta, int64_t W, int64_t flat,
              int tiles, int keys, int req, int g, int phase, int32_t& seg_counter, int64_t base,
              int n_obs) {
  int t0 = 0;
  while (t0 < tiles) {
    const int64_t f = flat + t0;
    int c = (int)(f * n_cta / W);
    while (c + 1 < n_cta && (int64_t)(c + 1) * W / n_cta <= f) ++c;
    while (c > 0 && (int64_t)c * W / n_cta > f) --c;
    const int64_t share_end = (int64_t)(c + 1) * W / n_cta;
    const int t1 = (int)((share_end - flat) < tiles ? (share_end - flat) : tiles);
    ScoreOp op;
    op.base = base; op.n = n_obs;
    op.req = req; op.g = g; op.key0 = t0 * TILE;
    op.nkeys = (t1 * TILE < keys ? t1 * TILE : keys) - t0 * TILE;
    op.phase = phase;
    op.seg = seg_counter++;
    per_cta[(c + rot) % (int)per_cta.size()].push_back(op);
    t0 = t1;
  }
}

// Waves of consecutive (request, KV head) pairs: K of the wave in pass B and of the wave in pass A
// must fit L2 together, so a wave is closed before the pair that would take it past kWaveBytes.
// (One wave for a whole layer of up to 64 MB was tried: no faster at 34 MB, slower at 64 MB.)
std::vector<int> tc_waves(const ReqInfo* reqs, int n_req, int Hkv, int head_dim) {
  const int n_pairs = n_req * Hkv;
  std::vector<int> wave_begin{0};
  int64_t bytes = 0;
  for (int p = 0; p < n_pairs; ++p) {
    const int64_t pb = (int64_t)reqs[p / Hkv].N * head_dim * 2;
    if (bytes > 0 && bytes + pb > kWaveBytes) {
      wave_begin.push_back(p);
      bytes = 0;
    }
    bytes += pb;
  }
  wave_begin.push_back(n_pairs);
  return wave_begin;
}

}  // namespace

// Exchanged rows of the current batch: merged rows of every pair, then the partial rows of every pass-A segment.
size_t tc_exchange_bytes(int64_t pairs, int64_t segs) {
  return (size_t)pairs * 128 * kLseStride * sizeof(uint2) + (size_t)segs * NWG * 128 * sizeof(float4);
}
static_assert(CAKE_MAX_LAYERS < 512, "a launch's mark has 9 bits");

size_t tc_index_size(int64_t pairs, int n_sm) { return 3 * (size_t)(pairs + 1) + 2 * (size_t)(n_sm + 1); }

bool tc_path_supported(const cake_config& c) {
  const int G = c.n_q_heads / c.n_kv_heads;
  const int rows = G * c.window;
  return c.dtype == CAKE_DTYPE_BF16 && (c.head_dim == 64 || c.head_dim == 128) && rows % 32 == 0 &&
         rows <= 128 && (G == 1 || G == 2 || G == 4 || G == 8) && c.window <= 256;
}

// Upper bound on the segments of one pass: every pair gives one segment plus one per CTA
// boundary inside its wave; two consecutive waves hold more than kWaveBytes of K, and there
// are no more waves than pairs.
int64_t tc_max_segments(const cake_config& c, int n_sm) {
  const int64_t pairs = (int64_t)c.max_requests * c.n_kv_heads;
  const int64_t bytes = (int64_t)c.n_kv_heads * c.max_total_tokens * c.head_dim * 2;
  int64_t waves = 2 * (bytes / kWaveBytes) + 2;
  if (waves > pairs) waves = pairs;
  return pairs + waves * n_sm;
}

// Builds the per-CTA programs of the batch in ctx->h_req[0..n_req): one with both passes, and one with
// pass B alone (denominators supplied by the caller).
int32_t tc_build_plan(cake_ctx* ctx, int32_t n_req) {
  const cake_config& c = ctx->cfg;
  const int Hkv = c.n_kv_heads;
  const int n_pairs = n_req * Hkv;
  const int64_t T = n_req > 0 ? ctx->h_req[n_req - 1].cu + ctx->h_req[n_req - 1].N : 0;
  int64_t tilesA_total = 0;
  for (int r = 0; r < n_req; ++r) tilesA_total += (int64_t)Hkv * ((ctx->h_req[r].N + TILE - 1) / TILE);
  int n_cta = (int)(tilesA_total < ctx->n_sm_score ? tilesA_total : ctx->n_sm_score);
  ctx->n_tc_ctas = n_cta;
  ctx->n_tc_ops_full = ctx->n_tc_ops_b = 0;
  ctx->n_tc_asegs = ctx->n_tc_bsegs = 0;
  ctx->n_tc_waves = 0;
  if (n_cta == 0) return CAKE_OK;

  const std::vector<int> wave_begin = tc_waves(ctx->h_req, n_req, Hkv, c.head_dim);
  const int n_waves = (int)wave_begin.size() - 1;
  ctx->n_tc_waves = n_waves;
  // Every wave ends when its slowest CTA does, i.e. after ceil(tiles / CTAs) tiles, and both
  // passes walk it.  Among the CTA counts down to three quarters of the SMs on offer, take the
  // smallest one that reaches the minimum of the summed quotients: the SMs left over shorten
  // nothing here and go to the cascade kernels that run beside this one.
  {
    std::vector<int64_t> w(n_waves, 0);
    for (int wv = 0; wv < n_waves; ++wv)
      for (int p = wave_begin[wv]; p < wave_begin[wv + 1]; ++p) w[wv] += (ctx->h_req[p / Hkv].N + TILE - 1) / TILE;
    int64_t best = -1;
    int best_n = n_cta;
    for (int n = n_cta; n >= 1 && n >= n_cta - n_cta / 4; --n) {
      int64_t steps = 0;
      for (int wv = 0; wv < n_waves; ++wv) steps += (w[wv] + n - 1) / n;
      if (best < 0 || steps <= best) { best = steps; best_n = n; }
      else break;
    }
    n_cta = best_n;
    ctx->n_tc_ctas = n_cta;
  }
  // A single wave with no more pairs than CTAs: if a tile more per CTA allows it, every CTA works for one pair.  A
  // second pair is another row-pass op, another wait for denominators and another column-pass op in a row
  // (8 heads of 7919 keys on 124 CTAs: most CTAs were done after 18.7 us, the four with two pairs after 23.4).
  std::vector<int> pair_cta;                         // first CTA of every pair, and their number
  if (n_waves == 1 && n_pairs <= ctx->n_sm_score) {
    int64_t W = 0;
    for (int p = 0; p < n_pairs; ++p) W += (ctx->h_req[p / Hkv].N + TILE - 1) / TILE;
    const int64_t steps = (W + n_cta - 1) / n_cta;
    for (int64_t most = steps; most <= steps + 1 && pair_cta.empty(); ++most) {
      std::vector<int> first(1, 0);
      for (int p = 0; p < n_pairs; ++p)
        first.push_back(first.back() + (int)(((ctx->h_req[p / Hkv].N + TILE - 1) / TILE + most - 1) / most));
      if (first.back() <= ctx->n_sm_score) pair_cta = first;
    }
    if (!pair_cta.empty()) ctx->n_tc_ctas = n_cta = pair_cta.back();
  }
  std::vector<std::vector<ScoreOp>> a_ops(n_cta), b_ops(n_cta);
  int32_t aseg = 0, bseg = 0;
  int32_t* pair_aseg = ctx->h_tc_index;                    // [pairs+1]
  int32_t* pair_bseg = ctx->h_tc_index + (n_pairs + 1);    // [pairs+1]
  int rot = 0;
  for (int wv = 0; wv < n_waves; ++wv) {
    int64_t WA = 0;
    for (int p = wave_begin[wv]; p < wave_begin[wv + 1]; ++p)
      WA += (ctx->h_req[p / Hkv].N + TILE - 1) / TILE;
    int64_t fa = 0;
    for (int p = wave_begin[wv]; p < wave_begin[wv + 1]; ++p) {
      const int r = p / Hkv, g = p % Hkv;
      const ReqInfo& rq = ctx->h_req[r];
      const int ta = (rq.N + TILE - 1) / TILE, tb = (rq.n + TILE - 1) / TILE;
      pair_aseg[p] = aseg;
      pair_bseg[p] = bseg;
      const int64_t base = (int64_t)g * T + rq.cu;
      const bool own = !pair_cta.empty();
      const int c0 = own ? pair_cta[p] : rot, nc = own ? pair_cta[p + 1] - c0 : n_cta;
      const int64_t w = own ? ta : WA, f = own ? 0 : fa;
      cut_pair(a_ops, c0, nc, w, f, ta, rq.N, r, g, 0, aseg, base, rq.n);
      // pass B walks the same flat tile positions, so a CTA re-reads the tiles it brought in
      if (tb > 0) cut_pair(b_ops, c0, nc, w, f, tb, rq.n, r, g, 1, bseg, base, rq.n);
      fa += ta;
    }
    // a wave's remainder tiles land on different CTAs each time (golden-ratio stride)
    rot = (rot + (int)(n_cta * 0.381966) + 1) % n_cta;
  }
  pair_aseg[n_pairs] = aseg;
  pair_bseg[n_pairs] = bseg;
  if (aseg > ctx->max_tc_segs || bseg > ctx->max_tc_segs) return CAKE_ERR_CAPACITY;

  // several rows at a time when there are pairs to take them from and a row has few partials
  {
    int max_segs = 0;
    for (int p = 0; p < n_pairs; ++p) max_segs = std::max(max_segs, pair_aseg[p + 1] - pair_aseg[p]);
    const int partials = max_segs * NWG;
    // at most 16 partials per lane (two batches of loads): 32 lanes / ways per row
    int ways = 1;
    while (ways < 32 && 2 * ways <= n_pairs && partials * 2 * ways <= 512) ways *= 2;
    if (n_pairs < 4) ways = 1;
    ctx->tc_merge_ways = ways;
    // The merger handles up to `ways` consecutive pairs at once and waits for the pass A of all of them, and
    // pass B of a pair for the whole group: a group lies inside a wave.
    int32_t* group_begin = ctx->h_tc_index + 2 * (n_pairs + 1);
    int ng = 0;
    for (int wv = 0, p0 = 0; wv < n_waves; ++wv) {
      const int p1 = wave_begin[wv + 1];
      for (; p0 < p1; p0 += std::min(ways, p1 - p0)) group_begin[ng++] = p0;
    }
    group_begin[ng] = n_pairs;
    ctx->n_tc_groups = ng;
    // With a single wave nothing runs between its pass A and its pass B, so a launch waits for the way
    // from the partial rows to the denominators.  As long as a pair's partials are few (a thread reads
    // one per segment, eight at a time) every CTA merges those of its own pass-B ops: the merged rows
    // are spared a trip through global memory (store, fence, count, poll, load: 4 us of 28 at 32 pairs
    // of 4K keys).
    bool all_b = true;                               // every pair has a pass-B op to write its entropy rows
    for (int p = 0; p < n_pairs; ++p) all_b = all_b && pair_bseg[p + 1] > pair_bseg[p];
    ctx->tc_direct = n_waves == 1 && all_b && max_segs <= kDirectSegs;
  }
  // Program of a CTA, by waves:  A0 A1 B0 A2 B1 ... A(n-1) B(n-2) B(n-1).  Pass B of a wave waits for the wave's merged
  // denominators, which trail the slowest CTA's pass A by some 4 us; the pass A in between covers that.  (Tiles of
  // A(w+1) and B(w) in turn, so that DRAM is never idle, and a lead of pass A of 4 to 16 tiles beyond the wave were
  // each no faster alone and 2 to 4 % slower in a long run, where the power cap sets the clock.)
  const int64_t n_full = (int64_t)aseg + bseg, total = n_full + bseg;
  if (total > ctx->max_tc_ops) return CAKE_ERR_CAPACITY;
  int32_t* cta_full = ctx->h_tc_index + 3 * (n_pairs + 1);   // [n_sm+1]
  int32_t* cta_b = cta_full + (ctx->n_sm + 1);               // [n_sm+1]
  int32_t o = 0, ob = (int32_t)n_full;
  auto wave_of = [&](const ScoreOp& op) {
    return (int)(std::upper_bound(wave_begin.begin(), wave_begin.end(), op.req * Hkv + op.g) - wave_begin.begin()) - 1;
  };
  for (int cta = 0; cta < n_cta; ++cta) {
    cta_full[cta] = o;
    cta_b[cta] = ob;
    size_t ib = 0;
    for (const ScoreOp& a : a_ops[cta]) {
      for (const int w = wave_of(a); ib < b_ops[cta].size() && wave_of(b_ops[cta][ib]) < w - 1; ++ib)
        ctx->h_tc_ops[o++] = b_ops[cta][ib];
      ctx->h_tc_ops[o++] = a;
    }
    for (; ib < b_ops[cta].size(); ++ib) ctx->h_tc_ops[o++] = b_ops[cta][ib];
    for (const ScoreOp& b : b_ops[cta]) ctx->h_tc_ops[ob++] = b;
  }
  cta_full[n_cta] = o;
  cta_b[n_cta] = ob;
  ctx->n_tc_ops_full = (int32_t)n_full;
  ctx->n_tc_ops_b = bseg;
  ctx->n_tc_asegs = aseg;
  ctx->n_tc_bsegs = bseg;
  return CAKE_OK;
}

// Builds the plan of a batch on the host alone (no device, no context) and checks the properties
// the kernel relies on.  Returns CAKE_OK, an error of the plan builder, or CAKE_ERR_STATE with
// info8[7] = the number of the violated property:
//   1  every key tile of every pair is covered exactly once by the pass-A ops, and every non-window
//      tile exactly once by the pass-B ops
//   2  inside every CTA's program the pass-B ops come in non-decreasing wave order and every
//      pass-A op of a wave w' <= w precedes the first pass-B op of wave w (so a wave's pass B can
//      only ever wait for pass-A ops that wait for nothing themselves)
//   3  the pairs the merger warps handle side by side lie in one wave
//   4  op counts and segment numbers stay inside the tables the context would allocate
//   5  no statistics warp writes a slot of the exchange rows that another may still read (xrow_slot)
int32_t tc_plan_check(const cake_config& c, int n_sm, int reserved, int32_t n_req, const int64_t* cu,
                      int32_t* info8) {
  if (!tc_path_supported(c)) return CAKE_ERR_ARG;
  cake_ctx x;
  memset(&x, 0, sizeof(x));
  x.cfg = c;
  x.rows = c.n_q_heads / c.n_kv_heads * c.window;
  x.n_sm = n_sm;
  x.n_sm_score = n_sm - reserved > 0 ? n_sm - reserved : 1;
  const int Hkv = c.n_kv_heads, n_pairs = n_req * Hkv;
  std::vector<ReqInfo> reqs(n_req > 0 ? n_req : 1);
  for (int r = 0; r < n_req; ++r) {
    memset(&reqs[r], 0, sizeof(ReqInfo));
    reqs[r].cu = cu[r];
    reqs[r].N = (int32_t)(cu[r + 1] - cu[r]);
    reqs[r].n = reqs[r].N - c.window;
  }
  x.h_req = reqs.data();
  x.max_tc_segs = (int32_t)tc_max_segments(c, n_sm);
  x.max_tc_ops = 3 * x.max_tc_segs + 8;
  std::vector<ScoreOp> ops((size_t)x.max_tc_ops);
  std::vector<int32_t> index(tc_index_size(n_pairs, n_sm));
  x.h_tc_ops = ops.data();
  x.h_tc_index = index.data();
  const int32_t rc = tc_build_plan(&x, n_req);
  info8[0] = x.n_tc_ctas; info8[1] = x.n_tc_waves; info8[2] = x.tc_merge_ways; info8[3] = x.n_tc_asegs;
  info8[4] = x.n_tc_bsegs; info8[5] = x.n_tc_ops_full; info8[6] = x.n_tc_ops_b; info8[7] = 0;
  if (rc != CAKE_OK || x.n_tc_ctas == 0) return rc;
  auto fail = [&](int what) { info8[7] = what; return (int32_t)CAKE_ERR_STATE; };
  if (x.n_tc_ops_full + x.n_tc_ops_b > x.max_tc_ops || x.n_tc_asegs > x.max_tc_segs ||
      x.n_tc_bsegs > x.max_tc_segs) return fail(4);
  // waves as the builder forms them
  std::vector<int> wave_of(n_pairs, 0);
  {
    const std::vector<int> wb = tc_waves(reqs.data(), n_req, Hkv, c.head_dim);
    for (int wv = 0; wv + 1 < (int)wb.size(); ++wv)
      for (int p = wb[wv]; p < wb[wv + 1]; ++p) wave_of[p] = wv;
  }
  const int32_t* cta_full = index.data() + 3 * (n_pairs + 1);
  // 1: coverage, per pair and pass, in tiles
  std::vector<std::vector<int>> cover[2];
  for (int ph = 0; ph < 2; ++ph) {
    cover[ph].resize(n_pairs);
    for (int p = 0; p < n_pairs; ++p) {
      const ReqInfo& rq = reqs[p / Hkv];
      cover[ph][p].assign(((ph ? rq.n : rq.N) + TILE - 1) / TILE, 0);
    }
  }
  for (int cta = 0; cta < x.n_tc_ctas; ++cta) {
    int last_b_wave = -1;
    std::vector<int> first_b_pos(x.n_tc_waves + 1, -1);
    std::vector<int> last_a_pos(x.n_tc_waves + 1, -1);
    for (int o = cta_full[cta]; o < cta_full[cta + 1]; ++o) {
      const ScoreOp& op = ops[o];
      const int p = op.req * Hkv + op.g;
      if (p < 0 || p >= n_pairs || op.key0 % TILE != 0 || op.nkeys <= 0) return fail(1);
      if (op.seg < 0 || op.seg >= (op.phase ? x.n_tc_bsegs : x.n_tc_asegs)) return fail(4);
      const int t0 = op.key0 / TILE, t1 = (op.key0 + op.nkeys + TILE - 1) / TILE;
      if (t1 > (int)cover[op.phase][p].size()) return fail(1);
      for (int t = t0; t < t1; ++t) cover[op.phase][p][t] += 1;
      const int wv = wave_of[p], pos = o - cta_full[cta];
      if (op.phase) {
        if (wv < last_b_wave) return fail(2);
        last_b_wave = wv;
        if (first_b_pos[wv] < 0) first_b_pos[wv] = pos;
      } else {
        last_a_pos[wv] = pos;
      }
    }
    for (int w = 0; w < x.n_tc_waves; ++w)
      if (first_b_pos[w] >= 0)
        for (int w2 = 0; w2 <= w; ++w2)
          if (last_a_pos[w2] > first_b_pos[w]) return fail(2);
    // 5: between two uses of a slot lies a use whose barrier the first one's readers and the second one's
    // writers both meet: any use after a pass-A op (its readers and writers are of one group), a pass-B op
    // after a direct merge
    if (tc_reps(x.rows) > 1 || x.tc_direct) {
      uint32_t n_a = 0, n_b = 0;
      int last[2] = {-1, -1}, last_phase[2] = {0, 0}, uses = 0, last_merge = -1;
      for (int o = cta_full[cta]; o < cta_full[cta + 1]; ++o) {
        const int phase = ops[o].phase;
        if (phase ? x.tc_direct : tc_reps(x.rows) > 1) {
          const int slot = xrow_slot(n_a, n_b);
          if (last[slot] >= 0 && (last_phase[slot] ? last_merge : uses - 1) <= last[slot]) return fail(5);
          last[slot] = uses;
          last_phase[slot] = phase;
          if (phase) last_merge = uses;
          ++uses;
        }
        // kbs counts the pass-B ops of the direct merge only
        if (!phase) ++n_a;
        else if (x.tc_direct) ++n_b;
      }
    }
  }
  for (int ph = 0; ph < 2; ++ph)
    for (int p = 0; p < n_pairs; ++p)
      for (int v : cover[ph][p])
        if (v != 1) return fail(1);
  // 3: merge groups
  const int32_t* group_begin = index.data() + 2 * (n_pairs + 1);
  if (group_begin[0] != 0 || group_begin[x.n_tc_groups] != n_pairs) return fail(3);
  for (int gi = 0; gi < x.n_tc_groups; ++gi) {
    const int p0 = group_begin[gi], p1 = group_begin[gi + 1] - 1;
    if (p1 < p0 || p1 - p0 >= x.tc_merge_ways || wave_of[p1] != wave_of[p0]) return fail(3);
    if (x.n_tc_waves == 1 && p0 != gi * x.tc_merge_ways) return fail(3);
  }
  return CAKE_OK;
}

int32_t launch_score_tc(cake_ctx* ctx, int32_t layer, const void* q_win, const void* k,
                        const float* lse, cudaStream_t st) {
  const cake_config& c = ctx->cfg;
  if (ctx->n_tc_ctas == 0) return CAKE_OK;
  if ((int64_t)c.n_kv_heads * ctx->total_tokens >= ((int64_t)1 << 31)) return CAKE_ERR_ARG;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return CAKE_ERR_CUDA;
  const int G = c.n_q_heads / c.n_kv_heads;
  CUtensorMap qmap, kmap;
  {
    // K [rows][d] seen as (64 elements, rows, d/64 slabs): one box of 128 rows brings both
    // 64-element halves of the rows, each as its own 128-byte-swizzled slab
    const cuuint64_t dims[3] = {64, (cuuint64_t)c.n_kv_heads * ctx->total_tokens, (cuuint64_t)(c.head_dim / 64)};
    const cuuint64_t strides[2] = {(cuuint64_t)c.head_dim * 2, 128};
    const cuuint32_t box[3] = {64, TILE, (cuuint32_t)(c.head_dim / 64)};
    const cuuint32_t es[3] = {1, 1, 1};
    if (enc(&kmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(k), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return CAKE_ERR_CUDA;
  }
  {
    // [req][head][i][d] viewed as (d, head, i, req) so that a box lands as rows r' = i*G + h
    const cuuint64_t dims[4] = {(cuuint64_t)c.head_dim, (cuuint64_t)c.n_q_heads, (cuuint64_t)c.window,
                                (cuuint64_t)ctx->n_req};
    const cuuint64_t strides[3] = {(cuuint64_t)c.window * c.head_dim * 2, (cuuint64_t)c.head_dim * 2,
                                   (cuuint64_t)c.n_q_heads * c.window * c.head_dim * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)G, (cuuint32_t)c.window, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    if (enc(&qmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(q_win), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return CAKE_ERR_CUDA;
  }
  const int n_pairs = ctx->n_req * c.n_kv_heads;
  TcParams P;
  P.ops = ctx->d_tc_ops;
  // with one wave the groups are those of the plain rule, which spares the merger a read per group
  P.group_begin = ctx->n_tc_waves > 1 ? ctx->d_tc_index + 2 * (n_pairs + 1) : nullptr;
  P.n_groups = ctx->n_tc_groups;
  P.pair_aseg = ctx->d_tc_index;
  P.lse2 = (uint2*)ctx->d_tc_exch;
  P.lse_ext = lse;
  P.rowpart = (float4*)(ctx->d_tc_exch + (size_t)n_pairs * 128 * kLseStride * sizeof(uint2));
  P.raw = ctx->d_raw[layer % ctx->score_depth];
  P.colpart = ctx->d_colpart[layer % ctx->score_depth];
  P.hrow = ctx->d_hrow[layer % ctx->score_depth];
  P.n_pairs = n_pairs;
  P.status = ctx->d_status;
  P.Hkv = c.n_kv_heads; P.Hq = c.n_q_heads; P.Sw = c.window; P.rows = ctx->rows; P.d = c.head_dim;
  P.scale2 = kLog2e / sqrtf((float)c.head_dim);
  P.inv_scale2 = 1.f / P.scale2;
  P.gamma = c.gamma;
  P.ind_mode = c.indicator_mode;
  P.merge_ways = ctx->tc_merge_ways;
  P.reps = tc_reps(ctx->rows);
  P.spin_limit = ctx->wait_limit_cycles > 0 ? ctx->wait_limit_cycles : kSpinLimit;
  P.bessel = c.var_ddof ? (float)c.window / (float)(c.window - 1) : 1.f;

  const int sp = prof_begin(ctx, CAKE_PROF_SCORE, st);
  P.cta_op = ctx->d_tc_index + 3 * (n_pairs + 1);
  if (lse) {
    // denominators supplied: pass B alone, entropy from its columns
    ctx->hhead_from_rows = false;
    P.cta_op += ctx->n_sm + 1;
    P.both = 0;
    P.tag = P.want = 0;
  } else {
    ctx->hhead_from_rows = true;
    P.both = 1;
    P.tag = ++ctx->tc_tag;
    P.want = P.tag + (uint32_t)ctx->debug_epoch_skew;
  }
  cudaError_t e;
  const bool eb = lse != nullptr;
  // An early start takes SMs from the cascade kernels.  The column pass of a single wave is so short that
  // these set the pace: it starts when the launch before it is done (32 layers of 16 heads and 12.7K keys:
  // 730 us with an early start, 690 without).
  const bool early = !(eb && ctx->n_tc_waves == 1);
  switch (G) {
    case 1: e = launch_g<1>(ctx->device, eb, P.reps > 1, ctx->tc_direct, early, ctx->n_tc_ctas, st, qmap, kmap, P); break;
    case 2: e = launch_g<2>(ctx->device, eb, P.reps > 1, ctx->tc_direct, early, ctx->n_tc_ctas, st, qmap, kmap, P); break;
    case 4: e = launch_g<4>(ctx->device, eb, P.reps > 1, ctx->tc_direct, early, ctx->n_tc_ctas, st, qmap, kmap, P); break;
    default: e = launch_g<8>(ctx->device, eb, P.reps > 1, ctx->tc_direct, early, ctx->n_tc_ctas, st, qmap, kmap, P); break;
  }
  count_launch();
  prof_end(ctx, sp, st);
  return cuda_status(e);
}

}  // namespace cake

// sm_103a masked prefill attention on the 5th-generation tensor cores (Sec. 3.1: the modified
// causal mask over every token of a prompt block).
//
// Work items are (sequence, head, 128-query tile); the queries are the last tokens of each
// sequence's history, the keys the sequence's stored rows of one layer, read straight from the
// ragged cache.  Persistent CTAs (two per SM for d_head 64 and 80, one otherwise) take the items one by
// one in the host's order.  Per CTA:
//
//   warps 0..3   softmax, one query row per thread: tcgen05.ld of its S row, the per-key rule on the
//                tiles that need it, an online softmax in the exp2 domain, P (16-bit) back into TMEM,
//                the rare rescale of its O row, and the final O / l
//   warp 4       takes the work items and sorts the keys of the tiles that need the per-key rule
//   warp 5       one thread issues tcgen05.mma: S = Q K^T into TMEM, then O += P V with P read from
//                TMEM; completions are signalled with tcgen05.commit
//   warps 6, 7   stream the K tiles and the V tiles, each through a ring of shared-memory stages
//
// Mask (Sec. 3.1, the same rows a decode at the query would see): stored row i is visible to the
// query at stored row iq exactly when i <= iq <= hid(i), except that a <CL> query sees only itself.
// hid(i) is the stored row of the <CR> that closes a span enclosing row i (its interior stops being
// visible after the <CR>), i itself for a <CL> row under the paper policy, and "never" otherwise;
// the host book computes it per stored row.
//
// Only keys that some query of a tile may see are fetched: the rows that no span hides, from a list of
// them, and the rows of the tile itself with the interior of a span it begins in.  A tile of keys whose
// rows lie side by side is one TMA copy (2-D tiled, swizzled); else its rows are gathered with 16-byte
// asynchronous copies into the same swizzled layout.
//
// What bounds it: the softmax warps' instructions (exp2, max and packing of 128 scores a row), and, since the
// eight warps of a CTA run five different programs, the instruction cache: every stretch of straight-line code
// taken out paid more than its instructions' issue slots.  So waits are one short loop, the epilogue and the
// masking exist once, and nothing but the softmax is unrolled far.  Time of a layer, against a kernel that read
// every stored row with masks over all of them: OPT-1.3B-shaped prompts (16 x 2048 tokens, 32 heads of 64,
// interiors of 32) 541 -> 250 us; 24 ragged rotary prompts (256 to 4096 tokens, heads of 80) 1587 -> 738 us; the
// last 512 of 32 x 4096 tokens, compacted before them, bf16 (heads of 80) 664 -> 327 us; the first with 96 and
// 128 columns 797 -> 385 and 1042 -> 421 us; one prompt of 300 tokens 13.2 -> 10.8 us.  (Copying the listed rows
// side by side first, for TMA tiles alone, took a second kernel and 381, 992 and 454 us on the first three when
// the gathers took 372, 1026 and 450.)
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "device_common.cuh"
#include "kernels.hpp"

namespace kvc {
namespace {

constexpr int kPfRows = 128;  // queries per tile (MMA M)
// Threads: a softmax warpgroup (one thread per query row), then a warpgroup of the four other roles' warps
// (so that registers can be moved between the two).
constexpr int kPfThreads = 256;
constexpr int kItemRing = 4;  // a power of two: the item in hand, the ones before and after it
constexpr int kClsRing = 2;  // sorted key tiles ahead of the softmax

// Shared-memory geometry for head dimension D.  Q ([128 rows][D]), K and V tiles ([KT rows][D]) are split into
// column subtiles of SW bytes per row, the widest swizzle (128 / 64 / 32 bytes) that divides a row;
// each subtile is the canonical K-major (Q, K) or MN-major (V) layout of that swizzle.
//
// SPLIT (bf16): the rotated query and the softmax weights P each go to the tensor cores as a high and
// a low 16-bit part (x = hi + lo with hi = bf16(x), lo = bf16(x - hi), 16 significant bits together),
// so q.k and P.V keep the precision that f16 operands give in one part.  With bf16's 8-bit
// significand a single part moves q.k and the P weights by up to 2^-9 relative, more than the
// decode tolerance allows; the low parts cost a second pass of each product on the tensor cores.
template <int D, bool SPLIT_ = false>
struct PfCfg {
  static constexpr bool SPLIT = SPLIT_;
  static constexpr int SW = (2 * D) % 128 == 0 ? 128 : (2 * D) % 64 == 0 ? 64 : 32;
  static constexpr int SUB = SW / 2;  // columns per subtile
  static constexpr int NSUB = D / SUB;
  // d_head 64 and 80 run two CTAs per SM (their softmax steps interleave), each with a single S
  // tile in TMEM; larger heads run one CTA per SM with a double-buffered S tile.
  static constexpr int CPS = (D == 64 || D == 80) ? 2 : 1;  // CTAs per SM
  static constexpr int SBUF = CPS == 2 ? 1 : 2;              // S tiles in TMEM
  static constexpr bool PSEP = CPS == 2;                     // P in TMEM columns of its own
  // Keys per tile (QK^T N, PV K): with two CTAs per SM as many as leave TMEM columns for a P of its own
  // (d_head 80, OPT-2.7B-shaped blocks in bf16: 128 keys with P over S 534 us, 64 with P apart 505).
  static constexpr int KT = !PSEP ? 128 : SPLIT ? 64 : D == 80 ? 112 : 128;
  static constexpr uint32_t QSUBB = kPfRows * SW;  // bytes of one subtile of Q
  static constexpr uint32_t SUBB = KT * SW;        // of K or V
  static constexpr uint32_t QTILE = kPfRows * D * 2;
  static constexpr uint32_t TILE = KT * D * 2;
  // SPLIT: the low part of the rotated query, the A operand of a second Q.K^T pass, lives in TMEM
  // with two CTAs per SM (whose shared memory is full) and in shared memory with one
  static constexpr bool QLO_TMEM = SPLIT && CPS == 2;
  static constexpr bool QLO_SMEM = SPLIT && CPS == 1;
  // stages of the K and of the V ring
  static constexpr int KST = CPS == 2 ? (SPLIT ? 3 : 2) : D <= 96 || !SPLIT ? 3 : 2;
  static constexpr int VST = CPS == 2 ? (SPLIT ? 3 : 2) : D <= 96 ? 3 : 2;
  static constexpr uint32_t Q_OFF = 0;
  static constexpr uint32_t QLO_OFF = QTILE;  // QLO_SMEM only
  static constexpr uint32_t K_OFF = QTILE * (QLO_SMEM ? 2 : 1);
  static constexpr uint32_t V_OFF = K_OFF + KST * TILE;
  static constexpr uint32_t SMEM = V_OFF + VST * TILE + 1024;  // + aligning the base
  // TMEM.  Two CTAs per SM, 256 columns each: S, O, P (16-bit, two per column; SPLIT: its high part, then
  // its low part) and SPLIT's low part of the query (D / 2 columns) in columns of their own, so S is
  // released as soon as the softmax has read it and the next Q.K^T overlaps the softmax.  One CTA per SM:
  // S0, S1, P written over the first half of its own S tile (SPLIT: the low part over the other), then
  // O0 and O1 (alternating per item).
  static constexpr int OBUF = SBUF == 1 ? 1 : 2;
  static constexpr uint32_t O_COL = SBUF == 2 ? 2 * KT : KT;
  static constexpr uint32_t P_COL = PSEP ? KT + D : 0;  // 0: P lives in its S tile
  static constexpr uint32_t PLO_COL = KT / 2;           // SPLIT: P's low part, after its high part
  static constexpr uint32_t QLO_COL = P_COL + KT;       // QLO_TMEM only
  static constexpr uint32_t TMEM_END = !PSEP ? O_COL + OBUF * D : SPLIT ? QLO_COL + D / 2 : P_COL + KT / 2;
  static constexpr uint32_t TMEM_COLS = TMEM_END <= 256 ? 256 : 512;
  static_assert(TMEM_END <= TMEM_COLS && TMEM_COLS * CPS <= 512, "TMEM budget");
  static_assert(D % 16 == 0 && SW * NSUB == 2 * D, "bad tile geometry");
  static_assert(SMEM <= 227 * 1024 && (CPS == 1 || SMEM + 6 * 1024 <= 113 * 1024), "shared memory budget");
  // Registers with two CTAs per SM: each thread is launched with REG_LAUNCH, then the other roles'
  // warpgroup gives registers up (setmaxnreg.dec to REG_OTHER) and the softmax warpgroup takes them
  // (setmaxnreg.inc to REG_SOFTMAX); the two shares add up to exactly what the CTA was launched with.
  static constexpr int REG_LAUNCH = 65536 / (CPS * kPfThreads);
  static constexpr int REG_OTHER = 56;
  static constexpr int REG_SOFTMAX = (REG_LAUNCH * kPfThreads - REG_OTHER * 128) / 128 / 8 * 8;
  static_assert(CPS == 1 || REG_SOFTMAX * 128 + REG_OTHER * 128 <= REG_LAUNCH * kPfThreads,
                "setmaxnreg shares exceed the launch allocation");
  static_assert(CPS == 1 || (REG_SOFTMAX <= 256 && REG_SOFTMAX % 8 == 0 && REG_OTHER % 8 == 0), "setmaxnreg range");
};

// ---------------------------------------------------------------------------------------------
// tcgen05 / TMA wrappers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D (TMEM) += A (TMEM, M rows in lanes, two 16-bit elements per column) x B (shared memory).
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// 16 TMEM lanes of 8 n columns: lane l gets of columns 8 c + 2 (l % 4) and the next those of rows l / 4 (v[4 c],
// v[4 c + 1]) and l / 4 + 8 (v[4 c + 2], v[4 c + 3]).
__device__ __forceinline__ void tmem_ld_16x256b_x2(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x2.b32 {"
      "%0,%1,%2,%3,%4,%5,%6,%7"
      "}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {"
      "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15"
      "}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st8u(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st4u(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Shared-memory matrix descriptor: start address, leading / stride byte offsets, version 1, and
// the swizzle (layout type 2 = 128 B, 4 = 64 B, 6 = 32 B).  Its low word holds the address and the leading
// offset, so a tile's descriptors are one word plus constants (addresses stay below 256 KB).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return addr >> 4 | (lbo >> 4) << 16; }
__device__ __forceinline__ uint64_t desc(uint32_t lo, uint32_t sbo, int sw) {
  const uint32_t hi = (sbo >> 4) | 1u << 14 | (sw == 128 ? 2u : sw == 64 ? 4u : 6u) << 29;
  return (uint64_t)hi << 32 | lo;
}
// Instruction descriptor of kind::f16 with an fp32 accumulator: A and B of one 16-bit type
// (0 = f16, 1 = bf16), A K-major, B K-major (0) or MN-major (1), N >> 3, M >> 4.
__host__ __device__ constexpr uint32_t mma_idesc(int ab_type, int b_mn_major, int M, int N) {
  return (1u << 4) | ((uint32_t)ab_type << 7) | ((uint32_t)ab_type << 10) | ((uint32_t)b_mn_major << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

template <typename T>
struct Pack16;
template <>
struct Pack16<F16T> {
  static constexpr int kType = 0;
  static __device__ __forceinline__ uint32_t two(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
  }
};
template <>
struct Pack16<BF16T> {
  static constexpr int kType = 1;
  static __device__ __forceinline__ uint32_t two(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
  }
};

// The two bf16 values of a packed pair as exact binary32 values (low half first).
__device__ __forceinline__ float2 bf16x2_to_float2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}
// SPLIT: x = hi + lo with hi, lo bf16 (a pair at a time): *hi = bf16(x) and the low part is the
// bf16 rounding of x - hi, which binary32 holds exactly (x and hi agree in their leading bits).
__device__ __forceinline__ uint32_t bf16_split2(float2 x, uint32_t* hi) {
  *hi = Pack16<BF16T>::two(x.x, x.y);
  const float2 h = bf16x2_to_float2(*hi);
  const float2 d = __ffma2_rn(h, make_float2(-1.f, -1.f), x);
  return Pack16<BF16T>::two(d.x, d.y);
}

// rope_sincos (device_common.cuh) of two frequencies (hi, hi, lo, lo) at position p, with packed instructions and the
// same roundings: sines, their negatives, cosines.  (Ragged rotary prompts 747 us a layer with rope_sincos, 740 so.)
// The turns' whole part comes off with scalar subtractions: a packed sum of a packed product is fused with it by the
// compiler, its explicit rounding notwithstanding, and loses the product's rounding error that e holds.
__device__ __forceinline__ void rope_sincos2(float p, float4 g, float2* s, float2* ns, float2* c) {
  const float2 p2 = make_float2(p, p), gh = make_float2(g.x, g.y);
  const float2 a = __fmul2_rn(p2, gh);
  const float2 e = __ffma2_rn(p2, gh, make_float2(-a.x, -a.y));
  const float2 turn = make_float2(__fsub_rn(a.x, rintf(a.x)), __fsub_rn(a.y, rintf(a.y)));
  const float2 f = __fadd2_rn(turn, __ffma2_rn(p2, make_float2(g.z, g.w), e));
  const float2 t = __fmul2_rn(make_float2(6.28318530717958647692f, 6.28318530717958647692f), f);
  __sincosf(t.x, &s->x, &c->x);
  __sincosf(t.y, &s->y, &c->y);
  *ns = make_float2(-s->x, -s->y);
}

template <typename T>
constexpr bool kSplit = false;
template <>
constexpr bool kSplit<BF16T> = true;

// 16-byte global -> shared copy that does not go through registers (src_bytes 0: zero fill).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// Arrives on the barrier (within its expected count) once this thread's asynchronous copies so far have
// completed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// Waits for every asynchronous copy of this thread, committed or not.
__device__ __forceinline__ void cp_async_wait_all_groups() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}


// Bits [0, n) of a 32-bit word, n clamped to [0, 32].
__device__ __forceinline__ uint32_t low_bits(int n) {
  uint32_t r;
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(r) : "r"(max(n, 0)));
  return r;
}
// The maximum, NaN if one of them is.
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// A value that is the warp's, so that the compiler knows it to be.
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xFFFFFFFFu, x, 0); }

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
  return one != 0;
}

// Bounded wait for the phase with the given parity: false after limit_ns (< 2^32).  A few instructions,
// because it is inlined at many places of one kernel whose warps run different code at the same time, and
// the instruction cache holds only so much of that; each role reports a wait that ran out when it ends.
__device__ __forceinline__ bool pf_wait(uint64_t* bar, uint32_t parity, uint32_t limit_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 t0, t;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra DONE;\n\t"
      "mov.u32 t0, %%globaltimer_lo;\n\t"
      "LOOP:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra DONE;\n\t"
      "mov.u32 t, %%globaltimer_lo;\n\t"
      "sub.u32 t, t, t0;\n\t"
      "setp.lt.u32 q, t, %3;\n\t"
      "@q bra LOOP;\n\t"
      "DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(limit_ns)
      : "memory");
  return ok != 0;
}

// One work item (kernels.hpp, PfItemRec and its PfTileRec), read from the host's tables; nk = 0: none left.
struct PfItem {
  int n_c, b0, tok0, moff;
  int s, h, qr0, qr_end, nk;
  int odd;       // the item's number is odd
  int row_base;  // K/V plane row of stored row 0 of (layer, s, h)
  int vb;
  // keys before the tile's own rows; the first of those (kt keys per tile); one past the last key
  __device__ __forceinline__ int before() const { return n_c + (qr0 - b0); }
  __device__ __forceinline__ int own(int kt) const {
    return kPfRows % kt == 0 ? (before() + kt - 1) / kt * kt : before();
  }
  __device__ __forceinline__ int keys(int kt) const { return own(kt) + (qr_end - qr0); }
  // Key tile of the j-th step: consecutive items run their key tiles in opposite directions, so an item
  // starts on the tiles its predecessor (same (sequence, head), most often) read last, while they are
  // still in L2.
  __device__ __forceinline__ int key_tile(int j) const { return odd ? nk - 1 - j : j; }
};

__device__ __forceinline__ PfItem pf_item(const PrefillArgs& a, int64_t it) {
  const int2 t = __ldg(reinterpret_cast<const int2*>(a.items + it));
  const int4* r = reinterpret_cast<const int4*>(a.tiles + t.x);
  const int4 x = __ldg(r), y = __ldg(r + 1), z = __ldg(r + 2);
  PfItem w;
  w.n_c = x.x;
  w.b0 = x.y;
  w.tok0 = x.z;
  w.moff = x.w;
  w.s = y.x;
  w.h = t.y;
  w.qr0 = y.z;
  w.qr_end = y.w;
  w.nk = z.x;
  w.odd = (int)(it & 1);
  w.row_base = (int)((int64_t)a.layer * a.H * a.C) + z.y + t.y * y.y;  // all planes' rows are below 2^31
  w.vb = z.z;
  return w;
}

// Gathers rows p0 .. p0 + 31 of a tile (row: lane's own, -1 none: zeros) below row kt, subtiles U0 .. U0 + NS - 1, with
// 16-byte asynchronous copies.  Each quarter of the warp, whose 128 bytes are written to shared memory together,
// covers the chunks of one subtile in as many rows as fill its swizzle pattern, so that they fall into different
// banks; its quarters lie side by side in the rows, as far as the row goes (96 columns: 621 us with lanes in
// row order, 577 so).  The gathers bound tiles of many short runs: few instructions a step and many steps in flight
// (OPT-1.3B-shaped prompts, interiors of 32 / 8: 292 / 445 us with the swizzle worked out per step and two steps
// unrolled, 271 / 393 so with four; 80, 96, 128 columns: 886, 458, 556 us with four, 867, 446, 490 with all).
template <int D, int SW, int U0, int NS>
__device__ __forceinline__ void gather_rows(uint32_t dst, uint32_t subb, const uint16_t* rows, int row, int p0, int kt,
                                            int lane) {
  constexpr int CH = SW / 16, RQ = 8 / CH;  // chunks of a subtile's row, rows of a quarter
  constexpr int RPS = RQ * 4 / NS;          // rows of a step
  const int q = lane >> 3, cw = lane % CH, u = U0 + q % NS, pr = q / NS * RQ + lane % 8 / CH;
  const uint16_t* src = rows + u * (SW / 2) + cw * 8;
  // the swizzle of row p = pr + i (a step's rows are aligned to their number) is that of pr and that of i
  constexpr int SH = SW == 128 ? 0 : SW == 64 ? 1 : 2;
  dst += u * subb + (p0 + pr) * SW;
  const int c0 = cw ^ (pr >> SH & (CH - 1));
#pragma unroll
  for (int i = 0; i < 32; i += RPS) {
    if (i >= 16 && kt - p0 < 32) break;  // 16 rows
    const int x = __shfl_sync(0xFFFFFFFFu, row, pr + i);
    const int phys = c0 ^ (i >> SH & (CH - 1));
    cp_async16(dst + i * SW + phys * 16, src + (int64_t)max(x, 0) * D, x < 0 ? 0u : 16u);
  }
}

// Persistent: the CTAs take items in the table's order from the launch's counter, one at a time (warp 4
// takes an item when the K warp is through with the last one and passes it on); every
// barrier phase counts tiles over all of the CTA's items, so the producer streams the next item's
// K/V while the current one finishes (with two S tiles, the O accumulator also alternates between
// two TMEM buffers per item).
// ROT: the queries are rotated (RoPE).  A kernel of its own without that code, because the instruction cache holds
// little more than one of them: OPT-1.3B-shaped prompts 327 -> 299 us, compacted bf16 prompts 441 -> 400.
template <typename T, int D, bool ROT>
__global__ void __launch_bounds__(kPfThreads, PfCfg<D>::CPS)
    prefill_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_q, const PrefillArgs a) {
  using Cf = PfCfg<D, kSplit<T>>;
  constexpr int SW = Cf::SW, SUB = Cf::SUB, KST = Cf::KST, VST = Cf::VST, SBUF = Cf::SBUF, KT = Cf::KT;
  extern __shared__ uint8_t pf_smem_raw[];
  __shared__ uint64_t k_full[KST], k_empty[KST], v_full[VST], v_empty[VST], s_full[SBUF], s_free;
  // the item's raw query rows are in; rotated (RoPE); its last Q.K^T is complete
  __shared__ uint64_t q_raw, q_full, q_empty;
  __shared__ uint64_t p_full, pv_done, drain;
  // the CTA's k-th item in slot k % kItemRing; full: warp 4 has written it, empty: the MMA thread, the K and V
  // warps and the four softmax warps are through with it, last: the K warp has issued its last tile
  __shared__ PfItem item_slot[kItemRing];
  __shared__ uint64_t item_full[kItemRing], item_empty[kItemRing], item_last;
  // For the key tiles that hold rows from b0 on, the tile's keys against its item's query tile
  // [qr0, qr_end): khid has bit c set when key c's bound holds for every query of the tile (hid >=
  // qr_end - 1).  The keys whose bound falls inside it (qr0 <= hid < qr_end - 1: a span closing among
  // the queries; a <CL> hidden from every later query) go by their bound: kend has bit hid - qr0 set for
  // each such bound, and kafter[i] are the keys whose bound is the i-th of those or a later one, so a
  // query finds all of them that it may see with one lookup (a loop over the spans in each softmax thread
  // before: OPT-1.3B-shaped prompts 333 us, 327 so).
  __shared__ uint4 khid[kClsRing], kend[kClsRing];
  __shared__ uint4 kafter[kClsRing][KT + 1];
  __shared__ int8_t bound[128];  // of the tile being sorted
  __shared__ int32_t kslow[kClsRing];  // the tile needs the per-key rule (else every key is visible)
  __shared__ uint64_t cls_full[kClsRing], cls_empty[kClsRing];
  // a.rope_g, two frequencies at a time: (hi, hi, lo, lo).  (Read from global memory in each item, with two words of
  // a row in flight: ragged rotary prompts 985 us, 949 so with eight.)
  __shared__ float4 rope_s[D / 4];
  __shared__ uint32_t tmem_slot;

  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(pf_smem_raw) + 1023) & ~uintptr_t(1023));
  // The warp's number and the TMEM base through a shuffle, which the compiler knows to be the warp's (OPT-1.3B-shaped
  // prompts 264 us a layer, 253 so; ragged rotary prompts 850 -> 753; heads of 96 430 -> 390, of 128 466 -> 426).
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(Cf::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (ROT && threadIdx.x >= 64 && threadIdx.x < 64 + a.rot / 4) {
    const float2 g0 = a.rope_g[2 * (threadIdx.x - 64)], g1 = a.rope_g[2 * (threadIdx.x - 64) + 1];
    rope_s[threadIdx.x - 64] = make_float4(g0.x, g1.x, g0.y, g1.y);
  }
  if (threadIdx.x == 32) {
    for (int i = 0; i < KST; ++i) {
      mbar_init(&k_full[i], 32);
      mbar_init(&k_empty[i], 1);
    }
    for (int i = 0; i < VST; ++i) {
      mbar_init(&v_full[i], 32);
      mbar_init(&v_empty[i], 1);
    }
    for (int i = 0; i < kClsRing; ++i) {
      mbar_init(&cls_full[i], 1);
      mbar_init(&cls_empty[i], 4);
    }
    for (int i = 0; i < SBUF; ++i) mbar_init(&s_full[i], 1);
    mbar_init(&s_free, 128);  // one S tile: the softmax has read it
    mbar_init(&q_raw, 1);
    mbar_init(&q_full, 128);
    mbar_init(&q_empty, 1);
    mbar_init(&p_full, 128);
    mbar_init(&pv_done, 1);
    mbar_init(&drain, 1);
    for (int i = 0; i < kItemRing; ++i) {
      mbar_init(&item_full[i], 1);
      mbar_init(&item_empty[i], 1 + 2 + 4);
    }
    mbar_init(&item_last, 1);
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(tmem_slot);
  const uint32_t limit_ns = (uint32_t)a.wait_limit_ns;
  bool ok = true;  // false once one of this role's waits has run out
  // At the two-CTA register cap, registers go from the other roles' warpgroup to the softmax: each
  // role starts with its setmaxnreg (every warp of a warpgroup executes the same one).
  auto regs_other = [] {
    if constexpr (Cf::CPS == 2) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Cf::REG_OTHER));
  };

  // Waits for the CTA's kk-th item, in item_slot[kk % kItemRing] (false: the wait gave up); done: a whole
  // warp is through with it.
  auto item_wait = [&](uint32_t kk) -> bool {
    return pf_wait(&item_full[kk % kItemRing], (kk / kItemRing) & 1, limit_ns);
  };
  auto item_done = [&](uint32_t kk) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&item_empty[kk % kItemRing]);
  };

  if (warp == 4) {
    regs_other();
    // ---------------- items and key classes ----------------
    uint32_t cg = 0;  // tiles sorted
    for (uint32_t k = 0; ok; ++k) {
      // take the next item, once the K warp is through with the last one (no CTA holds an item that
      // another could start on), and pass it on
      if (k >= 1) ok = pf_wait(&item_last, (k - 1) & 1, limit_ns);
      if (ok && k >= kItemRing) ok = pf_wait(&item_empty[k % kItemRing], (k / kItemRing - 1) & 1, limit_ns);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) break;
      if (lane == 0) {
        const unsigned long long t = atomicAdd(a.item_counter, 1ull);
        if (t < (unsigned long long)a.n_items)
          item_slot[k % kItemRing] = pf_item(a, (int64_t)t);
        else
          item_slot[k % kItemRing].nk = 0;
        mbar_arrive(&item_full[k % kItemRing]);
      }
      __syncwarp();
      const PfItem w = item_slot[k % kItemRing];
      if (w.nk == 0) break;
      const int own = w.own(KT), keys = w.keys(KT), before = w.before();
      for (int j = 0; j < w.nk; ++j) {
        const int v0 = KT * w.key_tile(j);
        if (v0 + KT <= w.n_c) continue;  // rows that no span hides, all before the queries
        const int cs = (int)(cg % kClsRing);
        // per-key mask bounds of the tile ((hid << 1) | is_cl) sorted into the classes above; the causal
        // part (i <= iq) is left to each query
        if (cg >= kClsRing && !(ok = __all_sync(0xFFFFFFFFu, pf_wait(&cls_empty[cs], (cg / kClsRing - 1) & 1, limit_ns))))
          break;
        uint32_t* hid_w = reinterpret_cast<uint32_t*>(&khid[cs]);
        uint32_t* end_w = reinterpret_cast<uint32_t*>(&kend[cs]);
        uint32_t my_end = 0u;  // word `lane` of kend
        constexpr int NW = (KT + 31) / 32;
        // (a rolled loop: this warp has some time, the instruction cache no room -- unrolled OPT-1.3B-shaped prompts
        // take 302 us, 293 so; with the loops below rolled too, 299, and one prompt of 300 tokens 12.0 for 11.0)
#pragma unroll 1
        for (int w4 = 0; w4 < NW; ++w4) {
          const int c = lane + 32 * w4, v = v0 + c;
          int hid = w.qr_end;  // a row that no span hides
          if (c >= KT || v >= keys || (v >= before && v < own))
            hid = -2;  // no key
          else if (v >= w.n_c)
            hid = a.meta[w.moff + (v >= own ? w.qr0 + (v - own) : w.b0 + (v - w.n_c))] >> 1;
          const uint32_t all = __ballot_sync(0xFFFFFFFFu, hid >= w.qr_end - 1);
          // the key's bound from the first query on when it falls among the queries, else -1
          const int h = hid >= w.qr0 && hid < w.qr_end - 1 ? hid - w.qr0 : -1;
          bound[c] = (int8_t)h;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t e = __reduce_or_sync(0xFFFFFFFFu, h >> 5 == u ? 1u << (h & 31) : 0u);
            if (lane == u) my_end |= e;
          }
          if (lane == 0) hid_w[w4] = all;
        }
        if (lane < 4) end_w[lane] = my_end;
        __syncwarp();
        int n_end = 0;
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
          for (uint32_t left = __shfl_sync(0xFFFFFFFFu, my_end, u); left != 0u; left &= left - 1u, ++n_end) {
            const int h = 32 * u + __ffs(left) - 1;
            uint32_t m[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int w4 = 0; w4 < NW; ++w4) m[w4] = __ballot_sync(0xFFFFFFFFu, bound[lane + 32 * w4] >= h);
            if (lane == 0) kafter[cs][n_end] = make_uint4(m[0], m[1], m[2], m[3]);
          }
        }
        __syncwarp();
        if (lane == 0) {
          kafter[cs][n_end] = make_uint4(0u, 0u, 0u, 0u);
          // per-key masking is needed when a key's visibility differs between the tile's queries: bounds
          // among them, and keys at or past the first query (the causal rule); and for columns without a key
          kslow[cs] = n_end > 0 || v0 + KT > before;
          mbar_arrive(&cls_full[cs]);
        }
        ++cg;
      }
    }
    // the last CTA to get here leaves the launch's counters at zero for the next launch
    if (lane == 0) {
      __threadfence();
      if (atomicAdd(a.item_counter + 1, 1ull) + 1 == gridDim.x) {
        a.item_counter[0] = 0;
        a.item_counter[1] = 0;
      }
    }
  } else if (warp >= 6) {
    regs_other();
    // ---------------- K (warp 6) and V (warp 7) tiles ----------------
    constexpr int NS1 = Cf::NSUB >= 4 ? 4 : Cf::NSUB >= 2 ? 2 : 1;  // subtiles of one step of a gather
    static_assert(Cf::NSUB - NS1 <= 1, "a gather's second pass takes one subtile");
    const bool is_v = warp == 7;
    const int nst = is_v ? VST : KST;
    uint64_t* full = is_v ? v_full : k_full;
    uint64_t* empty = is_v ? v_empty : k_empty;
    const uint32_t ring = smem_addr(sm + (is_v ? Cf::V_OFF : Cf::K_OFF));
    const CUtensorMap* tm = is_v ? &tm_v : &tm_k;
    const uint16_t* plane = is_v ? a.v : a.k;
    int st = 0;
    uint32_t ph = 1, issued = 0;  // parity of the stage's previous release; tiles issued
    uint32_t q_items = 0;         // items whose query rows were requested (warp 7)
    for (uint32_t k = 0; ok; ++k) {
      if (!(ok = __all_sync(0xFFFFFFFFu, item_wait(k)))) break;
      const PfItem w = item_slot[k % kItemRing];
      item_done(k);
      if (w.nk == 0) break;
      if (is_v) {
        // the item's query rows (past its last query another sequence's, or zeros past the last token: those
        // rows' results go nowhere), once the Q.K^T of the item before are complete
        if (k >= 1 && !(ok = __all_sync(0xFFFFFFFFu, pf_wait(&q_empty, (k - 1) & 1, limit_ns)))) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&q_raw, Cf::QTILE);
#pragma unroll
          for (int u = 0; u < Cf::NSUB; ++u)
            tma_load_3d(smem_addr(sm + Cf::Q_OFF) + u * Cf::QSUBB, &tm_q, u * SUB, w.h, w.tok0, &q_raw);
        }
        q_items = k + 1;
      }
      const int own = w.own(KT), keys = w.keys(KT), before = w.before();
      const uint16_t* rows = plane + (int64_t)w.row_base * D;
      for (int j = 0; j < w.nk; ++j) {
        const int v0 = KT * w.key_tile(j), v1 = v0 + KT;
        // rows side by side go in one copy: a tile of the list before its first gap, of the tile's own rows,
        // or of all rows up to its last one
        const bool in_list = v1 <= w.n_c && v1 <= w.vb, in_own = v0 >= own && v1 <= keys;
        const bool tiled = in_list || in_own || (w.n_c == w.b0 && own == before && v1 <= keys);
        int r0 = -1, r1 = -1, r2 = -1, r3 = -1;  // stored rows of keys v0 + 32 q + lane (-1: no key)
        if (!tiled) {
          auto key_row = [&](int v) -> int {
            if (v < w.n_c) return v < w.vb ? v : __ldg(a.klist + w.moff + v);
            if (v < before) return w.b0 + (v - w.n_c);
            return v >= own && v < keys ? w.qr0 + (v - own) : -1;
          };
          r0 = key_row(v0 + lane);
          r1 = key_row(v0 + 32 + lane);
          if (KT > 64) r2 = key_row(v0 + 64 + lane);
          if (KT > 96) r3 = key_row(v0 + 96 + lane);
        }
        if (issued >= (uint32_t)nst && !(ok = __all_sync(0xFFFFFFFFu, pf_wait(&empty[st], ph, limit_ns)))) break;
        const uint32_t dst = ring + st * Cf::TILE;
        if (tiled) {
          if (lane == 0) {
            mbar_expect_tx(&full[st], Cf::TILE);
            const int y = in_own ? w.row_base + w.qr0 + (v0 - own) : w.row_base + v0;
#pragma unroll
            for (int u = 0; u < Cf::NSUB; ++u) tma_load_2d(dst + u * Cf::SUBB, tm, u * SUB, y, &full[st]);
          }
          mbar_arrive(&full[st]);
        } else {
          // scattered rows
#pragma unroll 1
          for (int p0 = 0; p0 < KT; p0 += 32) {
            gather_rows<D, SW, 0, NS1>(dst, Cf::SUBB, rows, r0, p0, KT, lane);
            if constexpr (NS1 < Cf::NSUB) gather_rows<D, SW, NS1, 1>(dst, Cf::SUBB, rows, r0, p0, KT, lane);
            r0 = r1;
            r1 = r2;
            r2 = r3;
          }
          cp_async_arrive(&full[st]);
        }
        ++issued;
        if (++st == nst) {
          st = 0;
          ph ^= 1;
        }
      }
      if (ok && !is_v && lane == 0) mbar_arrive(&item_last);
    }
    cp_async_wait_all_groups();
    if (lane == 0) {
      // no copy is in flight when the CTA exits
      for (int n = issued < (uint32_t)nst ? (int)issued : nst; n > 0; --n) {
        if (st == 0) {
          st = nst;
          ph ^= 1;
        }
        --st;
        pf_wait(&full[st], ph ^ 1, limit_ns);
      }
      if (q_items > 0) pf_wait(&q_raw, (q_items - 1) & 1, limit_ns);
    }
  } else if (warp == 5) {
    regs_other();
    // ---------------- MMA issuer ----------------
    // The whole warp runs this role, and one lane of it issues (with the loop in one lane's branch compacted bf16
    // prompts, 13 products a tile, took 387 us a layer, 323 so; bf16 heads of 64 384 -> 342; heads of 128
    // 491 -> 466; OPT-1.3B-shaped prompts 272 -> 264).  Conditions are votes, so that the compiler knows them to be
    // the warp's.
    {
      constexpr uint32_t idS = mma_idesc(Pack16<T>::kType, 0, kPfRows, KT);
      constexpr uint32_t idO = mma_idesc(Pack16<T>::kType, 1, kPfRows, D);
      constexpr uint32_t SBO = 8 * SW;
      const uint32_t q_d = desc_lo(smem_addr(sm + Cf::Q_OFF), 16);
      [[maybe_unused]] const uint32_t qlo_d = desc_lo(smem_addr(sm + Cf::QLO_OFF), 16);
      auto uni_wait = [&](uint64_t* bar, uint32_t parity, uint32_t limit) -> bool {
        return __all_sync(0xFFFFFFFFu, pf_wait(bar, parity, limit));
      };
      // S = Q K^T of tile gj into its S tile.  One S tile: once the softmax has read S of tile
      // gj - 1.  Two: the tile last held P of tile gj - 2, whose P.V was issued before (tcgen05.mma
      // from one thread run in issue order).
      auto issue_qk = [&](uint32_t gj, bool last) -> bool {
        const int st = (int)(gj % KST), sb = (int)(gj % SBUF);
        if (!uni_wait(&k_full[st], (gj / KST) & 1, limit_ns)) return false;
        if (Cf::PSEP && gj >= 1 && !uni_wait(&s_free, (gj - 1) & 1, limit_ns)) return false;
        fence_proxy_async_smem();  // gathered rows were written through the generic proxy
        tc_fence_after();
        const uint32_t k_d = desc_lo(smem_addr(sm + Cf::K_OFF + st * Cf::TILE), 16);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t off = ((kk * 16) / SUB * Cf::SUBB + (kk * 16) % SUB * 2) >> 4;
            const uint32_t qoff = ((kk * 16) / SUB * Cf::QSUBB + (kk * 16) % SUB * 2) >> 4;
            tc_mma(tmem + sb * KT, desc(q_d + qoff, SBO, SW), desc(k_d + off, SBO, SW), idS, kk > 0);
          }
          // SPLIT with RoPE: + Q_lo K^T (without RoPE the query is exact in the cache type)
          if constexpr (Cf::SPLIT) {
            if constexpr (ROT) {
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t off = ((kk * 16) / SUB * Cf::SUBB + (kk * 16) % SUB * 2) >> 4;
                [[maybe_unused]] const uint32_t qoff = ((kk * 16) / SUB * Cf::QSUBB + (kk * 16) % SUB * 2) >> 4;
                if constexpr (Cf::QLO_TMEM)
                  tc_mma_ts(tmem + sb * KT, tmem + Cf::QLO_COL + 8 * kk, desc(k_d + off, SBO, SW), idS, 1);
                else
                  tc_mma(tmem + sb * KT, desc(qlo_d + qoff, SBO, SW), desc(k_d + off, SBO, SW), idS, 1);
              }
            }
          }
          tc_commit(&s_full[sb]);
          tc_commit(&k_empty[st]);
          if (last) tc_commit(&q_empty);
        }
        __syncwarp();
        return true;
      };
      // O += P V of tile gp (8 TMEM columns of P per 16 keys) into o_t; the first of an item: O = P V
      auto issue_pv = [&](uint32_t gp, uint32_t o_t, bool first) -> bool {
        const int st = (int)(gp % VST);
        if (!uni_wait(&v_full[st], (gp / VST) & 1, limit_ns)) return false;
        if (!uni_wait(&p_full, gp & 1, limit_ns)) return false;
        fence_proxy_async_smem();
        tc_fence_after();
        const uint32_t v_d = desc_lo(smem_addr(sm + Cf::V_OFF + st * Cf::TILE), Cf::SUBB);
        const uint32_t p_t = tmem + (Cf::PSEP ? Cf::P_COL : gp % SBUF * KT);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < KT / 16; ++kk)
            tc_mma_ts(o_t, p_t + 8 * kk, desc(v_d + kk * SW, SBO, SW), idO, (!first || kk > 0));
          if constexpr (Cf::SPLIT) {  // + P_lo V
#pragma unroll
            for (int kk = 0; kk < KT / 16; ++kk)
              tc_mma_ts(o_t, p_t + Cf::PLO_COL + 8 * kk, desc(v_d + kk * SW, SBO, SW), idO, 1);
          }
          tc_commit(&pv_done);
          tc_commit(&v_empty[st]);
        }
        __syncwarp();
        return true;
      };
      // Q K^T of a tile goes in ahead of P.V of the tile before, also when that is the last of its item: it
      // runs while the softmax works on that tile (an item's first scores were 1900 to 2900 cycles late with its
      // Q K^T after that P.V: OPT-1.3B-shaped prompts 362 us a layer, 348 so, with the cheaper descriptors).  The
      // rotated queries of an item come from the softmax warps after their last tile, whose P.V does not wait
      // for them.
      uint32_t gq = 0, gp = 0;  // Q K^T, P.V issued
      uint32_t kq = 0, kp = 0;  // their items
      int jq = 0, jp = 0, nkq = 0;
      bool items = true;  // there may be another one
      while (ok) {
        if (items && !(ROT && jq == 0 && gq != gp)) {
          if (jq == 0) {
            if (!(ok = __all_sync(0xFFFFFFFFu, item_wait(kq)))) break;
            nkq = item_slot[kq % kItemRing].nk;
            items = __any_sync(0xFFFFFFFFu, nkq > 0);
            if (items && !(ok = uni_wait(ROT ? &q_full : &q_raw, kq & 1, limit_ns))) break;
            tc_fence_after();
          }
          if (items) {
            const bool last = __any_sync(0xFFFFFFFFu, jq == nkq - 1);
            if (!(ok = issue_qk(gq, last))) break;
            ++gq;
            ++jq;
            if (last) {
              jq = 0;
              ++kq;
            }
            if (gq - gp == 1 && !(ROT && jq == 0)) continue;
          }
        }
        if (gq == gp) break;
        if (!(ok = issue_pv(gp, tmem + Cf::O_COL + (Cf::OBUF == 2 ? (kp & 1) * D : 0), jp == 0))) break;
        ++gp;
        if (__any_sync(0xFFFFFFFFu, ++jp == item_slot[kp % kItemRing].nk)) {
          item_done(kp);
          jp = 0;
          ++kp;
        }
      }
      // every MMA issued above has completed once this phase does
      if (elect_one()) tc_commit(&drain);
      __syncwarp();
      ok = uni_wait(&drain, 0, limit_ns) && ok;
    }
  } else if (warp < 4) {
    if constexpr (Cf::CPS == 2) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Cf::REG_SOFTMAX));
    // ---------------- softmax: one thread per query row ----------------
    constexpr int CW = KT;           // S columns of one thread
    const int r = warp * 32 + lane;  // tile row == TMEM lane
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    const float c2 = a.c2;
    // RoPE: row r of the K-major Q tile, rotated in place (pairs (e, e + rot/2), at the query's position,
    // rounded to the cache type) once item kk's raw rows are in, and released to the MMA thread.
    auto q_chunk = [&](int c8) -> uint32_t {  // shared address of 8-column chunk c8 of row r
      const int e0 = c8 * 8;
      const int u = e0 / SUB, cw = (e0 % SUB) / 8;
      const int phys = cw ^ ((r * SW >> 7) & (SW / 16 - 1));
      return smem_addr(sm + Cf::Q_OFF) + u * Cf::QSUBB + r * SW + phys * 16;
    };
    // SPLIT: the address of chunk c8 of row r in the query's low-part tile (QLO_SMEM)
    [[maybe_unused]] auto qlo_chunk = [&](int c8) -> uint32_t {
      return q_chunk(c8) - smem_addr(sm + Cf::Q_OFF) + smem_addr(sm + Cf::QLO_OFF);
    };
    [[maybe_unused]] auto qlo_store = [&](int c8, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
      if constexpr (Cf::QLO_TMEM)
        tmem_st4u(tl + Cf::QLO_COL + 4 * c8, w0, w1, w2, w3);  // warp-collective: every lane stores
      else
        st_shared_v4(qlo_chunk(c8), w0, w1, w2, w3);
    };
    [[maybe_unused]] auto q_rotate = [&](const PfItem& w, uint32_t kk) -> bool {
      if (!__all_sync(0xFFFFFFFFu, pf_wait(&q_raw, kk & 1, limit_ns))) return false;
      const int half = a.rot / 2;
      const int iq = w.qr0 + r;
      if constexpr (Cf::SPLIT) {
        // every row, so the TMEM stores are warp-wide (past the tile's queries another sequence's, or zeros: their
        // results go nowhere)
        {
          const float fpos = iq < w.qr_end ? (float)a.pos[a.off[w.s] + iq] : 0.f;
          const int hc = half / 8;  // chunks per rotated half
#pragma unroll 1
          for (int c8 = 0; c8 < D / 16; ++c8) {
            if (c8 < hc) {
              const uint32_t a1 = q_chunk(c8), a2 = q_chunk(c8 + hc);
              const uint4 u1 = ld_shared_v4(a1), u2 = ld_shared_v4(a2);
              const uint32_t w1[4] = {u1.x, u1.y, u1.z, u1.w}, w2[4] = {u2.x, u2.y, u2.z, u2.w};
              uint32_t h1[4], h2[4], l1[4], l2[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float2 x1 = T::f2(w1[e]), x2 = T::f2(w2[e]);
                float2 sn, ns, cs;
                rope_sincos2(fpos, rope_s[4 * c8 + e], &sn, &ns, &cs);
                l1[e] = bf16_split2(__ffma2_rn(x1, cs, __fmul2_rn(x2, ns)), &h1[e]);
                l2[e] = bf16_split2(__ffma2_rn(x2, cs, __fmul2_rn(x1, sn)), &h2[e]);
              }
              st_shared_v4(a1, h1[0], h1[1], h1[2], h1[3]);
              st_shared_v4(a2, h2[0], h2[1], h2[2], h2[3]);
              qlo_store(c8, l1[0], l1[1], l1[2], l1[3]);
              qlo_store(c8 + hc, l2[0], l2[1], l2[2], l2[3]);
            }
          }
          // the dimensions past the rotary ones are exact: their low part is zero
#pragma unroll 1
          for (int c8 = 0; c8 < D / 8; ++c8)
            if (c8 >= 2 * hc) qlo_store(c8, 0u, 0u, 0u, 0u);
        }
      } else if (iq < w.qr_end) {
        const float fpos = (float)a.pos[a.off[w.s] + iq];
#pragma unroll 1
        for (int c8 = 0; c8 < half / 8; ++c8) {
          const uint32_t a1 = q_chunk(c8), a2 = q_chunk(c8 + half / 8);
          const uint4 u1 = ld_shared_v4(a1), u2 = ld_shared_v4(a2);
          const uint32_t w1[4] = {u1.x, u1.y, u1.z, u1.w}, w2[4] = {u2.x, u2.y, u2.z, u2.w};
          uint32_t h1[4], h2[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 x1 = T::f2(w1[e]), x2 = T::f2(w2[e]);
            float2 sn, ns, cs;
            rope_sincos2(fpos, rope_s[4 * c8 + e], &sn, &ns, &cs);
            const float2 y1 = __ffma2_rn(x1, cs, __fmul2_rn(x2, ns)), y2 = __ffma2_rn(x2, cs, __fmul2_rn(x1, sn));
            h1[e] = Pack16<T>::two(y1.x, y1.y);
            h2[e] = Pack16<T>::two(y2.x, y2.y);
          }
          st_shared_v4(a1, h1[0], h1[1], h1[2], h1[3]);
          st_shared_v4(a2, h2[0], h2[1], h2[2], h2[3]);
        }
      }
      if constexpr (Cf::QLO_TMEM) {
        tmem_wait_st();  // the query's low part
        tc_fence_before();
      }
      fence_proxy_async_smem();
      mbar_arrive(&q_full);
      return true;
    };
    // the item's row r is a <CL> query
    auto is_cl = [&](const PfItem& w) -> bool {
      return w.qr0 + r < w.qr_end && (__ldg(a.meta + w.moff + w.qr0 + r) & 1);
    };

    uint32_t g = 0;   // tiles consumed
    uint32_t k = 0;   // items done
    uint32_t cg = 0;  // sorted key tiles consumed
    // waits of a whole warp -- with 64 keys a tile the lanes agree on them once a tile: as a share of its work a vote at
    // each is dear (compacted bf16 prompts 399 -> 387 us, bf16 heads of 64 396 -> 383; with more keys it is no gain)
    [[maybe_unused]] bool got_all = true;
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      const bool got = pf_wait(bar, parity, limit_ns);
      if constexpr (KT > 64) return __all_sync(0xFFFFFFFFu, got);
      got_all = got_all && got;
      __syncwarp();
      return true;
    };
    // Epilogue of item kk (row sum l_): O / l.  The 16-lane form of tcgen05.ld gives four neighbouring lanes 8 columns of
    // a row, so each store fills 32-byte sectors of eight queries' rows (OPT-1.3B-shaped prompts 333 us so, 348 when
    // each warp staged 16 columns at a time in shared memory for tensor stores).  All 32 rows of a few columns at a
    // time: the next tile's scores are in registers meanwhile, and 32 columns of 64 make the softmax spill (253 us
    // with 16 rows and 32 columns at a time, 248 with 32 and 16, 288 with 32 and 32).
    auto epilogue = [&](uint32_t kk, float l_) {
      const PfItem& w = item_slot[kk % kItemRing];
      const uint32_t o_t = tl + Cf::O_COL + (Cf::OBUF == 2 ? (kk & 1) * D : 0);
      const float inv = 1.f / l_;
      const int64_t row8 = (int64_t)8 * a.H * D;
      float* o_row = a.out + ((int64_t)(w.tok0 + warp * 32 + (lane >> 2)) * a.H + w.h) * D + 2 * (lane & 3);
      const int left = w.qr_end - w.qr0 - (warp * 32 + (lane >> 2));  // queries from this lane's first row on
      float inv8[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) inv8[i] = __shfl_sync(0xFFFFFFFFu, inv, 8 * i + (lane >> 2));
      constexpr int CO = Cf::PSEP ? 16 : 32;  // columns at a time
#pragma unroll 1
      for (int u = 0; u < D; u += CO, o_row += CO) {
        float o[2][CO / 2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if constexpr (CO == 32)
            tmem_ld_16x256b_x4(o_t + (i << 20) + u, o[i]);
          else
            tmem_ld_16x256b_x2(o_t + (i << 20) + u, o[i]);
        }
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int e = 0; e < CO / 2; ++e) asm volatile("" : "+f"(o[i][e]));  // no use of O moves above the wait
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (left > 8 * i) {
#pragma unroll
            for (int c = 0; c < CO / 8; ++c)
              *reinterpret_cast<float2*>(o_row + i * row8 + 8 * c) =
                  make_float2(o[i >> 1][4 * c + 2 * (i & 1)] * inv8[i], o[i >> 1][4 * c + 2 * (i & 1) + 1] * inv8[i]);
          }
        }
      }
      tc_fence_before();
      item_done(kk);
    };
    ok = __all_sync(0xFFFFFFFFu, item_wait(0));
    bool more = ok && item_slot[0].nk > 0;
    bool cl_next = false;  // is_cl of the next item
    float l_prev = 0.f;    // the item before's row sum: its epilogue comes once its last P.V is complete
    if (more) {
      cl_next = is_cl(item_slot[0]);
      if constexpr (ROT) ok = q_rotate(item_slot[0], 0);
    }
    // after the last item (!more) once more, for its epilogue alone
    while (ok && (more || k >= 1)) {
      const PfItem& w = item_slot[k % kItemRing];
      const int nk = more ? w.nk : 1, n_c = w.n_c, step = w.odd ? -KT : KT;
      int v0 = KT * w.key_tile(0);  // the tile's first key
      const int vq = w.own(KT) + r;  // its own key
      const bool cl_q = cl_next;
      bool next_ok = false;  // there is another item
      const uint32_t o_t = tl + Cf::O_COL + (Cf::OBUF == 2 ? (k & 1) * D : 0);
      float m = -INFINITY, l = 0.f;
      for (int j = 0; j < nk; ++j, v0 += step) {
        const uint32_t gj = g + j;
        const int sb = (int)(gj % SBUF);
        const uint32_t p_tl = tl + (Cf::PSEP ? Cf::P_COL : sb * KT);
        float sv[CW], alpha = 1.f, ref = 0.f, m_new = 0.f;
        float2 rs4[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        uint32_t pk[2][16];
        [[maybe_unused]] uint32_t pl[2][16];
        // P = 2^(s c2 - ref) of columns [32 q, 32 q + 32) (or their first 16) as 16-bit pairs; the row sum
        auto make_p = [&](int q) {
          const float2 c2v = make_float2(c2, c2), nref = make_float2(-ref, -ref);
#pragma unroll
          for (int c = 0; c < 32; c += 2) {
            if (32 * q + c >= CW) continue;
            const float2 x = __ffma2_rn(make_float2(sv[32 * q + c], sv[32 * q + c + 1]), c2v, nref);
            const float2 p = make_float2(ex2(x.x), ex2(x.y));
            rs4[(c >> 1) & 3] = __fadd2_rn(rs4[(c >> 1) & 3], p);
            if constexpr (Cf::SPLIT)
              pl[q & 1][c / 2] = bf16_split2(p, &pk[q & 1][c / 2]);
            else
              pk[q & 1][c / 2] = Pack16<T>::two(p.x, p.y);
          }
        };
        auto store_p = [&](int q) {  // into row r's lane
          if (CW - 32 * q >= 32)
            tmem_st16u(p_tl + 16 * q, pk[q & 1]);
          else
            tmem_st8u(p_tl + 16 * q, pk[q & 1]);
          if constexpr (Cf::SPLIT) tmem_st16u(p_tl + Cf::PLO_COL + 16 * q, pl[q & 1]);
        };
        // pv_done phases are consumed one by one, each while it is the only one that can be pending
        // (the next P.V waits for this tile's P): phase gj - 1 during tile gj, before O is rescaled and
        // before this tile's P is written where P.V of the tile before reads its P from.  The wait comes as
        // late as that allows: with P in columns of its own after the first 64 columns of P are made, with
        // two S tiles (P goes into its own) at the end.  An item's first tile then runs the epilogue of
        // the item before, whose last P.V that was.
        bool pv_wait = gj >= 1;
        if (more) {
          const bool sorted = v0 + KT > n_c;    // warp 4 has sorted its keys
          const int cs = (int)(cg % kClsRing);
          ok = warp_wait(&s_full[sb], (gj / SBUF) & 1) &&
               (!sorted || warp_wait(&cls_full[cs], (cg / kClsRing) & 1));
          // warp 4 takes the next item as soon as this item's last K tile is on its way
          if (ok && j == nk - 1) ok = __all_sync(0xFFFFFFFFu, item_wait(k + 1));
          // nothing is exchanged between the softmax warps: each stops by itself
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c + 32 <= CW; c += 32) tmem_ld32(tl + sb * KT + c, sv + c);
          if constexpr (CW % 32 == 16) tmem_ld16(tl + sb * KT + CW - 16, sv + CW - 16);
          const bool slow = sorted && kslow[cs] != 0;
          uint32_t vw[4];
          if (slow) {
            // visibility of the tile's keys to this query as 32-bit words: the causal prefix (keys up to the
            // query's own) with the tile-wide bound words plus the keys whose bound, among the
            // queries, is this one or a later one.  Every key of the other tiles is visible (to all but a <CL> query).
            const int t = vq - v0;  // the query's own column, the last visible one
            const uint4 hw = khid[cs], he = kend[cs];
            const uint4 af = kafter[cs][__popc(he.x & low_bits(r)) + __popc(he.y & low_bits(r - 32)) +
                                        __popc(he.z & low_bits(r - 64)) + __popc(he.w & low_bits(r - 96))];
            vw[0] = hw.x | af.x;
            vw[1] = hw.y | af.y;
            vw[2] = hw.z | af.z;
            vw[3] = hw.w | af.w;
            // the causal prefix; a <CL> query sees its own key alone
#pragma unroll
            for (int u = 0; u < 4; ++u) vw[u] &= low_bits(t + 1 - 32 * u) & ~low_bits(cl_q ? t - 32 * u : 0);
          }
          if (j == nk - 1) {
            next_ok = item_slot[(k + 1) % kItemRing].nk > 0;
            cl_next = next_ok && is_cl(item_slot[(k + 1) % kItemRing]);
          }
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < CW; ++c) asm volatile("" : "+f"(sv[c]));  // no use of S moves above the wait
          tc_fence_before();
          if (Cf::PSEP) mbar_arrive(&s_free);  // the next Q K^T may overwrite S
          if (sorted) {
            __syncwarp();  // every lane has read the tile's classes
            if (lane == 0) mbar_arrive(&cls_empty[cs]);
            ++cg;
          }
          // A <CL> query sees none of the keys of a tile without the per-key rule: an infinite reference makes
          // its P there 0.  Only if one of those scores is not below infinity the row is masked as well, in a
          // second round.
          const bool unseen = cl_q && !slow;
          bool masked = slow;
          float mx;
          // row max: a tree (eight partial maxima: columns 0-7, then pairs of 8-column blocks, then the
          // last block when one is left over)
          static_assert(CW % 8 == 0, "slice width");
          constexpr int kPairEnd = 8 + (CW - 8) / 16 * 16;  // columns [8, kPairEnd) go in pairs of blocks
          for (;;) {
            if (masked) {
#pragma unroll
              for (int u = 0; u < (CW + 31) / 32; ++u) {
                if (!__any_sync(0xFFFFFFFFu, vw[u] != 0xFFFFFFFFu)) continue;  // visible to the whole warp
#pragma unroll
                for (int c = 32 * u; c < 32 * u + 32; ++c)
                  if (c < CW) sv[c] = vw[u] & (1u << (c & 31)) ? sv[c] : -INFINITY;
              }
            }
            float mx8[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) mx8[u] = sv[u];
#pragma unroll
            for (int c = 8; c < kPairEnd; c += 16)
#pragma unroll
              for (int u = 0; u < 8; ++u) mx8[u] = max3(mx8[u], sv[c + u], sv[c + 8 + u]);
            if constexpr (kPairEnd < CW) {
#pragma unroll
              for (int u = 0; u < 8; ++u) mx8[u] = max3(mx8[u], sv[kPairEnd + u], sv[kPairEnd + u]);
            }
            mx = max3(max3(mx8[0], mx8[1], mx8[2]), max3(mx8[3], mx8[4], mx8[5]), max3(mx8[6], mx8[7], mx8[7]));
            masked = __any_sync(0xFFFFFFFFu, unseen && !(mx < INFINITY));
            if (!masked) break;
#pragma unroll
            for (int u = 0; u < 4; ++u) vw[u] = unseen ? 0u : 0xFFFFFFFFu;
          }
          // Reference maximum: moved only when the row maximum grows by more than 2^8 (log2 units), so
          // O is rescaled rarely; P stays below 2^8 and its scale cancels exactly in O / l.
          const float cand = unseen ? -INFINITY : mx * c2;
          const bool move = cand > m + 8.f;
          m_new = move ? cand : m;
          ref = unseen ? INFINITY : m_new == -INFINITY ? 0.f : m_new;
          // a row that has seen no key so far has O = 0 and l = 0: nothing to rescale
          alpha = !move || m == -INFINITY ? 1.f : ex2(m - ref);
          if (pv_wait && __any_sync(0xFFFFFFFFu, alpha != 1.f)) {
            pv_wait = false;
            ok = warp_wait(&pv_done, (gj - 1) & 1);
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int u = 0; u < D / 16; ++u) {
              float o[16];
              tmem_ld16(o_t + 16 * u, o);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 16; ++e) o[e] *= alpha;
              tmem_st16(o_t + 16 * u, o);
            }
          }
          make_p(0);
          if (!Cf::PSEP) store_p(0);
          make_p(1);
          if (!Cf::PSEP) {
            store_p(1);
#pragma unroll
            for (int q = 2; q < (CW + 31) / 32; ++q) {
              make_p(q);
              store_p(q);
            }
          }
        }
        if (pv_wait) {
          ok = warp_wait(&pv_done, (gj - 1) & 1);
          if (!ok) break;
        }
        tc_fence_after();
        if (Cf::PSEP && more) {
          store_p(0);
          store_p(1);
        }
        if (j == 0 && k >= 1) {
          // the item before is complete only if every wait up to its last P.V was
          if (KT == 64 && !(ok = __all_sync(0xFFFFFFFFu, got_all))) break;
          epilogue(k - 1, l_prev);
        }
        if (!more) break;
        if (Cf::PSEP) {
#pragma unroll
          for (int q = 2; q < (CW + 31) / 32; ++q) {
            make_p(q);
            store_p(q);
          }
        }
        const float rs =
            ((rs4[0].x + rs4[0].y) + (rs4[1].x + rs4[1].y)) + ((rs4[2].x + rs4[2].y) + (rs4[3].x + rs4[3].y));
        l = l * alpha + rs;
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&p_full);
        m = m_new;
        if (KT == 64 && !__all_sync(0xFFFFFFFFu, got_all)) {
          ok = false;
          break;
        }
      }
      if (!ok || !more) break;
      g += nk;
      l_prev = l;
      // the next item's queries came in after this item's last Q.K^T
      if constexpr (ROT) {
        if (next_ok) ok = q_rotate(item_slot[(k + 1) % kItemRing], k + 1);
      }
      more = next_ok;
      ++k;
    }
  }
  if (!ok) atomicOr(a.status, STATUS_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(Cf::TMEM_COLS) : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;
cudaError_t g_encode_err = cudaSuccess;

cudaError_t encode_plane(const Geometry& g, void* base, unsigned char* out) {
  const int sw = (2 * g.D) % 128 == 0 ? 128 : (2 * g.D) % 64 == 0 ? 64 : 32;
  cuuint64_t dims[2] = {(cuuint64_t)g.D, (cuuint64_t)((int64_t)g.M * g.H * g.C)};
  cuuint64_t strides[1] = {(cuuint64_t)g.D * 2};
  cuuint32_t box[2] = {(cuuint32_t)(sw / 2), (cuuint32_t)prefill_keys_per_tile(g.D, g.dtype)};
  cuuint32_t elem[2] = {1, 1};
  const CUtensorMapSwizzle swz =
      sw == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : sw == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
  CUtensorMap m;
  const CUresult r = g_encode(&m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, base, dims, strides, box, elem,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  std::memcpy(out, &m, sizeof m);
  return cudaSuccess;
}

template <typename T, int D, bool ROT>
cudaError_t launch_prefill_t(const PrefillMaps& maps, const PrefillArgs& a, int64_t grid, cudaStream_t stream) {
  using Cf = PfCfg<D, kSplit<T>>;
  static std::mutex mu;
  static bool attr_set[64] = {};  // per device: the shared-memory opt-in and the register check
  int dev = 0;
  {
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(prefill_kernel<T, D, ROT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)Cf::SMEM);
    if (e != cudaSuccess) return e;
    if (Cf::CPS == 2) {
      // the setmaxnreg shares assume each thread starts with exactly REG_LAUNCH registers; with
      // fewer the softmax warpgroup's increase could never be granted, so refuse to launch
      cudaFuncAttributes fa;
      const cudaError_t e2 = cudaFuncGetAttributes(&fa, prefill_kernel<T, D, ROT>);
      if (e2 != cudaSuccess) return e2;
      if (fa.numRegs != Cf::REG_LAUNCH) return cudaErrorInvalidConfiguration;
    }
    attr_set[dev] = true;
  }
  CUtensorMap mk, mv, mq;
  std::memcpy(&mk, maps.k, sizeof mk);
  std::memcpy(&mv, maps.v, sizeof mv);
  cuuint32_t elem[3] = {1, 1, 1};
  {
    // q as [token][head][D], in boxes of one column subtile x one head x 128 tokens
    cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)a.H, (cuuint64_t)a.n_qtok};
    cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)a.H * D * 2};
    cuuint32_t box[3] = {(cuuint32_t)Cf::SUB, 1, (cuuint32_t)kPfRows};
    const CUresult r = g_encode(&mq, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, const_cast<uint16_t*>(a.q), dims, strides, box, elem,
                                CU_TENSOR_MAP_INTERLEAVE_NONE,
                                Cf::SW == 128   ? CU_TENSOR_MAP_SWIZZLE_128B
                                : Cf::SW == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                               : CU_TENSOR_MAP_SWIZZLE_32B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  prefill_kernel<T, D, ROT><<<(unsigned)grid, kPfThreads, Cf::SMEM, stream>>>(mk, mv, mq, a);
  return cudaGetLastError();
}

template <typename T, int D>
cudaError_t launch_prefill_d(const PrefillMaps& maps, const PrefillArgs& a, int64_t grid, cudaStream_t stream) {
  return a.rot > 0 ? launch_prefill_t<T, D, true>(maps, a, grid, stream)
                   : launch_prefill_t<T, D, false>(maps, a, grid, stream);
}

}  // namespace

static cudaError_t load_encoder() {
  std::call_once(g_encode_once, [] {
    cudaDriverEntryPointQueryResult q;
    g_encode_err = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", reinterpret_cast<void**>(&g_encode),
                                                    12000, cudaEnableDefault, &q);
    if (g_encode_err == cudaSuccess && q != cudaDriverEntryPointSuccess) g_encode_err = cudaErrorNotSupported;
  });
  return g_encode_err;
}

cudaError_t encode_append_maps(const Geometry& g, const Buffers& buf, const int64_t* seq_row0, const int32_t* cap,
                               unsigned char* out) {
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  if (g.H > 256 || g.D > 256) return cudaErrorNotSupported;  // box dimensions hold at most 256 elements
  cudaError_t e = load_encoder();
  if (e != cudaSuccess) return e;
  for (int kv = 0; kv < 2; ++kv) {
    for (int s = 0; s < g.b; ++s) {
      uint16_t* base = (kv ? buf.v : buf.k) + seq_row0[s] * g.D;
      cuuint64_t dims[4] = {(cuuint64_t)g.D, (cuuint64_t)cap[s], (cuuint64_t)g.H, (cuuint64_t)g.M};
      cuuint64_t strides[3] = {(cuuint64_t)g.D * 2, (cuuint64_t)cap[s] * g.D * 2, (cuuint64_t)g.H * g.C * g.D * 2};
      cuuint32_t box[4] = {(cuuint32_t)g.D, 1, (cuuint32_t)g.H, 1};
      cuuint32_t elem[4] = {1, 1, 1, 1};
      CUtensorMap m;
      const CUresult r = g_encode(&m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, base, dims, strides, box, elem,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
      std::memcpy(out + 128 * ((size_t)kv * g.b + s), &m, sizeof m);
    }
  }
  return cudaSuccess;
}

cudaError_t encode_prefill_maps(const Geometry& g, const Buffers& buf, PrefillMaps* maps) {
  static_assert(sizeof(CUtensorMap) == sizeof(maps->k), "tensor map size");
  cudaError_t e = load_encoder();
  if (e != cudaSuccess) return e;
  e = encode_plane(g, buf.k, maps->k);
  if (e == cudaSuccess) e = encode_plane(g, buf.v, maps->v);
  maps->ready = e == cudaSuccess;
  return e;
}

int prefill_keys_per_tile(int D, int dtype) {
  switch (D) {
    case 64: return dtype ? PfCfg<64, true>::KT : PfCfg<64, false>::KT;
    case 80: return dtype ? PfCfg<80, true>::KT : PfCfg<80, false>::KT;
    case 96: return PfCfg<96>::KT;
    default: return PfCfg<128>::KT;
  }
}

int prefill_ctas_per_sm(int D) {
  switch (D) {
    case 64: return PfCfg<64>::CPS;
    case 80: return PfCfg<80>::CPS;
    case 96: return PfCfg<96>::CPS;
    case 128: return PfCfg<128>::CPS;
    default: return 1;
  }
}

cudaError_t launch_prefill(const Geometry& g, const PrefillMaps& maps, const PrefillArgs& a, cudaStream_t stream) {
  if (a.n_items <= 0 || a.n_ctas <= 0) return cudaSuccess;
  const int64_t grid = a.n_ctas;  // persistent
  const bool bf = g.dtype == 1;
  switch (g.D) {
    case 64:
      return bf ? launch_prefill_d<BF16T, 64>(maps, a, grid, stream) : launch_prefill_d<F16T, 64>(maps, a, grid, stream);
    case 80:
      return bf ? launch_prefill_d<BF16T, 80>(maps, a, grid, stream) : launch_prefill_d<F16T, 80>(maps, a, grid, stream);
    case 96:
      return bf ? launch_prefill_d<BF16T, 96>(maps, a, grid, stream) : launch_prefill_d<F16T, 96>(maps, a, grid, stream);
    case 128:
      return bf ? launch_prefill_d<BF16T, 128>(maps, a, grid, stream)
                : launch_prefill_d<F16T, 128>(maps, a, grid, stream);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace kvc

// GLIDE prefill outputs on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), bf16 I/O, head_dim 128.
//
// One CTA (19 warps) owns 256 query rows of one (layer, sequence, KV head) unit: two row tiles X = A, B of 128
// rows each, a row being (token, query head of the group), row = token * G + head.
//   warps 0-3, 8-11    softmax of tile A: two threads per row (TMEM lane), 64 columns each
//   warps 4-7, 12-15   softmax of tile B
//   warps 16, 17       issue the tcgen05.mma of A and of B (one elected lane), in turns.  Between two products a warp spends some 1000
//               cycles on waits, votes and commits, and the tensor core's queue is short: with one warp for both it idled half of
//               the time
//   warp 18     loads every operand (TMA; row by row where a 16-token group straddles two sources); Q of heads that do not lie
//               side by side is copied by the softmax threads
// Window part, per 128-key tile t (keys are tokens j0 + 0..127, j0 a multiple of 16):
//   loader    K_t and V_t (ring rows for tokens older than the call, the call's rows otherwise) into a ring of five
//             32 KiB buffers (kStages), 128-byte swizzle, completion on an mbarrier
//   MMA       S_X = Q_X K_t^T into TMEM (8 x m128n128k16), committed to an mbarrier the softmax warps wait on
//   softmax   tcgen05.ld of the own half row, mask, row maximum (the other half's by a barrier of two warps, and only when it
//             grows), P = 2^(s - m_ref) as bf16 over the consumed S columns; the reference m_ref is lazy: O is rescaled in TMEM only when the maximum grows by
//             more than 2^8
//   MMA       O_X += P_X V_t (V as the MN-major B operand), then S_X of the next tile: while one row tile is
//             in its softmax the tensor core works for the other
// TMEM columns: S_A [0,128) S_B [128,256) O_A [256,384) O_B [384,512).
// Linear part (after the window tiles, by the same warps in the same way): with a common reference M = max(m_ref, -64)
// per row, phi(Q) 2^-M as bf16 times a bf16 copy of the state (inter-chunk), and C = phi(Q) phi(K')^T masked to
// j' <= i, then C V' (intra-chunk); l accumulates the matching sums.  out = O / l.
// What bounds it: short windows, the fixed chain of a CTA (windows of 64, 23100 cycles: set-up 740, 6500 until Q and K_0 are there
// and the first product is done, one softmax 3600, phi 2700, its products 3000, C 2000, the last products 1300, the store 3200); long
// windows, per key tile and row tile the chain softmax (1770) -> P V and the next S (1050 to 1300) -> signals, 3500 cycles in which the
// two row tiles' products take 2048.  8 layers of 2048 tokens, 32 / 8 heads, windows of 64 / 256 / 1024: 255 / 316 / 479 us for all; with
// one softmax thread per row, one MMA warp and phi in one piece 292 / 379 / 576.
// Every mbarrier wait is bounded; on a time-out the CTA records kDevWaitTimeout, leaves its loops, frees its TMEM
// columns and returns.
#include <cuda.h>
#include <cstring>

#include <algorithm>
#include <type_traits>

#include "glide_prefill_rows.cuh"
#include "glide_tc.cuh"

namespace glide {

namespace {

constexpr int kD = 128;
constexpr int kRows = 128;            // rows per row tile
constexpr int kKT = 128;              // keys per tile
constexpr int kGroup = 16;            // tokens per TMA box
constexpr int kHalf = kD / 2;         // columns of a softmax thread: two threads per row
constexpr int kSoftmaxThreads = 512;
constexpr int kThreads = 608;
constexpr int kMmaWarp = 16, kLoadWarp = 18;   // (MMA warps: one per row tile)
constexpr uint32_t kTileBytes = 32768;   // [2 boxes][128 rows][64 bf16]
constexpr uint32_t kBoxBytes = 16384;
constexpr uint32_t kGroupBytes = kGroup * 128;   // one 16-token box of 64 columns
constexpr float kLazy = 8.0f;         // rescale O only when the row maximum grows by more than 2^8
constexpr int kStages = 5;

// byte offset of 16-byte chunk c16 (0..15) of row `row` inside a [2][128][64] bf16 tile with 128-byte swizzle
__device__ __forceinline__ uint32_t sw128(int row, int c16) {
  return uint32_t((c16 >> 3) * kBoxBytes + row * 128 + (((c16 & 7) ^ (row & 7)) << 4));
}
// instruction descriptor: fp32 accumulate, bf16 A and B, M = N = 128; b_mn: B operand is MN-major
__device__ __forceinline__ uint32_t make_idesc(bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn ? (1u << 16) : 0u) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
}
// 8 MMAs of one 128 x 128 x 128 product; B K-major (D = A B^T) or MN-major (D (+)= A B).  Called by the MMA warp as a
// whole, with operands that are the same in all lanes: the instruction takes them from uniform registers, and in code of
// one diverged lane every step moved them there anew (3400 cycles to issue the 32 MMAs of a key tile, which run in 2048).
__device__ __forceinline__ void issue_mma(bool leader, uint32_t tmem_d, uint32_t a_tile, uint32_t b_tile, bool b_mn, bool accumulate) {
  const uint32_t idesc = make_idesc(b_mn);
  const uint32_t a0 = desc_lo(a_tile, 16), b0 = desc_lo(b_tile, b_mn ? kBoxBytes : 16);
  if (leader) {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      const uint32_t step = uint32_t(((ks >> 2) * kBoxBytes + (ks & 3) * 32) >> 4);
      asm volatile(
          "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
          "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}" ::"r"(tmem_d),
          "r"(a0 + step), "r"(b0 + (b_mn ? uint32_t(ks * 2048 >> 4) : step)), "r"(idesc),
          "r"((accumulate || ks > 0) ? 1u : 0u), "r"(kDescHi)
          : "memory");
    }
  }
}
// the same product with the A operand in TMEM: lane = row, 32-bit column c = elements 2c (low half) and 2c+1 of
// the row, 8 columns per k16 step, elements 64 .. 127 from column 64 on (PAIRS: two steps, then a gap of 16 columns); B
// MN-major in shared memory
template <bool PAIRS>
__device__ __forceinline__ void issue_mma_ts(bool leader, uint32_t tmem_d, uint32_t tmem_a, uint32_t b_tile, bool accumulate) {
  const uint32_t idesc = make_idesc(true);
  const uint32_t b0 = desc_lo(b_tile, kBoxBytes);
  if (leader) {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
      asm volatile(
          "{\n\t.reg .pred p;\n\t.reg .b64 b;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b64 b, {%2, %5};\n\t"
          "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, p;\n\t}" ::"r"(tmem_d),
          "r"(tmem_a + (PAIRS ? (ks >> 1) * 32 + (ks & 1) * 8 : (ks >> 2) * 64 + (ks & 3) * 8)), "r"(b0 + uint32_t(ks * 2048 >> 4)), "r"(idesc), "r"((accumulate || ks > 0) ? 1u : 0u), "r"(kDescHi)
          : "memory");
  }
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *tmap, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(tmap), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void *tmap, int c0, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_2d(const void *tmap, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tmap), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_prefetch_4d(const void *tmap, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
// 32 columns of this thread's lane; the registers are valid only after tmem_wait_ld(r)
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// every load issued so far has landed; r (one of them) is an operand so that no use of it can move above the wait
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                 "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                 "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  tmem_ld32_nowait(taddr, r);
  tmem_wait_ld(r);
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]),
      "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]),
      "r"(r[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}


// (no wait: the caller issues tmem_wait_st() once after its last store)
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

#ifdef GLIDE_PF_CLOCKS
// debug builds only: clock cycles per phase of thread 0 of every CTA, summed over the CTAs ([8] = CTAs; [16] .. [20] the waits of
// the MMA thread and of the loader)
__device__ unsigned long long g_pf_clk[32];
#define PF_CLK(i)                                                   \
  do {                                                              \
    if (threadIdx.x == 0) {                                         \
      const long long now_ = clock64();                             \
      atomicAdd(&g_pf_clk[i], (unsigned long long)(now_ - pf_t_));  \
      pf_t_ = now_;                                                 \
    }                                                               \
  } while (0)
#define PF_LAP_INIT() long long pf_l_ = clock64()
#define PF_LAP(i)                                                 \
  do {                                                            \
    const long long now_ = clock64();                             \
    if ((threadIdx.x & 31) == 0) atomicAdd(&g_pf_clk[i], (unsigned long long)(now_ - pf_l_));  \
    pf_l_ = now_;                                                 \
  } while (0)
#else
#define PF_LAP_INIT() do { } while (0)
#define PF_LAP(i) do { } while (0)
#define PF_CLK(i) do { } while (0)
#endif

struct Smem {
  unsigned char q[2][kTileBytes];        // Q_A, Q_B; then phi(Q) 2^-M; then the output rows on their way out
  unsigned char kv[kStages][kTileBytes]; // K and V tiles in turn; linear part: state, phi(K') and V' tiles
  float z[2 * kD];                       // z of the unit (both halves with the learned map)
  uint64_t bar_full[kStages];            // the buffer's K or V tile has landed
  uint64_t bar_free[kStages];            // the MMAs that read the buffer have completed (one arrival per row tile)
  uint64_t bar_q[2];                     // Q_X staged (TMA, or the 256 threads that copied it)
  uint64_t bar_s[2];                     // MMA -> softmax threads of X: the products issued for X so far have completed
  uint64_t bar_p[2];                     // softmax threads of X -> MMA: the A operand of X's next products is ready (one arrival per warp)
  uint64_t bar_turn[2];                  // window part: the other row tile's batch of products has been issued
  uint64_t bar_done;                     // every window MMA has completed
  uint64_t bar_state;                    // the bf16 state and z of the unit have landed (learned map: phi(Q) as well)
  uint64_t bar_pk[2];                    // the phi(K') tile of an intra-chunk step has landed (even / odd steps)
  uint64_t bar_vp[2];                    // the V' tile of an intra-chunk step has landed (even / odd steps; 2 arrivals)
  uint64_t bar_lfree[2];                 // the MMAs that read an intra-chunk step's buffers have completed
  uint32_t tmem_base;
  int failed;
  float exch[kSoftmaxThreads / 2];       // a value of each row on its way between the row's two threads
};
static_assert(kLazy == 8.0f, "soft_tile's bound is 2^kLazy");
static_assert(sizeof(Smem) <= 232448, "shared memory of one CTA");

// the call's K (or V) rows as a 4-D tensor {d, Hkv, T, layers x sequences}: boxes of 16 tokens x 64 columns of one KV head
struct CallMaps {
  CUtensorMap k, v;         // boxes of 16 tokens
  CUtensorMap k128, v128;   // boxes of a whole 128-key tile
  CUtensorMap q;            // {d, H, T, layers x sequences}: boxes of one row tile's tokens x the G heads of a group x 64 columns
};

// Gated: the weights stay fp32 quantities (the gated recurrence has no other tensor-core form whose precision it could
// share): every A operand (P, phi(Q), C) and the state and phi(K') are split into two bf16 terms, hi + lo, and the
// products of two split operands leave out lo x lo (2^-18 of the result).  Against fp64 the outputs are as far off as those of the
// fp32 kernel to 1e-6 of that (1.64e-3, the rounding to bf16; 1000 tokens, windows of 64 and 256, gates of 0.95 to 1); l sums the
// weights before the split (their sums after it: the same figures, 2 % slower).
enum : int { kModeShared = 0, kModeSum = 1, kModeLearned = 2, kModeGated = 3 };

// the state at a chunk's start for a single row: the bf16 copies hi and lo (lo of an infinity is not a number) and z
struct SplitState {
  const __nv_bfloat16 *hi;
  size_t lo_half;
  const float *z0;
  template <int E>
  __device__ __forceinline__ void row(int r, int c, float (&x)[E]) const {
    float lo[E];
    load_elems<__nv_bfloat16, E>(hi + r * kD + c, x);
    load_elems<__nv_bfloat16, E>(hi + lo_half + r * kD + c, lo);
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = isfinite(x[e]) ? x[e] + lo[e] : x[e];
  }
  __device__ __forceinline__ float z(int r) const { return z0[r]; }
};

// Gated: the rows of `again` (bit i: row row0 + i of the CTA's 256, whose token 0 is chunk index tok0 of chunk `sub` of unit u)
// once more, by one warp, from the rows that count for them alone: in the tiles a masked row's weight of zero, and a lo
// weight of zero or of the other sign, meet whatever V holds.
template <int G>
__device__ __noinline__ void recompute_rows(const PrefillParams &p, unsigned again, int row0, int u, int sub, int tok0) {
  using bf16 = __nv_bfloat16;
  const int ug = u / p.Hkv, g = u - ug * p.Hkv, lrel = ug / p.B, b = ug - lrel * p.B;
  const LayerDev ld = p.layers[p.layer_begin + lrel];
  const size_t uc = size_t(u) * p.nsub + sub;
  for (; again; again &= again - 1) {
    const int rw = row0 + __ffs(int(again)) - 1, tl = tok0 + rw / G;
    const size_t token = (size_t(lrel) * p.B + b) * size_t(p.T) + size_t(p.c0 + sub * p.SC + tl);
    const size_t at = (token * p.H + p.heads_of[g * G + rw % G]) * kD;
    const RowJob<bf16, kD> job{Rows<bf16, kD>(p, ld, lrel, b, g), reinterpret_cast<const bf16 *>(p.q) + at, reinterpret_cast<bf16 *>(p.out) + at,
                               p.gcum + uc * p.SC, p.n0 + p.c0 + sub * p.SC, tl, ld.w, ld.wlin, ld.evicts, ld.merge, p.scale_log2};
    recompute_row(job, SplitState{reinterpret_cast<const bf16 *>(p.s16) + uc * kD * kD, size_t(p.units_cap) * kD * kD, p.zsnap + uc * kD});
  }
}

// bit i: column c + i of a key tile is valid for a row whose valid columns are lo .. hi
__device__ __forceinline__ uint32_t column_mask(int c, int lo, int hi) {
  const int a = lo - c, b = hi - c;
  const uint32_t ma = a <= 0 ? ~0u : (a >= 32 ? 0u : ~0u << a);
  const uint32_t mb = b < 0 ? 0u : (b >= 31 ? ~0u : (2u << b) - 1u);
  return ma & mb;
}
// two fp32 values at once (the packed instructions round like the scalar ones)
__device__ __forceinline__ void fma2(float &a0, float &a1, float x0, float x1, float s, float c) {
  asm("{\n\t.reg .b64 x, s, c, d;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 s, {%4, %4};\n\tmov.b64 c, {%5, %5};\n\t"
      "fma.rn.f32x2 d, x, s, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(a0), "=f"(a1)
      : "f"(x0), "f"(x1), "f"(s), "f"(c));
}
__device__ __forceinline__ void dot2(float &a0, float &a1, float x0, float x1, float y0, float y1) {   // a += x * y
  asm("{\n\t.reg .b64 a, x, y;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "fma.rn.f32x2 a, x, y, a;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(x0), "f"(x1), "f"(y0), "f"(y1));
}
__device__ __forceinline__ float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ float bf16_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }
__device__ __forceinline__ void add2(float &a0, float &a1, float x0, float x1) {
  asm("{\n\t.reg .b64 a, x;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 x, {%2, %3};\n\tadd.rn.f32x2 a, a, x;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(x0), "f"(x1));
}
// x0, x1 -> bf16 pairs hi (rounded) and lo (the rounded rest)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  hi = pack_bf16x2(x0, x1);
  lo = pack_bf16x2(x0 - __uint_as_float(hi << 16), x1 - __uint_as_float(hi & 0xffff0000u));
}

template <int G, int MODE>
__global__ void __launch_bounds__(kThreads, 1)   // 19 warps = 5 on one scheduler: 96 registers per thread at most
prefill_attn_tc_kernel(const __grid_constant__ PrefillParams p, const CUtensorMap *ring_maps, const __grid_constant__ CallMaps cm) {
  using bf16 = __nv_bfloat16;
  constexpr bool SUM = MODE == kModeSum;          // sum of two normalised terms instead of the shared normaliser
  constexpr bool PHI2 = MODE == kModeLearned;
  constexpr bool GATED = MODE == kModeGated;
  constexpr bool TWO = PHI2 || GATED;             // two tiles of phi(Q), S and phi(K'): the map's halves, or hi and lo
  constexpr int TOKT = kRows / G;    // tokens per row tile
  constexpr int TOKC = 2 * TOKT;     // tokens per CTA
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // CTAs of a unit: those of its full chunks, then those of the last one, the last tokens first (their windows are the
  // longest of a new prompt); from here on "the chunk" is the CTA's own
  const int ctas_per_chunk = (p.SC + TOKC - 1) / TOKC;
  const int ctas_per_unit = (p.nsub - 1) * ctas_per_chunk + (p.C - (p.nsub - 1) * p.SC + TOKC - 1) / TOKC;
  const int u = int(blockIdx.x / unsigned(ctas_per_unit));
  const int cta_u = ctas_per_unit - 1 - int(blockIdx.x - unsigned(u) * unsigned(ctas_per_unit));
  const int sub = cta_u / ctas_per_chunk;
  const int tok0 = (cta_u - sub * ctas_per_chunk) * TOKC;
  const int chunk_c0 = int(p.c0) + sub * p.SC;                // first token of the chunk, relative to the call
  const int chunk_n = min(p.SC, p.C - sub * p.SC);            // its tokens
  const int64_t uc = int64_t(u) * p.nsub + sub;                        // (unit, chunk): index into the scratch arrays
  const int ug = u / p.Hkv, g = u - ug * p.Hkv, lrel = ug / p.B, b = ug - lrel * p.B;
  const int layer = p.layer_begin + lrel;
  const int ntok = min(TOKC, chunk_n - tok0);
  const int ntokA = min(TOKT, ntok), ntokB = ntok - ntokA;
  const bool hasB = ntokB > 0;
  volatile int *failed = &sm.failed;
  const LayerDev ld = p.layers[layer];
  // The loader warp sets up the barriers and asks for Q before anything that waits for the layer table.
  const bool aligned = (smem_u32(smem_raw) & 1023u) == 0;   // (the swizzled tiles have to start on a multiple of 1024)
  const bool q_by_tma = p.q_tma && aligned;
  // one lane: Q_X, when the group's heads lie side by side.  (Tokens past the tile's last one are zeros or the next tile's rows:
  // their results are not stored.)
  auto ask_q = [&](int x) {
    const uint32_t bar = smem_u32(&sm.bar_q[x]), dst = smem_u32(sm.q[x]);
    mbar_expect_tx(bar, kTileBytes);
    tma_load_4d(dst, &cm.q, 0, g * G, chunk_c0 + tok0 + x * TOKT, lrel * p.B + b, bar);
    tma_load_4d(dst + kBoxBytes, &cm.q, 64, g * G, chunk_c0 + tok0 + x * TOKT, lrel * p.B + b, bar);
  };
  int status = 0;
  if (warp == kLoadWarp && lane == 0) {
    status = *reinterpret_cast<volatile int32_t *>(&p.ctl->status);
    const int n_rows = hasB ? 2 : 1;              // row tiles: each one frees a buffer
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sm.bar_full[s]), 2);
      mbar_init(smem_u32(&sm.bar_free[s]), n_rows);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(smem_u32(&sm.bar_q[x]), p.q_tma ? 1 : 2 * kRows);
      mbar_init(smem_u32(&sm.bar_s[x]), 1);
      mbar_init(smem_u32(&sm.bar_turn[x]), 1);
      mbar_init(smem_u32(&sm.bar_p[x]), kSoftmaxThreads / 32 / 2);
      mbar_init(smem_u32(&sm.bar_pk[x]), 1);
      mbar_init(smem_u32(&sm.bar_vp[x]), 2);
      mbar_init(smem_u32(&sm.bar_lfree[x]), n_rows);
    }
    mbar_init(smem_u32(&sm.bar_done), n_rows);
    mbar_init(smem_u32(&sm.bar_state), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // (Q_B behind K_0, which the first product needs before it: 8001 tokens layer by layer 2 %, 8 x 2048 1 % less, at commit 1790120)
    if (q_by_tma) ask_q(0);
  }
  // (positions stay below 2^30, the most tokens a context may hold; a longer window is no other than that)
  constexpr int64_t kMost = int64_t(1) << 30;
  const int n0 = int(p.n0);
  const int tq0 = n0 + chunk_c0 + tok0;
  const int tq_last = tq0 + ntok - 1;
  const int w = int(ld.w < kMost ? ld.w : kMost);
  const int wl = int(ld.wlin < kMost ? ld.wlin : kMost);   // delay of the linear stream: w, or 0 when the state holds every token
  const uint32_t cap = ld.cap > 0 ? uint32_t(ld.cap) : 1u;
  const size_t unit_rows = (size_t(b + p.b0) * p.Hkv + g) * size_t(ld.cap);   // b + b0: the sequence's slot in the context
  const size_t seq = (size_t(lrel) * p.B + b) * size_t(p.T);
#ifdef GLIDE_PF_CLOCKS
  long long pf_t_ = clock64();
  if (threadIdx.x == 0) atomicAdd(&g_pf_clk[8], 1ull);
#endif

  int j_lo = tq0 - w + 1;
  if (j_lo < 0) j_lo = 0;
  j_lo &= ~(kGroup - 1);   // key tiles start at a multiple of the TMA box
  const int n_tiles = w > 0 ? (tq_last - j_lo) / kKT + 1 : 0;
  // key tiles that row tile X has valid keys in: [t_first(X), t_end(X)) (A may end, B begin one tile off the CTA's range)
  auto t_first = [&](int x) {
    const int lo = tq0 + x * TOKT - w + 1;
    return lo <= j_lo ? 0 : (lo - j_lo) / kKT;
  };
  auto t_end = [&](int x) { return n_tiles == 0 ? 0 : (tq0 + x * TOKT + (x ? ntokB : ntokA) - 1 - j_lo) / kKT + 1; };

  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm.tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == kLoadWarp) {
    // a time-out recorded by an earlier CTA ends the launch quickly
    if (lane == 0) sm.failed = status == kDevWaitTimeout || !aligned;
    // The others may go on; this warp does not wait for them: it touches no TMEM and zeroes what has to be zero itself.  (A
    // barrier of its own: the one at the end of the CTA may be reached by this warp before the others have met here.)
    __syncwarp();
    asm volatile("barrier.cta.arrive 9, %0;" ::"n"(kThreads) : "memory");
    if (*failed) {   // (set before the meeting: the same for all)
      int alone = 0;
      if (q_by_tma) mbar_wait(smem_u32(&sm.bar_q[0]), 0u, &alone);   // no copy outlives the CTA
      if (lane == 0 && !aligned) atomicExch(&p.ctl->status, kDevWaitTimeout);
      return;
    }
    // Token groups past the CTA's last token are never loaded (only the last tile has such groups), and what a
    // masked key's V row holds is multiplied by a zero weight, so it has to be finite: those rows of the buffer that
    // will hold the last V tile start at zero (earlier tiles that pass through the buffer leave real rows behind).
    if (n_tiles > 0) {
      const int last_slot = (2 * (n_tiles - 1) + 1) % kStages;
      const int j0_last = j_lo + (n_tiles - 1) * kKT;
      const int first_skipped = (tq_last - j0_last) / kGroup + 1;   // groups [first_skipped, 8) are not loaded
      const int n16 = (kKT / kGroup - first_skipped) * int(kGroupBytes / 16);
      for (int half = 0; half < 2; ++half) {
        uint4 *dst = reinterpret_cast<uint4 *>(&sm.kv[last_slot][half * kBoxBytes + first_skipped * kGroupBytes]);
        for (int i = lane; i < n16; i += 32) dst[i] = make_uint4(0u, 0u, 0u, 0u);
      }
      fence_async_smem();
    }
    __syncwarp();
  }
  // Q_X otherwise: 128 rows x 16 chunks by the 256 threads of each row tile, asked for before the set-up's barrier so that the copy
  // runs while the other warps finish setting up (it needs nothing of that; nothing else writes these tiles).  A thread's
  // rows are 16 apart, so all of them belong to one head of the group (G divides 16).
  const int X = (warp >> 2) & 1, H = warp >> 3;   // row tile and column half of this thread (softmax warps only)
  const int row = tid & 127;
  const int ntokX = X ? ntokB : ntokA;
  const bool activeX = tid < kSoftmaxThreads && ntokX > 0;
  if (activeX && !p.q_tma) {
    const int c = row & 15, r0 = (row >> 4) + 8 * H, h2 = r0 % G;
    const bf16 *src = reinterpret_cast<const bf16 *>(p.q) +
                      ((seq + size_t(chunk_c0 + tok0 + X * TOKT)) * p.H + p.heads_of[g * G + h2]) * kD + c * 8;
    const uint32_t dst = smem_u32(sm.q[X]) + sw128(r0, c);   // (r & 7 is the same for all rows of the thread)
#pragma unroll 4
    for (int i = 0; i < 8; ++i) {
      const int tk = (r0 + 16 * i) / G;
      const bool valid = tk < ntokX;
      cp_async16(dst + uint32_t(i) * 16u * 128u, src + (valid ? size_t(tk) * p.H * kD : 0), valid);
    }
    cp_async_commit();
  }
  // the CTA's first meeting: barriers and TMEM are set up
  uint32_t tmem = 0;
  if (warp != kLoadWarp) {
    fence_async_smem();
    tc_fence_before();
    asm volatile("barrier.cta.sync 9, %0;" ::"n"(kThreads) : "memory");
    tc_fence_after();
    tmem = sm.tmem_base;
    PF_CLK(0);
    if (*failed) {
      cp_async_wait_all();
      if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
      return;
    }
  }
  const uint32_t sQ0 = smem_u32(sm.q[0]);
  const uint32_t sKV0 = smem_u32(sm.kv[0]);
  auto q_addr = [&](int x) { return sQ0 + uint32_t(x) * kTileBytes; };
  auto kv_addr = [&](int slot) { return sKV0 + uint32_t(slot) * kTileBytes; };
  // Linear part: what it needs is known now, so that the loader can fetch it behind the last key tiles.
  const bool linear = ld.evicts && tq_last >= wl;
  const int folded = n0 + chunk_c0 - wl;   // tokens below this index are in S, z at the start of the chunk
  const bool need_state = linear && folded > 0;
  // intra-chunk steps: delayed tokens of this chunk up to the CTA's last token, 128 at a time
  const int i_lo = folded < 0 ? min(-folded, chunk_n) : 0;
  const int i_hi = tok0 + ntok - 1;
  const int it0 = i_lo & ~(kKT - 1);
  const int n_itiles = (linear && it0 <= i_hi) ? (i_hi - it0) / kKT + 1 : 0;   // (linear without a state: at least one)
  // Roles of the five buffers after the window loop, by the order in which the loop stops using them (load number
  // 2 n_tiles - 5 + k; a negative number is a buffer the loop never used): the first to come free receives the bf16
  // copy of the unit's state, the next two the phi(K') tiles of the first two intra-chunk steps, the last two the V'
  // tiles of those steps; all are on their way while the last key tiles are still being processed.  Later steps take the
  // buffers of the step before the previous one.
  // Learned map and gated: twice the operands, so they come when every window product has completed: phi- (or phi's lo) of
  // the two row tiles in buffers 0 and 1 (phi+ or hi in the Q tiles), the state's two tiles and then the two phi(K') tiles
  // of each step in 2 and 3, V' in 4.
  auto late_seq = [&](int k) { return 2 * n_tiles - kStages + k; };
  auto late_slot = [&](int k) { const int sq = late_seq(k); return sq >= 0 ? sq % kStages : sq + kStages; };
  auto slot_state = [&]() { return TWO ? 2 : late_slot(0); };
  auto slot_pk = [&](int t) { return TWO ? 2 : late_slot(1 + (t & 1)); };
  auto slot_vp = [&](int t) { return TWO ? 4 : late_slot(3 + (t & 1)); };

  if (tid < kSoftmaxThreads) {
    // =========================== softmax threads: half a row each ===========================
    // Two threads per row, in warps that share a scheduler: thread (X, H, row) has columns 64 H .. 64 H + 63 of every 128-column
    // operand of the row.  One warp per scheduler and row tile waited on its own chain of loads, maxima, exponentials and stores (a
    // CTA took some 5000 issue slots of 29500 cycles); a pair of warps fills each other's gaps.  What the row has in common goes
    // through sm.exch behind barriers of the two warps, which every thread of a pair passes equally often: after a time-out the
    // waits return at once and the loops run on, storing nothing.
    // Every hand-over of row tile X is its own: the threads of A and of B meet only at the end of the CTA, so that one
    // tile's arithmetic runs beside the other's products.  bar_s completes once per batch of products of X, bar_p once
    // per operand that X's threads have written; both sides count in the same order.
    const int tok_r = row / G;
    const int tl = tok0 + X * TOKT + tok_r;         // chunk-relative token of this row
    const int tok_abs = n0 + chunk_c0 + tl;
    const uint32_t tS = tmem + (uint32_t((warp & 3) * 32) << 16) + uint32_t(X) * 128u + uint32_t(H) * 64u;
    const uint32_t tO = tS + 256u;
    float m_ref = -CUDART_INF_F, l_sum = 0.f;       // l: of this thread's columns
    uint32_t n_s = 0;                               // batches of products waited for
    bool ok = true;
    const int my_head = p.heads_of[g * G + lane % G];   // (head of group member h: lane h has it)
    auto wait_s = [&]() {
      if (ok) ok = mbar_wait(smem_u32(&sm.bar_s[X]), n_s & 1u, failed);
      ++n_s;
      tc_fence_after();
      ok = __all_sync(0xffffffffu, ok);             // warp-uniform
    };
    auto wait_once = [&](uint64_t &bar) { ok = ok && mbar_wait(smem_u32(&bar), 0u, failed); };
    // the operand that the MMA warp waits for is complete as far as this warp goes
    auto hand_over = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.bar_p[X]));
    };
    const int pair_bar = 1 + (warp & 7);            // named barrier of warps w and w + 8
    auto pair_sync = [&]() { asm volatile("barrier.cta.sync %0, 64;" ::"r"(pair_bar) : "memory"); };
    auto pair_any = [&](bool x) {
      uint32_t r;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbarrier.cta.red.or.pred p, %2, 64, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(r)
          : "r"(uint32_t(x)), "r"(pair_bar)
          : "memory");
      return r != 0;
    };
    // f(first thread's value, second thread's value) in both threads of a row
    auto combine = [&](float v, auto &&f) {
      float *slot = &sm.exch[tid & (kSoftmaxThreads / 2 - 1)];
      if (H == 0) *slot = v;
      pair_sync();
      if (H == 1) *slot = v = f(*slot, v);
      pair_sync();
      return H == 0 ? *slot : v;
    };
    auto row_sum_of = [&](float v) { return combine(v, [](float a, float b) { return a + b; }); };
    auto row_max_of = [&](float v) { return combine(v, [](float a, float b) { return fmaxf(a, b); }); };
    // multiply this thread's part of the O row by f (warp-collective TMEM read-modify-write)
    auto scale_o = [&](float f) {
#pragma unroll 1
      for (int c0 = 0; c0 < kHalf; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(tO + c0, r);
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
        tmem_st32(tO + c0, r);
      }
    };
    // weights of columns c .. c + 31 over columns c / 2 .. c / 2 + 15 (of the half); gated: hi over c .. c + 15, lo (first half
    // of x) over c + 16 .. c + 31
    auto store_p = [&](int c, const uint32_t (&pk)[16], const uint32_t (&x)[32]) {
      if constexpr (GATED) {
        uint32_t lo[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) lo[e] = x[e];
        tmem_st16(tS + c, pk);
        tmem_st16(tS + c + 16, lo);
      } else {
        tmem_st16(tS + (c >> 1), pk);
      }
    };
    // the lazy reference for a tile whose maximum over this thread's columns (raw) is mx: it moves, and O and l are rescaled, only
    // when the row's maximum grows by more than 2^kLazy; returns what the weights are taken against
    auto move_ref = [&](float mx, bool first) {
      auto grows = [&]() {
        const float ms = mx * p.scale_log2;   // (the scale is positive: it is applied to the maximum)
        return ms > m_ref + kLazy || (m_ref == -CUDART_INF_F && ms > -CUDART_INF_F);
      };
      if (pair_any(grows())) {
        mx = row_max_of(mx);
        float f = 1.f;
        if (grows()) {
          mx *= p.scale_log2;
          f = m_ref == -CUDART_INF_F ? 0.f : ex2(m_ref - mx);
          m_ref = mx;
        }
        if (!first && __any_sync(0xffffffffu, f != 1.f)) scale_o(f);
        l_sum *= f;
      }
      return m_ref == -CUDART_INF_F ? 0.f : m_ref;
    };
    auto row_max = [&](const uint32_t (&x)[32], float mx) {
      float m4[4] = {mx, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
      for (int i = 0; i < 32; i += 2) m4[(i >> 1) & 3] = max3(m4[(i >> 1) & 3], __uint_as_float(x[i]), __uint_as_float(x[i + 1]));
      return fmaxf(max3(m4[0], m4[1], m4[2]), m4[3]);
    };
    // weights of columns c .. c + 31 (scores x) over the S columns this thread has already consumed (columns c / 2 ..
    // c / 2 + 15); the sum uses the weights as the tensor core sees them
    auto weights = [&](int c, uint32_t (&x)[32], float mr, float &sum0, float &sum1) {
      uint32_t pk[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        float a0, a1;
        fma2(a0, a1, __uint_as_float(x[e * 2]), __uint_as_float(x[e * 2 + 1]), p.scale_log2, -mr);
        if constexpr (GATED) {
          a0 = ex2(a0), a1 = ex2(a1);
          add2(sum0, sum1, a0, a1);
          split2(a0, a1, pk[e], x[e]);   // (x[e] has been read: element e comes from x[2 e] and x[2 e + 1])
        } else {
          pk[e] = pack_bf16x2(ex2(a0), ex2(a1));
          add2(sum0, sum1, bf16_lo(pk[e]), bf16_hi(pk[e]));
        }
      }
      store_p(c, pk, x);
    };
    // A later key tile against the reference as it is, in one pass: no maximum is looked for.  The largest weight says afterwards whether
    // that was right: below 2^kLazy the reference stays, as it does in soft_tile_masked.  Otherwise (false, to both threads of all
    // rows of the pair) nothing has happened, the scores are still there, and the tile goes through soft_tile_masked.  (Two passes: 1840
    // cycles a tile, one 1770.  A row's first tile is taken against its maximum: against 0 a short window's tile took 2400 cycles
    // instead of 3500, but the rounding of the largest weights, which are 1 against the maximum, cost 6 % in precision.)
    auto soft_tile = [&](auto masked, int lo, int hi) {
      float sum0 = 0.f, sum1 = 0.f;
      const float mr = m_ref;
      uint32_t pk[32], mx2 = 0u;
#pragma unroll
      for (int c = 0; c < kHalf; c += 32) {
        uint32_t x[32];
        tmem_ld32(tS + c, x);
        if (decltype(masked)::value) {
          const uint32_t m = column_mask(c, lo, hi);
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i] = (m >> i) & 1u ? x[i] : 0xff800000u;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          float a0, a1;
          fma2(a0, a1, __uint_as_float(x[e * 2]), __uint_as_float(x[e * 2 + 1]), p.scale_log2, -mr);
          const uint32_t w2 = pack_bf16x2(ex2(a0), ex2(a1));
          mx2 = max_bf16x2(mx2, w2);
          add2(sum0, sum1, bf16_lo(w2), bf16_hi(w2));   // the sum uses the weights as the tensor core sees them
          pk[(c >> 1) + e] = w2;
        }
      }
      const float mx = fmaxf(bf16_lo(mx2), bf16_hi(mx2));
      if (pair_any(!(mx < 0x1p8f))) return false;
      tmem_st32(tS, pk);
      l_sum += sum0 + sum1;
      return true;
    };
    // One key tile with masked keys (valid columns lo .. hi of this row's half).  32 columns at a time, those in which no row of
    // the warp has a valid one left out; the loops stay rolled: with everything unrolled the kernel was 210 KB of code that a CTA
    // fetched once per phase (a CTA's first key tile took 12000 cycles, a later one 2500).  For the masked tiles of gated contexts, rows
    // that have no reference yet, and tiles that soft_tile leaves alone.
    auto soft_tile_masked = [&](int lo, int hi, bool first) {
      float mx = -CUDART_INF_F, sum0 = 0.f, sum1 = 0.f;
#pragma unroll 1
      for (int c = 0; c < kHalf; c += 32) {
        const uint32_t m = column_mask(c, lo, hi);
        if (!__any_sync(0xffffffffu, m)) continue;
        uint32_t x[32];
        tmem_ld32(tS + c, x);
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = (m >> i) & 1u ? x[i] : 0xff800000u;
        mx = row_max(x, mx);
      }
      const float mr = move_ref(mx, first);
#pragma unroll 1
      for (int c = 0; c < kHalf; c += 32) {
        const uint32_t m = column_mask(c, lo, hi);
        uint32_t x[32];
        if (!__any_sync(0xffffffffu, m)) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) pk[e] = x[e] = 0u;
          store_p(c, pk, x);
          continue;
        }
        tmem_ld32(tS + c, x);
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = (m >> i) & 1u ? x[i] : 0xff800000u;
        weights(c, x, mr, sum0, sum1);
      }
      tmem_wait_st();
      l_sum += sum0 + sum1;
    };
    // Gated: a key tile without a masked key, in the two passes of soft_tile_masked without its masks and votes.  4 layers, 4000 tokens
    // on windows of 1024 / 4096 / 16384: 1.61 / 2.55 / 5.03 ms; through soft_tile_masked 1.69 / 2.91 / 6.35, which was more than with
    // one thread per row (1.65 / 2.71 / 5.63).  (In one pass as soft_tile, hi and lo kept in 64 registers: 1.61 / 2.51 / 4.88, but with
    // 64 bytes more of spills 1.5 % longer at windows of 64.)
    auto soft_tile_gated = [&](bool first) {
      float mx = -CUDART_INF_F, sum0 = 0.f, sum1 = 0.f;
      uint32_t x[32];
      tmem_ld32(tS, x);
      mx = row_max(x, mx);
      tmem_ld32(tS + 32, x);
      mx = row_max(x, mx);
      const float mr = move_ref(mx, first);
#pragma unroll 1
      for (int c = 0; c < kHalf; c += 32) {
        tmem_ld32(tS + c, x);
        weights(c, x, mr, sum0, sum1);
      }
      tmem_wait_st();
      l_sum += sum0 + sum1;
    };
    if (activeX) {
      if (!p.q_tma) {
        cp_async_wait_all();   // Q_X (asked for before the set-up's barrier) has landed
        fence_async_smem();
        mbar_arrive(smem_u32(&sm.bar_q[X]));
      }
      // phi(q) of the parameter-free map is e^(q - max) / sum; both numbers come from the Q tile while the first product runs, the
      // values later (the tile is the products' operand until then)
      float q_mxl = 0.f, q_sum = 1.f;                // max log2(e); sum (over the row)
      auto load_q = [&](uint32_t (&v)[32]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 v4 = *reinterpret_cast<const uint4 *>(sm.q[X] + sw128(row, H * 8 + i));
          v[i * 4] = v4.x, v[i * 4 + 1] = v4.y, v[i * 4 + 2] = v4.z, v[i * 4 + 3] = v4.w;
        }
      };
      if (linear && !PHI2) {
        wait_once(sm.bar_q[X]);
        uint32_t v[32];
        load_q(v);
        uint32_t m2 = v[0];
#pragma unroll
        for (int i = 1; i < 32; ++i) m2 = max_bf16x2(m2, v[i]);
        q_mxl = row_max_of(fmaxf(bf16_lo(m2), bf16_hi(m2))) * kLog2e;
        if (!SUM) {
          float sum0 = 0.f, sum1 = 0.f;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float a0, a1;
            fma2(a0, a1, bf16_lo(v[i]), bf16_hi(v[i]), kLog2e, -q_mxl);
            add2(sum0, sum1, ex2(a0), ex2(a1));
          }
          q_sum = row_sum_of(sum0 + sum1);
        }
      }
      const int tqX0 = tq0 + X * TOKT, tqX_last = tqX0 + ntokX - 1;
      const int tf = t_first(X), te = t_end(X);
      for (int t = tf; t < te; ++t) {
        wait_s();
        if (tid == X * kRows) {   // S of the tile and P V of the tile before have completed
          mbar_arrive(smem_u32(&sm.bar_free[2 * t % kStages]));
          if (t > tf) mbar_arrive(smem_u32(&sm.bar_free[(2 * t - 1) % kStages]));
        }
        if (t == tf) PF_CLK(11); else PF_CLK(12);
        const int j0 = j_lo + t * kKT;
        const bool whole = j0 + kKT - 1 <= tqX0 && j0 > tqX_last - w;
        // valid columns of this row: lo <= c <= hi (a token more than 2^30 - 1 before another is none)
        const int lo = max(tok_abs - w + 1 - j0, 0), hi = min(tok_abs - j0, kKT - 1);
        bool done = false;
        if constexpr (GATED) {
          if (whole) soft_tile_gated(t == tf);
          done = whole;
        } else {
          // (what is asked here is the same in both warps of a pair: their threads share the rows)
          if (t > tf && !__any_sync(0xffffffffu, m_ref == -CUDART_INF_F)) {
            if (whole) done = soft_tile(std::false_type{}, 0, kHalf - 1);
            else done = soft_tile(std::true_type{}, lo - H * kHalf, hi - H * kHalf);
          }
        }
        if (!done) soft_tile_masked(lo - H * kHalf, hi - H * kHalf, t == tf);
        hand_over();            // this thread's TMEM accesses precede the MMAs that read P and overwrite S
        if (t == tf) PF_CLK(13); else PF_CLK(14);
      }
      const bool windowed = te > tf;               // O_X holds a valid accumulation
      if (linear) {
        // Any common reference M >= m_ref gives the same quotient O / l.  M = max(m_ref, 0) would rescale O for every
        // row whose window maximum is negative; a floor of -64 keeps 2^-M and everything scaled by it far inside the
        // fp32 / bf16 range (phi <= 1) and makes that rescale a rarity.
        // A row without evicted tokens (position below the window size) keeps its own reference and gets phi(q) = 0:
        // a floor there would only push its window weights towards underflow.
        // Sum of two normalised terms instead: the window part is normalised now (O / l), and phi(q) is divided by the
        // row's linear normaliser phi(q) . (z + running sum of phi(K') up to the row's own delayed token), so that what
        // the linear products add to O is the normalised linear term; the final division is by 1.
        const bool has_lin = tok_abs >= wl;
        const float M = has_lin ? fmaxf(m_ref, -64.f) : m_ref;
        float fw = m_ref == -CUDART_INF_F ? 0.f : ex2(m_ref - M);
        const float fl = has_lin ? ex2(-M) : 0.f;
        if (SUM) {
          const float l = row_sum_of(l_sum);
          fw = l > 0.f ? 1.0f / l : 0.f;
          l_sum = 0.5f;                             // (of each half: the final division is by 1)
        } else {
          l_sum *= fw;
        }
        if (PHI2 || (SUM && need_state)) wait_once(sm.bar_state);   // phi(Q); z
        unsigned char *tileX = sm.q[X];
        float dot = 0.f;
        const float g_own = GATED ? p.gcum[size_t(uc) * p.SC + min(tl, chunk_n - 1)] : 0.f;
        const float dec0 = GATED ? ex2(g_own * kLog2e) : 1.f;   // what the chunk-start state has decayed to
        if constexpr (!PHI2) {
          // this half row of Q is still in the shared tile, and every S product of X has completed: phi(q) takes its place
          uint32_t v[32];
          load_q(v);
          const bool with_z = !SUM && need_state;
          const float *zh = sm.z + H * kHalf;
          float dot1 = 0.f;
          if (SUM) {
            // sum of terms: phi(q) / (phi(q) . z_row) = e / (e . z_row)
            const float2 *zrow =
                reinterpret_cast<const float2 *>(p.zcum + (size_t(uc) * p.SC + size_t(tok_r < ntokX ? tl : tok0)) * kD + H * kHalf);
            float dz0 = 0.f, dz1 = 0.f;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              float a0, a1;
              fma2(a0, a1, bf16_lo(v[i]), bf16_hi(v[i]), kLog2e, -q_mxl);
              const float2 zc = __ldg(zrow + i);
              dot2(dz0, dz1, ex2(a0), ex2(a1), zc.x + (need_state ? zh[i * 2] : 0.f), zc.y + (need_state ? zh[i * 2 + 1] : 0.f));
            }
            q_sum = row_sum_of(dz0 + dz1);
          }
          if (with_z) wait_once(sm.bar_state);     // z has landed
          if constexpr (GATED) {
            // fp32 values, hi in place, lo in a buffer of the finished window part
            const float sc = fl * __frcp_rn(q_sum);
            wait_once(sm.bar_done);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              uint32_t hi4[4], lo4[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t x = v[c * 4 + e];
                float a0, a1;
                fma2(a0, a1, bf16_lo(x), bf16_hi(x), kLog2e, -q_mxl);
                a0 = ex2(a0) * sc, a1 = ex2(a1) * sc;
                split2(a0, a1, hi4[e], lo4[e]);
                if (with_z) dot2(dot, dot1, a0, a1, zh[c * 8 + e * 2], zh[c * 8 + e * 2 + 1]);
              }
              *reinterpret_cast<uint4 *>(tileX + sw128(row, H * 8 + c)) = make_uint4(hi4[0], hi4[1], hi4[2], hi4[3]);
              *reinterpret_cast<uint4 *>(sm.kv[X] + sw128(row, H * 8 + c)) = make_uint4(lo4[0], lo4[1], lo4[2], lo4[3]);
            }
            dot = (dot + dot1) * dec0;
          } else {
            // shared normaliser: phi(q) 2^-M.  The factor goes into the exponent, so that a value is rounded once.
            const bool some = has_lin && (!SUM || q_sum > 0.f);
            const float shift = some ? q_mxl + lg2(q_sum) + (SUM ? 0.f : M) : CUDART_INF_F;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              uint32_t o4[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t x = v[c * 4 + e];
                float a0, a1;
                fma2(a0, a1, bf16_lo(x), bf16_hi(x), kLog2e, -shift);
                o4[e] = pack_bf16x2(ex2(a0), ex2(a1));
                if (with_z) dot2(dot, dot1, bf16_lo(o4[e]), bf16_hi(o4[e]), zh[c * 8 + e * 2], zh[c * 8 + e * 2 + 1]);
              }
              *reinterpret_cast<uint4 *>(tileX + sw128(row, H * 8 + c)) = make_uint4(o4[0], o4[1], o4[2], o4[3]);
            }
            dot += dot1;
          }
        } else {
          // this thread's part of phi+ and of phi-: times 2^-M, back as bf16; the dot with z uses the rounded values
#pragma unroll 1
          for (int hf = 0; hf < 2; ++hf) {
            unsigned char *tile = hf == 0 ? tileX : sm.kv[X];
#pragma unroll 4
            for (int c = H * 8; c < H * 8 + 8; ++c) {
              uint4 *at = reinterpret_cast<uint4 *>(tile + sw128(row, c));
              const uint4 v4 = *at;
              uint32_t w4[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                w4[e] = pack_bf16x2(bf16_lo(w4[e]) * fl, bf16_hi(w4[e]) * fl);
                if (need_state)
                  dot += bf16_lo(w4[e]) * sm.z[hf * kD + c * 8 + e * 2] + bf16_hi(w4[e]) * sm.z[hf * kD + c * 8 + e * 2 + 1];
              }
              *at = make_uint4(w4[0], w4[1], w4[2], w4[3]);
            }
          }
        }
        l_sum += dot;
        if (windowed) {
          wait_s();                                // the last P V has completed
          if (__any_sync(0xffffffffu, fw != 1.f)) scale_o(fw);
        }
        fence_async_smem();
        hand_over();
        PF_CLK(10);
        if (GATED && need_state) {
          // phi(q) S is in the S columns: it has decayed by dec0 since the chunk began, row by row, so it is added here
          wait_s();
#pragma unroll 1
          for (int c0 = 0; c0 < kHalf; c0 += 32) {
            uint32_t o[32], x[32];
            tmem_ld32_nowait(tS + c0, x);
            if (windowed) tmem_ld32_nowait(tO + c0, o);
            tmem_wait_ld(x);
            if (windowed) tmem_wait_ld(o);
#pragma unroll
            for (int i = 0; i < 32; ++i)
              o[i] = __float_as_uint(fmaf(__uint_as_float(x[i]), dec0, windowed ? __uint_as_float(o[i]) : 0.f));
            tmem_st32(tO + c0, o);
          }
          hand_over();
        }
        // C row -> bf16 over the same TMEM columns, masked to the delayed tokens j' <= i of the row (the values already
        // carry 2^-M); the row's weight sum goes to l
        for (int t = 0; t < n_itiles; ++t) {
          wait_s();
          PF_CLK(3);
          const int i0 = it0 + t * kKT;
          float sum0 = 0.f, sum1 = 0.f;
          const int lo = i_lo - i0 - H * kHalf, hi = tl - i0 - H * kHalf;
          // a tile that lies wholly before the row tile's first token (and after the first delayed token) needs no mask
          const bool whole = i0 + kKT - 1 <= tok0 + X * TOKT && i0 >= i_lo;
#pragma unroll 1
          for (int c = 0; c < kHalf; c += 32) {
            uint32_t pk[16], x[32];
            const uint32_t m = whole ? ~0u : column_mask(c, lo, hi);
            // the running log-gates of the 32 columns' tokens, one per lane
            const float gl = GATED ? __ldg(p.gcum + size_t(uc) * p.SC + min(i0 + H * kHalf + c + lane, chunk_n - 1)) : 0.f;
            if (!__any_sync(0xffffffffu, m)) {   // no row of the warp has a delayed token here
#pragma unroll
              for (int e = 0; e < 16; ++e) pk[e] = x[e] = 0u;
              store_p(c, pk, x);
              continue;
            }
            tmem_ld32(tS + c, x);
            if (!GATED && !whole) {
#pragma unroll
              for (int i = 0; i < 32; ++i) x[i] = (m >> i) & 1u ? x[i] : 0u;
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              if constexpr (GATED) {
                // a delayed token ii <= i has decayed by exp(g_own - gc[ii]) <= 1; the others are left out after the product,
                // whatever it is (their factor is above 1 and may be infinite, or the gate of a later token not a number)
                const float g0 = __shfl_sync(0xffffffffu, gl, e * 2), g1 = __shfl_sync(0xffffffffu, gl, e * 2 + 1);
                float a0 = __uint_as_float(x[e * 2]) * ex2((g_own - g0) * kLog2e);
                float a1 = __uint_as_float(x[e * 2 + 1]) * ex2((g_own - g1) * kLog2e);
                if (!whole) a0 = (m >> (e * 2)) & 1u ? a0 : 0.f, a1 = (m >> (e * 2 + 1)) & 1u ? a1 : 0.f;
                add2(sum0, sum1, a0, a1);
                split2(a0, a1, pk[e], x[e]);
              } else {
                pk[e] = pack_bf16x2(__uint_as_float(x[e * 2]), __uint_as_float(x[e * 2 + 1]));
                add2(sum0, sum1, bf16_lo(pk[e]), bf16_hi(pk[e]));
              }
            }
            store_p(c, pk, x);
          }
          tmem_wait_st();
          if (!SUM) l_sum += sum0 + sum1;
          hand_over();
          PF_CLK(4);
        }
      }
      // ---- normalise and store: through the Q tile (every product that read it has completed), so that a warp's stores
      // are whole lines ----
      if (windowed || linear) {
        const float l_row = row_sum_of(l_sum);
        wait_s();                                  // every product of X has completed
        PF_CLK(5);
        const float inv = tok_r < ntokX ? 1.0f / l_row : 0.f;
        float chk0 = 0.f, chk1 = 0.f;   // gated: sums of the row's values, finite if all of them are
#pragma unroll 1
        for (int c0 = 0; c0 < kHalf; c0 += 32) {
          uint32_t r[32];
          tmem_ld32(tO + c0, r);
          if (GATED) {
#pragma unroll
            for (int i = 0; i < 32; i += 2) add2(chk0, chk1, __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
          }
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              pk[e] = pack_bf16x2(__uint_as_float(r[q4 * 8 + e * 2]) * inv, __uint_as_float(r[q4 * 8 + e * 2 + 1]) * inv);
            *reinterpret_cast<uint4 *>(sm.q[X] + sw128(row, H * 8 + (c0 >> 3) + q4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
        // a warp stores the 32 half rows its own threads have written, eight lanes to each; a lane's rows are 4 apart
        __syncwarp();
        const int c = H * 8 + (lane & 7), r0 = (row & ~31) + (lane >> 3);
        bf16 *obase = reinterpret_cast<bf16 *>(p.out) + (seq + size_t(chunk_c0 + tok0 + X * TOKT)) * p.H * kD + c * 8;
#pragma unroll 1
        for (int i0 = 0; i0 < 8; i0 += 4) {
          uint4 val[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) val[i] = *reinterpret_cast<const uint4 *>(sm.q[X] + sw128(r0 + 4 * (i0 + i), c));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int rr = r0 + 4 * (i0 + i), tk = rr / G;
            const int head = __shfl_sync(0xffffffffu, my_head, rr - tk * G);
            if (ok && tk < ntokX) *reinterpret_cast<uint4 *>(obase + (size_t(tk) * p.H + head) * kD) = val[i];
          }
        }
        if constexpr (GATED) {
          // rows of which either half is not finite, by the first warp of the pair when both have stored
          const bool bad = !isfinite((chk0 + chk1) * inv) && tok_r < ntokX;
          const unsigned again = __ballot_sync(0xffffffffu, row_sum_of(bad ? 1.f : 0.f) > 0.f);
          if (H == 0 && again && ok) recompute_rows<G>(p, again, X * kRows + (row & ~31), u, sub, tok0);
        }
      }
    }
  } else if (warp < kLoadWarp) {
    // =========================== MMA warps ===========================
    // A warp stays together (every wait ends in a vote), one elected lane issues.
    const bool leader = elect_one();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const int x = __shfl_sync(0xffffffffu, warp, 0) - kMmaWarp;   // the row tile
    const uint32_t tS = tm + uint32_t(x) * 128u, tO = tS + 256u;
    const int tf = t_first(x), te = t_end(x);
    uint32_t p_phase = 0;                          // parity of the next operand
    bool ok = x == 0 || hasB;
    auto wait = [&](uint64_t &bar, uint32_t parity) {
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), parity, failed));
      return ok;
    };
    auto wait_p = [&]() {
      const uint32_t par = p_phase;
      p_phase ^= 1u;
      wait(sm.bar_p[x], par);
      tc_fence_after();
      return ok;
    };
    auto commit = [&](uint64_t &bar) {
      if (leader) mma_commit(smem_u32(&bar));
    };
    // O (+)= A B with A in the S columns: packed bf16, or hi and lo in turn every 32 columns
    auto issue_ts = [&](uint32_t b_tile, bool accumulate) {
      if (!GATED) {
        issue_mma_ts<false>(leader, tO, tS, b_tile, accumulate);
      } else {
        issue_mma_ts<true>(leader, tO, tS, b_tile, accumulate);
        issue_mma_ts<true>(leader, tO, tS + 16, b_tile, true);
      }
    };
    // D (+)= [Q tile of X | buffer X] . [buffer 2 | buffer 3], the map's halves or hi and lo
    auto issue_two = [&](uint32_t d, bool b_mn, bool accumulate) {
      issue_mma(leader, d, q_addr(x), kv_addr(2), b_mn, accumulate);
      if (GATED) {
        issue_mma(leader, d, kv_addr(x), kv_addr(2), b_mn, true);
        issue_mma(leader, d, q_addr(x), kv_addr(3), b_mn, true);
      } else {
        issue_mma(leader, d, kv_addr(x), kv_addr(3), b_mn, true);
      }
    };
    PF_LAP_INIT();
    // t = -1: the first S product; then per key tile P V of the tile and S of the next one.  The two warps take turns: products of
    // A and B that run mixed end together, and then both tiles' softmax runs beside nothing (5000 cycles per key tile against
    // 3700).  Buffers are freed by the softmax threads when they see the next product's completion, and only those that no
    // later product follows here: a commit takes a place in the tensor core's queue.
    for (int t = -1; t < n_tiles && ok; ++t) {
      const int seqV = 2 * t + 1, seqK = 2 * t + 2;
      const bool more = t + 1 < n_tiles;
      const bool pv = t >= tf && t < te, qk = t + 1 >= tf && t + 1 < te;
      PF_LAP(18);
      if (t >= 0) wait(sm.bar_full[seqV % kStages], uint32_t(seqV / kStages) & 1u);
      if (ok && more) wait(sm.bar_full[seqK % kStages], uint32_t(seqK / kStages) & 1u);
      PF_LAP(16);
      if (ok && qk && t + 1 == tf) wait(sm.bar_q[x], 0u);
      if (ok && hasB && (x == 1 || t >= 0)) wait(sm.bar_turn[x], uint32_t(x == 1 ? t + 1 : t) & 1u);
      PF_LAP(17);
      if (ok && pv) wait_p();
      if (!ok) break;
      PF_LAP(19);
      if (pv) {
        issue_ts(kv_addr(seqV % kStages), t > tf);
        if (t + 1 == te) commit(sm.bar_s[x]);      // the window part of O
      }
      if (qk) {
        issue_mma(leader, tS, q_addr(x), kv_addr(seqK % kStages), false, false);
        commit(sm.bar_s[x]);
      }
      if (leader) {
        if (hasB) mbar_arrive(smem_u32(&sm.bar_turn[x ^ 1]));
        if (pv && t + 1 == te) mma_commit(smem_u32(&sm.bar_free[seqV % kStages]));
        if (!pv && t >= 0) mbar_arrive(smem_u32(&sm.bar_free[seqV % kStages]));   // (a tile without a valid key for this row tile)
        if (!qk && more) mbar_arrive(smem_u32(&sm.bar_free[seqK % kStages]));
      }
      // The query rows of the CTA that will take this place one wave later are asked into L2 (line by line: bulk prefetches of
      // the rows took the memory pipe 12000 cycles; before the first products the address arithmetic held them up by 1900).
      if (t < 0 && x == (hasB ? 1 : 0) && blockIdx.x + unsigned(p.sm_count) < gridDim.x) {
        const unsigned nb = blockIdx.x + unsigned(p.sm_count), nu = nb / unsigned(ctas_per_unit);
        const int ncta = ctas_per_unit - 1 - int(nb - nu * unsigned(ctas_per_unit)), nsub = ncta / ctas_per_chunk;
        const int ncol = (ncta - nsub * ctas_per_chunk) * TOKC, ntok0 = nsub * p.SC + ncol;   // relative to the pass
        const int nrows = min(TOKC, min(p.SC - ncol, p.C - ntok0)) * G;
        const int head = p.heads_of[(nu % unsigned(p.Hkv)) * G + (lane >> 1) % G];            // (rows are 16 apart: one head per lane)
        const bf16 *nq = reinterpret_cast<const bf16 *>(p.q) + (size_t(nu / unsigned(p.Hkv)) * size_t(p.T) + size_t(p.c0 + ntok0)) * p.H * kD +
                         size_t(head) * kD + (lane & 1) * 64;
#pragma unroll 4
        for (int r = lane >> 1; r < nrows; r += 16)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(nq + size_t(r / G) * p.H * kD));
      }
    }
    if (ok) commit(sm.bar_done);
    const bool windowed = te > tf;
    if (ok && linear && !TWO) {
      // the first C = phi(Q) phi(K')^T, then phi(Q) S (inter-chunk): the softmax threads convert C while the state's product
      // runs (its completion shows in the next batch)
      if (wait_p() && wait(sm.bar_pk[0], 0u)) {
        issue_mma(leader, tS, q_addr(x), kv_addr(slot_pk(0)), false, false);
        commit(sm.bar_s[x]);
      }
      if (ok && need_state && wait(sm.bar_state, 0u)) issue_mma(leader, tO, q_addr(x), kv_addr(slot_state()), true, windowed);
      for (int t = 0; t < n_itiles && ok; ++t) {
        wait(sm.bar_vp[t & 1], uint32_t(t >> 1) & 1u);
        if (ok && t + 1 < n_itiles) wait(sm.bar_pk[(t + 1) & 1], uint32_t((t + 1) >> 1) & 1u);
        if (!ok || !wait_p()) break;
        issue_ts(kv_addr(slot_vp(t)), windowed || need_state || t > 0);
        if (t + 1 < n_itiles) issue_mma(leader, tS, q_addr(x), kv_addr(slot_pk(t + 1)), false, false);
        commit(sm.bar_s[x]);
        commit(sm.bar_lfree[t & 1]);   // V'(t) has been read, and phi(K')(t) before it
      }
    }
    if (ok && linear && TWO) {
      // phi+ S+ and phi- S-, then per step C = phi+ phi+(K')^T + phi- phi-(K')^T (accumulated before the causal mask)
      // and C V'; the phi(K') halves of a step take the buffers of the state, or of the step before.  Gated: phi(Q) S goes
      // to the S columns, from where the softmax threads add it to O with the row's decay.
      if (GATED && need_state) wait(sm.bar_state, 0u);
      if (ok && wait_p()) {
        if (need_state) issue_two(GATED ? tS : tO, true, !GATED && windowed);
        if (GATED && need_state) commit(sm.bar_s[x]);
        commit(sm.bar_lfree[0]);
      }
      if (GATED && need_state && ok) wait_p();   // the state's part has left the S columns
      for (int t = 0; t < n_itiles && ok; ++t) {
        if (!wait(sm.bar_pk[0], uint32_t(t) & 1u)) break;
        issue_two(tS, false, false);
        commit(sm.bar_s[x]);
        if (!wait(sm.bar_vp[0], uint32_t(t) & 1u) || !wait_p()) break;
        issue_ts(kv_addr(4), windowed || need_state || t > 0);
        if (t + 1 == n_itiles) commit(sm.bar_s[x]);
        commit(sm.bar_lfree[0]);
      }
    }
  } else {
    // =========================== loader warp ===========================
    // A 128-key tile is eight groups of 16 tokens.  A group that lies in one source (ring or call) and is contiguous
    // there is fetched by TMA, lane gi issuing the two boxes (column halves) of group gi so that the address
    // arithmetic of the groups runs in parallel.  A group that straddles the call boundary or a ring wrap is copied
    // row by row by the whole warp (at most a few per tile).  Each buffer's barrier takes two arrivals: the
    // expect-tx one before the TMA boxes are issued and a plain one after the row copies.
    const CUtensorMap *ringK = ring_maps + 3 * layer, *ringV = ringK + 1;
    const CUtensorMap *ringK128 = ring_maps + 3 * p.L + 2 * layer, *ringV128 = ringK128 + 1;
    const CUtensorMap *map_pk = ring_maps + 5 * p.L, *map_s16 = map_pk + 1, *map_pq = map_pk + 2;
    const bf16 *ringKp = reinterpret_cast<const bf16 *>(p.ws + ld.ringK) + unit_rows * kD;
    const bf16 *ringVp = reinterpret_cast<const bf16 *>(p.ws + ld.ringV) + unit_rows * kD;
    const bf16 *callKp = reinterpret_cast<const bf16 *>(p.k) + (seq * p.Hkv + g) * kD;
    const bf16 *callVp = reinterpret_cast<const bf16 *>(p.v) + (seq * p.Hkv + g) * kD;
    const int64_t call_stride = int64_t(p.Hkv) * kD;
    const int gi = lane;
    bool ok = true;
    auto tma_tile = [&](uint32_t dst, const CUtensorMap *m, int y, uint32_t bar) {
      tma_load_2d(dst, m, 0, y, bar);
      tma_load_2d(dst + kBoxBytes, m, 64, y, bar);
    };
    // Jobs of the warp in order: the K and V tiles of the window (2 n_tiles), one job for the operands of the linear part
    // that one thread fetches, then the V' tiles of the intra-chunk steps (with the phi(K') tiles of later steps).
    const int n_window = 2 * n_tiles;
    const int n_jobs = n_window + (linear ? 1 + n_itiles : 0);
    const int job_qb = q_by_tma && hasB ? min(n_window, 1) : -1;   // the job before which Q_B is asked for
#pragma unroll 1
    for (int job = 0; job < n_jobs; ++job) {
      if (job == job_qb && lane == 0) ask_q(1);
      if (job == n_window) {
        if (lane == 0 && !TWO) {
          // the bf16 state (with z), then the phi(K') tiles of the first two intra-chunk steps
          const int n_late = 1 + (n_itiles < 2 ? n_itiles : 2);
#pragma unroll 1
          for (int k = 0; k < n_late && ok; ++k) {
            if (k == 0 && !need_state) continue;
            const int sq = late_seq(k);
            if (sq >= 0) ok = mbar_wait(smem_u32(&sm.bar_free[sq % kStages]), uint32_t(sq / kStages) & 1u, failed);
            if (!ok) break;
            const uint32_t bar = k == 0 ? smem_u32(&sm.bar_state) : smem_u32(&sm.bar_pk[k - 1]);
            mbar_expect_tx(bar, kTileBytes + (k == 0 ? uint32_t(kD * sizeof(float)) : 0u));
            if (k == 0) bulk_load(smem_u32(sm.z), p.zsnap + size_t(uc) * kD, uint32_t(kD * sizeof(float)), bar);
            tma_tile(kv_addr(late_slot(k)), k == 0 ? map_s16 : map_pk, k == 0 ? int(uc) * kD : int(uc) * p.SC + it0 + (k - 1) * kKT, bar);
          }
        }
        if (lane == 0 && TWO && (PHI2 || need_state)) {
          const uint32_t bar = smem_u32(&sm.bar_state);
          const int rows_q = int(p.units_cap) * p.SC * G, rows_s = int(p.units_cap) * kD;
          ok = mbar_wait(smem_u32(&sm.bar_done), 0u, failed);
          if (PHI2 && ok && n_tiles == 0) {        // no window: phi+ takes the place of Q when Q's copies have landed
            ok = mbar_wait(smem_u32(&sm.bar_q[0]), 0u, failed);
            if (ok && hasB) ok = mbar_wait(smem_u32(&sm.bar_q[1]), 0u, failed);
          }
          if (ok) {
            const uint32_t zbytes = uint32_t((PHI2 ? 2 : 1) * kD * sizeof(float));
            mbar_expect_tx(bar, (PHI2 ? (hasB ? 4u : 2u) * kTileBytes : 0u) + (need_state ? 2u * kTileBytes + zbytes : 0u));
#pragma unroll 1
            for (int i = 0; PHI2 && i < (hasB ? 4 : 2); ++i) {
              const int x = i >> 1, hf = i & 1;
              tma_tile(hf == 0 ? q_addr(x) : kv_addr(x), map_pq, hf * rows_q + (int(uc) * p.SC + tok0 + x * TOKT) * G, bar);
            }
            if (need_state) {
              tma_tile(kv_addr(2), map_s16, int(uc) * kD, bar);
              tma_tile(kv_addr(3), map_s16, rows_s + int(uc) * kD, bar);
              bulk_load(smem_u32(sm.z), p.zsnap + size_t(uc) * p.dp, zbytes, bar);
            }
          }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        continue;
      }
      // Rows of tokens j0 .. j0 + 127 (K or V) into buffer `slot` (the whole warp); 16-row groups that lie wholly above
      // the CTA's last token are not written in the window, but zero in a V' tile, as are rows of tokens below 0 (their
      // weights are zero, and 0 x anything must stay 0).  j0 need not be a multiple of the box size: a ring row or a token
      // of the call is a TMA coordinate like any other.
      const bool late = job > n_window;
      const int ts = late ? job - n_window - 1 : job >> 1;       // intra-chunk step, or key tile
      const bool is_v = late || (job & 1);
      const int slot = late ? slot_vp(ts) : job % kStages;
      const uint32_t bar = late ? smem_u32(&sm.bar_vp[TWO ? 0 : ts & 1]) : smem_u32(&sm.bar_full[slot]);
      const int j0 = late ? folded + it0 + ts * kKT : j_lo + ts * kKT;
      if (!late) {
        PF_LAP_INIT();
        if (job >= kStages) ok = mbar_wait(smem_u32(&sm.bar_free[slot]), uint32_t(job / kStages - 1) & 1u, failed);
        PF_LAP(20);
      } else if (!TWO) {
        const int sq = late_seq(3 + ts);
        if (ts < 2) {
          if (sq >= 0) ok = mbar_wait(smem_u32(&sm.bar_free[sq % kStages]), uint32_t(sq / kStages) & 1u, failed);
        } else {   // the buffers of step ts - 2: its phi(K') tile was read before its V' tile
          ok = mbar_wait(smem_u32(&sm.bar_lfree[ts & 1]), uint32_t((ts >> 1) - 1) & 1u, failed);
          if (ok && lane == 0) {
            const uint32_t pkb = smem_u32(&sm.bar_pk[ts & 1]);
            mbar_expect_tx(pkb, kTileBytes);
            tma_tile(kv_addr(slot_pk(ts)), map_pk, int(uc) * p.SC + it0 + ts * kKT, pkb);
          }
        }
      } else {   // learned map, gated: the state's or the previous step's products have completed
        ok = mbar_wait(smem_u32(&sm.bar_lfree[0]), uint32_t(ts) & 1u, failed);
        if (ok && lane == 0) {
          const uint32_t pkb = smem_u32(&sm.bar_pk[0]);
          const int rows_k = int(p.units_cap) * p.SC, y = int(uc) * p.SC + it0 + ts * kKT;
          mbar_expect_tx(pkb, 2u * kTileBytes);
          tma_tile(kv_addr(2), map_pk, y, pkb);
          tma_tile(kv_addr(3), map_pk, rows_k + y, pkb);
        }
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const int left = tq_last - j0;                         // >= 0: the tile holds at least one valid token
      const int ngroups = left >= kKT - 1 ? kKT / kGroup : left / kGroup + 1;
      // A full tile that lies in one source without a wrap takes two boxes of 128 rows (the layout in shared memory
      // is that of eight 16-row boxes).  Tiles that reach past the last token keep the 16-row path, which never
      // loads a later token's row.  (left >= kKT - 1: every row of the tile is a token up to the last one; eight groups
      // alone would also admit a last group that is only partly valid)
      if (j0 >= 0 && left >= kKT - 1) {
        const uint32_t slot_row0 = uint32_t(j0) % cap;
        const bool all_call = j0 >= n0;
        if (all_call || (j0 + kKT <= n0 && slot_row0 + kKT <= cap)) {
          if (lane == 0) {
            mbar_expect_tx(bar, kTileBytes);
            const uint32_t dst = kv_addr(slot);
            // (the same rows kAhead key tiles further on are asked into L2: a buffer is refilled one key tile before it is
            // needed, which covers a trip to L2 but not one to memory)
            constexpr int kAhead = 3;
            const bool ahead = !late && ts + kAhead < n_tiles;
            if (all_call) {
              const CUtensorMap *m = is_v ? &cm.v128 : &cm.k128;
              tma_load_4d(dst, m, 0, g, j0 - n0, lrel * p.B + b, bar);
              tma_load_4d(dst + kBoxBytes, m, 64, g, j0 - n0, lrel * p.B + b, bar);
              if (ahead) {
                tma_prefetch_4d(m, 0, g, j0 - n0 + kAhead * kKT, lrel * p.B + b);
                tma_prefetch_4d(m, 64, g, j0 - n0 + kAhead * kKT, lrel * p.B + b);
              }
            } else {
              const CUtensorMap *m = is_v ? ringV128 : ringK128;
              tma_tile(dst, m, int(unit_rows + slot_row0), bar);
              if (ahead && slot_row0 + (kAhead + 1) * kKT <= cap) {
                tma_prefetch_2d(m, 0, int(unit_rows + slot_row0) + kAhead * kKT);
                tma_prefetch_2d(m, 64, int(unit_rows + slot_row0) + kAhead * kKT);
              }
            }
            mbar_arrive(bar);   // the barrier's second arrival (after the row copies on the other path)
          }
          __syncwarp();
          continue;
        }
      }
      // this lane's group: where it comes from and whether one box covers it
      const int j = j0 + gi * kGroup;
      const bool mine = gi < kKT / kGroup && (late || gi < ngroups);
      const bool from_call = j >= n0;
      const uint32_t slot_row = j < 0 ? 0u : uint32_t(j) % cap;
      const bool boxed = mine && gi < ngroups && j >= 0 && (from_call || (j + kGroup <= n0 && slot_row + kGroup <= cap));
      const unsigned boxed_mask = __ballot_sync(0xffffffffu, boxed);
      const unsigned manual_mask = __ballot_sync(0xffffffffu, mine && !boxed);
      if (lane == 0) mbar_expect_tx(bar, uint32_t(__popc(boxed_mask)) * 2u * kGroupBytes);
      __syncwarp();
      if (boxed) {
        const uint32_t dst = kv_addr(slot) + uint32_t(gi) * kGroupBytes;
        if (from_call) {
          const CUtensorMap *m = is_v ? &cm.v : &cm.k;
          tma_load_4d(dst, m, 0, g, j - n0, lrel * p.B + b, bar);
          tma_load_4d(dst + kBoxBytes, m, 64, g, j - n0, lrel * p.B + b, bar);
        } else {
          tma_tile(dst, is_v ? ringV : ringK, int(unit_rows + slot_row), bar);
        }
      }
#pragma unroll 1
      for (unsigned mm = manual_mask; mm; mm &= mm - 1) {
        const int gm = __ffs(int(mm)) - 1;
        unsigned char *tile = sm.kv[slot];
#pragma unroll 2
        for (int i = 0; i < kGroup * 16 / 32; ++i) {
          const int id = lane + 32 * i;
          const int r = id >> 4, c = id & 15;
          const int jj = j0 + gm * kGroup + r;
          uint4 val = make_uint4(0u, 0u, 0u, 0u);
          if (jj >= 0 && jj <= tq_last) {
            const uint32_t sr = uint32_t(jj) % cap;
            const bf16 *src = jj >= n0 ? (is_v ? callVp : callKp) + size_t(jj - n0) * call_stride
                                         : (is_v ? ringVp : ringKp) + size_t(sr) * kD;
            val = *reinterpret_cast<const uint4 *>(src + c * 8);
          }
          *reinterpret_cast<uint4 *>(tile + sw128(gm * kGroup + r, c)) = val;
        }
      }
      fence_async_smem();   // the row copies are read by the tensor core (async proxy)
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    }
  }
  // after a time-out the waits return at once and nothing is stored; the CTA meets here either way
  tc_fence_before();
  __syncthreads();
  PF_CLK(6);
  if (tid == 0 && sm.failed) atomicExch(&p.ctl->status, kDevWaitTimeout);
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

}  // namespace


// The kernel needs the ring descriptors made for the tensor-core decode kernels.
#ifdef GLIDE_PF_CLOCKS
extern "C" int glide_debug_pf_clocks(unsigned long long *host32, int reset) {
  if (cudaMemcpyFromSymbol(host32, g_pf_clk, sizeof(g_pf_clk)) != cudaSuccess) return 6;
  if (reset) {
    unsigned long long z[32] = {};
    if (cudaMemcpyToSymbol(g_pf_clk, z, sizeof(z)) != cudaSuccess) return 6;
  }
  return 0;
}
#endif

bool prefill_attn_tc_supported(const glide_ctx *ctx) {
  return ctx->cfg.io_dtype == GLIDE_BF16 && ctx->cfg.head_dim == kD && ctx->decode_kind >= 1 && ctx->off_phik16 != 0;
}

namespace {
typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                             const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn tensor_map_encoder() {
  static EncodeFn fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess || !f ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;
    }
    return reinterpret_cast<EncodeFn>(f);
  }();
  return fn;
}
}  // namespace

int launch_prefill_attn_tc(glide_ctx *ctx, const PrefillParams &pass, cudaStream_t stream) {
  PrefillParams p = pass;
  EncodeFn encode = tensor_map_encoder();
  if (!encode) return GLIDE_ERR_CUDA;
  CallMaps cm;
  {
    const cuuint64_t dims[4] = {cuuint64_t(kD), cuuint64_t(p.Hkv), cuuint64_t(p.T), cuuint64_t(p.layer_count) * cuuint64_t(p.B)};
    const cuuint64_t strides[3] = {cuuint64_t(kD) * 2, cuuint64_t(p.Hkv) * kD * 2, cuuint64_t(p.T) * p.Hkv * kD * 2};
    const cuuint32_t box[4] = {64, 1, kGroup, 1}, box128[4] = {64, 1, kKT, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    memset(&cm, 0, sizeof(cm));
    // (a whole-tile box is used only for tiles that lie inside the call: calls shorter than a tile never need it)
    for (int kv = 0; kv < (p.T >= kKT ? 4 : 2); ++kv) {
      CUtensorMap *m = kv == 0 ? &cm.k : kv == 1 ? &cm.v : kv == 2 ? &cm.k128 : &cm.v128;
      CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>((kv & 1) == 0 ? p.k : p.v), dims,
                          strides, kv < 2 ? box : box128, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return GLIDE_ERR_UNSUPPORTED;
    }
    p.q_tma = 1;
    for (int h = 0; h < p.H; ++h) p.q_tma = p.q_tma && ctx->heads_of[size_t(h)] == h;   // groups of neighbouring heads
    if (p.q_tma) {
      const cuuint64_t qdims[4] = {cuuint64_t(kD), cuuint64_t(p.H), cuuint64_t(p.T), cuuint64_t(p.layer_count) * cuuint64_t(p.B)};
      const cuuint64_t qstrides[3] = {cuuint64_t(kD) * 2, cuuint64_t(p.H) * kD * 2, cuuint64_t(p.T) * p.H * kD * 2};
      const cuuint32_t qbox[4] = {64, cuuint32_t(ctx->G), cuuint32_t(kRows / ctx->G), 1};
      CUresult r = encode(&cm.q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(p.q), qdims, qstrides, qbox, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return GLIDE_ERR_UNSUPPORTED;
    }
  }
  const CUtensorMap *ring_maps = reinterpret_cast<const CUtensorMap *>(ctx->ws + ctx->off_tmaps);
  const int64_t units = int64_t(p.layer_count) * p.B * p.Hkv;
  auto launch = [&](auto gg) -> int {
    constexpr int G = decltype(gg)::value;
    constexpr int TOKC = 2 * kRows / G;
    const size_t smem = sizeof(Smem);
    const int64_t blocks = units * (int64_t(p.nsub - 1) * ((p.SC + TOKC - 1) / TOKC) + (p.C - (p.nsub - 1) * p.SC + TOKC - 1) / TOKC);
    auto run = [&](auto kern) -> int {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) {
        cudaGetLastError();
        return GLIDE_ERR_CUDA;
      }
      kern<<<unsigned(blocks), kThreads, smem, stream>>>(p, ring_maps, cm);
      return cudaGetLastError() == cudaSuccess ? GLIDE_OK : GLIDE_ERR_CUDA;
    };
    if (p.gated) return run(prefill_attn_tc_kernel<G, kModeGated>);      // (shared normaliser only, both)
    if (p.phiq16) return run(prefill_attn_tc_kernel<G, kModeLearned>);
    return p.merge == GLIDE_MERGE_SHARED ? run(prefill_attn_tc_kernel<G, kModeShared>) : run(prefill_attn_tc_kernel<G, kModeSum>);
  };
  switch (ctx->G) {
    case 1: return launch(IntTag<1>{});
    case 2: return launch(IntTag<2>{});
    case 4: return launch(IntTag<4>{});
    case 8: return launch(IntTag<8>{});
    default: return GLIDE_ERR_UNSUPPORTED;
  }
}

}  // namespace glide

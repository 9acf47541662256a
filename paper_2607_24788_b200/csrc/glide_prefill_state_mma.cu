// Chunk-scan carry of the prefill for bf16 I/O and d = 128 on the tensor cores, at fp32 accuracy:
//   S += phi(K')^T V',  z += sum phi(K')      over the chunk's delayed tokens (k'_i = k_{i-w}).
// For gates, and where another kernel makes phi (the learned map, sum-of-terms merges with outputs, outputs by the mma.sync or the
// CUDA-core kernel); all else is the kernel of glide_prefill_carry_tc.cu.
// V' is bf16 already.  phi(K') is fp32 in the chunk scratch; every value is split into three bf16 terms
// (x = hi + mid + lo, each the bf16 rounding of what the previous ones left: an error-free split of the 24-bit
// significand), so the three products phi_term^T V' are exact in fp32 and only the fp32 accumulation of the tensor
// core rounds.  The carry therefore stays an fp32 quantity, as the method's chunk scan requires, while the
// 2 C d^2 multiply-adds per KV head leave the CUDA cores (a bf16 or tf32 product of phi(K') itself would miss the
// 1e-5 state tolerance).  z is summed in fp32 on the CUDA cores from the same staged values.
//
// One CTA of 4 warps per (unit, chunk of the pass, 64 state rows); warp w owns rows 16 w .. 16 w + 15 and all 128 columns
// (16 n-tiles of m16n8k16, 64 accumulators per thread).  Tokens are staged 32 at a time through two shared-memory
// buffers filled by cp.async; row strides are padded (272 bytes) so that the scalar reads of the A fragments and
// the ldmatrix reads of V' are free of bank conflicts.  In gated contexts with the parameter-free map the kernel makes phi(K')
// itself from the staged K' rows (both CTAs of a unit's chunk the whole row, for its normaliser, each keeping its 64 columns) and
// leaves the bf16 rows for the attention kernel: as a kernel in front, phi cost a trip of 512 bytes per token through memory.
#include <algorithm>
#include <type_traits>

#include "glide_device.cuh"

namespace glide {

namespace {

constexpr int kD = 128;
constexpr int kThreads = 128;
constexpr int kRowsPerCta = 64;
constexpr int kTok = 32;                      // tokens per stage
constexpr int kPhiStride = 68;                // floats per staged phi row (64 + 4: conflict-free fragment reads)
constexpr int kVStride = 272;                 // bytes per staged V' row (256 + 16: conflict-free ldmatrix)
constexpr int kPhiBytes = kTok * kPhiStride * 4;
constexpr int kVBytes = kTok * kVStride;

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return uint32_t(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool valid) {
  const int bytes = valid ? 16 : 0;   // 0: writes zeros, reads nothing
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// x0, x1 -> three packed bf16 pairs (x0 in the low half) whose sums give x0, x1 back to fp32 accuracy
__device__ __forceinline__ void split3(float x0, float x1, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
  const float r0 = x0 - __low2float(h), r1 = x1 - __high2float(h);
  const __nv_bfloat162 m = __floats2bfloat162_rn(r0, r1);
  const float s0 = r0 - __low2float(m), s1 = r1 - __high2float(m);
  const __nv_bfloat162 l = __floats2bfloat162_rn(s0, s1);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  mid = *reinterpret_cast<const uint32_t *>(&m);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

// the bf16 copy of two values of S (gated: hi here and lo `lo_half` elements further on)
__device__ __forceinline__ void store_s16(__nv_bfloat16 *at, size_t lo_half, float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  *reinterpret_cast<__nv_bfloat162 *>(at) = h;
  if (lo_half) *reinterpret_cast<__nv_bfloat162 *>(at + lo_half) = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
}

// One element of a gated chunk's sum in fp32, token after token: what a split term times an infinity (0 x inf, or an infinity of
// the other sign) must not decide.  Row `row` of S and column `col` of V'; phi(k') of the row from `phi` (stride dp), or made
// from the K' rows with the tokens' maxima and 1 / sums.  Cold: called for sums that are not finite.
struct CarryRows {
  const __nv_bfloat16 *ringK, *ringV, *callK, *callV;
  int64_t n0, first, cap, call_stride;
  const float *gc;
  float g_end;
  int i_lo, chunk_n;
  __device__ __forceinline__ int64_t at(int i) const {
    const int64_t j = first + i;
    return j >= n0 ? (j - n0) * call_stride : int64_t(uint32_t(j) % uint32_t(cap)) * kD;
  }
  __device__ __forceinline__ const __nv_bfloat16 *k(int i) const { return (first + i >= n0 ? callK : ringK) + at(i); }
  __device__ __forceinline__ const __nv_bfloat16 *v(int i) const { return (first + i >= n0 ? callV : ringV) + at(i); }
};
__device__ __noinline__ float carry_element(const CarryRows &rows, const float *phi, int dp, const float2 *stats, int row, int col) {
  float sum = 0.f;
#pragma unroll 4
  for (int i = rows.i_lo; i < rows.chunk_n; ++i) {
    const float f = phi ? phi[size_t(i) * dp] : exp2f((__bfloat162float(rows.k(i)[row]) - stats[i].x) * kLog2e) * stats[i].y;
    sum = fmaf(f * expf(rows.g_end - rows.gc[i]), __bfloat162float(rows.v(i)[col]), sum);
  }
  return sum;
}

// PARTIAL (passes of several chunks): the chunk's own sum goes to the scratch rows that the CTA has just consumed instead
// of S (64 state rows x 128 values = 128 scratch rows x the CTA's 64 columns, z in row 128: chunks of more than 128
// tokens), and prefill_scan_kernel adds the sums up in chunk order.  Otherwise S is updated in place, and its value
// before the chunk is left as bf16 (z: fp32) for the attention kernel, which runs after this one.
// MAKE_PHI: phi(K') is made here (parameter-free map, gated, no sum-of-terms merge); otherwise it is in the scratch.
template <bool PARTIAL, bool MAKE_PHI, bool GATED>
__global__ void __launch_bounds__(kThreads, GATED ? 3 : 0) prefill_state_mma_kernel(const PrefillParams p) {
  if (!GATED) dependents_may_start();
  wait_for_predecessor();
  using bf16 = __nv_bfloat16;
  static_assert(!MAKE_PHI || GATED, "without gates glide_prefill_carry_tc.cu makes phi");
  // per stage phi columns (or K' rows, 16 bytes more per row) and V' rows; made phi columns
  constexpr int kInBytes = MAKE_PHI ? kVBytes : kPhiBytes;
  __shared__ __align__(16) unsigned char stage[2][kInBytes + kVBytes];
  __shared__ __align__(16) float made[MAKE_PHI ? kTok * kPhiStride : 4];
  __shared__ float decay[2][kTok];   // gated: what each staged token has decayed to by the end of the chunk
  const int blocks_per_unit = p.dp / kRowsPerCta;   // rows of S: d, or 2 d with the learned feature map
  const int64_t uc = blockIdx.x / blocks_per_unit;   // (unit, chunk of the pass)
  const int rb = blockIdx.x % blocks_per_unit;
  const int64_t u = PARTIAL ? uc / p.nsub : uc;
  const int chunk_c0 = PARTIAL ? int(uc - u * p.nsub) * p.SC : 0;   // first token of the chunk, relative to the pass
  const int chunk_n = min(p.SC, p.C - chunk_c0);
  const int g = int(u % p.Hkv);
  const int b = int((u / p.Hkv) % p.B);
  const int lrel = int(u / (int64_t(p.Hkv) * p.B));
  const LayerDev ld = p.layers[p.layer_begin + lrel];
  if (!ld.evicts) return;
  const int64_t first = p.n0 + p.c0 + chunk_c0 - ld.wlin;    // delayed token of chunk index 0
  const int i_lo = first < 0 ? int(first < -int64_t(chunk_n) ? chunk_n : -first) : 0;
  if (i_lo >= chunk_n) return;
  const int ub = (b + p.b0) * p.Hkv + g;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gid = lane >> 2, tig = lane & 3;
  // V' rows: the ring for tokens older than the call, the call's own rows otherwise
  const int64_t cap = ld.cap > 0 ? ld.cap : 1;
  const bf16 *ringV = reinterpret_cast<const bf16 *>(p.ws + ld.ringV) + size_t(ub) * size_t(ld.cap) * kD;
  const bf16 *callV = reinterpret_cast<const bf16 *>(p.v) + ((size_t(lrel) * p.B + b) * size_t(p.T) * p.Hkv + g) * kD;
  const bf16 *ringK = reinterpret_cast<const bf16 *>(p.ws + ld.ringK) + size_t(ub) * size_t(ld.cap) * kD;
  const bf16 *callK = reinterpret_cast<const bf16 *>(p.k) + ((size_t(lrel) * p.B + b) * size_t(p.T) * p.Hkv + g) * kD;
  const int64_t call_stride = int64_t(p.Hkv) * kD;
  bf16 *p16 = MAKE_PHI && p.phik16 ? reinterpret_cast<bf16 *>(p.phik16) + (size_t(u) * p.Cmax + chunk_c0) * kD + rb * kRowsPerCta : nullptr;
  float *pk = p.phik + (size_t(u) * p.Cmax + chunk_c0) * p.dp + rb * kRowsPerCta;

  float acc[kD / 8][4];
#pragma unroll
  for (int n = 0; n < kD / 8; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
  float zacc = 0.f;   // threads 0..63: z of row rb*64 + tid
  const float *gc = GATED ? p.gcum + size_t(u) * p.Cmax + chunk_c0 : nullptr;
  const float g_end = GATED ? gc[chunk_n - 1] : 0.f;

  // tokens past the chunk's end are filled with zeros
  auto issue = [&](int buf, int i0) {
    const int nt = min(kTok, chunk_n - i0);
    const uint32_t sphi = smem_addr(stage[buf]), sv = sphi + kInBytes;
    for (int e = tid; !MAKE_PHI && e < kTok * (kRowsPerCta / 4); e += kThreads) {
      const int i = e / (kRowsPerCta / 4), c4 = e % (kRowsPerCta / 4);
      cp16(sphi + uint32_t(i * kPhiStride + c4 * 4) * 4u, pk + size_t(i0 + (i < nt ? i : 0)) * p.dp + c4 * 4, i < nt);
    }
    for (int e = tid; e < kTok * 16; e += kThreads) {
      const int i = e >> 4, c = e & 15;
      const int64_t j = first + i0 + (i < nt ? i : 0);
      const int64_t at = j >= p.n0 ? (j - p.n0) * call_stride : int64_t(uint32_t(j) % uint32_t(cap)) * kD;   // (tokens stay below 2^31)
      cp16(sv + uint32_t(i * kVStride + c * 16), (j >= p.n0 ? callV : ringV) + at + c * 8, i < nt);
      if (MAKE_PHI) cp16(sphi + uint32_t(i * kVStride + c * 16), (j >= p.n0 ? callK : ringK) + at + c * 8, i < nt);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (tid < kTok) decay[buf][tid] = (GATED && tid < nt) ? expf(g_end - gc[i0 + tid]) : 1.f;   // (rows past the end are zero)
  };
  issue(0, i_lo);
  int buf = 0;
  for (int i0 = i_lo; i0 < chunk_n; i0 += kTok, buf ^= 1) {
    if (i0 + kTok < chunk_n) {
      issue(buf ^ 1, i0 + kTok);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    if constexpr (MAKE_PHI) {
      // four threads per token, 32 entries each; those of this CTA's columns go to `made`, rounded to the bf16 rows
      const int tok = tid >> 2, part = tid & 3;
      const uint4 *src = reinterpret_cast<const uint4 *>(stage[buf] + tok * kVStride + part * 64);
      float x[32];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint4 v = src[c];
        const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          x[c * 8 + e * 2] = __uint_as_float(w4[e] << 16);
          x[c * 8 + e * 2 + 1] = __uint_as_float(w4[e] & 0xffff0000u);
        }
      }
      float mx = x[0];
#pragma unroll
      for (int i = 1; i < 32; ++i) mx = fmaxf(mx, x[i]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        x[i] = exp2f((x[i] - mx) * kLog2e);
        sum += x[i];
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      const bool there = i0 + tok < chunk_n;
      const float inv = there ? 1.0f / sum : 0.f;   // (rows past the chunk's end stay zero)
      if (part >> 1 == rb) {
        float *dst = made + tok * kPhiStride + (part & 1) * 32;
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[i + e] *= inv;
          *reinterpret_cast<float4 *>(dst + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
        }
        if (p16 && there) {
          bf16 *out = p16 + size_t(i0 + tok) * kD + (part & 1) * 32;
#pragma unroll
          for (int hl = 0; hl < 2; ++hl) {   // (what the rounding left in the second half of the array)
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              uint32_t o[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(x[i + e * 2], x[i + e * 2 + 1]);
                o[e] = *reinterpret_cast<const uint32_t *>(&h);
                x[i + e * 2] -= __low2float(h);
                x[i + e * 2 + 1] -= __high2float(h);
              }
              *reinterpret_cast<uint4 *>(out + (hl ? size_t(p.units_cap) * p.SC * kD : 0) + i) = make_uint4(o[0], o[1], o[2], o[3]);
            }
          }
        }
      }
      __syncthreads();
    }
    const float *sphi = MAKE_PHI ? made : reinterpret_cast<const float *>(stage[buf]);
    const uint32_t sv = smem_addr(stage[buf]) + kInBytes;
    // A = phi(K')^T: element (row r, k i) = phi(k'_i)[r]; fragment registers a0: (gid, 2 tig + {0,1}),
    // a1: (gid + 8, ..), a2: (gid, 2 tig + 8 + {0,1}), a3: (gid + 8, ..)
    auto split_a = [&](int kk, uint32_t (&ah)[4], uint32_t (&am)[4], uint32_t (&al)[4]) {
      const float *base = sphi + (kk * 16 + 2 * tig) * kPhiStride + warp * 16 + gid;
      const float *dk = decay[buf] + kk * 16 + 2 * tig;   // (without gates: exact products with 1)
      split3(base[0] * dk[0], base[kPhiStride] * dk[1], ah[0], am[0], al[0]);
      split3(base[8] * dk[0], base[kPhiStride + 8] * dk[1], ah[1], am[1], al[1]);
      split3(base[8 * kPhiStride] * dk[8], base[9 * kPhiStride] * dk[9], ah[2], am[2], al[2]);
      split3(base[8 * kPhiStride + 8] * dk[8], base[9 * kPhiStride + 8] * dk[9], ah[3], am[3], al[3]);
    };
    // 16 tokens by 16 columns on top of d0, d1, smallest terms first
    auto product = [&](int kk, int dp, const uint32_t (&ah)[4], const uint32_t (&am)[4], const uint32_t (&al)[4], float (&d0)[4], float (&d1)[4]) {
      const int krow = kk * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
      uint32_t bfr[4];
      ldsm_x4_trans(bfr, sv + uint32_t(krow * kVStride + (2 * dp + (lane >> 4)) * 16));
      mma16816(d0, al, bfr[0], bfr[1]);
      mma16816(d1, al, bfr[2], bfr[3]);
      mma16816(d0, am, bfr[0], bfr[1]);
      mma16816(d1, am, bfr[2], bfr[3]);
      mma16816(d0, ah, bfr[0], bfr[1]);
      mma16816(d1, ah, bfr[2], bfr[3]);
    };
    if constexpr (GATED) {
      // The tensor core adds without rounding to nearest, and a gated state is held by other kernels to 2e-7 (S after 1000 tokens,
      // gates of 0.99 to 1, against fp64; this kernel 5.5e-7 with all sums in the tensor core, 1.5e-7 so): only the 32 tokens of
      // a stage are summed there, on top of zero, and the stages by the CUDA cores.  (Pass of 1000 tokens, 64 units:
      // 31.5 us -> 34.)
      uint32_t ah[kTok / 16][4], am[kTok / 16][4], al[kTok / 16][4];
#pragma unroll
      for (int kk = 0; kk < kTok / 16; ++kk) split_a(kk, ah[kk], am[kk], al[kk]);
#pragma unroll
      for (int dp = 0; dp < kD / 16; ++dp) {
        float part[2][4] = {};
#pragma unroll
        for (int kk = 0; kk < kTok / 16; ++kk) product(kk, dp, ah[kk], am[kk], al[kk], part[0], part[1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[2 * dp][e] += part[0][e], acc[2 * dp + 1][e] += part[1][e];
      }
    } else {
#pragma unroll
      for (int kk = 0; kk < kTok / 16; ++kk) {
        uint32_t ah[4], am[4], al[4];
        split_a(kk, ah, am, al);
#pragma unroll
        for (int dp = 0; dp < kD / 16; ++dp) product(kk, dp, ah, am, al, acc[2 * dp], acc[2 * dp + 1]);
      }
    }
    if (tid < kRowsPerCta) {
#pragma unroll 8
      for (int i = 0; i < kTok; ++i) zacc = fmaf(sphi[i * kPhiStride + tid], decay[buf][i], zacc);
    }
    __syncthreads();   // the stage is refilled by the next iteration's issue
  }
  if constexpr (GATED) {
    float chk[4] = {};   // finite if every sum of the thread is
#pragma unroll
    for (int n = 0; n < kD / 8; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) chk[e] += acc[n][e];
    if (__syncthreads_or(!isfinite(chk[0] + chk[1] + chk[2] + chk[3]))) {
      const CarryRows rows{ringK, ringV, callK, callV, p.n0, first, cap, call_stride, gc, g_end, i_lo, chunk_n};
      float2 *stats = reinterpret_cast<float2 *>(&stage[0][0]);   // [chunk token]: maximum of K', 1 / sum of its exponentials
      static_assert(sizeof(stage) >= 1024 * sizeof(float2), "as many as a chunk has tokens");
      for (int i = i_lo + tid; MAKE_PHI && i < chunk_n; i += kThreads) {
        const bf16 *kr = rows.k(i);
        float mx = __bfloat162float(kr[0]), sum = 0.f;
        for (int c = 1; c < kD; ++c) mx = fmaxf(mx, __bfloat162float(kr[c]));
        for (int c = 0; c < kD; ++c) sum += exp2f((__bfloat162float(kr[c]) - mx) * kLog2e);
        stats[i] = make_float2(mx, 1.0f / sum);
      }
      __syncthreads();
#pragma unroll
      for (int n = 0; n < kD / 8; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int row = warp * 16 + gid + (e >> 1) * 8;
          if (!isfinite(acc[n][e]))
            acc[n][e] = carry_element(rows, MAKE_PHI ? nullptr : pk + row, p.dp, stats, rb * kRowsPerCta + row, n * 8 + 2 * tig + (e & 1));
        }
      __syncthreads();   // (PARTIAL: the sums go over the scratch that was read)
    }
  }
  if (GATED) dependents_may_start();   // (8 layers of 8000 tokens, state only: 1.18 ms; at the kernel's top, and in the gcum kernel, 1.44, not at all 1.48)
  // accumulator fragment: c0, c1 -> (row gid, cols 2 tig + {0,1}); c2, c3 -> row gid + 8
  if (PARTIAL) {   // (every read of these scratch columns lies before the loop's last barrier)
#pragma unroll
    for (int n = 0; n < kD / 8; ++n)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = warp * 16 + gid + h * 8, col = n * 8 + 2 * tig;
        *reinterpret_cast<float2 *>(pk + size_t(2 * row + (col >> 6)) * p.dp + (col & 63)) =
            make_float2(acc[n][2 * h], acc[n][2 * h + 1]);
      }
    if (tid < kRowsPerCta) pk[size_t(kD) * p.dp + tid] = zacc;
    return;
  }
  float *Sb = reinterpret_cast<float *>(p.ws + ld.S) + size_t(ub) * p.dp * kD + size_t(rb * kRowsPerCta + warp * 16) * kD;
  // the halves of a state with 2 d rows are units_cap units apart in the bf16 copy, as are hi and lo of a gated one
  const size_t lo_half = GATED ? size_t(p.units_cap) * kD * kD : 0;
  const float dec_all = GATED ? expf(g_end) : 1.f;   // the state the chunk started from, after the whole chunk has entered
  bf16 *s16 = p.s16 ? reinterpret_cast<bf16 *>(p.s16) + (size_t(rb * kRowsPerCta / kD) * p.units_cap + u) * kD * kD +
                          size_t(rb * kRowsPerCta % kD + warp * 16) * kD
                    : nullptr;
#pragma unroll
  for (int n = 0; n < kD / 8; ++n)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const size_t at = size_t(gid + h * 8) * kD + n * 8 + 2 * tig;
      float2 *dst = reinterpret_cast<float2 *>(Sb + at);
      float2 c = *dst;
      if (s16) store_s16(s16 + at, lo_half, c.x, c.y);
      c.x = fmaf(c.x, dec_all, acc[n][2 * h]);
      c.y = fmaf(c.y, dec_all, acc[n][2 * h + 1]);
      *dst = c;
    }
  if (tid < kRowsPerCta) {
    float *zb = reinterpret_cast<float *>(p.ws + ld.z) + size_t(ub) * p.dp + rb * kRowsPerCta;
    const float z0 = zb[tid];
    if (s16) p.zsnap[size_t(u) * p.dp + rb * kRowsPerCta + tid] = z0;
    zb[tid] = fmaf(z0, dec_all, zacc);
  }
}

// The chunk sums of a pass added up in chunk order: S and z of the context move on by the whole pass, and their values at
// the start of every chunk are left for the attention kernel (bf16 copy of S, fp32 z) when there are outputs (SNAP).  One CTA per
// (unit, 4 rows of S): four warps with four columns of a row per thread, and a fifth for z, whose four chains of one value per chunk
// would hold up a warp that has its own.  The sums of the next four chunks are on their way while four are added.
template <bool GATED, bool SNAP>
__global__ void __launch_bounds__(kThreads + 32) prefill_scan_kernel(const PrefillParams p) {
  using bf16 = __nv_bfloat16;
  dependents_may_start();
  wait_for_predecessor();
  const unsigned ctas_per_unit = unsigned(p.dp) / 4;
  const int u = int(blockIdx.x / ctas_per_unit);
  const int j = int(blockIdx.x - unsigned(u) * ctas_per_unit), tid = threadIdx.x;
  const int ug = u / p.Hkv, g = u - ug * p.Hkv, lrel = ug / p.B, b = ug - lrel * p.B;
  const LayerDev &ld = p.layers[p.layer_begin + lrel];
  if (!ld.evicts) return;
  // chunks before the first delayed token add nothing (and have left no sum): k0 is the first that does
  const int64_t first = p.n0 + p.c0 - ld.wlin;
  if (first + p.C <= 0) return;
  const int k0 = first < 0 ? int(-first) / p.SC : 0;
  const int ub = (b + p.b0) * p.Hkv + g;
  const size_t step = size_t(p.SC) * p.dp;
  // gated: what the state has decayed by over chunk k (tokens before the first delayed one count as gates of 1)
  const float *gc = GATED ? p.gcum + size_t(u) * p.Cmax - 1 : nullptr;
  // f(k, value of the sum of chunk k) for every chunk, kAhead loads together
  auto over_chunks = [&](auto ahead, auto load, auto &&f) {
    constexpr int kAhead = decltype(ahead)::value;
    using Value = decltype(load(0));
    const int n = p.nsub;
    Value x[kAhead], y[kAhead];
#pragma unroll
    for (int a = 0; a < kAhead; ++a) x[a] = load(min(k0 + a, n - 1));
    int k = k0;
    for (; k + kAhead <= n; k += kAhead) {
#pragma unroll
      for (int a = 0; a < kAhead; ++a) y[a] = load(min(k + kAhead + a, n - 1));
#pragma unroll
      for (int a = 0; a < kAhead; ++a) f(k + a, GATED ? expf(gc[min((k + a + 1) * p.SC, p.C)]) : 1.f, x[a]);
#pragma unroll
      for (int a = 0; a < kAhead; ++a) x[a] = y[a];
    }
#pragma unroll
    for (int a = 0; a < kAhead; ++a)
      if (k + a < n) f(k + a, GATED ? expf(gc[min((k + a + 1) * p.SC, p.C)]) : 1.f, x[a]);
  };
  if (tid >= kThreads) {   // z of the CTA's four rows
    if (tid >= kThreads + 4) return;
    const int rz = j * 4 + tid - kThreads;
    const float *pz = p.phik + (size_t(u) * p.Cmax + kD) * p.dp + rz;
    float *zp = reinterpret_cast<float *>(p.ws + ld.z) + size_t(ub) * p.dp + rz;
    float z = *zp;
    over_chunks(IntTag<8>{}, [&](int k) { return pz[size_t(k) * step]; }, [&](int k, float dec, float x) {
      if (SNAP) p.zsnap[(size_t(u) * p.nsub + k) * p.dp + rz] = z;
      z = fmaf(z, dec, x);
    });
    *zp = z;
    return;
  }
  const int r = j * 4 + (tid >> 5), col = (tid & 31) * 4;
  const float *part = p.sums_by_row ? p.phik + size_t(u) * p.Cmax * kD + r * kD + col
                                    : p.phik + (size_t(u) * p.Cmax + 2 * (r & 63) + (col >> 6)) * p.dp + (r >> 6) * 64 + (col & 63);
  float4 *Sp = reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.ws + ld.S) + (size_t(ub) * p.dp + r) * kD + col);
  const int half = r / kD;
  bf16 *snap = SNAP ? reinterpret_cast<bf16 *>(p.s16) + ((size_t(half) * p.units_cap + size_t(u) * p.nsub) * kD + (r - half * kD)) * kD + col
                    : nullptr;
  const size_t lo_half = size_t(p.units_cap) * kD * kD;
  float4 s = *Sp;
  over_chunks(IntTag<4>{}, [&](int k) { return *reinterpret_cast<const float4 *>(part + size_t(k) * step); }, [&](int k, float dec, const float4 &x) {
    if (SNAP) {
      bf16 *at = snap + size_t(k) * kD * kD;
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(s.x, s.y), h1 = __floats2bfloat162_rn(s.z, s.w);
      *reinterpret_cast<uint2 *>(at) = make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
      if (GATED) {
        const __nv_bfloat162 l0 = __floats2bfloat162_rn(s.x - __low2float(h0), s.y - __high2float(h0));
        const __nv_bfloat162 l1 = __floats2bfloat162_rn(s.z - __low2float(h1), s.w - __high2float(h1));
        *reinterpret_cast<uint2 *>(at + lo_half) = make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
      }
    }
    s.x = fmaf(s.x, dec, x.x);
    s.y = fmaf(s.y, dec, x.y);
    s.z = fmaf(s.z, dec, x.z);
    s.w = fmaf(s.w, dec, x.w);
  });
  *Sp = s;
}

}  // namespace

bool prefill_state_mma_supported(const glide_ctx *ctx) {
  return ctx->cfg.io_dtype == GLIDE_BF16 && ctx->cfg.head_dim == kD;
}

int launch_prefill_state_mma(const PrefillParams &pass, bool make_phi, cudaStream_t stream) {
  PrefillParams p = pass;
  p.sums_by_row = make_phi && !p.gated;
  const int64_t units = int64_t(p.layer_count) * p.B * p.Hkv;
  auto scan = [&]() -> int {
    if (p.nsub > 1) {
      const unsigned ctas = unsigned(units * (p.dp / 4));
      auto run = [&](auto gated, auto snap) {
        launch_chained(prefill_scan_kernel<decltype(gated)::value, decltype(snap)::value>, ctas, kThreads + 32, 0, stream, p);
      };
      const std::true_type yes{};
      const std::false_type no{};
      if (p.gated) p.s16 ? run(yes, yes) : run(yes, no);
      else p.s16 ? run(no, yes) : run(no, no);
    }
    return cudaGetLastError() == cudaSuccess ? GLIDE_OK : GLIDE_ERR_CUDA;
  };
  if (p.sums_by_row) {
    const int rc = launch_prefill_carry_tc(p, stream);
    return rc ? rc : scan();
  }
  const unsigned blocks = unsigned(units * p.nsub * (p.dp / kRowsPerCta));
  auto run = [&](auto partial, auto make, auto gated) {
    launch_chained(prefill_state_mma_kernel<decltype(partial)::value, decltype(make)::value, decltype(gated)::value>, blocks, kThreads, 0, stream, p);
  };
  const std::true_type yes{};
  const std::false_type no{};
  if (p.gated) {   // (a gated pass of several chunks makes its own phi)
    if (p.nsub > 1) run(yes, yes, yes);
    else if (make_phi) run(no, yes, yes);
    else run(no, no, yes);
  } else {
    if (p.nsub > 1) run(yes, no, no);
    else run(no, no, no);
  }
  return scan();
}

}  // namespace glide

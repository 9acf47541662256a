// Chunk sums of the prefill's carry on the 5th-generation tensor cores (bf16 I/O, head_dim 128, parameter-free map, no gates):
//   S_c = phi(K'_c)^T V'_c,  z_c = sum phi(K'_c)      over a chunk's delayed tokens (k'_i = k_{i-w}).
// V' is bf16 already; every fp32 value of phi(K') is split without error into three bf16 terms (hi + mid + lo = the 24-bit
// significand, each the bf16 rounding of what the previous ones left), so the three products phi_term^T V' are exact in fp32 and
// only the fp32 accumulation in TMEM rounds (a bf16 or tf32 product of phi(K') itself would miss the 1e-5 state tolerance).
//
// One CTA of 9 warps per (unit, chunk of the pass), all 128 rows and columns of S in 128 TMEM columns, two CTAs per SM.  Stages of
// 32 tokens: warps 0-7 make phi (eight threads a token, 16 features each) from the staged K' rows, leave its terms in shared memory
// as the MN-major A operand (a token's row as it is) and its rounding for the attention kernel, and sum z on the way; warp 8 issues
// six m128n128k16 per stage with V' as the MN-major B operand.  K' and V' rows come by cp.async two stages ahead (rings of three and
// four buffers: V' is read until the products of its stage have completed), the terms are double-buffered.
// What bounds it: the chain of a CTA's stages.  8 x 2048 tokens of 4 layers take eight launches of 256 CTAs, 93 us (11.6 a launch), in
// which 268 MB of rows come from HBM and 256 MB of rounded phi and sums go to L2; 8001 tokens of one layer 20 us.  (ncu, one launch of
// 256 CTAs with cold caches: 23.6 us, 31 MB read, 0.7 written, 103 MB of L2 traffic, tensor pipe 12 %.)  The mma.sync form before it,
// two CTAs of 64 rows that both staged K' and made phi, took 185 and 43 us; it remains where phi comes from another kernel (the learned
// map, sum-of-terms merges with outputs, outputs by the mma.sync or CUDA-core kernel) and for gates.  Against fp64 S is as far
// off as with it (chunks of 256 tokens 7.9e-7, both; the tensor core adds without rounding to nearest, so with the chunk's length: 144 tokens
// 4.7e-7, 1024 2.5e-6 to 3.4e-6), z less (5.6e-8, 8.0e-8).
// Every mbarrier wait is bounded; after a time-out the CTA runs its loop out without waiting, stores nothing, records
// kDevWaitTimeout, frees its TMEM columns and returns.
#include <type_traits>

#include "glide_tc.cuh"

namespace glide {

namespace {

constexpr int kD = 128;
constexpr int kTok = 32;                         // tokens per stage
constexpr int kWorkers = 256;                    // threads that make phi
constexpr int kThreads = kWorkers + 32;          // and the MMA warp
constexpr uint32_t kTileB = kTok * kD * 2;       // bytes of a stage's K', V' or phi term: [2 column halves][32 tokens][64 bf16]
constexpr uint32_t kHalfB = kTileB / 2;
constexpr int kKBufs = 3, kVBufs = 4, kPhiBufs = 2;

struct CarrySmem {
  unsigned char phi[kPhiBufs][3][kTileB];        // hi, mid, lo of phi(K'); at the end the threads' sums of z
  unsigned char k[kKBufs][kTileB];
  unsigned char v[kVBufs][kTileB];
  uint64_t bar_full[kPhiBufs];                   // a stage's terms and V' rows are there (one arrival per worker warp)
  uint64_t bar_free[kPhiBufs];                   // its products have completed
  uint32_t tmem_base;
  int failed;
};
static_assert(2 * (sizeof(CarrySmem) + 1024) <= 233472, "two CTAs per SM");
static_assert(sizeof(float) * kTok * kD <= sizeof(CarrySmem::phi), "z of every token slot");

// byte offset of 16-byte chunk c16 (0..15) of row `row` inside a [2][32][64] bf16 tile with 128-byte swizzle
__device__ __forceinline__ uint32_t sw32(int row, int c16) {
  return uint32_t((c16 >> 3) * kHalfB + row * 128 + (((c16 & 7) ^ (row & 7)) << 4));
}
// fp32 accumulate, bf16 A and B, both MN-major, M = N = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

// 16 lanes x 64 columns: registers 4 n .. 4 n + 3 are columns 8 n + 2 (lane % 4) + {0, 1} of row lane / 4 and of row lane / 4 + 8
__device__ __forceinline__ void tmem_ld_16x64(uint32_t taddr, float (&r)[32]) {
  uint32_t x[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]), "=r"(x[9]),
        "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15]), "=r"(x[16]), "=r"(x[17]), "=r"(x[18]),
        "=r"(x[19]), "=r"(x[20]), "=r"(x[21]), "=r"(x[22]), "=r"(x[23]), "=r"(x[24]), "=r"(x[25]), "=r"(x[26]), "=r"(x[27]),
        "=r"(x[28]), "=r"(x[29]), "=r"(x[30]), "=r"(x[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __uint_as_float(x[i]);
}

// PARTIAL (passes of several chunks): the chunk's own sums go to its scratch rows (S row by row, z behind it: chunks of more than 128
// tokens), and prefill_scan_kernel adds them up in chunk order.  Otherwise S and z are updated in place, and their values
// before the chunk are left (bf16, fp32) for the attention kernel, which runs after this one.
template <bool PARTIAL>
__global__ void __launch_bounds__(kThreads, 2) prefill_carry_tc_kernel(const PrefillParams p) {
  using bf16 = __nv_bfloat16;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  CarrySmem &sm = *reinterpret_cast<CarrySmem *>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t uc = blockIdx.x;                                    // (unit, chunk of the pass)
  const int u = PARTIAL ? int(uc / p.nsub) : int(uc);
  const int chunk_c0 = PARTIAL ? int(uc - int64_t(u) * p.nsub) * p.SC : 0;   // first token of the chunk, relative to the pass
  const int chunk_n = min(p.SC, p.C - chunk_c0);
  const int ug = u / p.Hkv, g = u - ug * p.Hkv, lrel = ug / p.B, b = ug - lrel * p.B;
  const LayerDev &ld = p.layers[p.layer_begin + lrel];
  if (!ld.evicts) return;
  const int64_t first64 = p.n0 + p.c0 + chunk_c0 - ld.wlin;         // delayed token of chunk index 0
  if (first64 <= -int64_t(chunk_n)) return;
  const int first = int(first64), n0 = int(p.n0);                   // (positions stay below 2^30)
  const int i_lo = first < 0 ? -first : 0;
  const int ub = (b + p.b0) * p.Hkv + g;
  const uint32_t cap = ld.cap > 0 ? uint32_t(ld.cap) : 1u;
  const int n_stages = (chunk_n - i_lo + kTok - 1) / kTok;
  volatile int *failed = &sm.failed;

  if (warp == kWorkers / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_u32(&sm.tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if (lane == 0) {
      for (int i = 0; i < kPhiBufs; ++i) {
        mbar_init(smem_u32(&sm.bar_full[i]), kWorkers / 32);
        mbar_init(smem_u32(&sm.bar_free[i]), 1);
      }
      sm.failed = (smem_u32(smem_raw) & 1023u) != 0;                // (the swizzled tiles have to start on a multiple of 1024)
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
  }
  // K' and V' rows of stage s (tokens past the chunk's end as zeros): 16 threads per row, two rows per thread
  const bf16 *ringK = reinterpret_cast<const bf16 *>(p.ws + ld.ringK) + size_t(ub) * size_t(ld.cap) * kD;
  const bf16 *ringV = reinterpret_cast<const bf16 *>(p.ws + ld.ringV) + size_t(ub) * size_t(ld.cap) * kD;
  const size_t call0 = ((size_t(lrel) * p.B + b) * size_t(p.T) * p.Hkv + g) * kD;
  const bf16 *callK = reinterpret_cast<const bf16 *>(p.k) + call0, *callV = reinterpret_cast<const bf16 *>(p.v) + call0;
  auto issue = [&](int s) {
    if (s < n_stages) {
      const int c = tid & 15;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int t = (tid >> 4) + 16 * h, i = i_lo + s * kTok + t;
        const bool there = i < chunk_n;
        const int j = first + (there ? i : i_lo);
        const size_t at = (j >= n0 ? size_t(j - n0) * p.Hkv : size_t(uint32_t(j) % cap)) * kD + c * 8;
        cp_async16(smem_u32(sm.k[s % kKBufs]) + sw32(t, c), (j >= n0 ? callK : ringK) + at, there);
        cp_async16(smem_u32(sm.v[s % kVBufs]) + sw32(t, c), (j >= n0 ? callV : ringV) + at, there);
      }
    }
    cp_async_commit();
  };
  if (warp < kWorkers / 32) {
    issue(0);
    issue(1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  bool ok = !*failed;                                               // (the same for all here)

  if (warp == kWorkers / 32) {
    const bool leader = elect_one();
    for (int s = 0; s < n_stages && ok; ++s) {
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.bar_full[s & 1]), uint32_t(s >> 1) & 1u, failed));
      if (!ok) break;
      if (leader) {
        const uint32_t b0 = desc_lo(smem_u32(sm.v[s % kVBufs]), kHalfB);
#pragma unroll
        for (int ks = 0; ks < kTok / 16; ++ks)
#pragma unroll
          for (int term = 2; term >= 0; --term) {                   // smallest terms first
            const uint32_t a0 = desc_lo(smem_u32(sm.phi[s & 1][term]), kHalfB);
            asm volatile(
                "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}" ::"r"(tmem),
                "r"(a0 + uint32_t(ks * 2048 >> 4)), "r"(b0 + uint32_t(ks * 2048 >> 4)), "r"(kIdesc),
                "r"((s > 0 || ks > 0 || term < 2) ? 1u : 0u), "r"(kDescHi)
                : "memory");
          }
        mma_commit(smem_u32(&sm.bar_free[s & 1]));
      }
      __syncwarp();
    }
  } else {
    float zacc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) zacc[i] = 0.f;
    const int tok = tid >> 3, part = tid & 7;
    // the thread's two 16-byte chunks of a row, in the order that keeps a quarter warp on different banks
    const int c0 = part * 2 + (part >> 2), c1 = part * 2 + 1 - (part >> 2);
    bf16 *p16 = p.phik16 ? reinterpret_cast<bf16 *>(p.phik16) + (size_t(u) * p.Cmax + chunk_c0) * kD : nullptr;
    for (int s = 0; s < n_stages; ++s) {
      // the products of stage s - 2 have completed: its terms' and its V' rows' buffers are free
      if (s >= kPhiBufs && ok) ok = mbar_wait(smem_u32(&sm.bar_free[s & 1]), uint32_t((s >> 1) - 1) & 1u, failed);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      // everybody's rows of the stage have landed, and everybody has read the K' rows of the stage before
      asm volatile("barrier.cta.sync 1, %0;" ::"n"(kWorkers) : "memory");
      issue(s + 2);
      const unsigned char *kt = sm.k[s % kKBufs];
      const uint4 q0 = *reinterpret_cast<const uint4 *>(kt + sw32(tok, c0)), q1 = *reinterpret_cast<const uint4 *>(kt + sw32(tok, c1));
      const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
      float x[16];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[2 * i] = __uint_as_float(w[i] << 16), x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
      float mx = x[0];
#pragma unroll
      for (int i = 1; i < 16; ++i) mx = fmaxf(mx, x[i]);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        x[i] = exp2f((x[i] - mx) * kLog2e);
        sum += x[i];
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const int i = i_lo + s * kTok + tok;
      const bool there = i < chunk_n;
      const float inv = there ? 1.0f / sum : 0.f;                   // (rows past the chunk's end stay zero)
      uint32_t term[3][8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float a0 = x[2 * e] * inv, a1 = x[2 * e + 1] * inv;
        zacc[2 * e] += a0, zacc[2 * e + 1] += a1;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          term[t][e] = pack_bf16x2(a0, a1);
          a0 -= __uint_as_float(term[t][e] << 16), a1 -= __uint_as_float(term[t][e] & 0xffff0000u);
        }
      }
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        *reinterpret_cast<uint4 *>(sm.phi[s & 1][t] + sw32(tok, c0)) = make_uint4(term[t][0], term[t][1], term[t][2], term[t][3]);
        *reinterpret_cast<uint4 *>(sm.phi[s & 1][t] + sw32(tok, c1)) = make_uint4(term[t][4], term[t][5], term[t][6], term[t][7]);
      }
      fence_async_smem();   // the terms, and this thread's rows of V' (its copies have completed), are read by the tensor core
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.bar_full[s & 1]));
      if (p16 && there) {
        *reinterpret_cast<uint4 *>(p16 + size_t(i) * kD + c0 * 8) = make_uint4(term[0][0], term[0][1], term[0][2], term[0][3]);
        *reinterpret_cast<uint4 *>(p16 + size_t(i) * kD + c1 * 8) = make_uint4(term[0][4], term[0][5], term[0][6], term[0][7]);
      }
    }
    cp_async_wait_all();
    // every product has completed (the last stage's commit covers those before it)
    if (ok) ok = mbar_wait(smem_u32(&sm.bar_free[(n_stages - 1) & 1]), uint32_t((n_stages - 1) >> 1) & 1u, failed);
    tc_fence_after();
    float *zt = reinterpret_cast<float *>(sm.phi);                  // [32 token slots][128]
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 8; e += 4)
        *reinterpret_cast<float4 *>(zt + tok * kD + (h ? c1 : c0) * 8 + e) =
            make_float4(zacc[h * 8 + e], zacc[h * 8 + e + 1], zacc[h * 8 + e + 2], zacc[h * 8 + e + 3]);
  }
  ok = !__syncthreads_or(!ok);
  if (ok && warp < kWorkers / 32) {
    const int q = warp & 3, cols = (warp >> 2) * 64;
    float *sums = p.phik + (size_t(u) * p.Cmax + chunk_c0) * kD;
    float *Sb = reinterpret_cast<float *>(p.ws + ld.S) + size_t(ub) * kD * kD;
    bf16 *s16 = p.s16 ? reinterpret_cast<bf16 *>(p.s16) + size_t(u) * kD * kD : nullptr;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      float r[32];
      tmem_ld_16x64(tmem + (uint32_t(q * 32 + h * 16) << 16) + uint32_t(cols), r);
#pragma unroll
      for (int n = 0; n < 8; ++n)
#pragma unroll
        for (int lo = 0; lo < 2; ++lo) {
          const size_t at = size_t(q * 32 + h * 16 + (lane >> 2) + lo * 8) * kD + cols + n * 8 + 2 * (lane & 3);
          const float2 a = make_float2(r[4 * n + 2 * lo], r[4 * n + 2 * lo + 1]);
          if (PARTIAL) {
            *reinterpret_cast<float2 *>(sums + at) = a;
          } else {
            float2 c = *reinterpret_cast<const float2 *>(Sb + at);
            if (s16) *reinterpret_cast<uint32_t *>(s16 + at) = pack_bf16x2(c.x, c.y);
            c.x += a.x, c.y += a.y;
            *reinterpret_cast<float2 *>(Sb + at) = c;
          }
        }
    }
    if (tid < kD) {
      const float *zt = reinterpret_cast<const float *>(sm.phi);
      float z = 0.f;
#pragma unroll 8
      for (int t = 0; t < kTok; ++t) z += zt[t * kD + tid];
      if (PARTIAL) {
        sums[kD * kD + tid] = z;
      } else {
        float *zb = reinterpret_cast<float *>(p.ws + ld.z) + size_t(ub) * kD + tid;
        const float z0 = *zb;
        if (s16) p.zsnap[size_t(u) * kD + tid] = z0;
        *zb = z0 + z;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && !ok) atomicExch(&p.ctl->status, kDevWaitTimeout);
  if (warp == kWorkers / 32) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem) : "memory");
  }
}

}  // namespace

int launch_prefill_carry_tc(const PrefillParams &p, cudaStream_t stream) {
  const int64_t units = int64_t(p.layer_count) * p.B * p.Hkv;
  auto run = [&](auto kern) -> int {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(CarrySmem))) != cudaSuccess) {
      cudaGetLastError();
      return GLIDE_ERR_CUDA;
    }
    kern<<<unsigned(units * p.nsub), kThreads, sizeof(CarrySmem), stream>>>(p);
    return cudaGetLastError() == cudaSuccess ? GLIDE_OK : GLIDE_ERR_CUDA;
  };
  return p.nsub > 1 ? run(prefill_carry_tc_kernel<true>) : run(prefill_carry_tc_kernel<false>);
}

}  // namespace glide

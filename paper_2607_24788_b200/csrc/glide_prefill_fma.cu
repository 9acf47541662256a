// GLIDE prefill on the CUDA cores with fp32 arithmetic throughout (fp32 I/O, d = 64, and whenever the CUDA-core prefill is
// asked for) for the parameter-free feature map, gated or not.  A pass takes up to nsub chunks of CH tokens of every unit
// (unit = layer, sequence, KV head) in three launches, or four where it has many chunks:
//   1.  prefill_fma_sums_kernel    per chunk phi(K')^T V' and sum phi(K') of its delayed tokens k'_i = k_{i-w}
//   1b. prefill_fma_scan_kernel    (many chunks) the sums added up: S and z move on, the state at every chunk's start is left
//   2.  prefill_fma_attn_kernel    per 16 query rows: window softmax, the chunk's own delayed tokens, and the state at
//                                  the chunk's start, the scan's or S + the sums of the chunks before it; out
//   3.  prefill_fma_finish_kernel  S and z move on by the pass if no scan did it, the pass's newest tokens go to the ring,
//                                  counters advance
// A pass of one chunk needs no room for sums: 1 comes after 2 and adds to S and z in place.
// Gated: the running log-gates of the chunks' delayed tokens (gcum) come from a kernel in front; without gates every decay
// is an exact 1, so that a gated context driven without gates keeps the bits of a plain one.
// The kernels read K and V rows where they are (ring for tokens older than the call) and make phi in registers; the ring
// changes in the last only.  The problems are small (a few units of a few hundred tokens), so what bounds them is the
// length of the dependent chain and not the arithmetic: the rows of a tile are shared by 16 query rows and the next
// tile's loads are in flight while one is used, and a CTA's two groups of four warps work side by side on the window and
// the linear part (the sums kernel: on every other tile).  512 tokens of 4 units (fp32, d = 64, w = 64): attention 103 us
// per 256 tokens with a warp per query and one key row at a time, 20 us for all 512 now.
#include <algorithm>
#include <type_traits>

#include "glide_prefill_rows.cuh"

namespace glide {

namespace {

constexpr int kThreads = 128;     // of a group; the sums and the attention kernel run two groups per CTA
constexpr int kRows = 16;         // query rows (token, head of the group) per CTA: 8 half-warps of two rows
// Passes of more chunks than this are scanned.  Without a scan every CTA of 16 query rows reads S and the sums of all chunks
// before its own, which grows with the square of the chunks; the scan is a launch more (4 us).  Per layer of a 32-layer
// context with windows of 64, fp32, without / with a scan: 8 heads of 64, 8 chunks 42 / 45 us, 16 78 / 76, 64 383 / 223,
// 128 1153 / 433; 32 heads of 128 (8 KV heads), 4 chunks 107 / 107 us, 8 202 / 187, 125 7462 / 3288.
template <int D>
constexpr int kDirectChunks = 512 / D;

__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
  float x[4];
  load_elems<__nv_bfloat16, 4>(p, x);
  return make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void store4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16 *p, float4 v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}
// the barrier of one group of kThreads threads
__device__ __forceinline__ void group_sync(int grp) { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); }
// reductions over N consecutive lanes (N = 16 or 32), the result in all of them
template <int N>
__device__ __forceinline__ float lanes_max(float x) {
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
template <int N>
__device__ __forceinline__ float lanes_sum(float x) {
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// phi of a row whose D entries lie in D / 4 consecutive lanes, four in each
template <int D>
__device__ __forceinline__ float4 row_phi(float4 x) {
  const float mx = lanes_max<D / 4>(fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
  float4 e = make_float4(exp2f((x.x - mx) * kLog2e), exp2f((x.y - mx) * kLog2e), exp2f((x.z - mx) * kLog2e), exp2f((x.w - mx) * kLog2e));
  const float inv = 1.0f / lanes_sum<D / 4>(e.x + e.y + e.z + e.w);
  return make_float4(e.x * inv, e.y * inv, e.z * inv, e.w * inv);
}

struct UnitId {
  int64_t u;
  int g, b, lrel;
};
__device__ __forceinline__ UnitId unit_id(const PrefillParams &p, int64_t u) {
  return UnitId{u, int(u % p.Hkv), int((u / p.Hkv) % p.B), int(u / (int64_t(p.Hkv) * p.B))};
}
// delayed tokens exist from chunk index i_lo on (chunk_n: none); first: the delayed token of chunk index 0
__device__ __forceinline__ int first_delayed(int64_t first, int chunk_n) {
  return first >= 0 ? 0 : (first <= -int64_t(chunk_n) ? chunk_n : int(-first));
}

// gated: running log-gates of chunk uc of the pass (chunk index 0 on); null without gates
__device__ __forceinline__ const float *chunk_gates(const PrefillParams &p, int64_t uc) {
  return p.gated ? p.gcum + size_t(uc) * p.SC : nullptr;
}
// what a state has decayed by over chunk k of unit u
__device__ __forceinline__ float chunk_decay(const PrefillParams &p, int64_t u, int k) {
  return p.gated ? expf(chunk_gates(p, u * p.nsub + k)[min(p.SC, p.C - k * p.SC) - 1]) : 1.f;
}

// 1. One CTA per (unit, chunk, 16 rows of S): every half-warp owns two rows, a lane D / 16 columns of them.  The rows of phi
// are made from K' as they are loaded (all of them in every CTA of a unit: cheaper than a launch in front and a trip
// through memory), the CTA keeps its 16 columns of them.
constexpr int kSumTok = 32;    // tokens per tile
// IN_PLACE (passes of one chunk): behind the attention kernel, on top of S and z, so that such passes need no scratch.
template <typename T, int D, bool IN_PLACE>
__global__ void __launch_bounds__(2 * kThreads) prefill_fma_sums_kernel(const PrefillParams p) {
  constexpr int LD = kSumTok * D / 4 / kThreads;   // float4 per thread and tile
  constexpr int CG = D / 64;                       // groups of four columns per thread
  static_assert(2 * kThreads * (4 * CG + 1) <= kSumTok * D, "the second group's sums fit its tile");
  __shared__ __align__(16) float ph[2][kSumTok][16];   // [group]
  __shared__ __align__(16) float vt[2][kSumTok][D];
  wait_for_predecessor();
  const int grp = threadIdx.x / kThreads, tid = threadIdx.x % kThreads;
  const int rb = int(blockIdx.x % (D / 16));
  const int64_t uc = blockIdx.x / (D / 16);
  const UnitId id = unit_id(p, uc / p.nsub);
  const int chunk_c0 = int(uc - id.u * p.nsub) * p.SC, chunk_n = min(p.SC, p.C - chunk_c0);
  const LayerDev ld = p.layers[p.layer_begin + id.lrel];
  if (!ld.evicts) return;
  const int64_t first = p.n0 + p.c0 + chunk_c0 - ld.wlin;
  const int i_lo = first_delayed(first, chunk_n);
  if (i_lo >= chunk_n) return;                     // (the readers of the sums leave such chunks out as well)
  const Rows<T, D> rows(p, ld, id.lrel, id.b, id.g);
  const float *gc = chunk_gates(p, uc);
  const float g_end = gc ? gc[chunk_n - 1] : 0.f;
  float4 kr[LD], vr[LD];
  auto fetch = [&](int i0) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      kr[i] = vr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i0 + r < chunk_n) {
        const int64_t off = rows.at(first + i0 + r);
        kr[i] = load4(rows.k(off) + c);
        vr[i] = load4(rows.v(off) + c);
      }
    }
  };
  const int row = (tid >> 4) * 2, cg = tid & 15;
  float acc[2][4 * CG], zacc = 0.f;
#pragma unroll
  for (int c = 0; c < 4 * CG; ++c) acc[0][c] = acc[1][c] = 0.f;
  fetch(i_lo + grp * kSumTok);
  for (int i0 = i_lo + grp * kSumTok; i0 < chunk_n; i0 += 2 * kSumTok) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      float4 f = row_phi<D>(kr[i]);
      if (i0 + r >= chunk_n) f = make_float4(0.f, 0.f, 0.f, 0.f);
      else if (gc) {   // what the token has decayed to by the end of the chunk
        const float dec = expf(g_end - gc[i0 + r]);
        f = make_float4(f.x * dec, f.y * dec, f.z * dec, f.w * dec);
      }
      if (c >> 4 == rb) *reinterpret_cast<float4 *>(&ph[grp][r][c & 15]) = f;
      *reinterpret_cast<float4 *>(&vt[grp][r][c]) = vr[i];
    }
    group_sync(grp);
    if (i0 + 2 * kSumTok < chunk_n) fetch(i0 + 2 * kSumTok);
#pragma unroll 8
    for (int i = 0; i < kSumTok; ++i) {
      const float2 f = *reinterpret_cast<const float2 *>(&ph[grp][i][row]);
#pragma unroll
      for (int q = 0; q < CG; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(&vt[grp][i][q * 64 + cg * 4]);
        acc[0][q * 4 + 0] = fmaf(f.x, v.x, acc[0][q * 4 + 0]);
        acc[0][q * 4 + 1] = fmaf(f.x, v.y, acc[0][q * 4 + 1]);
        acc[0][q * 4 + 2] = fmaf(f.x, v.z, acc[0][q * 4 + 2]);
        acc[0][q * 4 + 3] = fmaf(f.x, v.w, acc[0][q * 4 + 3]);
        acc[1][q * 4 + 0] = fmaf(f.y, v.x, acc[1][q * 4 + 0]);
        acc[1][q * 4 + 1] = fmaf(f.y, v.y, acc[1][q * 4 + 1]);
        acc[1][q * 4 + 2] = fmaf(f.y, v.z, acc[1][q * 4 + 2]);
        acc[1][q * 4 + 3] = fmaf(f.y, v.w, acc[1][q * 4 + 3]);
      }
    }
    if (tid < 16) {
#pragma unroll 8
      for (int i = 0; i < kSumTok; ++i) zacc += ph[grp][i][tid];
    }
    group_sync(grp);
  }
  dependents_may_start();   // (8192 tokens of one fp32 layer, state only, d = 64 / 128 x 2 layers: 141 / 448 us; at every kernel's top 191 / 562, not at all 167 / 496)
  // the second group's sums on top of the first's, through the second group's tile
  float (*other)[4 * CG + 1] = reinterpret_cast<float (*)[4 * CG + 1]>(&vt[1][0][0]);   // [2 * kThreads]
  if (grp == 1) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4 * CG; ++c) other[r * kThreads + tid][c] = acc[r][c];
    if (tid < 16) ph[1][0][tid] = zacc;
  }
  __syncthreads();
  if (grp == 1) return;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < 4 * CG; ++c) acc[r][c] += other[r * kThreads + tid][c];
  if (tid < 16) zacc += ph[1][0][tid];
  const size_t ub = size_t(id.b + p.b0) * p.Hkv + id.g;
  float *dst = (IN_PLACE ? reinterpret_cast<float *>(p.ws + ld.S) + ub * D * D : p.phik + size_t(uc) * D * D) + (rb * 16 + row) * D + cg * 4;
  const float dec = IN_PLACE ? chunk_decay(p, id.u, 0) : 1.f;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < CG; ++q) {
      float4 x = make_float4(acc[r][q * 4], acc[r][q * 4 + 1], acc[r][q * 4 + 2], acc[r][q * 4 + 3]);
      if (IN_PLACE) {
        const float4 s = load4(dst + r * D + q * 64);
        x = make_float4(fmaf(s.x, dec, x.x), fmaf(s.y, dec, x.y), fmaf(s.z, dec, x.z), fmaf(s.w, dec, x.w));
      }
      store4(dst + r * D + q * 64, x);
    }
  if (tid < 16) {
    float *z = (IN_PLACE ? reinterpret_cast<float *>(p.ws + ld.z) + ub * D : p.zsnap + size_t(uc) * D) + rb * 16 + tid;
    *z = IN_PLACE ? fmaf(*z, dec, zacc) : zacc;
  }
}

// 2. Tiles of KT rows: group 0 takes the window's keys, group 1 the chunk's delayed tokens and the rows of the state; group
// 0 merges and stores.  Per tile a half-warp
// computes the weights of its two rows (a lane KT / 16 keys), keeps them in shared memory for itself, and adds the weighted
// V (or S) rows (a lane D / 16 columns).
template <int D>
struct AttnSmem {
  static constexpr int KT = 4096 / D;             // 64 rows for d = 64, 32 for d = 128: 16 float4 per thread and tile
  struct Group {
    float a[kRows][D + 4];                        // q in the log2 domain, or phi(q)
    float k[KT][D + 4];                           // (+ 4: rows start four banks apart)
    float v[KT][D];
    float p[kRows][KT + 4];
  } grp[2];
};

// The state at a chunk's start for a single row: S and z with the sums of chunks [sub0, sub) on top
template <int D>
struct SumsState {
  const float *S, *z0, *sums, *zs, *gates;   // gates: gcum of the unit's first chunk, or null
  int sub0, sub, SC;
  __device__ __forceinline__ float after(int k) const { return gates ? expf(gates[(k + 1) * SC - 1]) : 1.f; }   // (these chunks are whole)
  template <int E>
  __device__ __forceinline__ void row(int r, int c, float (&x)[E]) const {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      x[e] = S[r * D + c + e];
      for (int k = sub0; k < sub; ++k) x[e] = fmaf(x[e], after(k), sums[(size_t(k) * D + r) * D + c + e]);
    }
  }
  __device__ __forceinline__ float z(int r) const {
    float x = z0[r];
    for (int k = sub0; k < sub; ++k) x = fmaf(x, after(k), zs[size_t(k) * D + r]);
    return x;
  }
};

// (One CTA per SM is what fits with 170 registers a thread as with 250, which the second bound allows: 512 tokens of 4 units,
// fp32, d = 64, w = 64, 20.5 us without it, 18.2 with it.)
template <typename T, int D, int G>
__global__ void __launch_bounds__(2 * kThreads, 1) prefill_fma_attn_kernel(const PrefillParams p) {
  constexpr int KT = AttnSmem<D>::KT;
  constexpr int LD = KT * D / 4 / kThreads;        // float4 of K (and of V) per thread and tile
  constexpr int KPT = KT / 16;                     // keys per lane
  constexpr int CG = D / 64;
  constexpr int TOK = kRows / G;                   // tokens per CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  wait_for_predecessor();
  const int grp = threadIdx.x / kThreads, tid = threadIdx.x % kThreads;
  auto &all = *reinterpret_cast<AttnSmem<D> *>(smem_raw);
  typename AttnSmem<D>::Group &sm = all.grp[grp];
  const int per_chunk = (p.SC + TOK - 1) / TOK;
  const int per_unit = (p.nsub - 1) * per_chunk + (p.C - (p.nsub - 1) * p.SC + TOK - 1) / TOK;
  const UnitId id = unit_id(p, blockIdx.x / per_unit);
  const int cta = per_unit - 1 - int(blockIdx.x % per_unit);   // the longest windows of a new prompt first
  const int sub = cta / per_chunk, tok0 = (cta - sub * per_chunk) * TOK;
  const int chunk_c0 = sub * p.SC, chunk_n = min(p.SC, p.C - chunk_c0);
  const int ntok = min(TOK, chunk_n - tok0);
  const size_t seq_row = (size_t(id.lrel) * p.B + id.b) * size_t(p.T) + size_t(p.c0 + chunk_c0 + tok0);
  // the 16 query rows (D / 4 lanes of one row, as in the tiles), asked for before anything else
  constexpr int LQ = kRows * D / 4 / kThreads;
  float4 qr[LQ];
#pragma unroll
  for (int i = 0; i < LQ; ++i) {
    const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
    qr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r / G < ntok)
      qr[i] = load4(reinterpret_cast<const T *>(p.q) + ((seq_row + r / G) * p.H + p.heads_of[id.g * G + r % G]) * D + c);
  }
  const LayerDev ld = p.layers[p.layer_begin + id.lrel];
  const Rows<T, D> rows(p, ld, id.lrel, id.b, id.g);
  const int64_t tq0 = p.n0 + p.c0 + chunk_c0 + tok0, tq_last = tq0 + ntok - 1;

  // the group's tiles: n_st of state rows (they decay with the row, so they come first), then n_rows of key rows from token
  // j_lo on, up to token j_hi
  const bool linear = ld.evicts && tq_last >= ld.wlin;
  const int64_t first = p.n0 + p.c0 + chunk_c0 - ld.wlin;      // delayed token of chunk index 0
  const int64_t w_lo = tq0 - ld.w + 1;
  const int64_t j_lo = grp == 0 ? (w_lo < 0 ? 0 : w_lo) : (first < 0 ? 0 : first);
  const int64_t j_hi = grp == 0 ? tq_last : first + tok0 + ntok - 1;
  const bool any = grp == 0 ? ld.w > 0 : linear;
  const int n_rows = any && j_hi >= j_lo ? int((j_hi - j_lo) / KT) + 1 : 0;
  const int n_st = grp == 1 && linear && first > 0 ? D / KT : 0;
  const int n_tiles = n_rows + n_st;
  // The state at the chunk's start: left by the scan in the chunk's slot, or S and z with the sums of the chunks before this
  // one that hold delayed tokens, [sub0, sub), on top
  const bool scanned = p.nsub > kDirectChunks<D>;
  const int sub0 = scanned ? sub : (first - int64_t(chunk_c0) >= 0 ? 0 : int(-(first - chunk_c0) / p.SC));
  const float *sums = p.phik + size_t(id.u) * p.nsub * D * D, *zs = p.zsnap + size_t(id.u) * p.nsub * D;
  const int ub = (id.b + p.b0) * p.Hkv + id.g;
  const float *Sb = scanned ? sums + size_t(sub) * D * D : reinterpret_cast<const float *>(p.ws + ld.S) + size_t(ub) * D * D;
  const float *zb = scanned ? zs + size_t(sub) * D : reinterpret_cast<const float *>(p.ws + ld.z) + size_t(ub) * D;

  float4 kr[LD], vr[LD];
  auto fetch = [&](int t) {
    if (t >= n_st) {
#pragma unroll
      for (int i = 0; i < LD; ++i) {
        const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
        kr[i] = vr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int64_t j = j_lo + int64_t(t - n_st) * KT + r;
        if (j <= j_hi) {
          const int64_t off = rows.at(j);
          kr[i] = load4(rows.k(off) + c);
          vr[i] = load4(rows.v(off) + c);
        }
      }
    } else {
      const size_t at0 = size_t(t) * KT * D + tid * 4;   // (a tile's rows are contiguous)
#pragma unroll
      for (int i = 0; i < LD; ++i) vr[i] = *reinterpret_cast<const float4 *>(Sb + at0 + i * kThreads * 4);
      for (int k = sub0; k < sub; ++k) {
        const float dec = chunk_decay(p, id.u, k);
#pragma unroll
        for (int i = 0; i < LD; ++i) kr[i] = *reinterpret_cast<const float4 *>(sums + size_t(k) * D * D + at0 + i * kThreads * 4);
#pragma unroll
        for (int i = 0; i < LD; ++i)
          vr[i] = make_float4(fmaf(vr[i].x, dec, kr[i].x), fmaf(vr[i].y, dec, kr[i].y), fmaf(vr[i].z, dec, kr[i].z), fmaf(vr[i].w, dec, kr[i].w));
      }
    }
  };
  if (n_tiles > 0) fetch(0);
#pragma unroll
  for (int i = 0; i < LQ; ++i) {
    const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
    const float4 x = qr[i];
    *reinterpret_cast<float4 *>(&sm.a[r][c]) =
        grp ? row_phi<D>(x) : make_float4(x.x * p.scale_log2, x.y * p.scale_log2, x.z * p.scale_log2, x.w * p.scale_log2);
  }

  // o: window accumulator or linear one; l: the lane's part of the row's weight sum
  const int row = (tid >> 4) * 2, cg = tid & 15;
  float o[2][4 * CG], m[2], l[2];
  const float *gc = grp == 1 && linear ? chunk_gates(p, id.u * p.nsub + sub) : nullptr;
  float g_own[2];
  int64_t last[2];                                 // last token that counts for the row: its own, or its own delayed one
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    m[r] = -CUDART_INF_F;
    l[r] = 0.f;
    last[r] = (grp == 0 ? tq0 : first + tok0) + (row + r) / G;
    g_own[r] = gc ? gc[min(tok0 + (row + r) / G, chunk_n - 1)] : 0.f;
#pragma unroll
    for (int c = 0; c < 4 * CG; ++c) o[r][c] = 0.f;
  }
  // o[r] += the weights w0, w1 of rows row, row + 1 times the tile's V rows
  auto add_rows = [&](const float *w0, const float *w1) {
#pragma unroll 4
    for (int i = 0; i < KT; i += 4) {
      const float4 p0 = *reinterpret_cast<const float4 *>(w0 + i), p1 = *reinterpret_cast<const float4 *>(w1 + i);
      const float f0[4] = {p0.x, p0.y, p0.z, p0.w}, f1[4] = {p1.x, p1.y, p1.z, p1.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int q = 0; q < CG; ++q) {
          const float4 v = *reinterpret_cast<const float4 *>(&sm.v[i + e][q * 64 + cg * 4]);
          o[0][q * 4 + 0] = fmaf(f0[e], v.x, o[0][q * 4 + 0]);
          o[0][q * 4 + 1] = fmaf(f0[e], v.y, o[0][q * 4 + 1]);
          o[0][q * 4 + 2] = fmaf(f0[e], v.z, o[0][q * 4 + 2]);
          o[0][q * 4 + 3] = fmaf(f0[e], v.w, o[0][q * 4 + 3]);
          o[1][q * 4 + 0] = fmaf(f1[e], v.x, o[1][q * 4 + 0]);
          o[1][q * 4 + 1] = fmaf(f1[e], v.y, o[1][q * 4 + 1]);
          o[1][q * 4 + 2] = fmaf(f1[e], v.z, o[1][q * 4 + 2]);
          o[1][q * 4 + 3] = fmaf(f1[e], v.w, o[1][q * 4 + 3]);
        }
    }
  };

  for (int t = 0; t < n_tiles; ++t) {
    const bool keyed = t >= n_st;
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      if (keyed) *reinterpret_cast<float4 *>(&sm.k[r][c]) = grp ? row_phi<D>(kr[i]) : kr[i];   // (uniform over the group)
      *reinterpret_cast<float4 *>(&sm.v[r][c]) = vr[i];
    }
    group_sync(grp);
    if (t + 1 < n_tiles) fetch(t + 1);
    if (keyed) {
      // s[r][x] = a[row + r] . k[cg + 16 x]
      float s[2][KPT];
#pragma unroll
      for (int x = 0; x < KPT; ++x) s[0][x] = s[1][x] = 0.f;
#pragma unroll 4
      for (int c = 0; c < D; c += 4) {
        const float4 a0 = *reinterpret_cast<const float4 *>(&sm.a[row][c]), a1 = *reinterpret_cast<const float4 *>(&sm.a[row + 1][c]);
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const float4 b = *reinterpret_cast<const float4 *>(&sm.k[cg + 16 * x][c]);
          s[0][x] = fmaf(a0.w, b.w, fmaf(a0.z, b.z, fmaf(a0.y, b.y, fmaf(a0.x, b.x, s[0][x]))));
          s[1][x] = fmaf(a1.w, b.w, fmaf(a1.z, b.z, fmaf(a1.y, b.y, fmaf(a1.x, b.x, s[1][x]))));
        }
      }
      const int64_t j0 = j_lo + int64_t(t - n_st) * KT + cg;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (grp == 0) {
          float mx = -CUDART_INF_F;
#pragma unroll
          for (int x = 0; x < KPT; ++x) {
            const int64_t j = j0 + 16 * x;
            if (j > last[r] || j <= last[r] - ld.w) s[r][x] = -CUDART_INF_F;
            mx = fmaxf(mx, s[r][x]);
          }
          const float mn = fmaxf(m[r], lanes_max<16>(mx));
          const float f = m[r] == -CUDART_INF_F ? 0.f : exp2f(m[r] - mn);
          m[r] = mn;
          l[r] *= f;
#pragma unroll
          for (int c = 0; c < 4 * CG; ++c) o[r][c] *= f;
        }
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const int64_t j = j0 + 16 * x;
          float e = grp == 0 ? (s[r][x] == -CUDART_INF_F ? 0.f : exp2f(s[r][x] - m[r])) : (j <= last[r] ? s[r][x] : 0.f);
          if (gc && j <= last[r]) e *= expf(g_own[r] - gc[j - first]);   // what delayed token j has decayed to
          l[r] += e;
          sm.p[row + r][cg + 16 * x] = e;
        }
      }
      __syncwarp();
      add_rows(sm.p[row], sm.p[row + 1]);
    } else {
      add_rows(&sm.a[row][t * KT], &sm.a[row + 1][t * KT]);
      if (t + 1 == n_st) {   // the state's part is complete: phi(q) . z, and what both have decayed to by the row's token
        float z[D / 16];
#pragma unroll
        for (int i = 0; i < D / 16; ++i) z[i] = zb[cg + 16 * i];
        for (int k = sub0; k < sub; ++k) {
          const float dec = chunk_decay(p, id.u, k);
#pragma unroll
          for (int i = 0; i < D / 16; ++i) z[i] = fmaf(z[i], dec, zs[size_t(k) * D + cg + 16 * i]);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
          for (int i = 0; i < D / 16; ++i) l[r] = fmaf(sm.a[row + r][cg + 16 * i], z[i], l[r]);
          const float dec = gc ? expf(g_own[r]) : 1.f;
          l[r] *= dec;
#pragma unroll
          for (int c = 0; c < 4 * CG; ++c) o[r][c] *= dec;
        }
      }
    }
    group_sync(grp);
  }
  dependents_may_start();   // (512 tokens of 4 units, d = 64: 30 us with all; at the top 35, not at all 39)
#pragma unroll
  for (int r = 0; r < 2; ++r) l[r] = lanes_sum<16>(l[r]);
  // group 1 hands its part over in its V tile (16 x d floats) and the row sums in its weights
  float *lin = &all.grp[1].v[0][0], *lsum = &all.grp[1].p[0][0];
  if (grp == 1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
      for (int q = 0; q < CG; ++q)
        *reinterpret_cast<float4 *>(lin + (row + r) * D + q * 64 + cg * 4) = make_float4(o[r][q * 4], o[r][q * 4 + 1], o[r][q * 4 + 2], o[r][q * 4 + 3]);
      if (cg == 0) lsum[row + r] = l[r];
    }
  }
  __syncthreads();
  if (grp == 1) return;
  unsigned again[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const float L = l[r], Bl = lsum[row + r];
    const int tk = (row + r) / G, head = p.heads_of[id.g * G + (row + r) % G];
    // shared normaliser (reference max(window maximum, 0): the floor belongs to the linear terms, logit 0), or the sum of
    // the two separately normalised terms (an empty term counts as zero)
    float fa, fb;
    if (ld.merge != GLIDE_MERGE_SHARED) {
      fa = L > 0.f ? 1.0f / L : 0.f;
      fb = Bl > 0.f ? 1.0f / Bl : 0.f;
    } else {
      const float M = Bl > 0.f ? fmaxf(m[r], 0.f) : m[r];
      const float fw = m[r] == -CUDART_INF_F ? 0.f : exp2f(m[r] - M), fl = Bl > 0.f ? exp2f(-M) : 0.f;
      const float inv = 1.0f / fmaf(L, fw, fl * Bl);
      fa = fw * inv;
      fb = fl * inv;
    }
    bool bad = false;
    if (tk < ntok) {
      T *op = reinterpret_cast<T *>(p.out) + ((seq_row + tk) * p.H + head) * D + cg * 4;
#pragma unroll
      for (int q = 0; q < CG; ++q) {
        const float4 x = *reinterpret_cast<const float4 *>(lin + (row + r) * D + q * 64 + cg * 4);
        const float4 y = make_float4(fmaf(o[r][q * 4], fa, x.x * fb), fmaf(o[r][q * 4 + 1], fa, x.y * fb),
                                     fmaf(o[r][q * 4 + 2], fa, x.z * fb), fmaf(o[r][q * 4 + 3], fa, x.w * fb));
        store4(op + q * 64, y);
        bad = bad || !isfinite(y.x + y.y + y.z + y.w);
      }
    }
    again[r] = __ballot_sync(0xffffffffu, bad);
  }
  // rows with a result that is not finite (or a sum of four that is not): from the rows that count for them alone
  if (again[0] | again[1]) {
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {   // the warp's rows: lanes 0-15 have rows 0 and 1 of them, lanes 16-31 rows 2 and 3
      if (!((again[i & 1] >> (i >> 1) * 16) & 0xffffu)) continue;
      const int rw = (tid >> 5) * 4 + i, tk = rw / G, head = p.heads_of[id.g * G + rw % G];
      const size_t at = ((seq_row + tk) * p.H + head) * D;
      const RowJob<T, D> job{rows, reinterpret_cast<const T *>(p.q) + at, reinterpret_cast<T *>(p.out) + at,
                             chunk_gates(p, id.u * p.nsub + sub), p.n0 + p.c0 + chunk_c0, tok0 + tk, ld.w, ld.wlin, ld.evicts, ld.merge,
                             p.scale_log2};
      recompute_row(job, SumsState<D>{Sb, zb, sums, zs, chunk_gates(p, id.u * p.nsub), sub0, sub, p.SC});
    }
  }
}

// Four columns of one row of S (element index e over the units' states), and z for the first row's threads, move on by the
// pass's sums; SNAP: every sum gives way to the state at its chunk's start
template <int D, bool SNAP>
__device__ __forceinline__ void add_sums(const PrefillParams &p, int64_t e) {
  const UnitId id = unit_id(p, e / (D * D / 4));
  const int at = int(e % (D * D / 4)) * 4;
  const LayerDev ld = p.layers[p.layer_begin + id.lrel];
  const int64_t first = p.n0 + p.c0 - ld.wlin;
  if (!ld.evicts || first + p.C <= 0) return;
  const int k0 = first >= 0 ? 0 : int(-first / p.SC);
  const int ub = (id.b + p.b0) * p.Hkv + id.g;
  // the sums are `stride` floats apart; those of four chunks are asked for together
  auto run = [&](float *state, float *sum, size_t stride) {
    constexpr int kAhead = 4;
    float4 s = load4(state);
    for (int k = k0; k < p.nsub; k += kAhead) {
      float4 x[kAhead];
#pragma unroll
      for (int a = 0; a < kAhead; ++a)
        if (k + a < p.nsub) x[a] = load4(sum + size_t(k + a) * stride);
#pragma unroll
      for (int a = 0; a < kAhead; ++a) {
        if (k + a >= p.nsub) break;
        if (SNAP) store4(sum + size_t(k + a) * stride, s);
        const float dec = chunk_decay(p, id.u, k + a);
        s = make_float4(fmaf(s.x, dec, x[a].x), fmaf(s.y, dec, x[a].y), fmaf(s.z, dec, x[a].z), fmaf(s.w, dec, x[a].w));
      }
    }
    store4(state, s);
  };
  run(reinterpret_cast<float *>(p.ws + ld.S) + size_t(ub) * D * D + at, p.phik + size_t(id.u) * p.nsub * D * D + at, size_t(D) * D);
  if (at < D) run(reinterpret_cast<float *>(p.ws + ld.z) + size_t(ub) * D + at, p.zsnap + size_t(id.u) * p.nsub * D + at, D);
}

// 1b. (passes of more than kDirectChunks chunks) the sums are added up once: S and z move on by the pass, and every chunk's
// slot then holds the state at its start
template <int D>
__global__ void __launch_bounds__(kThreads) prefill_fma_scan_kernel(const PrefillParams p) {
  wait_for_predecessor();   // (the launch behind this one is let go as its CTAs end: they are short)
  add_sums<D, true>(p, int64_t(blockIdx.x) * kThreads + threadIdx.x);
}

// 3. The first blocks (passes without a scan): S and z plus the pass's sums; the others: the pass's newest min(C, cap) tokens
// to slot (position mod cap), one thread per four entries of a K and a V row.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) prefill_fma_finish_kernel(const PrefillParams p, unsigned state_blocks) {
  wait_for_predecessor();
  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && p.advance)
    for (int l = tid; l < p.layer_count; l += kThreads) p.n_dev[p.layer_begin + l] += p.advance;
  if (blockIdx.x < state_blocks) {
    add_sums<D, false>(p, int64_t(blockIdx.x) * kThreads + tid);
    return;
  }
  const int64_t e = int64_t(blockIdx.x - state_blocks) * kThreads + tid;
  const int c = int(e % (D / 4)) * 4;
  const int64_t ui = e / (D / 4);
  const int i = int(ui % p.C);
  if (ui / p.C >= int64_t(p.layer_count) * p.B * p.Hkv) return;
  const UnitId id = unit_id(p, ui / p.C);
  const LayerDev ld = p.layers[p.layer_begin + id.lrel];
  if (int64_t(i) < int64_t(p.C) - ld.cap) return;   // (a layer without a ring: every token)
  const size_t src = (((size_t(id.lrel) * p.B + id.b) * size_t(p.T) + size_t(p.c0 + i)) * p.Hkv + id.g) * D + c;
  const uint32_t slot = uint32_t(p.n0 + p.c0 + i) % uint32_t(ld.cap);
  const size_t dst = ((size_t(id.b + p.b0) * p.Hkv + id.g) * size_t(ld.cap) + slot) * D + c;
  store4(reinterpret_cast<T *>(p.ws + ld.ringK) + dst, load4(reinterpret_cast<const T *>(p.k) + src));
  store4(reinterpret_cast<T *>(p.ws + ld.ringV) + dst, load4(reinterpret_cast<const T *>(p.v) + src));
  if (p.gated && c == 0)   // the token's gate waits in the ring with it
    reinterpret_cast<float *>(p.ws + ld.ringG)[dst / D] = p.gate ? p.gate[src / D] : 1.f;   // ([layer][B][T][Hkv], as K's rows)
}

}  // namespace

// Pass p (SC, nsub, C set) of the CUDA-core prefill; outputs when p.out
int launch_prefill_fma(glide_ctx *ctx, const PrefillParams &p, cudaStream_t stream) {
  const int64_t units = int64_t(p.layer_count) * p.B * p.Hkv;
  bool any_evicts = false;
  for (int l = p.layer_begin; l < p.layer_begin + p.layer_count; ++l) any_evicts = any_evicts || ctx->layers[l].evicts;
  return dispatch_config(ctx->cfg.io_dtype, ctx->cfg.head_dim, ctx->G, [&](auto tt, auto dd, auto gg) -> int {
    using T = typename decltype(tt)::type;
    constexpr int D = decltype(dd)::value, G = decltype(gg)::value, TOK = kRows / G;
    const unsigned state_ctas = any_evicts ? unsigned(units * (D * D / 4 / kThreads)) : 0u;
    const bool in_place = p.nsub == 1, scan = any_evicts && p.nsub > kDirectChunks<D>;
    const unsigned sum_ctas = unsigned(units * p.nsub * (D / 16));
    if (any_evicts && !in_place) launch_chained(prefill_fma_sums_kernel<T, D, false>, sum_ctas, 2 * kThreads, 0, stream, p);
    if (scan) launch_chained(prefill_fma_scan_kernel<D>, state_ctas, kThreads, 0, stream, p);
    if (p.out) {
      auto kern = prefill_fma_attn_kernel<T, D, G>;
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(AttnSmem<D>))) != cudaSuccess) {
        cudaGetLastError();
        return GLIDE_ERR_CUDA;
      }
      const int64_t blocks = units * (int64_t(p.nsub - 1) * ((p.SC + TOK - 1) / TOK) + (p.C - (p.nsub - 1) * p.SC + TOK - 1) / TOK);
      launch_chained(kern, unsigned(blocks), 2 * kThreads, sizeof(AttnSmem<D>), stream, p);
    }
    if (any_evicts && in_place) launch_chained(prefill_fma_sums_kernel<T, D, true>, sum_ctas, 2 * kThreads, 0, stream, p);
    const unsigned state_blocks = scan || in_place ? 0u : state_ctas;
    const unsigned ring_blocks = unsigned((units * p.C * (D / 4) + kThreads - 1) / kThreads);
    launch_chained(prefill_fma_finish_kernel<T, D>, state_blocks + ring_blocks, kThreads, 0, stream, p, state_blocks);
    return cudaGetLastError() == cudaSuccess ? GLIDE_OK : GLIDE_ERR_CUDA;
  });
}

}  // namespace glide

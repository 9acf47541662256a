// GLIDE prefill on the CUDA cores with fp32 arithmetic throughout (fp32 I/O, d = 64, and whenever the CUDA-core prefill is
// asked for) for the parameter-free feature map without gates.  A pass takes up to nsub chunks of CH tokens of every unit
// (unit = layer, sequence, KV head) in three launches:
//   1. prefill_fma_sums_kernel    per chunk phi(K')^T V' and sum phi(K') of its delayed tokens k'_i = k_{i-w}
//   2. prefill_fma_attn_kernel    per 16 query rows: window softmax, the chunk's own delayed tokens, and the state at
//                                 the chunk's start = S + the sums of the chunks before it; out
//   3. prefill_fma_finish_kernel  S and z move on by the pass, the pass's newest tokens go to the ring, counters advance
// All three read K and V rows where they are (ring for tokens older than the call) and make phi in registers; the ring
// and S change in the third only.  The problems are small (a few units of a few hundred tokens), so what bounds them is the
// length of the dependent chain and not the arithmetic: the rows of a tile are shared by 16 query rows and the next
// tile's loads are in flight while one is used.  512 tokens of 4 units (fp32, d = 64, w = 64): attention 103 us per 256
// tokens with a warp per query and one key row at a time.
#include <algorithm>
#include <type_traits>

#include "glide_device.cuh"

namespace glide {

namespace {

constexpr int kThreads = 128;
constexpr int kRows = 16;         // query rows (token, head of the group) per CTA: 8 half-warps of two rows

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

// K and V rows of one unit by absolute token
template <typename T, int D>
struct Rows {
  const T *ringK, *ringV, *callK, *callV;
  int64_t n0, call_stride;
  uint32_t cap;
  __device__ __forceinline__ Rows(const PrefillParams &p, const LayerDev &ld, int lrel, int b, int g) {
    const size_t base = (size_t(b + p.b0) * p.Hkv + g) * size_t(ld.cap) * D;   // b + b0: the sequence's slot in the context
    ringK = reinterpret_cast<const T *>(p.ws + ld.ringK) + base;
    ringV = reinterpret_cast<const T *>(p.ws + ld.ringV) + base;
    const size_t seq = (size_t(lrel) * p.B + b) * size_t(p.T) * p.Hkv * D + size_t(g) * D;
    callK = reinterpret_cast<const T *>(p.k) + seq;
    callV = reinterpret_cast<const T *>(p.v) + seq;
    n0 = p.n0;
    call_stride = int64_t(p.Hkv) * D;
    cap = ld.cap > 0 ? uint32_t(ld.cap) : 1u;
  }
  // element offset of token j's row in the call's tensors (>= 0) or, as ~offset, in the rings; tokens stay below 2^31
  __device__ __forceinline__ int64_t at(int64_t j) const {
    return j >= n0 ? (j - n0) * call_stride : ~(int64_t(uint32_t(j) % cap) * D);
  }
  __device__ __forceinline__ float4 k(int64_t off, int c) const { return load4(off >= 0 ? callK + off + c : ringK + ~off + c); }
  __device__ __forceinline__ float4 v(int64_t off, int c) const { return load4(off >= 0 ? callV + off + c : ringV + ~off + c); }
};

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

// 1. One CTA per (unit, chunk, 16 rows of S): every half-warp owns two rows, a lane D / 16 columns of them.  The rows of phi
// are made from K' as they are loaded (all of them in every CTA of a unit: cheaper than a launch in front and a trip
// through memory), the CTA keeps its 16 columns of them.
constexpr int kSumTok = 32;    // tokens per tile
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) prefill_fma_sums_kernel(const PrefillParams p) {
  constexpr int LD = kSumTok * D / 4 / kThreads;   // float4 per thread and tile
  constexpr int CG = D / 64;                       // groups of four columns per thread
  __shared__ __align__(16) float ph[2][kSumTok][16];
  __shared__ __align__(16) float vt[2][kSumTok][D];
  const int tid = threadIdx.x;
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
  float4 kr[LD], vr[LD];
  auto fetch = [&](int i0) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      kr[i] = vr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i0 + r < chunk_n) {
        const int64_t off = rows.at(first + i0 + r);
        kr[i] = rows.k(off, c);
        vr[i] = rows.v(off, c);
      }
    }
  };
  const int row = (tid >> 4) * 2, cg = tid & 15;
  float acc[2][4 * CG], zacc = 0.f;
#pragma unroll
  for (int c = 0; c < 4 * CG; ++c) acc[0][c] = acc[1][c] = 0.f;
  fetch(i_lo);
  int buf = 0;
  for (int i0 = i_lo; i0 < chunk_n; i0 += kSumTok, buf ^= 1) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      float4 f = row_phi<D>(kr[i]);
      if (i0 + r >= chunk_n) f = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c >> 4 == rb) *reinterpret_cast<float4 *>(&ph[buf][r][c & 15]) = f;
      *reinterpret_cast<float4 *>(&vt[buf][r][c]) = vr[i];
    }
    __syncthreads();   // (two buffers: the tile before the previous one has been read by everyone)
    if (i0 + kSumTok < chunk_n) fetch(i0 + kSumTok);
#pragma unroll 8
    for (int i = 0; i < kSumTok; ++i) {
      const float2 f = *reinterpret_cast<const float2 *>(&ph[buf][i][row]);
#pragma unroll
      for (int q = 0; q < CG; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(&vt[buf][i][q * 64 + cg * 4]);
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
      for (int i = 0; i < kSumTok; ++i) zacc += ph[buf][i][tid];
    }
  }
  float *dst = p.phik + (size_t(uc) * D + rb * 16 + row) * D + cg * 4;
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < CG; ++q)
      *reinterpret_cast<float4 *>(dst + r * D + q * 64) = make_float4(acc[r][q * 4], acc[r][q * 4 + 1], acc[r][q * 4 + 2], acc[r][q * 4 + 3]);
  if (tid < 16) p.zsnap[size_t(uc) * D + rb * 16 + tid] = zacc;
}

// 2. Tiles of KT rows in turn: the window's keys, the chunk's delayed tokens, the rows of the state.  Per tile a half-warp
// computes the weights of its two rows (a lane KT / 16 keys), keeps them in shared memory for itself, and adds the weighted
// V (or S) rows (a lane D / 16 columns).
template <int D>
struct AttnSmem {
  static constexpr int KT = 4096 / D;             // 64 rows for d = 64, 32 for d = 128: 16 float4 per thread and tile
  float q[kRows][D + 4];                          // scaled to the log2 domain
  float pq[kRows][D + 4];                         // phi(q)
  float k[KT][D + 4];                             // (+ 4: rows start four banks apart)
  float v[KT][D];
  float p[kRows][KT + 4];
};

template <typename T, int D, int G>
__global__ void __launch_bounds__(kThreads) prefill_fma_attn_kernel(const PrefillParams p) {
  constexpr int KT = AttnSmem<D>::KT;
  constexpr int LD = KT * D / 4 / kThreads;        // float4 of K (and of V) per thread and tile
  constexpr int KPT = KT / 16;                     // keys per lane
  constexpr int CG = D / 64;
  constexpr int TOK = kRows / G;                   // tokens per CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  AttnSmem<D> &sm = *reinterpret_cast<AttnSmem<D> *>(smem_raw);
  const int tid = threadIdx.x;
  const int per_chunk = (p.SC + TOK - 1) / TOK;
  const int per_unit = (p.nsub - 1) * per_chunk + (p.C - (p.nsub - 1) * p.SC + TOK - 1) / TOK;
  const UnitId id = unit_id(p, blockIdx.x / per_unit);
  const int cta = per_unit - 1 - int(blockIdx.x % per_unit);   // the longest windows of a new prompt first
  const int sub = cta / per_chunk, tok0 = (cta - sub * per_chunk) * TOK;
  const int chunk_c0 = sub * p.SC, chunk_n = min(p.SC, p.C - chunk_c0);
  const int ntok = min(TOK, chunk_n - tok0);
  const LayerDev ld = p.layers[p.layer_begin + id.lrel];
  const Rows<T, D> rows(p, ld, id.lrel, id.b, id.g);
  const int64_t tq0 = p.n0 + p.c0 + chunk_c0 + tok0, tq_last = tq0 + ntok - 1;
  const size_t seq_row = (size_t(id.lrel) * p.B + id.b) * size_t(p.T) + size_t(p.c0 + chunk_c0 + tok0);

  // tiles: n_win of window keys from j_lo on, n_int of delayed tokens from chunk index i_lo on, n_st of state rows
  const int64_t w_lo = tq0 - ld.w + 1;
  const int64_t j_lo = w_lo < 0 ? 0 : w_lo;
  const int n_win = ld.w > 0 ? int((tq_last - j_lo) / KT) + 1 : 0;
  const bool linear = ld.evicts && tq_last >= ld.wlin;
  const int64_t first = p.n0 + p.c0 + chunk_c0 - ld.wlin;      // delayed token of chunk index 0
  const int i_lo = first_delayed(first, chunk_n), i_hi = tok0 + ntok - 1;
  const int n_int = linear && i_lo <= i_hi ? (i_hi - i_lo) / KT + 1 : 0;
  const int n_st = linear && first > 0 ? D / KT : 0;
  const int n_tiles = n_win + n_int + n_st;
  // sums of the chunks before this one that hold delayed tokens: [sub0, sub)
  const int sub0 = first - int64_t(chunk_c0) >= 0 ? 0 : int(-(first - chunk_c0) / p.SC);
  const float *sums = p.phik + size_t(id.u) * p.nsub * D * D;
  const int ub = (id.b + p.b0) * p.Hkv + id.g;
  const float *Sb = reinterpret_cast<const float *>(p.ws + ld.S) + size_t(ub) * D * D;

  float4 kr[LD], vr[LD];
  auto fetch = [&](int t) {
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      kr[i] = vr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (t < n_win + n_int) {
        const bool win = t < n_win;
        const int64_t j = win ? j_lo + int64_t(t) * KT + r : first + i_lo + (t - n_win) * KT + r;
        if (j <= (win ? tq_last : first + i_hi)) {
          const int64_t off = rows.at(j);
          kr[i] = rows.k(off, c);
          vr[i] = rows.v(off, c);
        }
      } else {
        const size_t at = size_t((t - n_win - n_int) * KT + r) * D + c;
        float4 s = *reinterpret_cast<const float4 *>(Sb + at);
        for (int k = sub0; k < sub; ++k) {
          const float4 x = *reinterpret_cast<const float4 *>(sums + size_t(k) * D * D + at);
          s.x += x.x, s.y += x.y, s.z += x.z, s.w += x.w;
        }
        vr[i] = s;
      }
    }
  };
  if (n_tiles > 0) fetch(0);
  // the 16 query rows, and phi of them (D / 4 lanes of one row, as in the tiles)
#pragma unroll
  for (int i = 0; i < kRows * D / 4 / kThreads; ++i) {
    const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
    const int tk = r / G, head = p.heads_of[id.g * G + r % G];
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tk < ntok) x = load4(reinterpret_cast<const T *>(p.q) + ((seq_row + tk) * p.H + head) * D + c);
    *reinterpret_cast<float4 *>(&sm.pq[r][c]) = row_phi<D>(x);
    *reinterpret_cast<float4 *>(&sm.q[r][c]) = make_float4(x.x * p.scale_log2, x.y * p.scale_log2, x.z * p.scale_log2, x.w * p.scale_log2);
  }

  const int row = (tid >> 4) * 2, cg = tid & 15;
  float acc[2][4 * CG], lin[2][4 * CG], m[2], l[2], bl[2];
  int64_t tq[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    m[r] = -CUDART_INF_F;
    l[r] = bl[r] = 0.f;
    tq[r] = tq0 + (row + r) / G;
#pragma unroll
    for (int c = 0; c < 4 * CG; ++c) acc[r][c] = lin[r][c] = 0.f;
  }
  // s[r][x] = a[row + r] . k[cg + 16 x]
  auto scores = [&](const float (*a)[D + 4], float (&s)[2][KPT]) {
#pragma unroll
    for (int x = 0; x < KPT; ++x) s[0][x] = s[1][x] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      const float4 a0 = *reinterpret_cast<const float4 *>(&a[row][c]), a1 = *reinterpret_cast<const float4 *>(&a[row + 1][c]);
#pragma unroll
      for (int x = 0; x < KPT; ++x) {
        const float4 b = *reinterpret_cast<const float4 *>(&sm.k[cg + 16 * x][c]);
        s[0][x] = fmaf(a0.w, b.w, fmaf(a0.z, b.z, fmaf(a0.y, b.y, fmaf(a0.x, b.x, s[0][x]))));
        s[1][x] = fmaf(a1.w, b.w, fmaf(a1.z, b.z, fmaf(a1.y, b.y, fmaf(a1.x, b.x, s[1][x]))));
      }
    }
  };
  // o[r] += weights of row + r (wt, row stride ws) times the tile's V rows
  auto add_rows = [&](const float *w0, const float *w1, float (&o)[2][4 * CG]) {
#pragma unroll 2
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
    const bool win = t < n_win, intra = !win && t < n_win + n_int;
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + kThreads * i, r = e / (D / 4), c = e % (D / 4) * 4;
      if (win) *reinterpret_cast<float4 *>(&sm.k[r][c]) = kr[i];
      if (intra) *reinterpret_cast<float4 *>(&sm.k[r][c]) = row_phi<D>(kr[i]);   // (uniform over the CTA)
      *reinterpret_cast<float4 *>(&sm.v[r][c]) = vr[i];
    }
    __syncthreads();
    if (t + 1 < n_tiles) fetch(t + 1);
    if (win) {
      float s[2][KPT];
      scores(sm.q, s);
      const int64_t j0 = j_lo + int64_t(t) * KT + cg;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float mx = -CUDART_INF_F;
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const int64_t j = j0 + 16 * x;
          if (j > tq[r] || j <= tq[r] - ld.w) s[r][x] = -CUDART_INF_F;
          mx = fmaxf(mx, s[r][x]);
        }
        const float mn = fmaxf(m[r], lanes_max<16>(mx));
        const float f = m[r] == -CUDART_INF_F ? 0.f : exp2f(m[r] - mn);
        m[r] = mn;
        l[r] *= f;
#pragma unroll
        for (int c = 0; c < 4 * CG; ++c) acc[r][c] *= f;
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const float e = s[r][x] == -CUDART_INF_F ? 0.f : exp2f(s[r][x] - mn);
          l[r] += e;
          sm.p[row + r][cg + 16 * x] = e;
        }
      }
      __syncwarp();
      add_rows(sm.p[row], sm.p[row + 1], acc);
    } else if (intra) {
      float s[2][KPT];
      scores(sm.pq, s);
      const int ii = i_lo + (t - n_win) * KT + cg;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int own = tok0 + (row + r) / G;      // delayed tokens up to and including the query's own
#pragma unroll
        for (int x = 0; x < KPT; ++x) {
          const float e = ii + 16 * x <= own ? s[r][x] : 0.f;
          bl[r] += e;
          sm.p[row + r][cg + 16 * x] = e;
        }
      }
      __syncwarp();
      add_rows(sm.p[row], sm.p[row + 1], lin);
    } else {
      const int r0 = (t - n_win - n_int) * KT;
      add_rows(&sm.pq[row][r0], &sm.pq[row + 1][r0], lin);
    }
    __syncthreads();
  }
  if (n_st > 0) {   // phi(q) . z
    const float *zb = reinterpret_cast<const float *>(p.ws + ld.z) + size_t(ub) * D;
    const float *zs = p.zsnap + size_t(id.u) * p.nsub * D;
#pragma unroll
    for (int i = 0; i < D / 16; ++i) {
      float z = zb[cg + 16 * i];
      for (int k = sub0; k < sub; ++k) z += zs[size_t(k) * D + cg + 16 * i];
      bl[0] = fmaf(sm.pq[row][cg + 16 * i], z, bl[0]);
      bl[1] = fmaf(sm.pq[row + 1][cg + 16 * i], z, bl[1]);
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const float L = lanes_sum<16>(l[r]), Bl = lanes_sum<16>(bl[r]);
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
    if (tk < ntok) {
      T *op = reinterpret_cast<T *>(p.out) + ((seq_row + tk) * p.H + head) * D + cg * 4;
#pragma unroll
      for (int q = 0; q < CG; ++q)
        store4(op + q * 64, make_float4(fmaf(acc[r][q * 4], fa, lin[r][q * 4] * fb), fmaf(acc[r][q * 4 + 1], fa, lin[r][q * 4 + 1] * fb),
                                        fmaf(acc[r][q * 4 + 2], fa, lin[r][q * 4 + 2] * fb), fmaf(acc[r][q * 4 + 3], fa, lin[r][q * 4 + 3] * fb)));
    }
  }
}

// 3. The first blocks: S and z plus the pass's sums (a thread four columns of one row); the others: the pass's newest
// min(C, cap) tokens to slot (position mod cap), one thread per four entries of a K and a V row.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) prefill_fma_finish_kernel(const PrefillParams p, unsigned state_blocks) {
  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && p.advance)
    for (int l = tid; l < p.layer_count; l += kThreads) p.n_dev[p.layer_begin + l] += p.advance;
  if (blockIdx.x < state_blocks) {
    const int64_t e = int64_t(blockIdx.x) * kThreads + tid;
    const UnitId id = unit_id(p, e / (D * D / 4));
    const int at = int(e % (D * D / 4)) * 4;
    const LayerDev ld = p.layers[p.layer_begin + id.lrel];
    const int64_t first = p.n0 + p.c0 - ld.wlin;
    if (!ld.evicts || first + p.C <= 0) return;
    const int k0 = first >= 0 ? 0 : int(-first / p.SC);
    const int ub = (id.b + p.b0) * p.Hkv + id.g;
    float4 *Sp = reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.ws + ld.S) + size_t(ub) * D * D + at);
    const float *sums = p.phik + size_t(id.u) * p.nsub * D * D + at;
    float4 s = *Sp;
#pragma unroll 4
    for (int k = k0; k < p.nsub; ++k) {
      const float4 x = *reinterpret_cast<const float4 *>(sums + size_t(k) * D * D);
      s.x += x.x, s.y += x.y, s.z += x.z, s.w += x.w;
    }
    *Sp = s;
    if (at < D) {
      float4 *zp = reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.ws + ld.z) + size_t(ub) * D + at);
      float4 z = *zp;
      for (int k = k0; k < p.nsub; ++k) {
        const float4 x = *reinterpret_cast<const float4 *>(p.zsnap + (size_t(id.u) * p.nsub + k) * D + at);
        z.x += x.x, z.y += x.y, z.z += x.z, z.w += x.w;
      }
      *zp = z;
    }
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
    if (any_evicts) prefill_fma_sums_kernel<T, D><<<unsigned(units * p.nsub * (D / 16)), kThreads, 0, stream>>>(p);
    if (p.out) {
      auto kern = prefill_fma_attn_kernel<T, D, G>;
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sizeof(AttnSmem<D>))) != cudaSuccess) {
        cudaGetLastError();
        return GLIDE_ERR_CUDA;
      }
      const int64_t blocks = units * (int64_t(p.nsub - 1) * ((p.SC + TOK - 1) / TOK) + (p.C - (p.nsub - 1) * p.SC + TOK - 1) / TOK);
      kern<<<unsigned(blocks), kThreads, sizeof(AttnSmem<D>), stream>>>(p);
    }
    const unsigned state_blocks = any_evicts ? unsigned(units * (D * D / 4 / kThreads)) : 0u;
    const unsigned ring_blocks = unsigned((units * p.C * (D / 4) + kThreads - 1) / kThreads);
    prefill_fma_finish_kernel<T, D><<<state_blocks + ring_blocks, kThreads, 0, stream>>>(p, state_blocks);
    return cudaGetLastError() == cudaSuccess ? GLIDE_OK : GLIDE_ERR_CUDA;
  });
}

}  // namespace glide

// K and V rows of a prefill pass by token, and one output row by itself: what the tiled attention kernels fall back to when a
// tile held a value that is not finite.
#pragma once

#include "glide_device.cuh"

namespace glide {

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
  __device__ __forceinline__ const T *k(int64_t off) const { return off >= 0 ? callK + off : ringK + ~off; }
  __device__ __forceinline__ const T *v(int64_t off) const { return off >= 0 ? callV + off : ringV + ~off; }
};

// One output row (token, query head) by one warp, from the rows that count for it and no others: the tiled kernels give a row
// that does not count the weight zero, which is not enough where it holds an infinity or a NaN (a padded tail of the call's
// V), and a split weight times an infinity may be NaN where the weight's product is not.  Cold: called for rows whose
// result is not finite.  State: the unit's state at the start of the token's chunk, row(r, c, x) E values of row r from
// column c on, z(r) of z.
template <typename T, int D>
struct RowJob {
  Rows<T, D> rows;
  const T *q;
  T *out;
  const float *gc;       // gated: running log-gates of the chunk's delayed tokens, or null
  int64_t chunk_first;   // absolute token of chunk index 0
  int tl;                // the token's chunk index
  int64_t w, wlin;
  int evicts, merge;
  float scale_log2;
};
template <typename T, int D, typename State>
__device__ __noinline__ void recompute_row(const RowJob<T, D> &job, const State &state) {
  constexpr int E = D / 32;
  const int c0 = (threadIdx.x & 31) * E;
  float q[1][E], f[E], acc[1][E], m[1] = {-CUDART_INF_F}, l[1] = {0.f}, lin[E], bl = 0.f;
  load_elems<T, E>(job.q + c0, q[0]);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    f[e] = q[0][e];
    q[0][e] *= job.scale_log2;
    acc[0][e] = lin[e] = 0.f;
  }
  warp_phi<E>(f);
  const int64_t tq = job.chunk_first + job.tl;
  for (int64_t j = tq - job.w + 1 < 0 ? 0 : tq - job.w + 1; j <= tq; ++j) {
    const int64_t off = job.rows.at(j);
    float kx[E], vx[E];
    load_elems<T, E>(job.rows.k(off) + c0, kx);
    load_elems<T, E>(job.rows.v(off) + c0, vx);
    online_row<E, 1>(q, kx, vx, m, l, acc);
  }
  if (job.evicts && tq >= job.wlin) {
    const int64_t first = job.chunk_first - job.wlin;   // delayed token of chunk index 0: tokens below it are in the state
    const float g_own = job.gc ? job.gc[job.tl] : 0.f;
    if (first > 0) {
      const float dec = job.gc ? expf(g_own) : 1.f;
      for (int r = 0; r < D; ++r) {
        float s[E];
        state.row(r, c0, s);
        const float fr = __shfl_sync(0xffffffffu, f[r % E], r / E) * dec;
#pragma unroll
        for (int e = 0; e < E; ++e) lin[e] = fmaf(fr, s[e], lin[e]);
      }
#pragma unroll
      for (int e = 0; e < E; ++e) bl = fmaf(f[e], state.z(c0 + e), bl);
      bl = warp_sum(bl) * dec;
    }
    for (int i = first < 0 ? int(-first) : 0; i <= job.tl; ++i) {
      const int64_t off = job.rows.at(first + i);
      float kx[E], vx[E], part = 0.f;
      load_elems<T, E>(job.rows.k(off) + c0, kx);
      load_elems<T, E>(job.rows.v(off) + c0, vx);
      warp_phi<E>(kx);
#pragma unroll
      for (int e = 0; e < E; ++e) part = fmaf(f[e], kx[e], part);
      const float c = warp_sum(part) * (job.gc ? expf(g_own - job.gc[i]) : 1.f);
      bl += c;
#pragma unroll
      for (int e = 0; e < E; ++e) lin[e] = fmaf(c, vx[e], lin[e]);
    }
  }
  // shared normaliser (the floor of the reference belongs to the linear terms, logit 0), or two separately normalised terms
  float fa, fb;
  if (job.merge != GLIDE_MERGE_SHARED) {
    fa = l[0] > 0.f ? 1.0f / l[0] : 0.f;
    fb = bl > 0.f ? 1.0f / bl : 0.f;
  } else {
    const float M = bl > 0.f ? fmaxf(m[0], 0.f) : m[0];
    const float fw = m[0] == -CUDART_INF_F ? 0.f : exp2f(m[0] - M), fl = bl > 0.f ? exp2f(-M) : 0.f;
    const float inv = 1.0f / fmaf(l[0], fw, fl * bl);
    fa = fw * inv;
    fb = fl * inv;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) from_f32(job.out + c0 + e, fmaf(acc[0][e], fa, lin[e] * fb));
}

}  // namespace glide

// The Adam update (§5.1) shared by k_adam and by the weight-gradient kernels
// that apply it to their own tiles.
#pragma once

#include "ff_internal.cuh"

namespace ff {

// One Adam step of the four weights at idx (16-byte aligned) from their
// gradient: W, m and v through registers, the bf16 copy at row n, column k.
// The state is touched once per step: evict-first, so that the stream leaves
// the GEMMs' operands in L2.
struct AdamVec {
  float4 w, m, v;
  __device__ __forceinline__ void load(const AdamArgs& a, size_t idx) {
    w = __ldcs(reinterpret_cast<const float4*>(a.W + idx));
    m = __ldcs(reinterpret_cast<const float4*>(a.mW + idx));
    v = __ldcs(reinterpret_cast<const float4*>(a.vW + idx));
  }
  __device__ __forceinline__ void update(const AdamArgs& a, const float4& g, float a1, float r2) {
    adam1(w.x, m.x, v.x, g.x, a1, a.beta1, a.beta2, a.eps, r2);
    adam1(w.y, m.y, v.y, g.y, a1, a.beta1, a.beta2, a.eps, r2);
    adam1(w.z, m.z, v.z, g.z, a1, a.beta1, a.beta2, a.eps, r2);
    adam1(w.w, m.w, v.w, g.w, a1, a.beta1, a.beta2, a.eps, r2);
  }
  __device__ __forceinline__ void store(const AdamArgs& a, size_t idx) const {
    __stcs(reinterpret_cast<float4*>(a.W + idx), w);
    __stcs(reinterpret_cast<float4*>(a.mW + idx), m);
    __stcs(reinterpret_cast<float4*>(a.vW + idx), v);
  }
  __device__ __forceinline__ uint2 packed() const {
    __nv_bfloat162 p0 = __floats2bfloat162_rn(w.x, w.y), p1 = __floats2bfloat162_rn(w.z, w.w);
    return make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1));
  }
};

// The bias elements, db from the local gradient's partials, and (blk 0) the
// step's loss and statistics; one block of whole warps (any number) per 32
// bias elements.  A fixed reduction order, with the loads batched: eight sums
// per column over row blocks w, w+8, ..., then the eight in order.
__device__ __forceinline__ void adam_bias_block(const AdamArgs& a, int blk, float a1, float r2) {
  __shared__ float part[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int j = blk * 32 + lane;
  for (int w = warp; w < 8; w += warps) {
    float acc = 0.f;
    if (j < a.N) {
      for (int rb0 = w; rb0 < a.nrb; rb0 += 64) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int rb = rb0 + 8 * u;
          v[u] = rb < a.nrb ? __ldg(a.dbpart + (size_t)rb * a.N + j) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) acc += v[u];
      }
    }
    part[w][lane] = acc;
  }
  __syncthreads();
  for (int w = warp; blk == 0 && w < 8; w += warps) {
    if (w == 1 && a.loss_part) {
      // the step's loss: grad_prep's per-row-block partials, lane-strided then
      // a fixed-order warp tree
      float tot = 0.f;
      for (int rb = lane; rb < a.nrb; rb += 32) tot += a.loss_part[rb];
      tot = warp_sum(tot);
      if (lane == 0) a.loss_out[0] = tot / (float)a.B;
    }
    if (w >= 2 && w <= 4 && a.stat_part) {
      // the step's statistics: mean goodness of the positive and of the
      // negative rows, and the fraction of active ReLUs
      const int n = w == 4 ? a.nrb * a.ncb : a.nrb;
      const float* src = a.stat_part + (w == 2 ? 0 : w == 3 ? a.nrb : 2 * a.nrb);
      float tot = 0.f;
      for (int k = lane; k < n; k += 32) tot += src[k];
      tot = warp_sum(tot);
      if (lane == 0) a.stats_out[w - 2] = w == 4 ? tot / (2.f * (float)a.B * (float)a.N) : tot / (float)a.B;
    }
  }
  if (warp != 0 || j >= a.N) return;
  float db = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) db += part[u][lane];
  if (a.db_out) a.db_out[j] = db;
  if (a.has_bias) {
    float b = a.b[j], m = a.mb[j], v = a.vb[j];
    adam1(b, m, v, db, a1, a.beta1, a.beta2, a.eps, r2);
    a.b[j] = b;
    a.mb[j] = m;
    a.vb[j] = v;
  }
}
inline int adam_bias_blocks(int N) { return cdiv(N, 32); }

}  // namespace ff

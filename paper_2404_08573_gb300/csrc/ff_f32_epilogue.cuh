// The end of the fp32 GEMMs (CUDA-core and tensor-core): a CTA's T x T partial
// tile sits in its shared memory, rows of f32_tile_ld(T) floats; the S CTAs
// of a cluster hold the partials of one tile over S slices of K, and each
// finishes T / S rows of the sum.
#pragma once

#include "ff_adam.cuh"
#include "ff_internal.cuh"
#include "ff_ptx.cuh"

namespace ff {

constexpr int NT = 256;  // threads of the epilogue
constexpr int MODE_FWD = 0, MODE_STORE = 1, MODE_ADAM = 2;
constexpr int kMaxSplit = 4;  // CTAs per cluster

__host__ __device__ constexpr int f32_tile_ld(int T) { return T + 4; }

__device__ __forceinline__ float4 ld_cluster4(const float* local, uint32_t rank) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(ptx::mapa_shared(ptx::smem_u32(local), rank))
               : "memory");
  return v;
}

// The slices' CTAs have cluster ranks rank0 + rank_step * slice (slice:
// blockIdx.z).  By threads 0 .. 255 (tid) of a CTA, after its own and its cluster's partials
// are in place (and before any CTA of the cluster leaves):
//   MODE_FWD    H = ReLU(s_r z + b), goodness partials per row and T columns
//   MODE_STORE  C = z
//   MODE_ADAM   z is the gradient of the weights W[gi, col]: Adam on them
template <int T, int MODE>
__device__ __forceinline__ void f32_tile_epilogue(const float* sm, int tid, int M, int N, int m0, int n0, int S,
                                                  const EpiArgs& ep, const AdamArgs& ad, uint32_t rank0 = 0,
                                                  uint32_t rank_step = 1) {
  constexpr int LD = f32_tile_ld(T);
  constexpr int LPR = T / 4;     // lanes per row, 4 columns each
  constexpr int RPP = NT / LPR;  // rows per pass
  const int lr = tid / LPR, lc = (tid % LPR) * 4;
  // the epilogue on this CTA's TM / S rows of the tile
  const int RS = T / S;
  const int col = n0 + lc;
  // four values of row r of the tile: the sum of the S partials in rank order
  auto tile4 = [&](int r, float (&v)[4]) {
    if (S > 1) {
      float4 u[kMaxSplit];
#pragma unroll
      for (int z = 0; z < kMaxSplit; ++z)
        if (z < S) u[z] = ld_cluster4(sm + r * LD + lc, rank0 + rank_step * (uint32_t)z);
      v[0] = v[1] = v[2] = v[3] = 0.f;
#pragma unroll
      for (int z = 0; z < kMaxSplit; ++z)
        if (z < S) {
          v[0] += u[z].x; v[1] += u[z].y; v[2] += u[z].z; v[3] += u[z].w;
        }
    } else {
      const float4 u = *reinterpret_cast<const float4*>(sm + r * LD + lc);
      v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
    }
  };
  if constexpr (MODE == MODE_ADAM) {
    // Adam on the tile's weights: the state of kBatch rows in flight at a time
    constexpr int kBatch = 4;
    const float a1 = ad.lr / ad.ds->bc1, r2 = 1.f / ad.ds->bc2;
    const bool vec = (ad.K & 3) == 0;
    for (int p = 0; p < RS; p += kBatch * RPP) {
      AdamVec st[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int o = p + q * RPP + lr;
        const int gi = m0 + (int)blockIdx.z * RS + o;
        if (vec && o < RS && gi < M && col < N) st[q].load(ad, (size_t)gi * N + col);
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int o = p + q * RPP + lr;
        const int gi = m0 + (int)blockIdx.z * RS + o;
        if (o >= RS || gi >= M || col >= N) continue;
        float v[4];
        tile4((int)blockIdx.z * RS + o, v);
        const size_t idx = (size_t)gi * N + col;
        if (vec) {
          const float4 dw = make_float4(v[0], v[1], v[2], v[3]);
          if (ad.keep_dW) *reinterpret_cast<float4*>(ad.keep_dW + idx) = dw;
          st[q].update(ad, dw, a1, r2);
          st[q].store(ad, idx);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (col + e >= N) break;
            float w = ad.W[idx + e], m = ad.mW[idx + e], vv = ad.vW[idx + e];
            adam1(w, m, vv, v[e], a1, ad.beta1, ad.beta2, ad.eps, r2);
            ad.W[idx + e] = w;
            ad.mW[idx + e] = m;
            ad.vW[idx + e] = vv;
            if (ad.keep_dW) ad.keep_dW[idx + e] = v[e];
          }
        }
      }
    }
  } else if constexpr (MODE == MODE_FWD) {
    // kBatch rows per thread at a time: their scales' loads together
    constexpr int kBatch = 4;
    float bias[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) bias[e] = ep.bias && col + e < N ? __ldg(ep.bias + col + e) : 0.f;
    for (int p = 0; p < RS; p += kBatch * RPP) {
      float s[kBatch], g[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int o = p + q * RPP + lr;
        const int gi = m0 + (int)blockIdx.z * RS + o;
        s[q] = o < RS && gi < M ? __ldg(ep.row_scale + gi) : 0.f;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int o = p + q * RPP + lr;
        const int gi = m0 + (int)blockIdx.z * RS + o;
        const bool row_ok = o < RS && gi < M;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (row_ok) tile4((int)blockIdx.z * RS + o, v);
        float own = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float h = 0.f;
          if (row_ok && col + e < N) {
            // both roundings spelled out, so that every GEMM form agrees
            float z = __fmul_rn(s[q], v[e]);
            if (ep.bias) z = __fadd_rn(z, bias[e]);
            h = z != z ? z : fmaxf(z, 0.f);  // ReLU, NaN kept for the non-finite check
          }
          own = fmaf(h, h, own);
          v[e] = h;
        }
        // the upper half of a row's lanes carries on the lower half's sums
        // (columns 4 l .. 4 l + 3, then T/2 + 4 l ..): LPR / 2 sums a row
        g[q] = __shfl_sync(0xffffffffu, own, (int)(threadIdx.x & 31) ^ (LPR / 2));
#pragma unroll
        for (int e = 0; e < 4; ++e) g[q] = fmaf(v[e], v[e], g[q]);
        // activation rows are padded to multiples of 8: whole 16-byte words
        if (row_ok && col < ep.ldo)
          *reinterpret_cast<float4*>(static_cast<float*>(ep.out) + (size_t)gi * ep.ldo + col) =
              make_float4(v[0], v[1], v[2], v[3]);
      }
      // the upper lanes' sums
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
#pragma unroll
        for (int o = LPR / 4; o > 0; o >>= 1) g[q] += __shfl_xor_sync(0xffffffffu, g[q], o);
        const int o = p + q * RPP + lr;
        const int gi = m0 + (int)blockIdx.z * RS + o;
        if (lc == T / 2 && o < RS && gi < M) ep.gpart[(size_t)(n0 / T) * M + gi] = g[q];
      }
    }
  } else {
    for (int p = 0; p < RS; p += RPP) {
      const int o = p + lr;
      const int gi = m0 + (int)blockIdx.z * RS + o;
      if (o >= RS || gi >= M) continue;
      float v[4];
      tile4((int)blockIdx.z * RS + o, v);
      float* out = static_cast<float*>(ep.out) + (size_t)gi * ep.ldo + col;
      if ((ep.ldo & 3) == 0 && col + 4 <= N) {
        *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (col + e < N) out[e] = v[e];
      }
    }
  }
}

}  // namespace ff

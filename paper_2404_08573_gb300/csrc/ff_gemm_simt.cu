// fp32 GEMMs of the FF layer step: the choice among the paths (plan_of), and
// the CUDA-core (FFMA) kernels, which run the outputs too small for the
// tensor-core ones (k_f32tc_gemm, k_f32tc_pair) and operands that these do
// not take.  The same contracts as the bf16 GEMMs (forward with the
// scale/bias/ReLU/goodness epilogue, plain fp32 store, weight gradient over
// the batch rows); either way fp32 operands and sums.
//
// Bound by the SM's shared-memory reads and FMA issue together (large
// outputs reach 45 to 50 TFLOP/s), small ones by latency.  FMAs are issued in
// pairs (fma.rn.f32x2, each rounded as fmaf): 10 % faster than single ones.
// A CTA of 256 threads computes a TM x TN tile over one slice of K, 8x8
// outputs per thread, operands staged 32 deep in K by a ring of cp.async
// copies.  Two shapes:
//   128 x 128, all threads on the same K: the fewest operand reads per FMA;
//   64 x 64, four groups of 64 threads that each take a quarter of every
//     stage's K (8x8 outputs per thread again) and add up in shared memory:
//     for outputs of few tiles.
// Either may further be cut over K: the S CTAs of a tile form a thread-block
// cluster, leave their partial tiles in their own shared memory, and each
// adds TM/S rows of all S partials (in rank order) through distributed
// shared memory and runs the epilogue on them -- no scratch in device memory
// and no counters.
#include "ff_adam.cuh"
#include "ff_f32_epilogue.cuh"
#include "ff_internal.cuh"
#include "ff_ptx.cuh"

namespace ff {
namespace {

constexpr int TKS = 32;  // K per stage

// Shape of one instance.  An operand's stage sits in shared memory as TKS
// rows (one per K) of the tile's T rows or columns, padded by 4 floats.
template <int T, int KGRP>
struct Cfg {
  static constexpr int TM = T, TN = T, KG = KGRP;
  static constexpr int TT = T / 8;                 // threads along each side of a K group's tile
  static constexpr int LD = f32_tile_ld(T);
  static constexpr int OP = TKS * LD;              // floats of one operand's stage
  static constexpr int STAGES = T == 128 ? 3 : 4;
  static constexpr int RING = 2 * OP * STAGES;
  static constexpr int PART = KG * TM * LD;        // the K groups' partial tiles, rows of LD floats
  static constexpr int SMEM = (RING > PART ? RING : PART) * 4;
  static_assert(TT * TT * KG == NT, "every thread owns 8x8 outputs of its K group");
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// Two fp32 FMAs in one instruction, each rounded as fmaf.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// Copies the slice [k0, k0 + TKS) of an operand whose tile rows start at r0
// into S[k][r].  MN == false: element (r, k) at P[r * ld + k], transposed by
// 4-byte copies (a warp takes 8 K of 4 rows: whole 32-byte sectors, and 32
// distinct banks).  MN == true: at P[k * ld + r], by 16-byte copies when
// `vec` (P and its row stride 16-byte aligned).  Elements past `rows` or K
// read as zero (a copy of fewer source bytes than it writes fills the rest
// with zeros, so row padding is never read).
template <int T, bool MN>
__device__ __forceinline__ void load_tile(float* S, const float* __restrict__ P, int ld, int rows, int K, int r0,
                                          int k0, bool vec) {
  constexpr int LD = T + 4;
  const int tid = threadIdx.x;
  if (MN && vec) {
#pragma unroll
    for (int i = 0; i < T * TKS / 4 / NT; ++i) {
      const int c = tid + i * NT;
      const int k = c / (T / 4), r = (c % (T / 4)) * 4;
      const int left = k0 + k < K ? rows - (r0 + r) : 0;
      const int n = left < 0 ? 0 : left > 4 ? 4 : left;
      cp_async16(S + k * LD + r, n ? P + (size_t)(k0 + k) * ld + r0 + r : P, n * 4);
    }
  } else {
#pragma unroll 8
    for (int i = 0; i < T * TKS / NT; ++i) {
      // !MN: warp w of step i takes K 8 (w % 4) .. and rows 4 (w / 4 + 2 i) ..
      const int c = tid + i * NT;
      const int r = MN ? c % T : (tid >> 7) * 4 + i * 8 + ((tid >> 3) & 3);
      const int k = MN ? c / T : ((tid >> 5) & 3) * 8 + (tid & 7);
      const bool ok = r0 + r < rows && k0 + k < K;
      const float* src = MN ? P + (size_t)(k0 + k) * ld + r0 + r : P + (size_t)(r0 + r) * ld + k0 + k;
      cp_async4(S + k * LD + r, ok ? src : P, ok ? 4 : 0);
    }
  }
}

// MN: both operands MN-major (the weight gradient), else both K-major.
template <int T, int KGRP, bool MN, int MODE>
__global__ void __launch_bounds__(NT, 2)
    k_simt_gemm(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int M, int N, int K,
                int vecs, EpiArgs ep, AdamArgs ad) {
  using C = Cfg<T, KGRP>;
  extern __shared__ __align__(16) float sm[];
  const int m0 = blockIdx.x * C::TM, n0 = blockIdx.y * C::TN;
  // this CTA's share of K: split blockIdx.z of gridDim.z (whole stages)
  const int S = gridDim.z;
  const int steps = (K + TKS - 1) / TKS;
  const int per = (steps + S - 1) / S;
  const int s0 = min(steps, (int)blockIdx.z * per), ns = min(steps, s0 + per) - s0;
  const int tid = threadIdx.x;
  const int grp = tid / (C::TT * C::TT), t = tid % (C::TT * C::TT);
  const int tx = t % C::TT, ty = t / C::TT;
  const bool va = vecs & 1, vb = vecs & 2;
  if constexpr (MODE == MODE_ADAM) {
    if (blockIdx.y + 1 == gridDim.y) {
      // the last row of CTAs: the bias elements, loss and statistics
      ptx::griddep_wait();
      const float a1 = ad.lr / ad.ds->bc1, r2 = 1.f / ad.ds->bc2;
      for (int blk = blockIdx.x * S + blockIdx.z; blk * 32 < ad.N; blk += gridDim.x * S) {
        adam_bias_block(ad, blk, a1, r2);
        __syncthreads();
      }
      return;
    }
  }
  ptx::griddep_wait();  // launched with programmatic stream serialization

  auto stage = [&](int s) {
    float* a = sm + (s % C::STAGES) * 2 * C::OP;
    load_tile<T, MN>(a, A, lda, M, K, m0, (s0 + s) * TKS, va);
    load_tile<T, MN>(a + C::OP, B, ldb, N, K, n0, (s0 + s) * TKS, vb);
  };
#pragma unroll
  for (int s = 0; s < C::STAGES - 1; ++s) {
    if (s < ns) stage(s);
    cp_commit();
  }

  // outputs of row pair (rows 4 ty + {0,1}, {2,3}, TM/2 + 4 ty + {0,1}, {2,3})
  // and column j (4 tx + j for j < 4, TN/2 + 4 tx + j - 4 above)
  unsigned long long acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;

  for (int s = 0; s < ns; ++s) {
    cp_wait<C::STAGES - 2>();
    __syncthreads();  // stage s has landed for everyone, and everyone is done with stage s - 1
    if (s + C::STAGES - 1 < ns) stage(s + C::STAGES - 1);
    cp_commit();
    const float* as = sm + (s % C::STAGES) * 2 * C::OP;
    const float* bs = as + C::OP;
    constexpr int KPG = TKS / C::KG;  // K per group and stage
    const float* ap = as + grp * KPG * C::LD + ty * 4;
    const float* bp = bs + grp * KPG * C::LD + tx * 4;
#pragma unroll 8
    for (int k = 0; k < KPG; ++k) {
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(ap + k * C::LD);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(ap + k * C::LD + T / 2);
      const float4 b0 = *reinterpret_cast<const float4*>(bp + k * C::LD);
      const float4 b1 = *reinterpret_cast<const float4*>(bp + k * C::LD + T / 2);
      const unsigned long long a[4] = {a0.x, a0.y, a1.x, a1.y};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const unsigned long long bb = pack2(b[j], b[j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) fma2(acc[i][j], a[i], bb);
      }
    }
  }
  cp_wait<0>();
  if (tid == 0) ptx::griddep_launch_dependents();  // the mainloop is done
  __syncthreads();  // the ring is idle: the partial tile takes its place

  float* mine = sm + grp * C::TM * C::LD;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = unpack2(acc[i][j]);
    float* p = mine + ((i >> 1) * (C::TM / 2) + ty * 4 + (i & 1) * 2) * C::LD + tx * 4;
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
    *reinterpret_cast<float4*>(p + C::TN / 2) = make_float4(v[4].x, v[5].x, v[6].x, v[7].x);
    *reinterpret_cast<float4*>(p + C::LD) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
    *reinterpret_cast<float4*>(p + C::LD + C::TN / 2) = make_float4(v[4].y, v[5].y, v[6].y, v[7].y);
  }
  __syncthreads();
  constexpr int LPR = C::TN / 4;   // lanes per row in the steps below (4 columns each)
  constexpr int RPP = NT / LPR;    // rows per pass
  const int lr = tid / LPR, lc = (tid % LPR) * 4;
  if constexpr (C::KG > 1) {
    // the K groups' partials, in group order, into the first
#pragma unroll
    for (int r = lr; r < C::TM; r += RPP) {
      float* p = sm + r * C::LD + lc;
      float4 v = *reinterpret_cast<const float4*>(p);
#pragma unroll
      for (int g = 1; g < C::KG; ++g) {
        const float4 u = *reinterpret_cast<const float4*>(p + g * C::TM * C::LD);
        v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
      }
      *reinterpret_cast<float4*>(p) = v;
    }
  }
  if (S > 1)
    ptx::cluster_sync();  // every partial of the tile is in place
  else
    __syncthreads();

  f32_tile_epilogue<T, MODE>(sm, tid, M, N, m0, n0, S, ep, ad);
  if (S > 1) ptx::cluster_sync();  // no CTA leaves while another reads its partial tile
}

// How an M x N output over K is computed: on the CUDA cores in 64 x 64 or
// 128 x 128 tiles, or on the tensor cores (ff_gemm_f32tc.cu) in 128 x 128
// tiles or, by CTA pairs, 256 x 256 ones, and in how many K slices: the least
// modelled time.  Measured: a CTA
// takes 0.95 us per 32-deep stage of a 64 x 64 tile and 3.3 us of a 128 x 128
// one (42 and 48 TFLOP/s over 152 SMs) whether or not it shares its SM -- the
// shared-memory operand reads and the FMAs fill the SM's time -- and 1.7 us
// per 64-deep chunk of a tensor-core tile, an SM to itself (a pair's, of four
// times the output, 2.7 us), with about 9 us before and after its mainloop
// against 5.  A GEMM takes the stages that the
// fullest SM runs; a split costs about 1 us more.  Eight slices measured no
// faster than four at any size (clusters of 8 find fewer places).
// Rows x K -> N, us: one 128 x 128 tile per CTA and partial tiles through
// device memory (as before) / CUDA cores / tensor cores / by pairs:
//   128 x 784 -> 500    22 / 15 / 20 / --     (CUDA cores chosen)
//   128 x 2000 -> 2000  -- / 39 / 27 / 35     (tensor cores from here on)
//   512 x 2000 -> 2000  122 / 113 / 43 / 57   weight gradient 118 / 94 / 42 / 33
//   2048 x 2000 -> 2000 480 / 367 / 130 / 99  weight gradient 416 / 322 / 121 / 97
enum Kind { TILE_64, TILE_128, TENSOR, TENSOR_PAIR };
struct Plan {
  Kind kind;
  int S;
};
Plan plan_of(int M, int N, int K, bool tensor) {
  Plan best{TILE_128, 1};
  double bt = 0.0;
  for (int kind = tensor ? TENSOR_PAIR : TILE_128; kind >= TILE_64; --kind) {
    const int T = kind == TILE_64 ? 64 : kind == TENSOR_PAIR ? 256 : 128;
    const int steps = cdiv(K, kind >= TENSOR ? 64 : TKS);
    const double tiles = (double)cdiv(M, T) * cdiv(N, T);
    for (int S = 1; S <= kMaxSplit; S *= 2) {
      if (S > 1 && steps < 2 * S) break;
      if (kind == TENSOR_PAIR && S > 2) break;  // no clusters of 8
      // CTAs (pairs) an SM (two SMs) runs in all
      const double per_sm = cdiv((long long)(tiles * S), kind == TENSOR_PAIR ? 76 : 152);
      const double step = kind == TILE_64 ? 0.95 : kind == TILE_128 ? 3.3 : kind == TENSOR ? 1.7 : 2.7;
      const double t = (kind >= TENSOR ? per_sm * (cdiv(steps, S) * step + 9.0) : per_sm * cdiv(steps, S) * step + 5.0) +
                       (S > 1 ? 1.0 : 0.0);
      if (bt == 0.0 || t < bt) {
        bt = t;
        best = Plan{(Kind)kind, S};
      }
    }
  }
  return best;
}
// The tensor-core form needs 16-byte aligned rows of both operands: for the
// forward and store, of the weights (rows of K).
Plan plan_kmajor(int M, int N, int K) { return plan_of(M, N, K, (K & 3) == 0); }

// plan_rows = kF32InOrder: each output one ascending chain of FMAs over K.
Plan plan_fwd(int plan_rows, int N, int K) {
  return plan_rows == kF32InOrder ? Plan{TILE_128, 1} : plan_kmajor(plan_rows, N, K);
}

bool aligned(const float* p, int ld) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && (ld & 3) == 0; }
bool on_tensor_cores(const Plan& p, const float* A, int lda, const float* B, int ldb) {
  return p.kind >= TENSOR && aligned(A, lda) && aligned(B, ldb);
}
Plan plan_wgrad(int R, int N, int K, bool in_order) { return in_order ? Plan{TILE_128, 1} : plan_of(N, K, R, true); }

template <int T, int KGRP, bool MN, int MODE>
cudaError_t launch_plan(const float* A, int lda, const float* B, int ldb, int M, int N, int K, int S, const EpiArgs& ep,
                        const AdamArgs& ad, cudaStream_t st) {
  using C = Cfg<T, KGRP>;
  const cudaError_t attr = allow_smem<k_simt_gemm<T, KGRP, MN, MODE>>(C::SMEM);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cdiv(M, T), cdiv(N, T) + (MODE == MODE_ADAM ? 1 : 0), S);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = S;
  cfg.attrs = at;
  cfg.numAttrs = S > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_simt_gemm<T, KGRP, MN, MODE>, A, lda, B, ldb, M, N, K,
                            (aligned(A, lda) ? 1 : 0) | (aligned(B, ldb) ? 2 : 0), ep, ad);
}

template <bool MN, int MODE>
cudaError_t launch(const float* A, int lda, const float* B, int ldb, int M, int N, int K, Plan p, const EpiArgs& ep,
                   const AdamArgs& ad, cudaStream_t st) {
  if (p.kind != TILE_64) return launch_plan<128, 1, MN, MODE>(A, lda, B, ldb, M, N, K, p.S, ep, ad, st);
  return launch_plan<64, 4, MN, MODE>(A, lda, B, ldb, M, N, K, p.S, ep, ad, st);
}

}  // namespace

int f32_fwd_ntiles(int plan_rows, int N, int K) { return cdiv(N, plan_fwd(plan_rows, N, K).kind == TILE_64 ? 64 : 128); }
int f32_fwd_ntiles_max(int N) { return cdiv(N, 64); }
bool f32_fwd_on_tensor_cores(const float* A, int lda, const float* B, int ldb, int plan_rows, int N, int K) {
  return on_tensor_cores(plan_fwd(plan_rows, N, K), A, lda, B, ldb);
}
bool f32_wgrad_on_tensor_cores(const float* G, int ldg, const float* X, int ldx, int R, int N, int K, bool in_order) {
  return on_tensor_cores(plan_wgrad(R, N, K, in_order), G, ldg, X, ldx);
}

cudaError_t f32_gemm_fwd(const float* A, int lda, const float* B, int ldb, int M, int N, int K, int plan_rows,
                         const EpiArgs& ep, int* err, cudaStream_t st) {
  const Plan p = plan_fwd(plan_rows, N, K);
  if (on_tensor_cores(p, A, lda, B, ldb))
    return f32tc_gemm_fwd(A, lda, B, ldb, M, N, K, p.S, p.kind == TENSOR_PAIR, ep, err, st);
  return launch<false, MODE_FWD>(A, lda, B, ldb, M, N, K, p, ep, AdamArgs{}, st);
}

cudaError_t f32_gemm_store(const float* A, int lda, const float* B, int ldb, int M, int N, int K, float* C, int ldc,
                           int* err, cudaStream_t st) {
  const Plan p = plan_kmajor(M, N, K);
  if (on_tensor_cores(p, A, lda, B, ldb))
    return f32tc_gemm_store(A, lda, B, ldb, M, N, K, p.S, p.kind == TENSOR_PAIR, C, ldc, err, st);
  EpiArgs ep{nullptr, nullptr, C, ldc, nullptr};
  return launch<false, MODE_STORE>(A, lda, B, ldb, M, N, K, p, ep, AdamArgs{}, st);
}

// C[n, k] = sum_r G[r, n] X[r, k]: rows of C index G's columns (MN-major A),
// columns of C index X's columns (MN-major B), contraction over R.
cudaError_t f32_gemm_wgrad(const float* G, int ldg, const float* X, int ldx, int R, int N, int K, float* C, int ldc,
                           bool in_order, int* err, cudaStream_t st) {
  const Plan p = plan_wgrad(R, N, K, in_order);
  if (on_tensor_cores(p, G, ldg, X, ldx))
    return f32tc_gemm_wgrad(G, ldg, X, ldx, R, N, K, p.S, p.kind == TENSOR_PAIR, C, ldc, err, st);
  EpiArgs ep{nullptr, nullptr, C, ldc, nullptr};
  return launch<true, MODE_STORE>(G, ldg, X, ldx, N, K, R, p, ep, AdamArgs{}, st);
}

bool f32_wgrad_adam_fits(int R, int N, int K) {
  const Plan p = plan_of(N, K, R, true);
  const int T = p.kind == TILE_64 ? 64 : 128;
  return p.kind < TENSOR && (long long)cdiv(N, T) * cdiv(K, T) * p.S <= 2 * 152;
}

cudaError_t f32_gemm_wgrad_adam(const float* G, int ldg, const float* X, int ldx, int R, const AdamArgs& a,
                                cudaStream_t st) {
  return launch<true, MODE_ADAM>(G, ldg, X, ldx, a.N, a.K, R, plan_of(a.N, a.K, R, true), EpiArgs{}, a, st);
}

}  // namespace ff

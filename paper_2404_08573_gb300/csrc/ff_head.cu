// Softmax prediction head of §3 "Prediction" (Softmax method).
//
// The unlabelled input carries the neutral label (0.1 in each of the 10
// label features) and runs once through every FF layer; the activities of
// all but the first hidden layer, each normalised like a layer input
// (h / max(||h||, 1e-12)), are the features A of a linear softmax layer
// z = A V^T + c.  The head is trained by backpropagation through itself only
// (cross-entropy averaged over the rows, Adam with its own learning rate,
// §5.1): no gradient reaches the FF layers.  Prediction is the class with the
// largest logit.
//
// Kernels (all fixed-order reductions, no floating-point atomics):
//   k_head_dot     partial logits A V^T over feature splits of the
//                  segments; A is never materialised -- it is read as the
//                  stored activities H_k times their row scales s_k.  The
//                  last block of each 64-row block to finish then forms
//                  z = c + the splits' partials (in split order), softmax,
//                  per-row loss and dz = (softmax(z) - onehot(y)) / n, and
//                  the row block's partials of dc and of the loss
//   k_head_dot_mma the same on bf16 activities, with tensor-core MMAs
//   k_head_wgrad   dV partials per 64-row block: dz^T (s_k H_k) (fp32)
//   k_head_adam    reduces the partials in a fixed order, Adam on V and c,
//                  the step's loss
//   k_head_wgrad_adam  both in one launch on bf16 activities
//   k_po_grad      the Performance-Optimized step (§4): the gradient through
//                  a layer's own block into the layer and the block's dV
//                  partials; with bf16 layers it first finishes its rows'
//                  softmax from the partial logits that the forward GEMM's
//                  epilogue wrote (no k_head_dot pass)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "ff_api_internal.h"
#include "ff_internal.cuh"
#include "ff_mma.cuh"
#include "ff_prof.h"
#include "ff_ptx.cuh"

namespace ff {
namespace {

constexpr int kClasses = 10;
constexpr int kMaxSegs = 16;
constexpr int kDotRows = 64;     // rows per block of k_head_dot (eight per warp)
constexpr int kSplit = 1024;     // widest feature split of one segment per k_head_dot block (fp32)
constexpr int kMmaSplit = 512;   // and per k_head_dot_mma block (bf16)
constexpr int kDotMinBlocks = 152 / 2;  // k_head_dot grids narrower than this split features finer
constexpr int kWgRows = 64;      // rows per block of k_head_wgrad (8 per warp)
constexpr int kWgChunk = 128;    // features per block of k_head_wgrad (4 per lane)
constexpr int kPart = kClasses + 1;  // per-block partials: dc[10], loss

// The feature segments: segment k is layer (k+2)'s activity (layer 1's when
// there is one layer), features off[k] .. off[k] + F[k] of A, scaled per row
// by s[k] (a null s[k] reads the activity unscaled).
struct Segs {
  const void* H[kMaxSegs];
  const float* s[kMaxSegs];
  int ld[kMaxSegs];
  int F[kMaxSegs];
  int off[kMaxSegs];
  int nseg;
  int F_total;
};


// h[0..4) = H[row, f .. f+4), zero past the segment or the rows.
__device__ __forceinline__ void load_feats4(const float* __restrict__ H, int ld, int row, int n, int f, int F, float* h) {
  if (row < n && f + 4 <= F) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(H + (size_t)row * ld + f));
    h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = (row < n && f + i < F) ? H[(size_t)row * ld + f + i] : 0.f;
  }
}

// Softmax, loss and dz of one row with label y from its logits (z has the bias added).
// Writes logits/dz when given; returns the row's loss (0 without a label).
__device__ __forceinline__ float finish_row(const float (&z)[kClasses], int row, bool labelled, int y,
                                            float inv_n, float* __restrict__ logits, float* __restrict__ dz,
                                            float (&dzr)[kClasses], int* err) {
  bool finite = true;
#pragma unroll
  for (int c = 0; c < kClasses; ++c) {
    if (logits) logits[(size_t)row * kClasses + c] = z[c];
    finite = finite && isfinite(z[c]);
    dzr[c] = 0.f;
  }
  if (!finite) atomicOr(err, DEVERR_NONFINITE);
  if (!labelled) return 0.f;
  float m = z[0];
#pragma unroll
  for (int c = 1; c < kClasses; ++c) m = fmaxf(m, z[c]);
  float e[kClasses], sum = 0.f;
#pragma unroll
  for (int c = 0; c < kClasses; ++c) {
    e[c] = expf(z[c] - m);
    sum += e[c];
  }
  const float inv = 1.f / sum;
  float zy = 0.f;
#pragma unroll
  for (int c = 0; c < kClasses; ++c) {
    const float p = e[c] * inv;
    dzr[c] = (p - (c == y ? 1.f : 0.f)) * inv_n;
    if (c == y) zy = z[c];
    if (dz) dz[(size_t)row * kClasses + c] = dzr[c];
  }
  return (m + logf(sum)) - zy;
}

// Number of feature splits of width `split`: segment k has ceil(F_k / split).
__host__ __device__ inline int head_splits(const int* F, int nseg, int split) {
  int S = 0;
  for (int k = 0; k < nseg; ++k) S += (F[k] + split - 1) / split;
  return S;
}

// Split width of the logits kernels for n rows: the widest (kSplit features,
// bf16 kMmaSplit), halved (down to 128, bf16 256) while the grid would cover
// less than half the SMs, so that few rows are spread over the SMs by
// features.
int dot_split(const int* F, int nseg, int n, int es) {
  const int ch = es == 2 ? 256 : 128;
  const long long rb = (n + kDotRows - 1) / kDotRows;
  int split = es == 2 ? kMmaSplit : kSplit;
  while (split > ch && head_splits(F, nseg, split) * rb < kDotMinBlocks) split /= 2;
  return split;
}

// Floats of partial logits k_head_dot writes for any row count up to `rows`.
size_t zpart_floats(const int* F, int nseg, int rows, int es) {
  size_t mx = 0;
  for (int rb = 1; (rb - 1) * kDotRows < rows; ++rb) {
    const int n = rb * kDotRows < rows ? rb * kDotRows : rows;
    const size_t z = (size_t)head_splits(F, nseg, dot_split(F, nseg, n, es)) * n * kClasses;
    if (z > mx) mx = z;
  }
  return mx;
}

// What the last block of a row block needs to finish its rows: the bias,
// labels (null: logits only), outputs, the head's step counter (advanced by
// row block 0 when training) and one arrival counter per row block (zero
// between launches; the finishing block resets it).
struct FinishArgs {
  const float* cb;
  const int* labels;
  float inv_n;
  float* logits;  // [n, 10] or null
  int* pred;      // [n] or null: the class with the largest logit, the lowest on ties
  float* dz;      // [n, 10] or null
  float* part;    // [row blocks, 11] or null
  uint4* dzfrag;  // [segment][16-row group][part][lane]: A operands of k_head_wgrad_adam, or null
  ff_dev_state* ds;
  float beta1, beta2;
  int* counter;
  int S;          // blocks (splits) per row block
};

// ------------------------------------------------ bf16 activities: tensor cores
// The head's two contractions are thin (10 classes) and latency-bound: 1024
// rows of 6000 features are 12 MB of activity from L2 and 0.06 GFLOP each.
// They run as warp-level m16n8k16 MMAs fed straight from L2: a 128-row
// tcgen05 tile would leave most SMs idle and wait on TMEM and barrier set-up.
// The fp32 operand (V, or dz times the row scale) enters as three bf16 parts
// of 8 mantissa bits each, x = hi + mid + lo exactly, whose products with the
// activity are exact.  The tensor cores' running sum is not rounded to nearest:
// kept in it for a whole batch it drifted by 1.5e-6 of dV at 1024 rows and
// 1.9e-5 at 16384.  So only 32 features, or 16 rows with the small parts first,
// are summed there, and each such sum is added to fp32 registers with rounded
// adds (mma_add).
__device__ __forceinline__ void split3(float x, bf16 (&p)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float top = __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
    p[i] = __float2bfloat16_rn(top);  // exact
    x = isfinite(top) ? __fsub_rn(x, top) : 0.f;
  }
}
__device__ __forceinline__ uint32_t pack_bf16(bf16 lo, bf16 hi) {
  const __nv_bfloat162 v = __halves2bfloat162(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// The end of every logits block (256 threads) of row block blockIdx.y, rows
// rblk .. rblk + 63: the last of the row block's fa.S blocks to arrive forms
// its rows' logits from the splits' partials and finishes them.
__device__ __forceinline__ void finish_row_block(const Segs& sg, const float* __restrict__ zpart, int n, int rblk,
                                                 const FinishArgs& fa, int* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Every block arrives (an aborted one too, so that the counter is reset);
  // the last of the row block's S blocks finishes its rows.
  __shared__ int last;
  __shared__ float fred[kDotRows / 32][kPart];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(fa.counter + blockIdx.y, 1) == fa.S - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) {
    fa.counter[blockIdx.y] = 0;
    if (blockIdx.y == 0 && fa.labels && fa.ds) {
      // this step's Adam counter and bias corrections, read by k_head_adam
      fa.ds->t += 1;
      fa.ds->pow1 *= (double)fa.beta1;
      fa.ds->pow2 *= (double)fa.beta2;
      fa.ds->bc1 = (float)(1.0 - fa.ds->pow1);
      fa.ds->bc2 = (float)(1.0 - fa.ds->pow2);
    }
  }
  // z = c + the splits' partials in split order, a thread per row and class
  // (read past L1: other blocks wrote them during this launch), sixteen splits'
  // loads in flight at a time
  __shared__ float zs[kDotRows][kClasses];
  // the segments' row scales and the labels, loaded beside the partials
  __shared__ float ss[kMaxSegs][kDotRows];
  __shared__ int ys[kDotRows];
  {
    constexpr int NI = (kDotRows * kClasses + 255) / 256, SP = 16;
    const int items = min(kDotRows, n - rblk) * kClasses;
    const float* zp = zpart + (size_t)rblk * kClasses + threadIdx.x;
    const size_t zs_stride = (size_t)n * kClasses;
    float z[NI], v[NI][SP];
    auto load = [&](int sp0) {
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int u = 0; u < SP; ++u)
          v[i][u] = sp0 + u < fa.S && (int)threadIdx.x + i * 256 < items ? __ldcg(zp + i * 256 + (sp0 + u) * zs_stride)
                                                                         : 0.f;
    };
    load(0);
#pragma unroll
    for (int i = 0; i < NI; ++i) z[i] = __ldg(fa.cb + (threadIdx.x + i * 256) % kClasses);
    if (fa.dzfrag)
      for (int u = threadIdx.x; u < sg.nseg * kDotRows; u += 256) {
        const int k = u / kDotRows, r = u % kDotRows;
        ss[k][r] = rblk + r < n ? (sg.s[k] ? __ldg(sg.s[k] + rblk + r) : 1.f) : 0.f;
      }
    if (fa.labels && threadIdx.x < kDotRows && rblk + (int)threadIdx.x < n)
      ys[threadIdx.x] = __ldg(fa.labels + rblk + threadIdx.x);
    for (int sp0 = 0;;) {
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int u = 0; u < SP; ++u)
          if (sp0 + u < fa.S) z[i] += v[i][u];
      sp0 += SP;
      if (sp0 >= fa.S) break;
      load(sp0);
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if ((int)threadIdx.x + i * 256 < items) (&zs[0][0])[threadIdx.x + i * 256] = z[i];
  }
  __syncthreads();
  // a thread per row: softmax, loss and dz (left in zs too)
  if (threadIdx.x < kDotRows) {
    const int row = rblk + (int)threadIdx.x;
    float dzr[kClasses];
    float loss = 0.f;
#pragma unroll
    for (int c = 0; c < kClasses; ++c) dzr[c] = 0.f;
    if (row < n) {
      float z[kClasses];
#pragma unroll
      for (int c = 0; c < kClasses; ++c) z[c] = zs[threadIdx.x][c];
      if (fa.pred) {
        int best = 0;
        float bv = z[0];
#pragma unroll
        for (int c = 1; c < kClasses; ++c)
          if (z[c] > bv) {
            bv = z[c];
            best = c;
          }
        fa.pred[row] = best;
      }
      loss = finish_row(z, row, fa.labels != nullptr, fa.labels ? ys[threadIdx.x] : 0, fa.inv_n, fa.logits, fa.dz, dzr, err);
    }
    if (fa.part) {
      // the row block's sums of dz (for dc) and of the loss, in a fixed order
#pragma unroll
      for (int c = 0; c < kClasses; ++c) zs[threadIdx.x][c] = dzr[c];
#pragma unroll
      for (int c = 0; c < kClasses; ++c) dzr[c] = warp_sum(dzr[c]);
      loss = warp_sum(loss);
      if (lane == 0) {
#pragma unroll
        for (int c = 0; c < kClasses; ++c) fred[warp][c] = dzr[c];
        fred[warp][kClasses] = loss;
      }
    }
  }
  if (!fa.part) return;
  __syncthreads();
  if (threadIdx.x < kPart) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kDotRows / 32; ++w) t += fred[w][threadIdx.x];
    fa.part[(size_t)blockIdx.y * kPart + threadIdx.x] = t;
  }
  if (!fa.dzfrag) return;
  // dz times each segment's row scale as the weight gradient's A operands
  // (k_head_wgrad_adam): a lane's four words at a time; rows past n and
  // classes past 9 are zero
  const int groups = (n + 15) / 16;
  for (int u = threadIdx.x; u < sg.nseg * (kDotRows / 16) * 32; u += 256) {
    const int l = u & 31, gl = (u >> 5) % (kDotRows / 16), k = (u >> 5) / (kDotRows / 16);
    const int group = rblk / 16 + gl;
    if (group >= groups) continue;
    uint32_t w[3][4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      // a0: class < 8, slots 2t, 2t+1; a1: class >= 8; a2, a3: slots 8 further
      const int c = (l >> 2) + 8 * (a & 1), r = 16 * gl + 2 * (l & 3) + 8 * (a >> 1);
      bf16 x[2][3];
#pragma unroll
      for (int e = 0; e < 2; ++e) split3(c < kClasses ? zs[r + e][c] * ss[k][r + e] : 0.f, x[e]);
#pragma unroll
      for (int q = 0; q < 3; ++q) w[q][a] = pack_bf16(x[0][q], x[1][q]);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
      fa.dzfrag[(((size_t)k * groups + group) * 3 + q) * 32 + l] = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
  }
}

// fp32 activities.  One tensor map per segment: H_k as [n, ld_k] with 64-row
// boxes of 512 bytes (128 features), no swizzle.
struct HeadMaps {
  CUtensorMap m[kMaxSegs];
};

constexpr int kDotStages = 2;
constexpr int kDotStageBytes = kDotRows * 512;
constexpr int kDotSmem = kDotStages * kDotStageBytes + kSplit * kClasses * 4 + 64;

// zpart[split, row, c] = sum over the split's features f of s_k[row] H_k[row, f] V[c, off_k + f].
// One block per (split, 64 rows), eight rows per warp.  Thread 0 streams the
// split's 512-byte-wide row tiles of H_k into a two-stage shared-memory ring
// with TMA (mbarrier completion; a stage is refilled once all eight warps
// have arrived on its `empty` barrier); the split's slice of V sits in shared
// memory interleaved so that lane l's features (FPL consecutive ones per
// chunk) are read without bank conflicts.  Every wait is bounded.
__global__ void __launch_bounds__(256, 1) k_head_dot(const __grid_constant__ HeadMaps maps, Segs sg, int split, int n,
                                                     const float* __restrict__ V, float* __restrict__ zpart,
                                                     FinishArgs fa, int* err) {
  constexpr int CH = 512 / 4;  // features per chunk
  constexpr int FPL = CH / 32;              // features per lane
  constexpr int NCH = kSplit / CH;          // chunks in the widest split
  extern __shared__ __align__(128) uint8_t dsm[];
  uint8_t* ring = dsm;
  float* Vs = reinterpret_cast<float*>(dsm + kDotStages * kDotStageBytes);
  uint64_t* full = reinterpret_cast<uint64_t*>(Vs + NCH * kClasses * CH);
  uint64_t* empty = full + kDotStages;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + kDotStages);
  volatile int* never_set = abort_flag + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int k = 0, sp = blockIdx.x;
  while (k + 1 < sg.nseg && sp >= (sg.F[k] + split - 1) / split) {
    sp -= (sg.F[k] + split - 1) / split;
    ++k;
  }
  const int off = sg.off[k];
  const int fs = sp * split;
  const int fe = min(fs + split, sg.F[k]);
  const int nch = (fe - fs + CH - 1) / CH;
  const int rblk = blockIdx.y * kDotRows;
  const CUtensorMap* map = &maps.m[k];
  int issued = 0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kDotStages; ++i) {
      ptx::mbar_init(&full[i], 1);
      ptx::mbar_init(&empty[i], 8);
    }
    *abort_flag = 0;
    *never_set = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(map);
  }
  __syncthreads();
  ptx::griddep_wait();  // launched with programmatic stream serialization
  if (threadIdx.x == 0) {
    for (; issued < kDotStages && issued < nch; ++issued) {
      if (!ff_dcheck(tma_x_aligned(fs + issued * CH, 4), err)) {
        *abort_flag = 1;
        break;
      }
      ptx::mbar_arrive_expect_tx(&full[issued], kDotStageBytes);
      ptx::tma_load_2d(ring + issued * kDotStageBytes, map, &full[issued], fs + issued * CH, rblk);
    }
  }
  // the split's slice of V, zero past the segment
  for (int idx = threadIdx.x; idx < nch * kClasses * CH; idx += 256) {
    const int ch = idx / (kClasses * CH), rem = idx % (kClasses * CH);
    const int c = rem / CH, j = rem % CH;
    const int f = fs + ch * CH + j;
    Vs[((ch * kClasses + c) * FPL + j % FPL) * 32 + j / FPL] = f < fe ? __ldg(V + (size_t)c * sg.F_total + off + f) : 0.f;
  }
  const int r0 = rblk + warp * 8;
  float srow[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) srow[r] = (r0 + r < n) ? (sg.s[k] ? __ldg(sg.s[k] + r0 + r) : 1.f) : 0.f;
  __syncthreads();
  float acc[8][kClasses];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < kClasses; ++c) acc[r][c] = 0.f;
  for (int ch = 0; ch < nch; ++ch) {
    const int s = ch % kDotStages;
    const uint32_t ph = (uint32_t)(ch / kDotStages) & 1u;
    if (!ptx::mbar_wait(&full[s], ph, kWaitTimeoutNs, abort_flag)) {
      *abort_flag = 1;
      atomicOr(err, DEVERR_TIMEOUT);
      break;
    }
    const uint8_t* tile = ring + s * kDotStageBytes;
    const float* vch = Vs + ch * kClasses * FPL * 32;
    // the warp's 8 rows of this chunk (scaled by s_k), then every V value
    // read once from shared memory serves all 8 rows
    float h[8][FPL];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint8_t* rowp = tile + (warp * 8 + r) * 512 + lane * 16;
      const float4 q = *reinterpret_cast<const float4*>(rowp);
      h[r][0] = q.x * srow[r];
      h[r][1] = q.y * srow[r];
      h[r][2] = q.z * srow[r];
      h[r][3] = q.w * srow[r];
    }
#pragma unroll
    for (int c = 0; c < kClasses; ++c)
#pragma unroll
      for (int e = 0; e < FPL; ++e) {
        const float v = vch[(c * FPL + e) * 32 + lane];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r][c] = fmaf(h[r][e], v, acc[r][c]);
      }
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&empty[s]);
    if (threadIdx.x == 0 && issued < nch) {
      // stage s is refilled with chunk `issued` (= ch + kDotStages) once every warp is done with it
      if (!ptx::mbar_wait(&empty[s], ph, kWaitTimeoutNs, abort_flag)) {
        *abort_flag = 1;
        atomicOr(err, DEVERR_TIMEOUT);
        break;
      }
      if (!ff_dcheck(tma_x_aligned(fs + issued * CH, 4), err)) {
        *abort_flag = 1;
        break;
      }
      ptx::mbar_arrive_expect_tx(&full[s], kDotStageBytes);
      ptx::tma_load_2d(ring + s * kDotStageBytes, map, &full[s], fs + issued * CH, rblk);
      ++issued;
    }
  }
  if (*abort_flag) {
    // copies already issued land before the block's shared memory goes away
    if (threadIdx.x == 0)
      for (int ch = issued - kDotStages < 0 ? 0 : issued - kDotStages; ch < issued; ++ch)
        ptx::mbar_wait(&full[ch % kDotStages], (uint32_t)(ch / kDotStages) & 1u, 10000000ull, never_set);
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < kClasses; ++c) acc[r][c] = warp_sum(acc[r][c]);
    // lane c writes class c of the warp's rows
#pragma unroll
    for (int c = 0; c < kClasses; ++c) {
      if (lane != c) continue;
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r0 + r < n) zpart[((size_t)blockIdx.x * n + r0 + r) * kClasses + c] = acc[r][c];
    }
  }
  finish_row_block(sg, zpart, n, rblk, fa, err);
}

// zpart as k_head_dot writes it, from bf16 activities.  A block takes 64 rows
// x one split of at most 512 features: warp w the 16 rows 16 (w % 4) .. and
// half w / 4 of the split.  A lane's 16-byte load of a row (8 features) feeds
// the K slots of two MMAs, so K runs in a permuted order that the staged V
// parts follow.  The three parts of the 10 classes are 30 of 32 columns: four
// MMA tiles a K step (six, with a part's classes padded to 16, took a third
// longer: the MMAs' own rate counts here).  Bound by a chain of round trips
// (loads, partials, arrival, the finishing block's loads), so each phase
// issues all of its loads before it uses one.
// 1024 rows x 6000 features: 192 blocks (see dot_split), 12.1 us with labels,
// 9.0 without; 14.1 and 11.2 with padded parts and V loaded a unit at a time.
constexpr int kMmaLd = 40;  // floats of a row of the halves' sums: no bank conflicts
int mma_smem(int split) { return std::max(split / 16 * 2 * 32 * 16, 2 * kDotRows * kMmaLd * 4); }

__global__ void __launch_bounds__(256, 2) k_head_dot_mma(Segs sg, int split, int n, const float* __restrict__ V,
                                                      float* __restrict__ zpart, FinishArgs fa, int* err) {
  extern __shared__ __align__(16) uint4 vfrag[];  // [K step of 16][column tiles 0-1, 2-3][lane]: b0, b1 of either tile
  __shared__ float rs[kDotRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  int k = 0, sp = blockIdx.x;
  while (k + 1 < sg.nseg && sp >= (sg.F[k] + split - 1) / split) {
    sp -= (sg.F[k] + split - 1) / split;
    ++k;
  }
  const bf16* H = static_cast<const bf16*>(sg.H[k]);
  const int ld = sg.ld[k];
  const int fs = sp * split, fe = min(fs + split, sg.F[k]);
  const int rblk = blockIdx.y * kDotRows;
  ptx::griddep_wait();  // launched with programmatic stream serialization
  // The split's V: unit u (block of 32 features, class, quarter) is 8 features
  // of one class.  All of a thread's loads are issued first, without branches
  // between them, then its rows' activities; V is split while those arrive.
  constexpr int NU = (kMmaSplit / 32 * 4 * kClasses + 255) / 256;
  const int units = split / 32 * 4 * kClasses;
  const float* Vk = V + sg.off[k];
  const bool vec = ((sg.F_total | sg.off[k] | sg.F[k]) & 3) == 0;  // V itself is 256-byte aligned
  float v[NU][8];
#pragma unroll
  for (int i = 0; i < NU; ++i) {
    const int u = threadIdx.x + 256 * i, r = u >> 2;
    const int c = r % kClasses, f = fs + 32 * (r / kClasses) + 8 * (u & 3);
    const float* vp = Vk + (size_t)c * sg.F_total + f;
    if (vec) {
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 lo = u < units && f < fe ? __ldg(reinterpret_cast<const float4*>(vp)) : z;
      const float4 hi = u < units && f + 4 < fe ? __ldg(reinterpret_cast<const float4*>(vp) + 1) : z;
      v[i][0] = lo.x; v[i][1] = lo.y; v[i][2] = lo.z; v[i][3] = lo.w;
      v[i][4] = hi.x; v[i][5] = hi.y; v[i][6] = hi.z; v[i][7] = hi.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[i][e] = u < units && f + e < fe ? __ldg(vp + e) : 0.f;
    }
  }
  const float scale = threadIdx.x < kDotRows && rblk + (int)threadIdx.x < n && sg.s[k]
                          ? __ldg(sg.s[k] + rblk + threadIdx.x) : 1.f;
  // this warp's rows over its half of the split, 8 features a lane and row
  constexpr int NB = kMmaSplit / 2 / 32;  // blocks of 32 features per warp
  const int half = split / 2;             // a multiple of 32
  const int f0 = fs + (warp >> 2) * half + 8 * t;
  const int ra = rblk + (warp & 3) * 16 + g, rb = ra + 8;
  uint4 ha[NB], hb[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    // rows are padded to whole 8-feature words, the padding zero
    const bool ok = 32 * i < half && f0 + 32 * i < fe;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    ha[i] = ok && ra < n ? __ldg(reinterpret_cast<const uint4*>(H + (size_t)ra * ld + f0 + 32 * i)) : z;
    hb[i] = ok && rb < n ? __ldg(reinterpret_cast<const uint4*>(H + (size_t)rb * ld + f0 + 32 * i)) : z;
  }
  // V as B operands: part q of class c is column 10 q + c of 32 (30 and 31 are
  // never read)
#pragma unroll
  for (int i = 0; i < NU; ++i) {
    const int u = threadIdx.x + 256 * i, ut = u & 3, r = u >> 2, c = r % kClasses, b = r / kClasses;
    if (u >= units) break;
    bf16 p[8][3];
#pragma unroll
    for (int e = 0; e < 8; ++e) split3(v[i][e], p[e]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int col = kClasses * q + c;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        uint2* dst = reinterpret_cast<uint2*>(&vfrag[((2 * b + s) * 2 + (col >> 4)) * 32 + (col & 7) * 4 + ut]) + ((col >> 3) & 1);
        *dst = make_uint2(pack_bf16(p[4 * s][q], p[4 * s + 1][q]), pack_bf16(p[4 * s + 2][q], p[4 * s + 3][q]));
      }
    }
  }
  if (threadIdx.x < kDotRows) rs[threadIdx.x] = scale;
  __syncthreads();
  float d[4][4] = {};  // column tile
  const uint4* vf = vfrag + (warp >> 2) * (half / 16) * 2 * 32 + lane;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    if (32 * i >= half) break;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint4 v0 = vf[(2 * i * 2 + j) * 32], v1 = vf[((2 * i + 1) * 2 + j) * 32];
      float t0[4] = {}, t1[4] = {};
      mma16816(t0, ha[i].x, hb[i].x, ha[i].y, hb[i].y, v0.x, v0.y);
      mma16816(t1, ha[i].x, hb[i].x, ha[i].y, hb[i].y, v0.z, v0.w);
      mma16816(t0, ha[i].z, hb[i].z, ha[i].w, hb[i].w, v1.x, v1.y);
      mma16816(t1, ha[i].z, hb[i].z, ha[i].w, hb[i].w, v1.z, v1.w);
      mma_add(d[2 * j], t0);
      mma_add(d[2 * j + 1], t1);
    }
  }
  __syncthreads();  // the operands' memory takes the sums
  float* red = reinterpret_cast<float*>(vfrag);  // [half][row][column], rows of kMmaLd floats
  const int lr = (warp & 3) * 16 + g;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int r = 0; r < 2; ++r)
      *reinterpret_cast<float2*>(&red[((warp >> 2) * kDotRows + lr + 8 * r) * kMmaLd + 8 * j + 2 * t]) =
          make_float2(d[j][2 * r], d[j][2 * r + 1]);
  __syncthreads();
  // a thread per row and class: the small parts first, times the row scale
  for (int i = threadIdx.x; i < kDotRows * kClasses; i += 256) {
    const int row = i / kClasses, c = i % kClasses;
    const float *a = red + row * kMmaLd + c, *b = a + kDotRows * kMmaLd;
    const float lo = a[2 * kClasses] + b[2 * kClasses], mid = a[kClasses] + b[kClasses], hi = a[0] + b[0];
    if (rblk + row < n) zpart[((size_t)blockIdx.x * n + rblk) * kClasses + i] = rs[row] * (lo + mid + hi);
  }
  finish_row_block(sg, zpart, n, rblk, fa, err);
}

// dV partials of one 128-row block for one 128-feature chunk of one segment:
// dVpart[rb, c, f] = sum over the block's rows i of dz[i, c] s_k[i] H_k[i, f].
// Eight warps take 16 rows each (lane = 4 features); the eight partial sums
// are added in warp order.
__global__ void __launch_bounds__(256) k_head_wgrad(Segs sg, int n, const float* __restrict__ dz,
                                                    float* __restrict__ dVpart) {
  __shared__ float dzs[kWgRows][kClasses];
  __shared__ float red[8][kClasses][kWgChunk];
  ptx::griddep_wait();  // launched with programmatic stream serialization
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // segment and chunk of this block
  int k = 0, chunk = blockIdx.x;
  while (k + 1 < sg.nseg && chunk >= (sg.F[k] + kWgChunk - 1) / kWgChunk) {
    chunk -= (sg.F[k] + kWgChunk - 1) / kWgChunk;
    ++k;
  }
  const float* H = static_cast<const float*>(sg.H[k]);
  const int ld = sg.ld[k], Fk = sg.F[k], off = sg.off[k];
  const int f0 = chunk * kWgChunk;
  const int rb0 = blockIdx.y * kWgRows;
  for (int idx = threadIdx.x; idx < kWgRows * kClasses; idx += 256) {
    const int i = idx / kClasses, c = idx % kClasses;
    const int row = rb0 + i;
    dzs[i][c] = row < n ? __ldg(dz + (size_t)row * kClasses + c) * (sg.s[k] ? __ldg(sg.s[k] + row) : 1.f) : 0.f;
  }
  __syncthreads();
  float acc[kClasses][4];
#pragma unroll
  for (int c = 0; c < kClasses; ++c)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[c][e] = 0.f;
  const int f = f0 + 4 * lane;
#pragma unroll 4
  for (int i = warp * (kWgRows / 8); i < (warp + 1) * (kWgRows / 8); ++i) {
    float h[4];
    load_feats4(H, ld, rb0 + i, n, f, Fk, h);
#pragma unroll
    for (int c = 0; c < kClasses; ++c) {
      const float d = dzs[i][c];
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[c][e] = fmaf(d, h[e], acc[c][e]);
    }
  }
#pragma unroll
  for (int c = 0; c < kClasses; ++c)
#pragma unroll
    for (int e = 0; e < 4; ++e) red[warp][c][4 * lane + e] = acc[c][e];
  __syncthreads();
  for (int idx = threadIdx.x; idx < kClasses * kWgChunk; idx += 256) {
    const int c = idx / kWgChunk, j = idx % kWgChunk;
    if (f0 + j >= Fk) continue;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += red[w][c][j];
    dVpart[((size_t)blockIdx.y * kClasses + c) * sg.F_total + off + f0 + j] = v;
  }
}

// ------------------------------------------ Performance-Optimized layer (§4)
// The gradient that a layer's softmax block sends back into the layer, one
// block per 32 rows x 256 columns (block 32 x 8; thread (x, y) owns columns
// 8x..8x+7 of rows y, y+8, y+16, y+24):
//   dZ_ij = (sum_c dz_ic V_cj) [h_ij > 0],  G_ij = s_i dZ_ij (weight-gradient
//   operand, in the activity type),  db partials = sum over the block's rows,
//   and the block's own weight-gradient partials dV_cj = sum_i dz_ic h_ij
//   over the same rows (the block reads the raw activity).
// V (before this step's update) and dz are staged in shared memory.  Lead
// blocks (x == 0) also write the next layer's row scale from the forward's
// goodness partials; block (0, 0) advances the layer's Adam step.
// With zpart set (bf16 layers), dz is not given: the forward GEMM wrote the
// block's partial logits, and every block finishes its own rows from them
// (bias + partials in tile order, softmax, cross-entropy; the blocks of a row
// block compute identical values); lead blocks then write the row block's dz
// and loss sums, and block (0, 0) also advances the block's Adam step.
// Bound by its chain of round trips (partials, softmax, dV, db), not by
// memory (1024 x 2000 bf16: 8.2 MB).  dV rows stored as octets and db summed
// by the whole block: 13.9 -> 11.6 us, an epoch of the 2000x4 network at
// batch 1024 1576 -> 1552 us.
struct PoGradArgs {
  const float* dz;      // [n, 10], or null with zpart
  const float* zpart;   // [zt, n, 10] partial logits, or null
  int zt;
  const float* cb;      // [10] block bias
  const int* labels;    // [n]
  float inv_n;
  float* part;          // [row blocks, 11]: sums of dz and of the loss (with zpart)
  ff_dev_state* hds;    // the block's Adam state (with zpart)
  float hbeta1, hbeta2;
  const float* V;       // [10, N] (before this step's update)
  const float* s;       // [n] row scale of the layer input
  const float* gpart;   // forward goodness partials [ntiles, n]
  int ntiles, n, N, ld;
  float* s_next;        // [n] or null
  float* dbpart;        // [row blocks, N]
  float* dVpart;        // [row blocks, 10, N]: the block's dV partials
  ff_dev_state* ds;     // the layer's
  float beta1, beta2;
  int* err;
};

constexpr int kPoRows = 32;

template <typename T>
__global__ void __launch_bounds__(256) k_po_grad(PoGradArgs a, const T* __restrict__ H, T* __restrict__ G) {
  __shared__ __align__(16) float Vsh[kClasses][2][32][4];  // V[c][c0 + 8 l + 4 q + e] at [c][q][l][e]
  __shared__ float dzs[kPoRows][kClasses];
  // the block's activity tile in its own type (for the dV partials), then
  // the db reduction in the same memory
  __shared__ __align__(16) T Hs[kPoRows][256 + 8];
  static_assert(sizeof(Hs) >= 8 * (256 + 4) * sizeof(float), "the db reduction fits in the tile's memory");
  const int r0 = blockIdx.y * kPoRows;
  const int lane = threadIdx.x, tid = threadIdx.y * 32 + threadIdx.x;
  const int c0 = blockIdx.x * 256;
  const int cg = c0 + lane * 8;
  const bool cols_ok = cg < a.ld;
  ptx::griddep_wait();  // launched with programmatic stream serialization
  // this thread's activity (rows y, y+8, y+16, y+24; 8 columns) and its rows'
  // scales, loaded first so that their latency overlaps the logits and softmax
  float hv[4][8], sr[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = r0 + threadIdx.y + 8 * k;
    sr[k] = i < a.n ? __ldg(a.s + i) : 0.f;
    if (cols_ok && i < a.n) {
      Vec8<T>::load(H + (size_t)i * a.ld + cg, hv[k]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) hv[k][e] = 0.f;
    }
  }
  for (int idx = tid; idx < kClasses * 256; idx += 256) {
    const int c = idx / 256, j = idx % 256;
    Vsh[c][(j >> 2) & 1][j >> 3][j & 3] = (c0 + j < a.N) ? __ldg(a.V + (size_t)c * a.N + c0 + j) : 0.f;
  }
  if (a.zpart) {
    // logits of the block's rows: thread per (row, class), partials in tile
    // order, both of a thread's sums and 8 partials each in flight together
    constexpr int NI = (kPoRows * kClasses + 255) / 256;
    const int items = min(kPoRows, a.n - r0) * kClasses;
    const float* zp = a.zpart + (size_t)r0 * kClasses + tid;
    const size_t stride = (size_t)a.n * kClasses;
    float z[NI] = {};
    for (int t0 = 0; t0 < a.zt; t0 += 8) {
      float v[NI][8];
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[i][u] = t0 + u < a.zt && tid + 256 * i < items ? __ldg(zp + 256 * i + (t0 + u) * stride) : 0.f;
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (t0 + u < a.zt) z[i] += v[i][u];
    }
    const int y = threadIdx.y == 0 && r0 + lane < a.n ? __ldg(a.labels + r0 + lane) : 0;
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (tid + 256 * i < kPoRows * kClasses)
        (&dzs[0][0])[tid + 256 * i] =
            tid + 256 * i < items ? __ldg(a.cb + (tid + 256 * i) % kClasses) + z[i] : 0.f;
    __syncthreads();
    if (threadIdx.y == 0) {
      // warp 0: softmax, loss and dz of row r0 + lane, in place
      float z[kClasses], dzr[kClasses];
#pragma unroll
      for (int c = 0; c < kClasses; ++c) z[c] = dzs[lane][c];
      float loss = 0.f;
      if (r0 + lane < a.n) {
        loss = finish_row(z, r0 + lane, true, y, a.inv_n, nullptr, nullptr, dzr, &a.hds->err);
      } else {
#pragma unroll
        for (int c = 0; c < kClasses; ++c) dzr[c] = 0.f;
      }
#pragma unroll
      for (int c = 0; c < kClasses; ++c) dzs[lane][c] = dzr[c];
      if (blockIdx.x == 0) {
        // the row block's sums of dz (for dc) and of the loss, in a fixed order
#pragma unroll
        for (int c = 0; c < kClasses; ++c) dzr[c] = warp_sum(dzr[c]);
        loss = warp_sum(loss);
        if (lane < kPart) {
          float t = loss;
#pragma unroll
          for (int c = 0; c < kClasses; ++c)
            if (lane == c) t = dzr[c];
          a.part[(size_t)blockIdx.y * kPart + lane] = t;
        }
        if (blockIdx.y == 0 && lane == 0) {
          a.hds->t += 1;
          a.hds->pow1 *= (double)a.hbeta1;
          a.hds->pow2 *= (double)a.hbeta2;
          a.hds->bc1 = (float)(1.0 - a.hds->pow1);
          a.hds->bc2 = (float)(1.0 - a.hds->pow2);
        }
      }
    }
  } else {
    for (int idx = tid; idx < kPoRows * kClasses; idx += 256) {
      const int i = idx / kClasses, c = idx % kClasses;
      dzs[i][c] = (r0 + i < a.n) ? __ldg(a.dz + (size_t)(r0 + i) * kClasses + c) : 0.f;
    }
  }
  // beside warp 0's softmax: warp 1 the next layer's scales, warp 2 the step
  if (blockIdx.x == 0 && threadIdx.y == 1 && r0 + lane < a.n) {
    const float g = sum_partials(a.gpart, a.ntiles, a.n, r0 + lane);
    if (!isfinite(g)) atomicOr(a.err, DEVERR_NONFINITE);
    if (a.s_next) {
      const float r = sqrtf(g);
      a.s_next[r0 + lane] = r != r ? r : 1.f / fmaxf(r, 1e-12f);
    }
  }
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 64) {
    a.ds->t += 1;
    a.ds->pow1 *= a.beta1;
    a.ds->pow2 *= a.beta2;
    a.ds->bc1 = (float)(1.0 - a.ds->pow1);
    a.ds->bc2 = (float)(1.0 - a.ds->pow2);
  }
  __syncthreads();
  // d_ke = sum over the classes in order: a class's 8 weights are read once
  // for the thread's 4 rows (with a row's classes innermost the kernel was
  // bound by its 640 shared-memory reads a thread; now 60)
  float d[4][8];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int e = 0; e < 8; ++e) d[k][e] = 0.f;
#pragma unroll
  for (int c = 0; c < kClasses; ++c) {
    const float4 v0 = *reinterpret_cast<const float4*>(Vsh[c][0][lane]);
    const float4 v1 = *reinterpret_cast<const float4*>(Vsh[c][1][lane]);
    const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float z = dzs[threadIdx.y + 8 * k][c];
#pragma unroll
      for (int e = 0; e < 8; ++e) d[k][e] = fmaf(z, v[e], d[k][e]);
    }
  }
  float db[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) db[e] = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int li = threadIdx.y + 8 * k;
    const int i = r0 + li;
    Vec8<T>::store(&Hs[li][lane * 8], hv[k]);
    if (!cols_ok || i >= a.n) continue;
    float z[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float t = hv[k][e] > 0.f ? d[k][e] : 0.f;
      db[e] += t;
      z[e] = sr[k] * t;
    }
    Vec8<T>::store(G + (size_t)i * a.ld + cg, z);
  }
  __syncthreads();
  // dV partials from the staged tile, each the block's 32 rows in order:
  // thread (x, y) sums class y over its 8 columns and, of classes 8 and 9, two
  // columns (64 (y % 4) + 2 x, + 1 of class 8 + y / 4)
  {
    const int y = threadIdx.y, c2 = 8 + (y >> 2), j2 = 64 * (y & 3) + 2 * lane;
    float dv[8], dw[2] = {0.f, 0.f};
#pragma unroll
    for (int e = 0; e < 8; ++e) dv[e] = 0.f;
#pragma unroll 4
    for (int li = 0; li < kPoRows; ++li) {
      const float d = dzs[li][y], d2 = dzs[li][c2];
      float h[8];
      Vec8<T>::load(&Hs[li][lane * 8], h);
      float h0, h1;
      if constexpr (sizeof(T) == 2) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&Hs[li][j2]));
        h0 = f.x;
        h1 = f.y;
      } else {
        h0 = Hs[li][j2];
        h1 = Hs[li][j2 + 1];
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) dv[e] = fmaf(d, h[e], dv[e]);
      dw[0] = fmaf(d2, h0, dw[0]);
      dw[1] = fmaf(d2, h1, dw[1]);
    }
    float* out = a.dVpart + (size_t)blockIdx.y * kClasses * a.N;
    if ((a.N & 7) == 0) {  // whole octets, rows 16-byte aligned
      if (cg < a.N) Vec8<float>::store(out + (size_t)y * a.N + cg, dv);
      if (c0 + j2 < a.N) *reinterpret_cast<float2*>(out + (size_t)c2 * a.N + c0 + j2) = make_float2(dw[0], dw[1]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (cg + e < a.N) out[(size_t)y * a.N + cg + e] = dv[e];
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (c0 + j2 + e < a.N) out[(size_t)c2 * a.N + c0 + j2 + e] = dw[e];
    }
  }
  __syncthreads();
  // db partials: the eight row groups added in order, through the tile's memory
  float (*red)[256 + 4] = reinterpret_cast<float (*)[256 + 4]>(&Hs[0][0]);
  Vec8<float>::store(&red[threadIdx.y][lane * 8], db);
  __syncthreads();
  const int j = c0 + tid;
  float t = 0.f;
#pragma unroll
  for (int y = 0; y < 8; ++y) t += red[y][tid];
  if (j < a.N) a.dbpart[(size_t)blockIdx.y * a.N + j] = t;
}

struct HeadAdamArgs {
  float *V, *mV, *vV, *c, *mc, *vc;
  const float* dVpart;  // [nrb, 10, F]
  int nrb, F;
  const float* part;    // [nlb, 11]
  int nlb;
  float inv_n;
  float lr, beta1, beta2, eps;
  const ff_dev_state* ds;
  float* loss_out;
  float* dV_out;        // [10, F] or null
  float* dc_out;        // [10] or null
};


// One Adam step of one element of V, and its gradient kept.
__device__ __forceinline__ void head_adam_v(const HeadAdamArgs& a, int idx, float g, float a1, float r2) {
  if (a.dV_out) a.dV_out[idx] = g;
  float w = a.V[idx], m = a.mV[idx], v = a.vV[idx];
  adam1(w, m, v, g, a1, a.beta1, a.beta2, a.eps, r2);
  a.V[idx] = w;
  a.mV[idx] = m;
  a.vV[idx] = v;
}

// The 10 biases and the loss, by one block of 256 threads (warp w: columns w
// and w + 8 of the partials, column 10 being the loss).
__device__ __forceinline__ void head_adam_c(const HeadAdamArgs& a, float a1, float r2) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int col = warp; col < kPart; col += 8) {
    float t = 0.f;
    for (int b = lane; b < a.nlb; b += 32) t += __ldg(a.part + (size_t)b * kPart + col);
    t = warp_sum(t);
    if (lane != 0) continue;
    if (col == kClasses) {
      if (a.loss_out) a.loss_out[0] = t * a.inv_n;
      continue;
    }
    if (a.dc_out) a.dc_out[col] = t;
    float w = a.c[col], m = a.mc[col], v = a.vc[col];
    adam1(w, m, v, t, a1, a.beta1, a.beta2, a.eps, r2);
    a.c[col] = w;
    a.mc[col] = m;
    a.vc[col] = v;
  }
}

// Threads 0 .. 10F-1 of the grid own one V element each; the last block owns
// the 10 biases.
__global__ void __launch_bounds__(256) k_head_adam(HeadAdamArgs a) {
  ptx::griddep_wait();  // launched with programmatic stream serialization
  const float a1 = a.lr / a.ds->bc1, r2 = 1.f / a.ds->bc2;
  const int total = kClasses * a.F;
  const int vblocks = (total + 255) / 256;
  if ((int)blockIdx.x >= vblocks) {
    head_adam_c(a, a1, r2);
    return;
  }
  const int idx = blockIdx.x * 256 + threadIdx.x;
  // the row blocks' partials in order, eight loads in flight
  if (idx < total) head_adam_v(a, idx, sum_partials(a.dVpart, a.nrb, total, idx), a1, r2);
}

// The head's weight gradient and Adam of bf16 activities in one kernel: a
// block owns 32 features of one segment over all n rows (so its dV is
// complete: no partials through memory, no second launch), the last block the
// biases.  dV is 16 (classes) x 32 (features) per block, K = the rows: warp w
// takes every eighth group of 16 rows.  dz times the segment's row scale
// comes as A operands of three bf16 parts, written once by the logits
// kernel's finishing blocks; the activity is loaded as 8 bytes of four rows
// per lane -- 64 contiguous bytes per row -- and pairs of rows are interleaved
// into B operands.  No staging: every load is independent of the others.
// 1024 rows x 6000 features: 8 us, bound by the latency of these loads and of
// Adam's state (issue slots 19 % active, tensor pipe 13 %).
constexpr int kWgaFeats = 32;

__global__ void __launch_bounds__(256, 2) k_head_wgrad_adam(Segs sg, int n, const uint4* __restrict__ dzfrag,
                                                         HeadAdamArgs a) {
  __shared__ float red[8][kClasses][kWgaFeats + 1];
  ptx::griddep_wait();  // launched with programmatic stream serialization
  const float a1 = a.lr / a.ds->bc1, r2 = 1.f / a.ds->bc2;
  if (blockIdx.x + 1 == gridDim.x) {
    head_adam_c(a, a1, r2);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  int k = 0, chunk = blockIdx.x;
  while (k + 1 < sg.nseg && chunk >= (sg.F[k] + kWgaFeats - 1) / kWgaFeats) {
    chunk -= (sg.F[k] + kWgaFeats - 1) / kWgaFeats;
    ++k;
  }
  const bf16* H = static_cast<const bf16*>(sg.H[k]);
  const int ld = sg.ld[k], Fk = sg.F[k], off = sg.off[k];
  const int f0 = chunk * kWgaFeats;
  // rows are padded to whole 8-feature words, the padding zero
  const bool f_ok = f0 + 4 * g < ld;
  const int groups = (n + 15) / 16;
  const uint4* df = dzfrag + (size_t)k * groups * 3 * 32 + lane;
  float d[4][4] = {};  // feature f0 + 4 (column) + j of column tile j
#pragma unroll 4
  for (int gr = warp; gr < groups; gr += 8) {
    const int row = gr * 16 + 2 * t;
    uint2 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = row + (e & 1) + (e >> 1) * 8;
      h[e] = f_ok && r < n ? __ldg(reinterpret_cast<const uint2*>(H + (size_t)r * ld + f0 + 4 * g)) : make_uint2(0u, 0u);
    }
    uint4 av[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) av[q] = __ldg(df + (gr * 3 + q) * 32);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t sel = j & 1 ? 0x7632u : 0x5410u;
      const uint32_t b0 = __byte_perm(j < 2 ? h[0].x : h[0].y, j < 2 ? h[1].x : h[1].y, sel);
      const uint32_t b1 = __byte_perm(j < 2 ? h[2].x : h[2].y, j < 2 ? h[3].x : h[3].y, sel);
      float sum16[4] = {};
#pragma unroll
      for (int q = 2; q >= 0; --q) mma16816(sum16, av[q].x, av[q].y, av[q].z, av[q].w, b0, b1);
      mma_add(d[j], sum16);
    }
  }
  // the eight warps' sums in warp order, then Adam: a thread per element
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      red[warp][g][4 * (2 * t + e) + j] = d[j][e];
      if (g < kClasses - 8) red[warp][8 + g][4 * (2 * t + e) + j] = d[j][2 + e];
    }
  __syncthreads();
  for (int idx = threadIdx.x; idx < kClasses * kWgaFeats; idx += 256) {
    const int c = idx / kWgaFeats, j = idx % kWgaFeats;
    if (f0 + j >= Fk) continue;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += red[w][c][j];
    head_adam_v(a, c * a.F + off + f0 + j, v, a1, r2);
  }
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace
}  // namespace ff

// The head object behind the opaque handle.
struct ff_head {
  ff_head_config cfg;
  int F;
  int device;
  cudaStream_t last_stream;
  float *V, *c, *mV, *vV, *mc, *vc;  // one allocation: V, mV, vV [10, F]; c, mc, vc [10]
  float *dV, *dc;                    // gradient of the last train step [10, F], [10]
  ff::ff_dev_state* ds;
  void* ws;
  size_t ws_bytes;
  int* counters;    // k_head_dot arrival counters, one per 64-row block (zero between launches)
  int counter_cap;
  // ff_head_train_epoch: a second feature workspace and a side stream, so
  // that the next pass's neutral forward runs while the head steps read the
  // current one (created on first use)
  void* ws2;
  size_t ws2_bytes;
  cudaStream_t side;
  cudaEvent_t ev_start, ev_fwd[2], ev_use[2];
  // ff_po_train_step: the block's Adam on the side stream (fork, join)
  cudaEvent_t ev_fork, ev_join;
};

namespace ff {
namespace {

// Validates the layer chain for the head and describes its feature segments
// (without buffers).  Returns FF_OK or FF_ERR_INVALID_ARG.
ff_status head_layers(const ff_head* hd, ff_layer* const* layers, int n_layers) {
  if (!layers || n_layers < 1 || n_layers > kMaxSegs + 1) return FF_ERR_INVALID_ARG;
  int F = 0;
  for (int k = 0; k < n_layers; ++k) {
    if (!layers[k]) return FF_ERR_INVALID_ARG;
    if (layers[k]->is_bf16 != layers[0]->is_bf16) return FF_ERR_INVALID_ARG;
    if (k > 0 && layers[k]->K != layers[k - 1]->N) return FF_ERR_INVALID_ARG;
    if (k >= 1 || n_layers == 1) F += layers[k]->N;
  }
  if (layers[0]->K < kClasses) return FF_ERR_INVALID_ARG;
  if (F != hd->F) return FF_ERR_INVALID_ARG;
  return FF_OK;
}

struct HeadWork {
  void* X0;
  float* S[kMaxSegs + 2];   // S[k]: row scale of layer k's input (S[L]: of the last activity)
  void* Hk[kMaxSegs + 1];
  float* gpart;
  float* gpart2;   // the tensor-core forward alternates between gpart and gpart2
  float* zpart;
  float* dz;
  float* part;
  float* dVpart;   // fp32 layers
  uint4* dzfrag;   // bf16 layers
};

// Partial-logit floats for up to `rows` rows of the layer chain's segments.
size_t chain_zpart_floats(ff_layer* const* layers, int L, int rows) {
  int F[kMaxSegs + 1], nseg = 0;
  for (int k = (L == 1 ? 0 : 1); k < L; ++k) F[nseg++] = layers[k]->N;
  return zpart_floats(F, nseg, rows, layers[0]->is_bf16 ? 2 : 4);
}

// Carves the head's workspace for `rows` rows (grown on demand); buf 1: the
// second workspace of ff_head_train_epoch.
ff_status head_workspace(ff_head* hd, ff_layer* const* layers, int L, int rows, bool train, HeadWork* w,
                         int buf = 0) {
  void*& wsp = buf ? hd->ws2 : hd->ws;
  size_t& wsb = buf ? hd->ws2_bytes : hd->ws_bytes;
  const bool b16 = layers[0]->is_bf16;
  const size_t es = b16 ? 2 : 4;
  int ntmax = 0;
  for (int k = 0; k < L; ++k) {
    const int nt = b16 ? tc_fwd_ntiles_max(layers[k]->N) : f32_fwd_ntiles_max(layers[k]->N);
    if (nt > ntmax) ntmax = nt;
  }
  size_t off = 0;
  size_t oX = off; off += align256((size_t)rows * layers[0]->ldK * es);
  size_t oS[kMaxSegs + 2];
  for (int k = 0; k <= L; ++k) { oS[k] = off; off += align256((size_t)rows * 4); }
  size_t oH[kMaxSegs + 1];
  for (int k = 0; k < L; ++k) { oH[k] = off; off += align256((size_t)rows * layers[k]->ldN * es); }
  size_t oG = off; off += align256((size_t)ntmax * rows * 4);
  size_t oG2 = off; off += align256(b16 ? (size_t)ntmax * rows * 4 : 0);
  size_t oZP = off; off += align256(chain_zpart_floats(layers, L, rows) * 4);
  size_t oD = off; off += align256(train && !b16 ? (size_t)rows * kClasses * 4 : 0);
  const int nseg = L > 1 ? L - 1 : 1;
  size_t oF = off; off += align256(train && b16 ? (size_t)nseg * cdiv(rows, 16) * 3 * 32 * sizeof(uint4) : 0);
  size_t oP = off; off += align256(train ? (size_t)cdiv(rows, kDotRows) * kPart * 4 : 0);
  size_t oV = off; off += align256(train && !b16 ? (size_t)cdiv(rows, kWgRows) * kClasses * hd->F * 4 : 0);
  if (off > wsb) {
    FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync before head workspace growth");
    if (hd->side) FF_TRY(cudaStreamSynchronize(hd->side), "sync before head workspace growth");
    dev_free(wsp);
    wsp = nullptr;
    wsb = 0;
    FF_TRY(dev_alloc(&wsp, off), "head workspace");
    wsb = off;
  }
  char* base = static_cast<char*>(wsp);
  w->X0 = base + oX;
  for (int k = 0; k <= L; ++k) w->S[k] = reinterpret_cast<float*>(base + oS[k]);
  for (int k = 0; k < L; ++k) w->Hk[k] = base + oH[k];
  w->gpart = reinterpret_cast<float*>(base + oG);
  w->gpart2 = reinterpret_cast<float*>(base + (b16 ? oG2 : oG));
  w->zpart = reinterpret_cast<float*>(base + oZP);
  w->dz = train && !b16 ? reinterpret_cast<float*>(base + oD) : nullptr;
  w->dzfrag = train && b16 ? reinterpret_cast<uint4*>(base + oF) : nullptr;
  w->part = train ? reinterpret_cast<float*>(base + oP) : nullptr;
  w->dVpart = train ? reinterpret_cast<float*>(base + oV) : nullptr;
  return FF_OK;
}

// Neutral-labelled forward of `rows` raw input rows through every layer:
// H_k and the row scale of every activity.  narrow: the forward GEMMs may take
// 128-column tiles when their grid is small (predict); training keeps
// 256-column tiles at every row count, so that a row's goodness partials --
// and with them every activity scale -- do not depend on how many rows share
// the GEMM (ff_head_train_epoch runs many steps' rows at once); the fp32
// GEMMs then take the tile shape of kTrainPlanRows rows at any row count.
constexpr int kTrainPlanRows = 1024;
ff_status head_forward(ff_layer* const* layers, int L, const float* x, int rows, const HeadWork& w, int* err,
                       cudaStream_t st, bool narrow) {
  ff_layer* L0 = layers[0];
  const bool b16 = L0->is_bf16;
  const double es = b16 ? 2.0 : 4.0;
  FF_LAUNCH(K_OVERLAY, (double)rows * (L0->K * 4.0 + L0->ldK * es + 4), st,
            launch_overlay(x, nullptr, rows, L0->K, w.X0, L0->ldK, b16, w.S[0], 2, st), "neutral-label overlay");
  const void* in = w.X0;
  int nt_prev = 0;
  for (int k = 0; k < L; ++k) {
    ff_layer* Lk = layers[k];
    float* gpart = b16 && (k & 1) ? w.gpart2 : w.gpart;
    EpiArgs ep{w.S[k], Lk->cfg.has_bias ? Lk->b : nullptr, w.Hk[k], Lk->ldN, gpart};
    ep.narrow = narrow;
    int nt;
    if (b16) {
      if (k >= 1) {
        // layer k-1's activity scale S[k] comes from its goodness partials
        // inside this GEMM (no separate finalize)
        ep.row_scale = nullptr;
        ep.gpart_in = (k - 1) & 1 ? w.gpart2 : w.gpart;
        ep.ntiles_in = nt_prev;
        ep.s_out = w.S[k];
      }
      nt = tc_fwd_ntiles(rows, Lk->N, narrow);
      FF_LAUNCH(K_FWD_TC, 2.0 * rows * Lk->N * Lk->K, st,
                tc_gemm_fwd(static_cast<const bf16*>(in), Lk->ldK, Lk->Wb, Lk->ldK, rows, Lk->N, Lk->K, ep, err, st),
                "head forward GEMM (tcgen05)");
    } else {
      const int plan_rows = narrow ? rows : kTrainPlanRows;
      nt = f32_fwd_ntiles(plan_rows, Lk->N, Lk->K);
      const bool tc = f32_fwd_on_tensor_cores(static_cast<const float*>(in), Lk->ldK, Lk->W, Lk->K, plan_rows, Lk->N,
                                              Lk->K);
      FF_LAUNCH(tc ? K_FWD_F32TC : K_FWD_SIMT, 2.0 * rows * Lk->N * Lk->K, st,
                f32_gemm_fwd(static_cast<const float*>(in), Lk->ldK, Lk->W, Lk->K, rows, Lk->N, Lk->K, plan_rows, ep,
                             err, st),
                "head forward GEMM (fp32)");
    }
    nt_prev = nt;
    if (!b16 || k + 1 == L) {
      FinalizeArgs fa{};
      fa.gpart = gpart;
      fa.ntiles = nt;
      fa.M = rows;
      fa.s_next = w.S[k + 1];
      fa.err = err;
      FF_LAUNCH(K_FINALIZE, (double)rows * (nt * 4.0 + 4), st, launch_finalize(fa, st), "head activity scale");
    }
    in = w.Hk[k];
  }
  return FF_OK;
}

Segs make_segs(ff_layer* const* layers, int L, const HeadWork& w, int F) {
  Segs sg{};
  int off = 0, j = 0;
  for (int k = (L == 1 ? 0 : 1); k < L; ++k, ++j) {
    sg.H[j] = w.Hk[k];
    sg.s[j] = w.S[k + 1];
    sg.ld[j] = layers[k]->ldN;
    sg.F[j] = layers[k]->N;
    sg.off[j] = off;
    off += layers[k]->N;
  }
  sg.nseg = j;
  sg.F_total = F;
  return sg;
}

// One arrival counter per 64-row block of k_head_dot, all zero (grown on
// demand; the kernel leaves them zero).
ff_status ensure_counters(ff_head* hd, int blocks) {
  if (blocks <= hd->counter_cap) return FF_OK;
  FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync before counter growth");
  dev_free(hd->counters);
  hd->counters = nullptr;
  hd->counter_cap = 0;
  FF_TRY(dev_alloc(reinterpret_cast<void**>(&hd->counters), (size_t)blocks * sizeof(int)), "head counters");
  FF_TRY(cudaMemset(hd->counters, 0, (size_t)blocks * sizeof(int)), "zero head counters");
  hd->counter_cap = blocks;
  return FF_OK;
}

// Logits (and, with labels, softmax, loss, dz and the per-row-block
// partials) of n rows: k_head_dot over the feature splits, whose last block
// per row block finishes the rows.
ff_status head_logits(ff_head* hd, const Segs& sg, bool b16, int n, const int* labels, float* logits, int* pred,
                      float* zpart, float* dz, float* part, uint4* dzfrag, int* err, cudaStream_t st) {
  const int es = b16 ? 2 : 4;
  const int split = dot_split(sg.F, sg.nseg, n, es);
  const int S = head_splits(sg.F, sg.nseg, split);
  ff_status s = ensure_counters(hd, cdiv(n, kDotRows));
  if (s != FF_OK) return s;
  FinishArgs fa{};
  fa.cb = hd->c;
  fa.labels = labels;
  fa.inv_n = 1.f / (float)n;
  fa.logits = logits;
  fa.pred = pred;
  fa.dz = dz;
  fa.part = part;
  fa.dzfrag = dzfrag;
  fa.ds = labels ? hd->ds : nullptr;
  fa.beta1 = hd->cfg.beta1;
  fa.beta2 = hd->cfg.beta2;
  fa.counter = hd->counters;
  fa.S = S;
  const float* V = hd->V;
  dim3 grid(S, cdiv(n, kDotRows));
  const double work = (double)n * sg.F_total * es + (double)n * (2 * S + 2) * kClasses * 4;
  if (b16) {
    FF_TRY(allow_smem<k_head_dot_mma>(mma_smem(kMmaSplit)), "head kernel attributes");
    PdlLaunch l(grid, dim3(256), st, mma_smem(split));
    FF_LAUNCH(K_HEAD_LOGITS, work, st, cudaLaunchKernelEx(&l.cfg, k_head_dot_mma, sg, split, n, V, zpart, fa, err),
              "head logits, softmax and cross-entropy");
    return FF_OK;
  }
  HeadMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int k = 0; k < sg.nseg; ++k)
    if (!make_plain_map(&maps.m[k], sg.H[k], es, sg.ld[k], n, sg.ld[k], 512 / es, kDotRows))
      return FF_ERR_INVALID_ARG;
  FF_TRY(allow_smem<k_head_dot>(kDotSmem), "head kernel attributes");
  PdlLaunch l(grid, dim3(256), st, kDotSmem);
  FF_LAUNCH(K_HEAD_LOGITS, work, st, cudaLaunchKernelEx(&l.cfg, k_head_dot, maps, sg, split, n, V, zpart, fa, err),
            "head logits, softmax and cross-entropy");
  return FF_OK;
}

cudaError_t launch_head_wgrad(const Segs& sg, int n, const float* dz, float* dVpart, cudaStream_t st) {
  int chunks = 0;
  for (int k = 0; k < sg.nseg; ++k) chunks += cdiv(sg.F[k], kWgChunk);
  PdlLaunch l(dim3(chunks, cdiv(n, kWgRows)), dim3(256), st);
  return cudaLaunchKernelEx(&l.cfg, k_head_wgrad, sg, n, dz, dVpart);
}

cudaError_t launch_head_wgrad_adam(const Segs& sg, int n, const uint4* dzfrag, const HeadAdamArgs& a, cudaStream_t st) {
  int chunks = 0;
  for (int k = 0; k < sg.nseg; ++k) chunks += cdiv(sg.F[k], kWgaFeats);
  PdlLaunch l(dim3(chunks + 1), dim3(256), st);
  return cudaLaunchKernelEx(&l.cfg, k_head_wgrad_adam, sg, n, dzfrag, a);
}

}  // namespace
}  // namespace ff

using namespace ff;

namespace ff {

int head_features(const ff_head* h) { return h->F; }
void head_forget_stream(ff_head* h, cudaStream_t st) {
  if (h->last_stream == st) h->last_stream = nullptr;
}

namespace {

// Scratch of a softmax block for n rows of a layer of width N, carved from
// the head's workspace (grown on demand).
struct PoWork {
  float *zpart, *dz, *part, *dVpart;
};

ff_status po_workspace(ff_head* hd, int n, int N, int es, PoWork* w) {
  size_t off = 0;
  // partial logits: k_head_dot's (fp32 layers) or the forward GEMM's (bf16)
  size_t zf = zpart_floats(&N, 1, n, es);
  if (es == 2) zf = std::max(zf, (size_t)tc_fwd_ntiles_max(N) * n * kClasses);
  const size_t oZ = off; off += align256(zf * 4);
  const size_t oD = off; off += align256((size_t)n * kClasses * 4);
  const size_t oP = off; off += align256((size_t)cdiv(n, std::min(kDotRows, kPoRows)) * kPart * 4);
  const size_t oV = off; off += align256((size_t)cdiv(n, kPoRows) * kClasses * N * 4);
  if (off > hd->ws_bytes) {
    FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync before workspace growth");
    if (hd->side) FF_TRY(cudaStreamSynchronize(hd->side), "sync before workspace growth");
    dev_free(hd->ws);
    hd->ws = nullptr;
    hd->ws_bytes = 0;
    FF_TRY(dev_alloc(&hd->ws, off), "block workspace");
    hd->ws_bytes = off;
  }
  char* base = static_cast<char*>(hd->ws);
  w->zpart = reinterpret_cast<float*>(base + oZ);
  w->dz = reinterpret_cast<float*>(base + oD);
  w->part = reinterpret_cast<float*>(base + oP);
  w->dVpart = reinterpret_cast<float*>(base + oV);
  return FF_OK;
}

// Adam arguments of the head / block from its state and this step's partials.
HeadAdamArgs head_adam_args(ff_head* hd, const float* dVpart, int nrb, const float* part, int nlb, int n,
                            float* loss) {
  HeadAdamArgs a{};
  a.V = hd->V;
  a.mV = hd->mV;
  a.vV = hd->vV;
  a.c = hd->c;
  a.mc = hd->mc;
  a.vc = hd->vc;
  a.dVpart = dVpart;
  a.nrb = nrb;
  a.F = hd->F;
  a.part = part;
  a.nlb = nlb;
  a.inv_n = 1.f / (float)n;
  a.lr = hd->cfg.lr;
  a.beta1 = hd->cfg.beta1;
  a.beta2 = hd->cfg.beta2;
  a.eps = hd->cfg.eps;
  a.ds = hd->ds;
  a.loss_out = loss ? loss : &hd->ds->loss;
  a.dV_out = hd->dV;
  a.dc_out = hd->dc;
  return a;
}

}  // namespace
}  // namespace ff

extern "C" {

ff_status ff_head_create(const ff_head_config* cfg, ff_head** out) {
  if (!out) return FF_ERR_INVALID_ARG;
  *out = nullptr;
  if (!cfg || cfg->n_features < 1 || cfg->max_rows < 0) return FF_ERR_INVALID_ARG;
  if (!std::isfinite(cfg->lr) || !(cfg->beta1 >= 0.f && cfg->beta1 < 1.f) || !(cfg->beta2 >= 0.f && cfg->beta2 < 1.f) ||
      !(cfg->eps > 0.f))
    return FF_ERR_INVALID_ARG;
  ff_head* hd = new (std::nothrow) ff_head();
  if (!hd) return FF_ERR_OOM;
  hd->cfg = *cfg;
  if (hd->cfg.max_rows == 0) hd->cfg.max_rows = 4096;
  hd->F = cfg->n_features;
  cudaGetDevice(&hd->device);
  const size_t nv = (size_t)kClasses * hd->F;
  const size_t total = 4 * nv + 5 * kClasses;  // V, mV, vV, dV; c, mc, vc, dc (+ pad)
  void* p = nullptr;
  ff_status s = cuda_status(dev_alloc(&p, total * 4), "head parameters");
  if (s != FF_OK) {
    delete hd;
    return s;
  }
  float* f = static_cast<float*>(p);
  hd->V = f;
  hd->mV = f + nv;
  hd->vV = f + 2 * nv;
  hd->dV = f + 3 * nv;
  hd->c = f + 4 * nv;
  hd->mc = hd->c + kClasses;
  hd->vc = hd->mc + kClasses;
  hd->dc = hd->vc + kClasses;
  void* dsp = nullptr;
  s = cuda_status(dev_alloc(&dsp, sizeof(ff_dev_state)), "head device state");
  if (s != FF_OK) {
    dev_free(p);
    delete hd;
    return s;
  }
  hd->ds = static_cast<ff_dev_state*>(dsp);
  const ff_dev_state init{0, 1.0, 1.0, 0.f, 0.f, 0, 0.f};
  cudaError_t e = cudaMemcpy(hd->ds, &init, sizeof(init), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(p, 0, total * 4);  // V and c start at zero (the head's reading)
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    dev_free(p);
    dev_free(dsp);
    delete hd;
    return cuda_status(e, "head initialisation");
  }
  *out = hd;
  return FF_OK;
}

ff_status ff_head_destroy(ff_head* hd) {
  if (!hd) return FF_OK;
  cudaStreamSynchronize(hd->last_stream);
  if (hd->side) {
    cudaStreamSynchronize(hd->side);
    cudaStreamDestroy(hd->side);
    cudaEventDestroy(hd->ev_start);
    cudaEventDestroy(hd->ev_fork);
    cudaEventDestroy(hd->ev_join);
    for (int i = 0; i < 2; ++i) {
      cudaEventDestroy(hd->ev_fwd[i]);
      cudaEventDestroy(hd->ev_use[i]);
    }
  }
  dev_free(hd->ws2);
  dev_free(hd->ws);
  dev_free(hd->counters);
  dev_free(hd->V);
  dev_free(hd->ds);
  delete hd;
  return FF_OK;
}

// Rows of stored features ff_head_train_epoch forms per forward pass: whole
// steps of B rows, at least one, at most kEpochFeatureRows; with bf16 layers
// also at most what the widest layer's GEMM does in two full waves of CTAs.
// The first pass's forward has nothing to run beside, and a pass's activities
// are read again by its steps, from L2 if they still are there: 20000 rows of
// 784-2000x4 in steps of 1024 take 891 us with 16384 rows a pass, 827 with
// 9728 (two waves), 816 with 4864, 1112 with 2432.
constexpr int kEpochFeatureRows = 16384;
static int epoch_pass_steps(ff_layer* const* layers, int n_layers, int B) {
  int steps = kEpochFeatureRows / B > 0 ? kEpochFeatureRows / B : 1;
  if (!layers[0]->is_bf16) return steps;
  int dev = 0, sms = 0, Nw = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return steps;
  for (int k = 0; k < n_layers; ++k) Nw = std::max(Nw, layers[k]->N);
  while (steps > 1 && tc_gemm_fwd_ctas(steps * B, Nw, false) > 2 * sms) --steps;
  return steps;
}

// The head's side stream and its events (created on first use).
static ff_status ensure_side(ff_head* hd) {
  if (hd->side) return FF_OK;
  FF_TRY(cudaStreamCreateWithFlags(&hd->side, cudaStreamNonBlocking), "head side stream");
  cudaEvent_t* evs[] = {&hd->ev_start, &hd->ev_fork, &hd->ev_join, &hd->ev_fwd[0], &hd->ev_fwd[1], &hd->ev_use[0],
                        &hd->ev_use[1]};
  for (cudaEvent_t* e : evs) FF_TRY(cudaEventCreateWithFlags(e, cudaEventDisableTiming), "head event");
  return FF_OK;
}

// The head's part of one train step on n rows of the features in w, starting
// at row r0 of the stored activities: logits, softmax, loss and dz
// (k_head_dot), dV partials (k_head_wgrad), Adam on V and c (k_head_adam).
static ff_status head_step_on_features(ff_head* hd, ff_layer* const* layers, int n_layers, const HeadWork& w, int r0,
                                       const int* labels, int n, float* loss, cudaStream_t st) {
  Segs sg = make_segs(layers, n_layers, w, hd->F);
  const bool b16 = layers[0]->is_bf16;
  const double es = b16 ? 2.0 : 4.0;
  for (int j = 0; j < sg.nseg; ++j) {
    sg.H[j] = static_cast<const char*>(sg.H[j]) + (size_t)r0 * sg.ld[j] * (size_t)es;
    sg.s[j] += r0;
  }
  int* err = &hd->ds->err;
  ff_status s = head_logits(hd, sg, b16, n, labels, nullptr, nullptr, w.zpart, w.dz, w.part, w.dzfrag, err, st);
  if (s != FF_OK) return s;
  const HeadAdamArgs a =
      head_adam_args(hd, w.dVpart, b16 ? 0 : cdiv(n, kWgRows), w.part, cdiv(n, kDotRows), n, loss);
  if (b16) {
    FF_LAUNCH(K_HEAD_WGRAD, (double)n * hd->F * es + (double)kClasses * hd->F * 28, st,
              launch_head_wgrad_adam(sg, n, w.dzfrag, a, st), "head weight gradient and Adam");
    return FF_OK;
  }
  FF_LAUNCH(K_HEAD_WGRAD, (double)n * hd->F * es + (double)cdiv(n, kWgRows) * kClasses * hd->F * 4, st,
            launch_head_wgrad(sg, n, w.dz, w.dVpart, st), "head weight gradient");
  const int vblocks = cdiv((long long)kClasses * hd->F, 256);
  PdlLaunch l(dim3(vblocks + 1), dim3(256), st);
  FF_LAUNCH(K_HEAD_ADAM, (double)kClasses * hd->F * (a.nrb * 4.0 + 28), st, cudaLaunchKernelEx(&l.cfg, k_head_adam, a),
            "head Adam");
  return FF_OK;
}

ff_status ff_head_train_step(ff_head* hd, ff_layer* const* layers, int n_layers, const float* x, const int* labels,
                             int n, float* loss, void* stream) {
  ff::NvtxRange nvtx_("ff_head_train_step");
  if (!hd || n < 0) return FF_ERR_INVALID_ARG;
  ff_status s = head_layers(hd, layers, n_layers);
  if (s != FF_OK) return s;
  if (n == 0) return FF_OK;
  if (!x || !labels || n > hd->cfg.max_rows) return FF_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  HeadWork w;
  s = head_workspace(hd, layers, n_layers, n, true, &w);
  if (s != FF_OK) return s;
  hd->last_stream = st;
  int* err = &hd->ds->err;
  s = head_forward(layers, n_layers, x, n, w, err, st, false);
  if (s != FF_OK) return s;
  return head_step_on_features(hd, layers, n_layers, w, 0, labels, n, loss, st);
}

ff_status ff_head_train_epoch(ff_head* hd, ff_layer* const* layers, int n_layers, const float* x, const int* labels,
                              int n, int B, float* loss, void* stream) {
  ff::NvtxRange nvtx_("ff_head_train_epoch");
  if (!hd || n < 0 || B < 1) return FF_ERR_INVALID_ARG;
  ff_status s = head_layers(hd, layers, n_layers);
  if (s != FF_OK) return s;
  if (n == 0) return FF_OK;
  if (!x || !labels || B > hd->cfg.max_rows) return FF_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int steps_per_chunk = epoch_pass_steps(layers, n_layers, B);
  const int R = (int)((long long)steps_per_chunk * B < n ? (long long)steps_per_chunk * B : n);
  const int npass = cdiv(n, R);
  if (npass > 1) {
    s = ensure_side(hd);
    if (s != FF_OK) return s;
  }
  HeadWork w[2];
  for (int i = 0; i < (npass > 1 ? 2 : 1); ++i) {
    s = head_workspace(hd, layers, n_layers, R, true, &w[i], i);
    if (s != FF_OK) return s;
  }
  hd->last_stream = st;
  int* err = &hd->ds->err;
  const int K0 = layers[0]->K;
  // Pass p's forward fills workspace p % 2 on the side stream (after the
  // head steps of pass p - 2 have read it); its head steps run on `stream`
  // after that forward, while the side stream forms pass p + 1.  One pass:
  // everything on `stream`.
  cudaStream_t fs = npass > 1 ? hd->side : st;
  if (npass > 1) {
    FF_TRY(cudaEventRecord(hd->ev_start, st), "event record");
    FF_TRY(cudaStreamWaitEvent(fs, hd->ev_start, 0), "stream wait");
  }
  for (int p = 0, r0 = 0, t = 0; p < npass; ++p, r0 += R) {
    const int rows = n - r0 < R ? n - r0 : R;
    const int buf = p & 1;
    if (npass > 1 && p >= 2) FF_TRY(cudaStreamWaitEvent(fs, hd->ev_use[buf], 0), "stream wait");
    s = head_forward(layers, n_layers, x + (size_t)r0 * K0, rows, w[buf], err, fs, false);
    if (s != FF_OK) return s;
    if (npass > 1) {
      FF_TRY(cudaEventRecord(hd->ev_fwd[buf], fs), "event record");
      FF_TRY(cudaStreamWaitEvent(st, hd->ev_fwd[buf], 0), "stream wait");
    }
    for (int q = 0; q < rows; q += B, ++t) {
      const int b = rows - q < B ? rows - q : B;
      s = head_step_on_features(hd, layers, n_layers, w[buf], q, labels + r0 + q, b, loss ? loss + t : nullptr, st);
      if (s != FF_OK) return s;
    }
    if (npass > 1) FF_TRY(cudaEventRecord(hd->ev_use[buf], st), "event record");
  }
  return FF_OK;
}

ff_status ff_head_predict(ff_head* hd, ff_layer* const* layers, int n_layers, const float* x, int n, int* pred,
                          float* logits, void* stream) {
  ff::NvtxRange nvtx_("ff_head_predict");
  if (!hd || n < 0) return FF_ERR_INVALID_ARG;
  ff_status s = head_layers(hd, layers, n_layers);
  if (s != FF_OK) return s;
  if (n == 0) return FF_OK;
  if (!x || (!pred && !logits)) return FF_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int C = n < hd->cfg.max_rows ? n : hd->cfg.max_rows;
  HeadWork w;
  s = head_workspace(hd, layers, n_layers, C, false, &w);
  if (s != FF_OK) return s;
  hd->last_stream = st;
  int* err = &hd->ds->err;
  const bool b16 = layers[0]->is_bf16;
  const int K0 = layers[0]->K;
  for (int r0 = 0; r0 < n; r0 += C) {
    const int cn = (n - r0) < C ? (n - r0) : C;
    s = head_forward(layers, n_layers, x + (size_t)r0 * K0, cn, w, err, st, true);
    if (s != FF_OK) return s;
    const Segs sg = make_segs(layers, n_layers, w, hd->F);
    s = head_logits(hd, sg, b16, cn, nullptr, logits ? logits + (size_t)r0 * kClasses : nullptr,
                    pred ? pred + r0 : nullptr, w.zpart, nullptr, nullptr, nullptr, err, st);
    if (s != FF_OK) return s;
  }
  return FF_OK;
}

static ff_status head_copy(void* dst, const void* src, size_t bytes) {
  if (!dst || !src) return FF_OK;
  FF_TRY(cudaMemcpy(dst, src, bytes, cudaMemcpyDefault), "head state copy");
  return FF_OK;
}

ff_status ff_head_get_state(const ff_head* hdc, float* V, float* c, float* mV, float* vV, float* mc, float* vc,
                            long long* step) {
  if (!hdc) return FF_ERR_INVALID_ARG;
  ff_head* hd = const_cast<ff_head*>(hdc);
  FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync");
  const size_t nv = (size_t)kClasses * hd->F * 4, nc = kClasses * 4;
  ff_status s;
  if ((s = head_copy(V, hd->V, nv)) != FF_OK) return s;
  if ((s = head_copy(mV, hd->mV, nv)) != FF_OK) return s;
  if ((s = head_copy(vV, hd->vV, nv)) != FF_OK) return s;
  if ((s = head_copy(c, hd->c, nc)) != FF_OK) return s;
  if ((s = head_copy(mc, hd->mc, nc)) != FF_OK) return s;
  if ((s = head_copy(vc, hd->vc, nc)) != FF_OK) return s;
  if (step) {
    ff_dev_state d;
    FF_TRY(cudaMemcpy(&d, hd->ds, sizeof(d), cudaMemcpyDeviceToHost), "head step counter");
    *step = d.t;
  }
  return FF_OK;
}

ff_status ff_head_set_state(ff_head* hd, const float* V, const float* c, const float* mV, const float* vV,
                            const float* mc, const float* vc, long long step) {
  if (!hd || step < 0) return FF_ERR_INVALID_ARG;
  FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync");
  const size_t nv = (size_t)kClasses * hd->F * 4, nc = kClasses * 4;
  ff_status s;
  if ((s = head_copy(hd->V, V, nv)) != FF_OK) return s;
  if ((s = head_copy(hd->mV, mV, nv)) != FF_OK) return s;
  if ((s = head_copy(hd->vV, vV, nv)) != FF_OK) return s;
  if ((s = head_copy(hd->c, c, nc)) != FF_OK) return s;
  if ((s = head_copy(hd->mc, mc, nc)) != FF_OK) return s;
  if ((s = head_copy(hd->vc, vc, nc)) != FF_OK) return s;
  ff_dev_state d;
  FF_TRY(cudaMemcpy(&d, hd->ds, sizeof(d), cudaMemcpyDeviceToHost), "head device state");
  d.t = step;
  d.pow1 = std::pow((double)hd->cfg.beta1, (double)step);
  d.pow2 = std::pow((double)hd->cfg.beta2, (double)step);
  FF_TRY(cudaMemcpy(hd->ds, &d, sizeof(d), cudaMemcpyHostToDevice), "head device state");
  return FF_OK;
}

ff_status ff_head_get_grad(const ff_head* hdc, float* dV, float* dc) {
  if (!hdc) return FF_ERR_INVALID_ARG;
  ff_head* hd = const_cast<ff_head*>(hdc);
  FF_TRY(cudaStreamSynchronize(hd->last_stream), "sync");
  ff_status s;
  if ((s = head_copy(dV, hd->dV, (size_t)kClasses * hd->F * 4)) != FF_OK) return s;
  return head_copy(dc, hd->dc, kClasses * 4);
}

ff_status ff_head_check(ff_head* hd) {
  if (!hd) return FF_ERR_INVALID_ARG;
  FF_TRY(cudaStreamSynchronize(hd->last_stream), "check sync");
  int err = 0;
  FF_TRY(cudaMemcpy(&err, &hd->ds->err, sizeof(int), cudaMemcpyDeviceToHost), "read error word");
  if (err) {
    const int zero = 0;
    FF_TRY(cudaMemcpy(&hd->ds->err, &zero, sizeof(int), cudaMemcpyHostToDevice), "clear error word");
  }
  if (err & DEVERR_CHECK) return FF_ERR_DEVICE_CHECK;  // a skipped copy also runs waits out
  if (err & DEVERR_TIMEOUT) return FF_ERR_TIMEOUT;
  if (err & DEVERR_NONFINITE) return FF_ERR_NONFINITE;
  return FF_OK;
}

// ------------------------------------------ Performance-Optimized layer (§4)
ff_status ff_po_train_step(ff_layer* L, ff_head* hd, const void* x, int raw_input, const float* row_scale,
                           const int* labels, int n, void* h_out, float* next_scale, float* loss, void* stream) {
  ff::NvtxRange nvtx_("ff_po_train_step");
  if (!L || !hd || n < 0) return FF_ERR_INVALID_ARG;
  if (hd->F != L->N) return FF_ERR_INVALID_ARG;
  if (raw_input && L->K < kClasses) return FF_ERR_INVALID_ARG;
  if (n == 0) return FF_OK;
  if (!x || !labels) return FF_ERR_INVALID_ARG;
  if (h_out && (reinterpret_cast<uintptr_t>(h_out) & 15u)) return FF_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ff_status s = ensure_capacity(L, n);
  if (s != FF_OK) return s;
  PoWork w;
  s = po_workspace(hd, n, L->N, L->is_bf16 ? 2 : 4, &w);
  if (s != FF_OK) return s;
  L->last_stream = st;
  hd->last_stream = st;
  const bool b16 = L->is_bf16;
  const double es = b16 ? 2.0 : 4.0;
  const int K = L->K, N = L->N;
  // the layer's forward pass (layer 1: the neutral-labelled raw input)
  const void* X;
  const float* sc;
  if (raw_input) {
    FF_LAUNCH(K_OVERLAY, (double)n * (K * 4.0 + L->ldK * es + 4), st,
              launch_overlay(static_cast<const float*>(x), nullptr, n, K, L->X, L->ldK, b16, L->s_in, 2, st),
              "neutral-label overlay");
    X = L->X;
    sc = L->s_in;
  } else {
    X = x;
    if (row_scale) {
      sc = row_scale;
    } else {
      FF_LAUNCH(K_ROW_SCALE, (double)n * (K * es + 4), st, launch_row_scale(x, L->ldK, b16, n, K, L->s_in, st),
                "row scale");
      sc = L->s_in;
    }
  }
  void* H = h_out ? h_out : L->H;
  EpiArgs ep{sc, L->cfg.has_bias ? L->b : nullptr, H, L->ldN, L->gpart};
  int ntiles;
  if (b16) {
    // the block's partial logits come out of the forward GEMM's epilogue
    ep.logit_V = hd->V;
    ep.logit_ldV = N;
    ep.zpart = w.zpart;
    ntiles = tc_fwd_ntiles(n, N, false);
    FF_LAUNCH(K_FWD_TC, 2.0 * n * N * K, st,
              tc_gemm_fwd(static_cast<const bf16*>(X), L->ldK, L->Wb, L->ldK, n, N, K, ep, &L->ds->err, st),
              "forward GEMM (tcgen05)");
  } else {
    ntiles = f32_fwd_ntiles(kF32InOrder, N, K);
    FF_LAUNCH(K_FWD_SIMT, 2.0 * n * N * K, st,
              f32_gemm_fwd(static_cast<const float*>(X), L->ldK, L->W, K, n, N, K, kF32InOrder, ep,
                           &L->ds->err, st), "forward GEMM (fp32)");
  }
  if (!b16) {
    // the block on the raw activity: logits, cross-entropy, dz
    Segs sg{};
    sg.H[0] = H;
    sg.s[0] = nullptr;
    sg.ld[0] = L->ldN;
    sg.F[0] = N;
    sg.off[0] = 0;
    sg.nseg = 1;
    sg.F_total = N;
    s = head_logits(hd, sg, b16, n, labels, nullptr, nullptr, w.zpart, w.dz, w.part, nullptr, &hd->ds->err, st);
    if (s != FF_OK) return s;
  }
  // the gradient reaching the layer, with the block's weights before its
  // update, and the block's weight-gradient partials (bf16: after finishing
  // the block's rows from the GEMM's partial logits)
  PoGradArgs pa{};
  if (b16) {
    pa.zpart = w.zpart;
    pa.zt = ntiles;
    pa.cb = hd->c;
    pa.labels = labels;
    pa.inv_n = 1.f / (float)n;
    pa.part = w.part;
    pa.hds = hd->ds;
    pa.hbeta1 = hd->cfg.beta1;
    pa.hbeta2 = hd->cfg.beta2;
  } else {
    pa.dz = w.dz;
  }
  pa.V = hd->V;
  pa.s = sc;
  pa.gpart = L->gpart;
  pa.ntiles = ntiles;
  pa.n = n;
  pa.N = N;
  pa.ld = L->ldN;
  pa.s_next = next_scale;
  pa.dbpart = L->dbpart;
  pa.dVpart = w.dVpart;
  pa.ds = L->ds;
  pa.beta1 = L->cfg.beta1;
  pa.beta2 = L->cfg.beta2;
  pa.err = &L->ds->err;
  PdlLaunch pl(dim3(cdiv(L->ldN, 256), cdiv(n, kPoRows)), dim3(32, 8), st);
  FF_LAUNCH(K_GRAD_PREP, (double)n * L->ldN * es * 2 + (double)cdiv(n, kPoRows) * (kClasses + 1) * N * 4, st,
            (b16 ? cudaLaunchKernelEx(&pl.cfg, k_po_grad<bf16>, pa, static_cast<const bf16*>(H),
                                      static_cast<bf16*>(L->dZ))
                 : cudaLaunchKernelEx(&pl.cfg, k_po_grad<float>, pa, static_cast<const float*>(H),
                                      static_cast<float*>(L->dZ))),
            "block gradient into the layer");
  // The block's Adam needs only what k_po_grad wrote, and nothing later in
  // this step reads the block's weights: it runs on the head's side stream,
  // beside the layer's weight gradient and Adam, and `stream` joins it at the
  // end of the step.
  s = ensure_side(hd);
  if (s != FF_OK) return s;
  FF_TRY(cudaEventRecord(hd->ev_fork, st), "event record");
  FF_TRY(cudaStreamWaitEvent(hd->side, hd->ev_fork, 0), "stream wait");
  {
    const HeadAdamArgs ha =
        head_adam_args(hd, w.dVpart, cdiv(n, kPoRows), w.part, cdiv(n, b16 ? kPoRows : kDotRows), n, loss);
    const int vblocks = cdiv((long long)kClasses * hd->F, 256);
    // a plain launch: after an event wait, programmatic serialization has
    // nothing to overlap (griddepcontrol.wait is then a no-op)
    FF_LAUNCH(K_HEAD_ADAM, (double)kClasses * hd->F * (ha.nrb * 4.0 + 28), hd->side,
              (k_head_adam<<<vblocks + 1, 256, 0, hd->side>>>(ha), cudaGetLastError()), "block Adam");
  }
  FF_TRY(cudaEventRecord(hd->ev_join, hd->side), "event record");
  AdamArgs aa = adam_args(L, n);
  aa.B = n;
  s = weight_update(L, X, n, aa, st, true);
  if (s != FF_OK) return s;
  FF_TRY(cudaStreamWaitEvent(st, hd->ev_join, 0), "stream wait");
  return FF_OK;
}

ff_status ff_po_predict(ff_layer* const* layers, int n_layers, ff_head* hd, const float* x, int n, int* pred,
                        float* logits, void* stream) {
  ff::NvtxRange nvtx_("ff_po_predict");
  if (!layers || n_layers < 1 || n_layers > kMaxSegs + 1 || !hd || n < 0) return FF_ERR_INVALID_ARG;
  for (int k = 0; k < n_layers; ++k) {
    if (!layers[k]) return FF_ERR_INVALID_ARG;
    if (layers[k]->is_bf16 != layers[0]->is_bf16) return FF_ERR_INVALID_ARG;
    if (k > 0 && layers[k]->K != layers[k - 1]->N) return FF_ERR_INVALID_ARG;
  }
  if (layers[0]->K < kClasses || hd->F != layers[n_layers - 1]->N) return FF_ERR_INVALID_ARG;
  if (n == 0) return FF_OK;
  if (!x || (!pred && !logits)) return FF_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int C = n < hd->cfg.max_rows ? n : hd->cfg.max_rows;
  HeadWork w;
  ff_status s = head_workspace(hd, layers, n_layers, C, false, &w);
  if (s != FF_OK) return s;
  hd->last_stream = st;
  int* err = &hd->ds->err;
  const bool b16 = layers[0]->is_bf16;
  ff_layer* top = layers[n_layers - 1];
  for (int r0 = 0; r0 < n; r0 += C) {
    const int cn = (n - r0) < C ? (n - r0) : C;
    s = head_forward(layers, n_layers, x + (size_t)r0 * layers[0]->K, cn, w, err, st, true);
    if (s != FF_OK) return s;
    Segs sg{};
    sg.H[0] = w.Hk[n_layers - 1];
    sg.s[0] = nullptr;
    sg.ld[0] = top->ldN;
    sg.F[0] = top->N;
    sg.nseg = 1;
    sg.F_total = top->N;
    s = head_logits(hd, sg, b16, cn, nullptr, logits ? logits + (size_t)r0 * kClasses : nullptr,
                    pred ? pred + r0 : nullptr, w.zpart, nullptr, nullptr, nullptr, err, st);
    if (s != FF_OK) return s;
  }
  return FF_OK;
}

}  // extern "C"

// fp32 GEMMs on the tensor cores without loss of precision, for the exact fp32
// mode's larger training GEMMs (the contracts of ff_gemm_simt.cu).
//
// Each fp32 operand value enters as three bf16 parts, hi = rn(x) (at most the
// largest finite bf16), mid = rn(x - hi), lo = x - hi - mid: exact, 24 bits in
// all, but for what lies below bf16's smallest number, 2^-133.  Six of the nine
// part products are formed (lo-hi, mid-mid, mid-hi and hi-hi, both ways); the
// three dropped ones are below 2^-25 of the term.  Every product is exact in
// fp32.  The tensor cores' running sum is not rounded to nearest, and a sum of
// K terms left in it drifts by up to K/16 6 2^-24 of its size (the three-TF32
// forward of goodness predict shows that drift, 2e-5 at K = 2000): so only 64
// terms are summed there, the small products first, and each such chunk is
// added to fp32 registers with ordinary rounded adds.  Measured against 64
// bits (2-norm), 2000-wide activities over K = 2000: 1.2e-7 with one K slice,
// 1.0e-7 with four; the CUDA-core GEMM 7.3e-7 and 3.3e-7.
//
// Split of the work: a CTA makes a 128 x 128 tile over one slice of K (up to
// four slices, the CTAs of a cluster, added through distributed shared memory
// as in ff_gemm_simt.cu), with
//   warps 0..7   load both operands' 128 x 64 fp32 tiles from L2 into
//                registers, half a stage ahead, and write the three parts as
//                128-byte-swizzled tiles into a two-stage ring (96 KB a stage)
//   warp 8       one lane issues the MMAs of each 64-deep chunk (24 of M = N
//                = 128, K = 16) into one of four TMEM buffers
//   warps 8..15  add each finished chunk to their registers (a 32-row quarter
//                of TMEM and half the columns each), then run the epilogue
// Bound by the chain of a chunk, no unit being full: its loads from L2, the
// split (about 7 instructions for each of its 16,384 values), the 96 KB of
// parts stored and the 24 MMAs' 192 KB of operand reads follow one another with
// two stages in flight (512 x 2000 over 2000: tensor pipe 36 % active, the
// tensor cores' shared-memory wavefronts 22 % of peak, the load/store unit's
// 30 %, issue slots 40 %); measured 1.7 us a chunk, 136 TFLOP/s of fp32 terms
// on the 2048-row weight gradient (the CUDA-core GEMM reaches 50).
// An infinite operand comes out as NaN (its parts are an infinity and inf -
// inf), which the non-finite check reports as it does infinities.
#include "ff_f32_epilogue.cuh"
#include "ff_internal.cuh"
#include "ff_ptx.cuh"

namespace ff {
namespace {

constexpr int T = 128;          // rows and columns of a CTA's tile
constexpr int KC = 64;          // K per chunk: one 128-byte row of bf16
constexpr int STAGES = 2;
constexpr int PART_BYTES = T * KC * 2;      // one part of one operand
constexpr int OP_BYTES = 3 * PART_BYTES;
constexpr int STAGE_BYTES = 2 * OP_BYTES;
constexpr int BUFS = 4;         // TMEM chunk buffers of T columns
constexpr int LOAD_WARPS = 8, SUM_WARPS = 8;
constexpr int NTHREADS = 32 * (LOAD_WARPS + SUM_WARPS);
constexpr int LD = f32_tile_ld(T);
constexpr int SMEM = STAGES * STAGE_BYTES + 1024 /*alignment*/ + 256 /*barriers*/;
static_assert(T * LD * 4 <= STAGES * STAGE_BYTES, "the partial tile takes the ring's place");
static_assert(SMEM > 113 * 1024 && SMEM <= 227 * 1024, "one tensor-core GEMM CTA per SM: no TMEM allocation waits");

// The three bf16 parts of x0 (low halves) and x1 (high halves).
__device__ __forceinline__ uint32_t cvt2(float x0, float x1) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(x0, x1);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t cvt2_finite(float x0, float x1) {
  uint32_t v;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(x1), "f"(x0));
  return v;
}
__device__ __forceinline__ void split2(float x0, float x1, uint32_t (&p)[3]) {
  p[0] = cvt2_finite(x0, x1);
  x0 = __fsub_rn(x0, __uint_as_float(p[0] << 16));
  x1 = __fsub_rn(x1, __uint_as_float(p[0] & 0xFFFF0000u));
  p[1] = cvt2(x0, x1);
  x0 = __fsub_rn(x0, __uint_as_float(p[1] << 16));
  x1 = __fsub_rn(x1, __uint_as_float(p[1] & 0xFFFF0000u));
  p[2] = cvt2(x0, x1);
}

// One of 16 RPP loader threads' share of one operand's 128 x 64 fp32 tile:
// NV = 128 / RPP words of 4 values, RPP tile rows at a time.  Tile row i of 128
// holds 64 values contiguous in memory: K-major operands, row r0 + i, K k0 ..;
// MN-major ones, K k0 + i % 64, rows r0 + 64 (i / 64) ...  16 lanes take a row,
// a warp two rows at a time.
template <bool MN, int NV>
__device__ __forceinline__ void load_part(float4 (&v)[NV], const float* __restrict__ P, int ld, int rows, int K, int r0,
                                          int k0, int t) {
  constexpr int RPP = T / NV;
  const int c = 4 * (t & 15), r = t >> 4;
  if (r0 + T <= rows && k0 + KC <= K) {  // the whole tile exists
    const float* p = MN ? P + (size_t)(k0 + r) * ld + r0 + c : P + (size_t)(r0 + r) * ld + k0 + c;
    const size_t step = (size_t)RPP * ld;
    constexpr int H = 64 / RPP;  // words per 64-row half of an MN-major tile
#pragma unroll
    for (int i = 0; i < NV; ++i)
      v[i] = __ldg(reinterpret_cast<const float4*>(MN ? p + (i % H) * step + (i / H) * 64 : p + i * step));
    return;
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int row = r + RPP * i;
    const int slow = MN ? k0 + (row & 63) : r0 + row;
    const int fast = MN ? r0 + (row >> 6) * 64 + c : k0 + c;
    const bool ok = slow < (MN ? K : rows) && fast < (MN ? rows : K);
    v[i] = ok ? __ldg(reinterpret_cast<const float4*>(P + (size_t)slow * ld + fast)) : make_float4(0.f, 0.f, 0.f, 0.f);
    // a row's padding is never used
    const int left = (MN ? rows : K) - fast;
    if (left < 2) v[i].y = 0.f;
    if (left < 3) v[i].z = 0.f;
    if (left < 4) v[i].w = 0.f;
  }
}
// Its three parts into the operand's tiles (128-byte rows, 16-byte words
// permuted by the row's low three bits, the same for all of a thread's rows).
template <int NV>
__device__ __forceinline__ void store_part(uint8_t* op, const float4 (&v)[NV], int t) {
  constexpr int RPP = T / NV;
  const int c = t & 15, r = t >> 4;
  uint8_t* dst = op + r * 128 + (((c >> 1) ^ (r & 7)) << 4) + (c & 1) * 8;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    uint32_t a[3], b[3];
    split2(v[i].x, v[i].y, a);
    split2(v[i].z, v[i].w, b);
#pragma unroll
    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(dst + i * RPP * 128 + p * PART_BYTES) = make_uint2(a[p], b[p]);
  }
}

__device__ __forceinline__ void latch(int* err, volatile int* abort_flag) {
  *abort_flag = 1;
  atomicOr(err, DEVERR_TIMEOUT);
}

// The MMAs of one chunk (a stage's parts) into the accumulator at acc: the six
// part products, the smallest first.  PAIR: M = N = 256 over the CTA pair.
template <bool MN, bool PAIR>
__device__ __forceinline__ void issue_chunk(uint32_t acc, const uint8_t* stage) {
  constexpr uint32_t idesc = ptx::idesc_bf16_f32(PAIR ? 2 * T : T, PAIR ? 2 * T : T, MN ? 1 : 0, MN ? 1 : 0);
  constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
  const uint32_t ab = ptx::smem_u32(stage), bb = ab + OP_BYTES;
#pragma unroll
  for (int p = 0; p < 6; ++p)
#pragma unroll
    for (int k = 0; k < KC / 16; ++k) {
      // K-major: 32 bytes along the swizzled rows, 8-row groups 1024 bytes
      // apart; MN-major: 16 K rows further, the 64-element halves 64 rows apart
      const uint32_t aa = ab + pa[p] * PART_BYTES, ba = bb + pb[p] * PART_BYTES;
      const uint64_t ad = MN ? ptx::sdesc_sw128(aa + k * 2048, 64 * 128, 1024) : ptx::sdesc_sw128(aa + k * 32, 16, 1024);
      const uint64_t bd = MN ? ptx::sdesc_sw128(ba + k * 2048, 64 * 128, 1024) : ptx::sdesc_sw128(ba + k * 32, 16, 1024);
      if constexpr (PAIR)
        ptx::umma_f16_pair(acc, ad, bd, idesc, (p | k) != 0 ? 1u : 0u);
      else
        ptx::umma_f16(acc, ad, bd, idesc, (p | k) != 0 ? 1u : 0u);
    }
}

template <bool MN, int MODE>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_f32tc_gemm(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int M, int N, int K,
                 EpiArgs ep, int* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + BUFS;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tempty + BUFS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * T, n0 = blockIdx.y * T;
  const int S = gridDim.z;
  const int chunks = (K + KC - 1) / KC;
  const int per = (chunks + S - 1) / S;
  const int c0 = min(chunks, (int)blockIdx.z * per), nc = min(chunks, c0 + per) - c0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(&full[s], LOAD_WARPS);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < BUFS; ++b) {
      ptx::mbar_init(&tfull[b], 1);
      ptx::mbar_init(&tempty[b], SUM_WARPS);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(tslot, BUFS * T);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tslot;
  ptx::griddep_wait();  // launched with programmatic stream serialization

  if (warp < LOAD_WARPS) {
    const int t = threadIdx.x;
    float4 va[8], vb[8];
    if (nc > 0) {
      load_part<MN>(va, A, lda, M, K, m0, c0 * KC, t);
      load_part<MN>(vb, B, ldb, N, K, n0, c0 * KC, t);
    }
    for (int c = 0; c < nc; ++c) {
      const int s = c % STAGES;
      const bool ok = ptx::mbar_wait(&empty[s], ((uint32_t)(c / STAGES) & 1u) ^ 1u, kWaitTimeoutNs, abort_flag);
      if (!ok) latch(err, abort_flag);
      if (!__all_sync(0xffffffffu, ok && !*abort_flag)) break;
      uint8_t* op = smem + s * STAGE_BYTES;
      store_part(op, va, t);
      if (c + 1 < nc) load_part<MN>(va, A, lda, M, K, m0, (c0 + c + 1) * KC, t);
      store_part(op + OP_BYTES, vb, t);
      if (c + 1 < nc) load_part<MN>(vb, B, ldb, N, K, n0, (c0 + c + 1) * KC, t);
      ptx::fence_async_smem();  // read by the MMAs (async proxy)
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&full[s]);
    }
  } else {
    const bool issuer = warp == LOAD_WARPS && lane == 0;
    // 32 rows (TMEM lanes 32 q ..) x 64 columns of the tile
    const int q = warp & 3, half = (warp - LOAD_WARPS) >> 2;
    float acc[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0.f;
    bool good = true;
    // chunk c's MMAs are issued before chunk c - 1 is added
    for (int c = 0; c <= nc; ++c) {
      if (issuer && c < nc) {
        const int s = c % STAGES, b = c % BUFS;
        if (ptx::mbar_wait(&full[s], (uint32_t)(c / STAGES) & 1u, kWaitTimeoutNs, abort_flag) &&
            ptx::mbar_wait(&tempty[b], ((uint32_t)(c / BUFS) & 1u) ^ 1u, kWaitTimeoutNs, abort_flag)) {
          ptx::tc_fence_after();
          issue_chunk<MN, false>(tmem + (uint32_t)(b * T), smem + s * STAGE_BYTES);
          ptx::umma_commit(&empty[s]);
          ptx::umma_commit(&tfull[b]);
        } else {
          latch(err, abort_flag);
        }
      }
      __syncwarp();
      if (c == 0) continue;
      const int b = (c - 1) % BUFS;
      const bool ok = ptx::mbar_wait(&tfull[b], (uint32_t)((c - 1) / BUFS) & 1u, kWaitTimeoutNs, abort_flag);
      if (!ok) latch(err, abort_flag);
      good = __all_sync(0xffffffffu, ok && !*abort_flag);
      if (!good) break;
      ptx::tc_fence_after();
      const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * T + half * 64);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t r[32];
        ptx::tmem_ld32(src + 32 * h, r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[32 * h + j] = __fadd_rn(acc[32 * h + j], __uint_as_float(r[j]));
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&tempty[b]);
    }
    if (!good) {
      // MMAs already issued finish before TMEM is released
      const uint64_t t0 = ptx::globaltimer();
      while (ptx::globaltimer() - t0 < 1000000ull) {
      }
    }
    // every chunk is summed, so every MMA has read the ring: the partial tile
    // takes its place (all warps of this role first)
    ptx::named_bar(1, 32 * SUM_WARPS);
    float* row = reinterpret_cast<float*>(smem) + (q * 32 + lane) * LD + half * 64;
    if (good) {
#pragma unroll
      for (int j = 0; j < 64; j += 4)
        *reinterpret_cast<float4*>(row + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
    }
  }
  if (threadIdx.x == 0) ptx::griddep_launch_dependents();
  ptx::tc_fence_before();
  if (S > 1)
    ptx::cluster_sync();  // every partial of the tile is in place
  else
    __syncthreads();
  if (warp >= LOAD_WARPS) {
    if (!*abort_flag)
      f32_tile_epilogue<T, MODE>(reinterpret_cast<const float*>(smem), (int)threadIdx.x - 32 * LOAD_WARPS, M, N, m0, n0,
                                 S, ep, AdamArgs{});
  } else if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, BUFS * T);
  }
  if (S > 1) ptx::cluster_sync();  // no CTA leaves while another reads its partial tile
}

// The same by CTA pairs (cta_group::2), for outputs of more than 128 rows and
// columns: a pair makes a 256 x 256 tile, each CTA its 128 rows, splitting
// 128 x 64 of A and of B per chunk as above -- half the splitting, half the
// shared-memory reads and writes per output.  All 16 warps do the same: write
// chunk c's parts, (one lane of the even CTA issues its MMAs once both CTAs
// have written,) add chunk c - 1 from TMEM to their registers (a 32-row quarter
// and 64 columns each), load chunk c + 1.  Measured 2.7 us a chunk (its 24
// MMAs of M = N = 256 take 3072 clocks; the rest is the chain of barriers,
// loads and splitting between them): 165 to 188 TFLOP/s of fp32 terms on 2048
// to 4600 rows of a 2000-wide layer, where 128 x 128 tiles reach 126 to 147.
template <bool MN, int MODE>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_f32tc_pair(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb, int M, int N, int K,
                 EpiArgs ep, int* err) {
  static_assert(2 * T * LD * 4 <= STAGES * STAGE_BYTES, "both halves of the partial tile take the ring's place");
  constexpr int WARPS = NTHREADS / 32;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);  // both CTAs have written the stage
  uint64_t* done = full + STAGES;                                             // the stage's MMAs have finished
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + STAGES);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank(), lead = rank & ~1u;
  const bool leader = rank == lead;
  const int m0 = blockIdx.x * T;
  const int n0 = blockIdx.y * 2 * T;
  const int nb = n0 + (int)(rank & 1u) * T;  // the columns whose B this CTA supplies
  const int S = gridDim.z;
  const int chunks = (K + KC - 1) / KC;
  const int per = (chunks + S - 1) / S;
  const int c0 = min(chunks, (int)blockIdx.z * per), nc = min(chunks, c0 + per) - c0;
  ptx::tmem_alloc_pair(tslot, STAGES * 2 * T, warp == 1);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(&full[s], 2 * WARPS);
      ptx::mbar_init(&done[s], 1);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // every CTA's barriers and TMEM exist before any cross-CTA use
  ptx::tc_fence_after();
  const uint32_t tmem = *tslot;
  ptx::griddep_wait();  // launched with programmatic stream serialization

  const int q = warp & 3, cg = warp >> 2;
  float acc[64];
#pragma unroll
  for (int j = 0; j < 64; ++j) acc[j] = 0.f;
  float4 va[4], vb[4];
  if (nc > 0) {
    load_part<MN>(va, A, lda, M, K, m0, c0 * KC, threadIdx.x);
    load_part<MN>(vb, B, ldb, N, K, nb, c0 * KC, threadIdx.x);
  }
  bool good = true;
  for (int c = 0; c <= nc; ++c) {
    const int s = c % STAGES;
    if (c < nc) {
      // stage s and its TMEM buffer are free: this warp added chunk c - STAGES,
      // whose MMAs had then finished, and the MMAs wait for every warp
      uint8_t* op = smem + s * STAGE_BYTES;
      store_part(op, va, threadIdx.x);
      store_part(op + OP_BYTES, vb, threadIdx.x);
      ptx::fence_async_smem();  // read by the MMAs (async proxy)
      ptx::tc_fence_before();   // this warp's TMEM reads come before the buffer's next MMAs
      __syncwarp();
      if (lane == 0) {
        if (leader)
          ptx::mbar_arrive(&full[s]);
        else
          ptx::mbar_arrive_remote(&full[s], lead);
      }
      if (leader && threadIdx.x == 0) {
        if (ptx::mbar_wait_cluster(&full[s], (uint32_t)(c / STAGES) & 1u, kWaitTimeoutNs, abort_flag)) {
          ptx::tc_fence_after();
          issue_chunk<MN, true>(tmem + (uint32_t)(s * 2 * T), op);
          ptx::umma_commit_pair(&done[s], (uint16_t)(3u << lead));
        } else {
          latch(err, abort_flag);
        }
      }
      __syncwarp();
    }
    if (c > 0) {
      const int sp = (c - 1) % STAGES;
      const bool ok = ptx::mbar_wait(&done[sp], (uint32_t)((c - 1) / STAGES) & 1u, kWaitTimeoutNs, abort_flag);
      if (!ok) latch(err, abort_flag);
      good = __all_sync(0xffffffffu, ok && !*abort_flag);
      if (!good) break;
      ptx::tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t r[32];
        ptx::tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(sp * 2 * T + cg * 64 + h * 32), r);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[32 * h + j] = __fadd_rn(acc[32 * h + j], __uint_as_float(r[j]));
      }
    }
    if (c + 1 < nc) {
      load_part<MN>(va, A, lda, M, K, m0, (c0 + c + 1) * KC, threadIdx.x);
      load_part<MN>(vb, B, ldb, N, K, nb, (c0 + c + 1) * KC, threadIdx.x);
    }
  }
  if (!good) {
    // MMAs already issued finish before shared memory and TMEM are released
    const uint64_t t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 1000000ull) {
    }
  }
  // every warp has seen the last chunk's MMAs finish, so nothing reads the
  // ring any more: the partial tile takes its place, as two 128-column halves
  __syncthreads();
  if (good) {
    float* row = reinterpret_cast<float*>(smem) + ((cg >> 1) * T + q * 32 + lane) * LD + (cg & 1) * 64;
#pragma unroll
    for (int j = 0; j < 64; j += 4)
      *reinterpret_cast<float4*>(row + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
  }
  if (threadIdx.x == 0) ptx::griddep_launch_dependents();
  ptx::tc_fence_before();
  ptx::cluster_sync();  // every partial of the tile is in place; the pair is done with TMEM
  ptx::tc_fence_after();
  if (warp == 1) ptx::tmem_dealloc_pair(tmem, STAGES * 2 * T);
  const int half = threadIdx.x / NT;
  if (!*abort_flag && n0 + half * T < N)
    f32_tile_epilogue<T, MODE>(reinterpret_cast<const float*>(smem) + half * T * LD, threadIdx.x % NT, M, N, m0,
                               n0 + half * T, S, ep, AdamArgs{}, rank & 1u, 2u);
  ptx::cluster_sync();  // no CTA leaves while another reads its partial tile
}

template <bool MN, int MODE>
cudaError_t launch(const float* A, int lda, const float* B, int ldb, int M, int N, int K, int S, bool pair,
                   const EpiArgs& ep, int* err, cudaStream_t st) {
  const cudaError_t attr = pair ? allow_smem<k_f32tc_pair<MN, MODE>>(SMEM) : allow_smem<k_f32tc_gemm<MN, MODE>>(SMEM);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = pair ? dim3(2 * cdiv(M, 2 * T), cdiv(N, 2 * T), S) : dim3(cdiv(M, T), cdiv(N, T), S);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = pair ? 2 : 1;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = S;
  cfg.attrs = at;
  cfg.numAttrs = pair || S > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, pair ? k_f32tc_pair<MN, MODE> : k_f32tc_gemm<MN, MODE>, A, lda, B, ldb, M, N, K, ep,
                            err);
}

}  // namespace

cudaError_t f32tc_gemm_fwd(const float* A, int lda, const float* B, int ldb, int M, int N, int K, int S, bool pair,
                           const EpiArgs& ep, int* err, cudaStream_t st) {
  return launch<false, MODE_FWD>(A, lda, B, ldb, M, N, K, S, pair, ep, err, st);
}

cudaError_t f32tc_gemm_store(const float* A, int lda, const float* B, int ldb, int M, int N, int K, int S, bool pair,
                             float* C, int ldc, int* err, cudaStream_t st) {
  EpiArgs ep{nullptr, nullptr, C, ldc, nullptr};
  return launch<false, MODE_STORE>(A, lda, B, ldb, M, N, K, S, pair, ep, err, st);
}

cudaError_t f32tc_gemm_wgrad(const float* G, int ldg, const float* X, int ldx, int R, int N, int K, int S, bool pair,
                             float* C, int ldc, int* err, cudaStream_t st) {
  EpiArgs ep{nullptr, nullptr, C, ldc, nullptr};
  return launch<true, MODE_STORE>(G, ldg, X, ldx, N, K, R, S, pair, ep, err, st);
}

}  // namespace ff

// a2 (materialized) and operand staging for the tensor-core paths.
//
//   encode_f32    A_coded row (i h + j) = sum_{s in supp(c_i)} A[s h + j]  (FP32)
//   encode_split  the same sum, then split into bf16 hi = RN(x) and
//                 lo = RN(x - hi) (or hi only for plain bf16), K-major rows
//                 ready for the TMA loads of the tcgen05 GEMM
//   b_split       B (K x N, FP32) -> B^T hi / lo (N x K, bf16, K-major)
//   encode_f16    the same sum per coded row, scaled by 2^e (e from the
//                 row's largest magnitude, f16_scale_exp), split into fp16
//                 hi = RN(x) and lo = RN(x - hi); e stored per coded row
//   b_colmax / b_split_f16
//                 max |B| per column, then B^T hi / lo in fp16 under the
//                 column's 2^e
//
// c_i is the i-th surviving cell of the plan.  Rows of A past M read as zero
// (the zero padding of the last source blocks).  All are HBM-bound streams.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "device_common.cuh"

namespace bpx {
namespace {

constexpr int kEncThreads = 128;
constexpr int kEncVec = 8;  // consecutive K elements per thread (two float4 loads per source)

// An FP32 value as three bf16 parts: p1 = RN(x), p2 = RN(x - p1), p3 = x - p1
// - p2, whose sum is x exactly (8 significand bits each) while x lies in
// [2^-102, 2^127): p1 does not round up to infinity and p3's last bit is a
// normal bf16.  Zero is exact too; any other value is reported.

// |x| lies outside [2^-102, 2^(top - 127)) and is not zero.
template <uint32_t top>
__device__ __forceinline__ bool parts_outside(float x) {
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
  return u != 0u && u - (25u << 23) >= (top - 25u) << 23;
}
// Splits eight elements; returns whether one is outside [2^-102, 2^32).
__device__ __forceinline__ bool parts_split8(const float (&v)[8], __nv_bfloat16* o1, __nv_bfloat16* o2,
                                             __nv_bfloat16* o3) {
  uint32_t w1[4], w2[4], w3[4];
  bool odd = false;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float x0 = v[2 * q], x1 = v[2 * q + 1];
    odd |= parts_outside<127 + 32>(x0) | parts_outside<127 + 32>(x1);
    const __nv_bfloat162 p1 = __floats2bfloat162_rn(x0, x1);
    const float2 f1 = __bfloat1622float2(p1);
    const float r0 = x0 - f1.x, r1 = x1 - f1.y;
    const __nv_bfloat162 p2 = __floats2bfloat162_rn(r0, r1);
    const float2 f2 = __bfloat1622float2(p2);
    const __nv_bfloat162 p3 = __floats2bfloat162_rn(r0 - f2.x, r1 - f2.y);
    w1[q] = *reinterpret_cast<const uint32_t*>(&p1);
    w2[q] = *reinterpret_cast<const uint32_t*>(&p2);
    w3[q] = *reinterpret_cast<const uint32_t*>(&p3);
  }
  *reinterpret_cast<uint4*>(o1) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  *reinterpret_cast<uint4*>(o2) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
  *reinterpret_cast<uint4*>(o3) = make_uint4(w3[0], w3[1], w3[2], w3[3]);
  return odd;
}
// Of eight elements with one outside that range: notes an element that the
// parts cannot hold, else raises ctr[word] to their largest magnitude (float
// bits).  Ordinary operands come here never; where all are large a warp reads
// the word every time (1000 x 1416 x 1100 62 -> 67 us, 4096 cubed 665 -> 688).
static_assert(kF32Plain == 0x1p32f, "magnitudes below are not noted");
__device__ __noinline__ void note_parts8(int32_t* ctr, int word, const float4 a, const float4 b) {
  const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  bool unfit = false;
  uint32_t most = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    unfit |= parts_outside<254>(v[q]);
    most = max(most, __float_as_uint(fabsf(v[q])));
  }
  if (unfit) {
    ctr[CTR_F32_SIMT] = 1;
    return;
  }
  const unsigned lanes = __activemask();
  most = __reduce_max_sync(lanes, most);
  auto* at = reinterpret_cast<uint32_t*>(ctr + word);
  if ((threadIdx.x & 31) == __ffs(lanes) - 1 && *reinterpret_cast<volatile uint32_t*>(at) < most)
    atomicMax(at, most);
}
__device__ __forceinline__ void note_parts8(int32_t* ctr, int word, const float (&v)[8]) {
  note_parts8(ctr, word, make_float4(v[0], v[1], v[2], v[3]), make_float4(v[4], v[5], v[6], v[7]));
}

// A CTA covers `rows` coded rows x `cols` columns (cols = min(1024, K rounded
// up to a power of two), rows = 1024 / cols): short K still fills the CTA.
// blockIdx.x walks the coded rows fastest so that CTAs resident together read
// the same K-chunk of A (L2 reuse of a source block across the cells that
// contain it).
template <int kMode>  // 0: FP32 out, 1: bf16 hi only, 2: bf16 hi + lo, 3: three bf16 parts
__device__ __forceinline__ void encode_body(const DevGraph& g, const DevPlan& p,
                                            const float* __restrict__ A, int M, int K, int h,
                                            float* out_f32, __nv_bfloat16* out_hi,
                                            __nv_bfloat16* out_lo, int rblock, int kchunk,
                                            __nv_bfloat16* out_3 = nullptr) {
  const int tpr = enc_threads_per_row(K);  // threads per row
  const int row = rblock * (kEncThreads / tpr) + threadIdx.x / tpr;  // coded row, compacted order
  const int nsurv = p.ctr[CTR_NSURV];
  if (row >= nsurv * h) return;
  const int ci = row / h, j = row - ci * h;
  const int cell = p.surv[ci];
  const int e0 = g.cell_ptr[cell], e1 = g.cell_ptr[cell + 1];
  const int k8 = (kchunk * tpr + threadIdx.x % tpr) * kEncVec;
  if (k8 >= K) return;
  const bool full = k8 + kEncVec <= K;  // K % 8 == 0, so a chunk is full or absent
  // the 8 sums as packed pairs (add.rn.f32x2: two FP32 adds an issue slot,
  // each rounded as a scalar add; the same ascending order per element)
  uint64_t acc2[kEncVec / 2] = {0, 0, 0, 0};
  if (full) {
    for (int e = e0; e < e1; ++e) {
      const long long arow = static_cast<long long>(__ldg(g.cell_src + e)) * h + j;
      if (arow >= M) continue;
      const float* src = A + arow * K + k8;
      uint64_t x[kEncVec / 2];
      asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[0]), "=l"(x[1]) : "l"(src));
      asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[2]), "=l"(x[3]) : "l"(src + 4));
#pragma unroll
      for (int q = 0; q < kEncVec / 2; ++q) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc2[q]) : "l"(x[q]));
    }
  }
  if (!full) return;
  float acc[kEncVec];
#pragma unroll
  for (int q = 0; q < kEncVec / 2; ++q) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * q]), "=f"(acc[2 * q + 1]) : "l"(acc2[q]));
  const long long o = static_cast<long long>(row) * K + k8;
  if (kMode == 0) {
    float4* d = reinterpret_cast<float4*>(out_f32 + o);
    d[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    d[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  } else if constexpr (kMode == 3) {
    if (parts_split8(acc, out_hi + o, out_lo + o, out_3 + o)) note_parts8(p.ctr, CTR_F32_AMAX, acc);
  } else {
    uint32_t hv[4], lv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const __nv_bfloat162 hh = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
      hv[q] = *reinterpret_cast<const uint32_t*>(&hh);
      if (kMode == 2) {
        const float2 f = __bfloat1622float2(hh);
        const __nv_bfloat162 ll = __floats2bfloat162_rn(acc[2 * q] - f.x, acc[2 * q + 1] - f.y);
        lv[q] = *reinterpret_cast<const uint32_t*>(&ll);
      }
    }
    *reinterpret_cast<uint4*>(out_hi + o) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
    if (kMode == 2) *reinterpret_cast<uint4*>(out_lo + o) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
  }
}

template <int kMode>
__global__ void __launch_bounds__(kEncThreads)
encode_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h,
              float* out_f32, __nv_bfloat16* out_hi, __nv_bfloat16* out_lo) {
  chain_wait();
  encode_body<kMode>(g, p, A, M, K, h, out_f32, out_hi, out_lo, blockIdx.x, blockIdx.y);
}

__global__ void __launch_bounds__(kEncThreads)
encode_parts_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h, __nv_bfloat16* o1,
                    __nv_bfloat16* o2, __nv_bfloat16* o3) {
  chain_wait();
  encode_body<3>(g, p, A, M, K, h, nullptr, o1, o2, blockIdx.x, blockIdx.y, o3);
}

// The FP32 encode behind the tensor-core FP32 GEMM: a fixed grid walks the
// (row block, k-chunk) blocks when the staged operands are left to the CUDA
// cores.
__global__ void __launch_bounds__(kEncThreads)
encode_f32_flagged_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h, float* out,
                          long long row_blocks, long long blocks) {
  chain_wait();
  if (!f32_on_cuda_cores(p.ctr + CTR_F32_SIMT, K)) return;
  for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
    const long long kc = b / row_blocks;
    encode_body<0>(g, p, A, M, K, h, out, nullptr, nullptr, static_cast<int>(b - kc * row_blocks), static_cast<int>(kc));
  }
}

// B (K x N row-major FP32) -> Bt (N x K row-major bf16) through a 64 x 64
// shared-memory tile: float4 reads along N, 16-byte bf16 writes along K.
constexpr int kTile = 64;
template <bool kParts3 = false>
__device__ __forceinline__ void b_split_body(const float* __restrict__ B, int K, int N, int ldb,
                                             __nv_bfloat16* bt_hi, __nv_bfloat16* bt_lo, int bx,
                                             int by, __nv_bfloat16* bt_3 = nullptr, int32_t* ctr = nullptr) {
  __shared__ float tile[kTile][kTile + 1];
  const int n0 = bx * kTile, k0 = by * kTile;
  {
    // 64 rows (k) x 16 float4 (n): 4 float4 per thread
    const int c4 = threadIdx.x & 15, r0 = threadIdx.x >> 4;  // 16 x 16
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + 16 * i, k = k0 + r, n = n0 + 4 * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < K && n < N) v = __ldg(reinterpret_cast<const float4*>(B + static_cast<long long>(k) * ldb + n));
      tile[r][4 * c4 + 0] = v.x;
      tile[r][4 * c4 + 1] = v.y;
      tile[r][4 * c4 + 2] = v.z;
      tile[r][4 * c4 + 3] = v.w;
    }
  }
  __syncthreads();
  // 64 n-rows x 8 chunks of 8 k: thread -> (n = t / 8, chunk = t % 8), two rounds
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t = threadIdx.x + 256 * i;
    const int r = t >> 3, kc = t & 7;
    const int n = n0 + r, k = k0 + 8 * kc;
    if (n >= N || k >= K) continue;
    if constexpr (kParts3) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = tile[8 * kc + q][r];
      const long long o = static_cast<long long>(n) * K + k;
      if (parts_split8(v, bt_hi + o, bt_lo + o, bt_3 + o)) note_parts8(ctr, CTR_F32_BMAX, v);
    } else {
      uint32_t hv[4], lv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float x0 = tile[8 * kc + 2 * q][r], x1 = tile[8 * kc + 2 * q + 1][r];
        const __nv_bfloat162 hh = __floats2bfloat162_rn(x0, x1);
        hv[q] = *reinterpret_cast<const uint32_t*>(&hh);
        const float2 f = __bfloat1622float2(hh);
        const __nv_bfloat162 ll = __floats2bfloat162_rn(x0 - f.x, x1 - f.y);
        lv[q] = *reinterpret_cast<const uint32_t*>(&ll);
      }
      const long long o = static_cast<long long>(n) * K + k;
      *reinterpret_cast<uint4*>(bt_hi + o) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
      if (bt_lo) *reinterpret_cast<uint4*>(bt_lo + o) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
    }
  }
}

__global__ void __launch_bounds__(256)
b_parts_kernel(DevPlan p, const float* __restrict__ B, int K, int N, int ldb, __nv_bfloat16* o1, __nv_bfloat16* o2,
               __nv_bfloat16* o3, bool early) {
  chain_begin_staging(early);
  b_split_body<true>(B, K, N, ldb, o1, o2, blockIdx.x, blockIdx.y, o3, p.ctr);
  chain_end_staging(early);
}

__global__ void __launch_bounds__(256)
b_split_kernel(const float* __restrict__ B, int K, int N, int ldb, __nv_bfloat16* bt_hi, __nv_bfloat16* bt_lo,
               bool early) {
  chain_begin_staging(early);
  b_split_body(B, K, N, ldb, bt_hi, bt_lo, blockIdx.x, blockIdx.y);
  chain_end_staging(early);
}

// Grouped launches: a flat grid over every job's CTAs; each CTA finds its job
// and its local (x, y) block, x fastest as in the single-job grids.
__global__ void __launch_bounds__(256)
b_split_group_kernel(const GJob* __restrict__ jobs, const long long* __restrict__ bases, int njobs) {
  const long long b = blockIdx.x;
  const int j = find_base(bases, njobs, b);
  const GJob& J = jobs[j];
  const uint32_t local = static_cast<uint32_t>(b - __ldg(bases + j));  // < 2^31: one launch's CTAs
  const uint32_t gx = (J.N + kTile - 1) / kTile, by = local / gx;
  b_split_body(J.B, J.K, J.N, J.N, static_cast<__nv_bfloat16*>(J.b_hi), static_cast<__nv_bfloat16*>(J.b_lo),
               static_cast<int>(local - by * gx), static_cast<int>(by));
}

// The grouped encode: a CTA takes kEncGroupRows row blocks of one job over
// every k-chunk.  Its rows' cells, source lists and positions are looked up
// once, all rows at the same time, into shared memory; the rows then cost no
// dependent loads but their sources'.  (Looked up row block after row block,
// four dependent loads each, the CTA waited longer for them than for its
// data.)  Each thread's 8-element chunk sums the same sources in the same
// ascending order as encode_body: the same bits.  48-job batch: 517 -> 433 us
// (509 with one source's loads at a time; the single-job encode, whose resident
// CTAs share a k-chunk, is slower with four: 127 -> 151 us on the benchmark).
template <int kMode>
__device__ __forceinline__ void sum_split_store(const DevGraph& g, const float* __restrict__ A, int M, int K, int h,
                                                int e0, int e1, int j, int k8, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  uint64_t acc2[kEncVec / 2] = {0, 0, 0, 0};
  int e = e0;
  for (; e + 4 <= e1; e += 4) {  // four sources' loads in flight (rows past M add +0, which changes no sum)
    uint64_t x[4][kEncVec / 2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long arow = static_cast<long long>(__ldg(g.cell_src + e + u)) * h + j;
#pragma unroll
      for (int q = 0; q < kEncVec / 2; ++q) x[u][q] = 0;
      if (arow < M) {
        const float* src = A + arow * K + k8;
        asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[u][0]), "=l"(x[u][1]) : "l"(src));
        asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[u][2]), "=l"(x[u][3]) : "l"(src + 4));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int q = 0; q < kEncVec / 2; ++q) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc2[q]) : "l"(x[u][q]));
  }
  for (; e < e1; ++e) {
    const long long arow = static_cast<long long>(__ldg(g.cell_src + e)) * h + j;
    if (arow >= M) continue;
    const float* src = A + arow * K + k8;
    uint64_t x[kEncVec / 2];
    asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[0]), "=l"(x[1]) : "l"(src));
    asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(x[2]), "=l"(x[3]) : "l"(src + 4));
#pragma unroll
    for (int q = 0; q < kEncVec / 2; ++q) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc2[q]) : "l"(x[q]));
  }
  float acc[kEncVec];
#pragma unroll
  for (int q = 0; q < kEncVec / 2; ++q)
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * q]), "=f"(acc[2 * q + 1]) : "l"(acc2[q]));
  uint32_t hv[4], lv[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const __nv_bfloat162 hh = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
    hv[q] = *reinterpret_cast<const uint32_t*>(&hh);
    if (kMode == 2) {
      const float2 f = __bfloat1622float2(hh);
      const __nv_bfloat162 ll = __floats2bfloat162_rn(acc[2 * q] - f.x, acc[2 * q + 1] - f.y);
      lv[q] = *reinterpret_cast<const uint32_t*>(&ll);
    }
  }
  *reinterpret_cast<uint4*>(hi) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
  if (kMode == 2) *reinterpret_cast<uint4*>(lo) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
}

template <int kMode>
__global__ void __launch_bounds__(kEncThreads)
encode_group_kernel(const GJob* __restrict__ jobs, const long long* __restrict__ bases, int njobs, int max_rows) {
  extern __shared__ int2 span[];                       // a row's sources: [x, y) of cell_src
  int* pos = reinterpret_cast<int*>(span + max_rows);  // and its position in its block
  const long long b = blockIdx.x;
  const int jb = find_base(bases, njobs, b);
  const GJob& J = jobs[jb];
  const int K = J.K, h = J.h, tpr = enc_threads_per_row(K), rpc = kEncThreads / tpr;
  const long long row0 = (b - __ldg(bases + jb)) * (static_cast<long long>(kEncGroupRows) * rpc);
  const long long live = static_cast<long long>(J.p.ctr[CTR_NSURV]) * h;
  if (row0 >= live) return;  // coded rows beyond the surviving cells'
  const int rows = static_cast<int>(min(static_cast<long long>(kEncGroupRows) * rpc, live - row0));
  for (int r = threadIdx.x; r < rows; r += kEncThreads) {
    const int row = static_cast<int>(row0) + r, ci = row / h, cell = J.p.surv[ci];
    span[r] = make_int2(J.g.cell_ptr[cell], J.g.cell_ptr[cell + 1]);
    pos[r] = row - ci * h;
  }
  __syncthreads();
  const DevGraph g = J.g;
  const float* A = J.A;
  const int M = J.M;
  auto* hi = static_cast<__nv_bfloat16*>(J.a_hi);
  auto* lo = static_cast<__nv_bfloat16*>(J.a_lo);
  for (int r = threadIdx.x / tpr; r < rows; r += rpc) {
    const long long o = (row0 + r) * K;
    const int2 e = span[r];
    for (int k8 = (threadIdx.x % tpr) * kEncVec; k8 < K; k8 += tpr * kEncVec)
      sum_split_store<kMode>(g, A, M, K, h, e.x, e.y, pos[r], k8, hi + o + k8, lo + o + k8);
  }
}

// ---- split-fp16 staging (BPX_FP16X3) --------------------------------------
//
// One CTA per coded row: the threads sum 8 consecutive K-elements of every
// source of the row's cell at a time (ascending sources, RN FP32 adds, as the
// other encodes), take the row's largest magnitude with a block reduction,
// and write the scaled fp16 halves.  Up to kF16Keep chunks per thread stay in
// registers between the two steps: 256 threads hold rows of K <= 8192, 512
// threads K <= 16384; longer rows sum their later chunks a second time.
constexpr int kF16Keep = 4;
// Codes with at least this many sources per cell on average take the
// K-chunked form (below).
constexpr int kF16ChunkedDegree = 4;
bool encode_f16_chunked(const DevGraph& g) {
  return static_cast<long long>(g.num_edges) >= kF16ChunkedDegree * static_cast<long long>(g.num_cells);
}

__device__ __forceinline__ void coded_chunk(const DevGraph& g, const float* __restrict__ A, int M, int K, int h,
                                            int e0, int e1, int j, int k8, float (&acc)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll 4
  for (int e = e0; e < e1; ++e) {
    const long long arow = static_cast<long long>(__ldg(g.cell_src + e)) * h + j;
    if (arow >= M) continue;
    const float4* src = reinterpret_cast<const float4*>(A + arow * K + k8);
    const float4 x0 = __ldg(src), x1 = __ldg(src + 1);
    acc[0] += x0.x; acc[1] += x0.y; acc[2] += x0.z; acc[3] += x0.w;
    acc[4] += x1.x; acc[5] += x1.y; acc[6] += x1.z; acc[7] += x1.w;
  }
}

// 8 scaled values -> fp16 hi and lo (16 bytes each)
__device__ __forceinline__ void f16_split8(const float (&v)[8], int e, __half* hi, __half* lo) {
  uint32_t hv[4], lv[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float x0 = scale_pow2(v[2 * q], e), x1 = scale_pow2(v[2 * q + 1], e);
    const __half2 hh = __floats2half2_rn(x0, x1);
    const float2 f = __half22float2(hh);
    const __half2 ll = __floats2half2_rn(x0 - f.x, x1 - f.y);
    hv[q] = *reinterpret_cast<const uint32_t*>(&hh);
    lv[q] = *reinterpret_cast<const uint32_t*>(&ll);
  }
  *reinterpret_cast<uint4*>(hi) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
  *reinterpret_cast<uint4*>(lo) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
}

template <int kF16Threads>
__global__ void __launch_bounds__(kF16Threads)
encode_f16_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h, __half* out_hi,
                  __half* out_lo, int32_t* a_exp) {
  __shared__ float red[kF16Threads / 32];
  chain_wait();
  const int row = blockIdx.x;  // coded row, compacted order
  if (row >= p.ctr[CTR_NSURV] * h) return;
  const int ci = row / h, j = row - ci * h;
  const int cell = p.surv[ci];
  const int e0 = g.cell_ptr[cell], e1 = g.cell_ptr[cell + 1];
  const int nchunks = K / 8;  // K % 8 == 0
  float keep[kF16Keep][8];
#pragma unroll
  for (int it = 0; it < kF16Keep; ++it)
#pragma unroll
    for (int i = 0; i < 8; ++i) keep[it][i] = 0.f;
  // sources outermost: a thread's loads of one source are all in flight at once
  for (int e = e0; e < e1; ++e) {
    const long long arow = static_cast<long long>(__ldg(g.cell_src + e)) * h + j;
    if (arow >= M) continue;
    const float* src = A + arow * K;
    float4 x[kF16Keep][2];
#pragma unroll
    for (int it = 0; it < kF16Keep; ++it) {
      const int c = it * kF16Threads + static_cast<int>(threadIdx.x);
      if (c < nchunks) {
        x[it][0] = __ldg(reinterpret_cast<const float4*>(src + 8 * c));
        x[it][1] = __ldg(reinterpret_cast<const float4*>(src + 8 * c) + 1);
      }
    }
#pragma unroll
    for (int it = 0; it < kF16Keep; ++it) {
      const int c = it * kF16Threads + static_cast<int>(threadIdx.x);
      if (c < nchunks) {
        float* a = keep[it];
        a[0] += x[it][0].x; a[1] += x[it][0].y; a[2] += x[it][0].z; a[3] += x[it][0].w;
        a[4] += x[it][1].x; a[5] += x[it][1].y; a[6] += x[it][1].z; a[7] += x[it][1].w;
      }
    }
  }
  float amax = 0.f;
#pragma unroll
  for (int it = 0; it < kF16Keep; ++it)
#pragma unroll
    for (int i = 0; i < 8; ++i) amax = fmaxf(amax, fabsf(keep[it][i]));
  for (int c = kF16Keep * kF16Threads + static_cast<int>(threadIdx.x); c < nchunks; c += kF16Threads) {
    float v[8];
    coded_chunk(g, A, M, K, h, e0, e1, j, 8 * c, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) amax = fmaxf(amax, fabsf(v[i]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
  __syncthreads();
  amax = red[0];
#pragma unroll
  for (int w = 1; w < kF16Threads / 32; ++w) amax = fmaxf(amax, red[w]);
  const int e = f16_scale_exp(amax);
  if (threadIdx.x == 0) a_exp[row] = e;
  const long long base = static_cast<long long>(row) * K;
#pragma unroll
  for (int it = 0; it < kF16Keep; ++it) {
    const int c = it * kF16Threads + static_cast<int>(threadIdx.x);
    if (c < nchunks) f16_split8(keep[it], e, out_hi + base + 8 * c, out_lo + base + 8 * c);
  }
  for (int c = kF16Keep * kF16Threads + static_cast<int>(threadIdx.x); c < nchunks; c += kF16Threads) {
    float v[8];
    coded_chunk(g, A, M, K, h, e0, e1, j, 8 * c, v);
    f16_split8(v, e, out_hi + base + 8 * c, out_lo + base + 8 * c);
  }
}

// High-degree codes (sources in many cells) take a K-chunked form instead, in
// the encode grid (coded rows fastest, so that CTAs resident together read
// the same K-chunk of A and a source chunk read for one cell is still in L2
// for the next cells that contain it).  One CTA per coded row reads every
// source row of a cell from DRAM again for each later cell that contains
// it.  Three steps:
//   1. each thread's 8 coded sums, stored unscaled as their FP32 bit patterns
//      (upper halves in the hi buffer, lower halves in the lo buffer); their
//      largest magnitude, reduced over the row's lanes of a warp, folded into
//      the row's word by atomicMax on the float bits (non-negative floats
//      order like their bits);
//   2. per row, the word becomes the exponent e (f16_scale_exp);
//   3. per 8 elements, the sums read back, scaled by 2^e and split into fp16
//      hi / lo in place: the same bits as the one-CTA-per-row form.
__global__ void __launch_bounds__(kEncThreads)
encode_f16_sum_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h, uint16_t* out_hi,
                      uint16_t* out_lo, uint32_t* row_max) {
  chain_wait();
  const int tpr = enc_threads_per_row(K);
  const int row = blockIdx.x * (kEncThreads / tpr) + threadIdx.x / tpr;
  const bool live = row < p.ctr[CTR_NSURV] * h;
  const int k8 = (blockIdx.y * tpr + threadIdx.x % tpr) * kEncVec;
  float m = 0.f;
  if (live && k8 < K) {
    const int ci = row / h, j = row - ci * h;
    const int cell = p.surv[ci];
    float v[8];
    coded_chunk(g, A, M, K, h, g.cell_ptr[cell], g.cell_ptr[cell + 1], j, k8, v);
    uint32_t hv[4], lv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t b0 = __float_as_uint(v[2 * q]), b1 = __float_as_uint(v[2 * q + 1]);
      hv[q] = (b0 >> 16) | (b1 & 0xffff0000u);
      lv[q] = (b0 & 0xffffu) | (b1 << 16);
      m = fmaxf(m, fmaxf(fabsf(v[2 * q]), fabsf(v[2 * q + 1])));
    }
    const long long o = static_cast<long long>(row) * K + k8;
    *reinterpret_cast<uint4*>(out_hi + o) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
    *reinterpret_cast<uint4*>(out_lo + o) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
  }
  const int span = tpr < 32 ? tpr : 32;  // a row's lanes: an aligned power-of-two group
  for (int o = 1; o < span; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (live && threadIdx.x % span == 0 && m > 0.f) atomicMax(row_max + row, __float_as_uint(m));
}

__global__ void __launch_bounds__(256) encode_f16_exp_kernel(DevPlan p, int h, int32_t* a_exp) {
  chain_wait();
  const long long row = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;
  if (row < static_cast<long long>(p.ctr[CTR_NSURV]) * h)
    a_exp[row] = f16_scale_exp(__uint_as_float(static_cast<uint32_t>(a_exp[row])));
}

__global__ void __launch_bounds__(256)
encode_f16_rescale_kernel(DevPlan p, int K, int h, __half* out_hi, __half* out_lo, const int32_t* __restrict__ a_exp) {
  chain_wait();
  const long long c = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x;  // 8-element chunk
  const int per_row = K / 8;
  const long long row = c / per_row;
  if (row >= static_cast<long long>(p.ctr[CTR_NSURV]) * h) return;
  const long long o = c * 8;
  const uint4 hv = *reinterpret_cast<const uint4*>(out_hi + o);
  const uint4 lv = *reinterpret_cast<const uint4*>(out_lo + o);
  const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w}, lw[4] = {lv.x, lv.y, lv.z, lv.w};
  float v[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[2 * q] = __uint_as_float((hw[q] << 16) | (lw[q] & 0xffffu));
    v[2 * q + 1] = __uint_as_float((hw[q] & 0xffff0000u) | (lw[q] >> 16));
  }
  f16_split8(v, a_exp[row], out_hi + o, out_lo + o);
}

// max |B| per column: a cluster of eight CTAs takes 32 columns (8 float4, 32
// row phases a CTA), each CTA every eighth run of kColRows rows; the partial
// maxima meet in the first CTA's shared memory, which stores them: no clearing
// of the words before, no atomics.  HBM-bound when large; N = 1024, K = 4096
// 40 -> 7 us against 16 CTAs of 256 rows each.  The grid also clears `clear`
// words for a later kernel.
constexpr int kColRows = 128, kColSplit = 8;
__global__ void __cluster_dims__(1, kColSplit, 1) __launch_bounds__(256)
b_colmax_kernel(const float* __restrict__ B, int K, int N, int ldb, uint32_t* bmax, uint32_t* cleared,
                long long clear, bool early) {
  __shared__ float4 red[32][8];
  __shared__ float4 part[kColSplit][8];
  // another CTA's shared memory may be stored to once that CTA has started:
  // arrived here, waited for before the store, behind the column loads
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  chain_begin_staging(early);
  const int c4 = threadIdx.x & 7, ph = threadIdx.x >> 3;
  const int n = blockIdx.x * 32 + 4 * c4;
  for (long long i = (blockIdx.x * gridDim.y + blockIdx.y) * 256LL + threadIdx.x; i < clear;
       i += 256LL * gridDim.x * gridDim.y)
    cleared[i] = 0;
  float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int k0 = blockIdx.y * kColRows; n < N && k0 < K; k0 += kColSplit * kColRows) {
    const int k1 = min(K, k0 + kColRows);
#pragma unroll 4
    for (int k = k0 + ph; k < k1; k += 32) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(B + static_cast<long long>(k) * ldb + n));
      m.x = fmaxf(m.x, fabsf(v.x));
      m.y = fmaxf(m.y, fabsf(v.y));
      m.z = fmaxf(m.z, fabsf(v.z));
      m.w = fmaxf(m.w, fabsf(v.w));
    }
  }
  auto more = [&](const float4& x) {
    m.x = fmaxf(m.x, x.x);
    m.y = fmaxf(m.y, x.y);
    m.z = fmaxf(m.z, x.z);
    m.w = fmaxf(m.w, x.w);
  };
  red[ph][c4] = m;
  __syncthreads();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (ph == 0) {
#pragma unroll
    for (int q = 1; q < 32; ++q) more(red[q][c4]);
    // to part[rank] of the cluster's first CTA
    uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(&part[blockIdx.y % kColSplit][c4]));
    asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(to));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to), "f"(m.x), "f"(m.y), "f"(m.z), "f"(m.w)
                 : "memory");
  }
  __syncwarp();  // (aligned: whole warps arrive)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (blockIdx.y % kColSplit == 0 && ph == 0 && n < N) {
#pragma unroll
    for (int q = 0; q < kColSplit; ++q) more(part[q][c4]);
    bmax[n] = __float_as_uint(m.x);  // (words: the exact path's follow h others, so 4-byte aligned only)
    bmax[n + 1] = __float_as_uint(m.y);
    bmax[n + 2] = __float_as_uint(m.z);
    bmax[n + 3] = __float_as_uint(m.w);
  }
  chain_end_staging(early);
}

// B (K x N) -> B^T fp16 hi / lo (N x K) under each column's 2^e, through the
// same 64 x 64 shared-memory transpose as b_split; the first k-tile's CTAs
// also record each column's exponent for the GEMM epilogue.
__global__ void __launch_bounds__(256)
b_split_f16_kernel(const float* __restrict__ B, int K, int N, int ldb, const uint32_t* __restrict__ bmax,
                   __half* bt_hi, __half* bt_lo, int32_t* b_exp) {
  __shared__ float tile[kTile][kTile + 1];
  chain_wait();
  const int n0 = blockIdx.x * kTile, k0 = blockIdx.y * kTile;
  {
    const int c4 = threadIdx.x & 15, r0 = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + 16 * i, k = k0 + r, n = n0 + 4 * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < K && n < N) v = __ldg(reinterpret_cast<const float4*>(B + static_cast<long long>(k) * ldb + n));
      tile[r][4 * c4 + 0] = v.x;
      tile[r][4 * c4 + 1] = v.y;
      tile[r][4 * c4 + 2] = v.z;
      tile[r][4 * c4 + 3] = v.w;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t = threadIdx.x + 256 * i;
    const int r = t >> 3, kc = t & 7;
    const int n = n0 + r, k = k0 + 8 * kc;
    if (n >= N || k >= K) continue;
    const int e = f16_scale_exp(__uint_as_float(__ldg(bmax + n)));
    if (blockIdx.y == 0 && kc == 0) b_exp[n] = e;
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = tile[8 * kc + q][r];
    const long long o = static_cast<long long>(n) * K + k;
    f16_split8(v, e, bt_hi + o, bt_lo + o);
  }
}

// ---- MXFP8 staging -------------------------------------------------------
//
// Every run of 32 consecutive K-elements of a row gets one UE8M0 scale 2^e,
// e = the smallest integer with amax / 2^e <= 448 (the largest finite E4M3),
// and its elements become RN-satfinite E4M3 of x / 2^e.  The four threads
// that own a 32-run (8 elements each) agree on amax through shuffles.

__device__ __forceinline__ int ue8m0_of(float amax) {
  if (!(amax > 0.f)) return 0;
  const float y = amax / 448.f;
  const uint32_t bits = __float_as_uint(y);
  int e = static_cast<int>((bits >> 23) & 0xFF) - 127;
  if ((bits & 0x7FFFFF) != 0 || ((bits >> 23) & 0xFF) == 0) e += 1;  // ceil(log2 y)
  return max(0, min(254, e + 127));
}

__device__ __forceinline__ uint2 e4m3x8(const float (&v)[8], int sbyte) {
  const int e = sbyte - 127;
  uint32_t w[2] = {0u, 0u};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_fp8x2_storage_t q = __nv_cvt_float2_to_fp8x2(
        make_float2(ldexpf(v[2 * i], -e), ldexpf(v[2 * i + 1], -e)), __NV_SATFINITE, __NV_E4M3);
    w[i >> 1] |= static_cast<uint32_t>(q) << (16 * (i & 1));
  }
  return make_uint2(w[0], w[1]);
}

// Coded A -> E4M3 rows + A scale blocks (512 B per 128-row tile and 128-wide
// K stage: byte 16 l + 4 q + j holds row 32 q + l, K-run 4 s + j).
__device__ __forceinline__ void encode_mx_body(const DevGraph& g, const DevPlan& p,
                                               const float* __restrict__ A, int M, int K, int h,
                                               uint8_t* out, uint8_t* sfa, int rblock, int kchunk) {
  const int tpr = enc_threads_per_row(K);
  const int row = rblock * (kEncThreads / tpr) + threadIdx.x / tpr;
  const int nsurv = p.ctr[CTR_NSURV];
  const int k8 = (kchunk * tpr + threadIdx.x % tpr) * kEncVec;
  const bool valid = row < nsurv * h && k8 < K;
  float acc[kEncVec];
#pragma unroll
  for (int i = 0; i < kEncVec; ++i) acc[i] = 0.f;
  if (valid) {
    const int ci = row / h, j = row - ci * h;
    const int cell = p.surv[ci];
    for (int e = g.cell_ptr[cell]; e < g.cell_ptr[cell + 1]; ++e) {
      const long long arow = static_cast<long long>(__ldg(g.cell_src + e)) * h + j;
      if (arow >= M) continue;
      const float4* src = reinterpret_cast<const float4*>(A + arow * K + k8);
      const float4 x0 = __ldg(src), x1 = __ldg(src + 1);
      acc[0] += x0.x; acc[1] += x0.y; acc[2] += x0.z; acc[3] += x0.w;
      acc[4] += x1.x; acc[5] += x1.y; acc[6] += x1.z; acc[7] += x1.w;
    }
  }
  float am = 0.f;
#pragma unroll
  for (int i = 0; i < kEncVec; ++i) am = fmaxf(am, fabsf(acc[i]));
  am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, 1));
  am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, 2));
  if (!valid) return;
  const int sbyte = ue8m0_of(am);
  *reinterpret_cast<uint2*>(out + static_cast<long long>(row) * K + k8) = e4m3x8(acc, sbyte);
  if ((k8 & 31) == 0) {
    const int kblk = k8 >> 5, ks = kblk >> 2, kb = kblk & 3, KS = K / 128;
    const int mt = row >> 7, rr = row & 127;
    sfa[(static_cast<long long>(mt) * KS + ks) * 512 + 16 * (rr & 31) + 4 * (rr >> 5) + kb] =
        static_cast<uint8_t>(sbyte);
  }
}

__global__ void __launch_bounds__(kEncThreads)
encode_mx_kernel(DevGraph g, DevPlan p, const float* __restrict__ A, int M, int K, int h, uint8_t* out,
                 uint8_t* sfa) {
  chain_wait();
  encode_mx_body(g, p, A, M, K, h, out, sfa, blockIdx.x, blockIdx.y);
}

// B (K x N FP32) -> B^T E4M3 (N x K) + B scale blocks (1 KB per 256-column
// tile and 128-wide K stage: byte 512 t + 16 l + 4 c + j holds column
// 128 t + 32 c + l, K-run 4 s + j).
__global__ void __launch_bounds__(256)
b_mx_kernel(const float* __restrict__ B, int K, int N, uint8_t* bt, uint8_t* sfb, bool early) {
  __shared__ float tile[kTile][kTile + 1];
  chain_begin_staging(early);
  const int n0 = blockIdx.x * kTile, k0 = blockIdx.y * kTile;
  {
    const int c4 = threadIdx.x & 15, r0 = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + 16 * i, k = k0 + r, n = n0 + 4 * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < K && n < N) v = __ldg(reinterpret_cast<const float4*>(B + static_cast<long long>(k) * N + n));
      tile[r][4 * c4 + 0] = v.x;
      tile[r][4 * c4 + 1] = v.y;
      tile[r][4 * c4 + 2] = v.z;
      tile[r][4 * c4 + 3] = v.w;
    }
  }
  __syncthreads();
  const int KS = K / 128;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t = threadIdx.x + 256 * i;
    const int r = t >> 3, kc = t & 7;  // 8 consecutive lanes share a column; 4 lanes = one 32-run
    const int n = n0 + r, k = k0 + 8 * kc;
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = tile[8 * kc + q][r];
    float am = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) am = fmaxf(am, fabsf(v[q]));
    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, 1));
    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, 2));
    if (n >= N || k >= K) continue;
    const int sbyte = ue8m0_of(am);
    *reinterpret_cast<uint2*>(bt + static_cast<long long>(n) * K + k) = e4m3x8(v, sbyte);
    if ((kc & 3) == 0) {
      const int kblk = k >> 5, ks = kblk >> 2, kb = kblk & 3;
      const int nt = n >> 8, nn = n & 255;
      sfb[(static_cast<long long>(nt) * KS + ks) * 1024 + 512 * (nn >> 7) + 16 * (nn & 31) +
          4 * ((nn & 127) >> 5) + kb] = static_cast<uint8_t>(sbyte);
    }
  }
  chain_end_staging(early);
}

}  // namespace

cudaError_t launch_encode_mx(const DevGraph& g, const DevPlan& p, const float* A, int M, int K, int h,
                             void* out, void* sfa, cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(enc_row_blocks(rows, K)), static_cast<unsigned>(enc_k_chunks(K)));
  return launch(encode_mx_kernel, grid, kEncThreads, 0, st, g, p, A, M, K, h, static_cast<uint8_t*>(out),
                static_cast<uint8_t*>(sfa));
}

cudaError_t launch_b_mx(const float* B, int K, int N, void* bt, void* sfb, cudaStream_t st, bool early) {
  if (K == 0 || N == 0) return cudaSuccess;
  dim3 grid((N + kTile - 1) / kTile, (K + kTile - 1) / kTile);
  return launch(b_mx_kernel, grid, 256, 0, st, B, K, N, static_cast<uint8_t*>(bt), static_cast<uint8_t*>(sfb), early);
}

cudaError_t launch_encode_f32(const DevGraph& g, const DevPlan& p, const float* A, int M, int K,
                              int h, float* out, cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(enc_row_blocks(rows, K)), static_cast<unsigned>(enc_k_chunks(K)));
  return launch(encode_kernel<0>, grid, kEncThreads, 0, st, g, p, A, M, K, h, out, nullptr, nullptr);
}

cudaError_t launch_encode_split(const DevGraph& g, const DevPlan& p, const float* A, int M, int K,
                                int h, void* a_hi, void* a_lo, cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(enc_row_blocks(rows, K)), static_cast<unsigned>(enc_k_chunks(K)));
  auto hi = static_cast<__nv_bfloat16*>(a_hi);
  auto lo = static_cast<__nv_bfloat16*>(a_lo);
  return launch(lo ? encode_kernel<2> : encode_kernel<1>, grid, kEncThreads, 0, st, g, p, A, M, K, h, nullptr, hi, lo);
}

cudaError_t launch_b_split_group(const GJob* d_jobs, const long long* d_bases, int njobs, long long total_ctas,
                                 cudaStream_t st) {
  if (total_ctas <= 0) return cudaSuccess;
  b_split_group_kernel<<<static_cast<unsigned>(total_ctas), 256, 0, st>>>(d_jobs, d_bases, njobs);
  return cudaGetLastError();
}

cudaError_t launch_encode_split_group(const GJob* d_jobs, const long long* d_bases, int njobs,
                                      long long total_ctas, int min_K, bool split, cudaStream_t st) {
  if (total_ctas <= 0) return cudaSuccess;
  const int max_rows = kEncGroupRows * (kEncThreads / enc_threads_per_row(min_K));
  const size_t smem = static_cast<size_t>(max_rows) * (sizeof(int2) + sizeof(int));
  const unsigned grid = static_cast<unsigned>(total_ctas);
  // plain bf16 jobs have no lo buffer: the hi-only variant never touches it
  if (split)
    encode_group_kernel<2><<<grid, kEncThreads, smem, st>>>(d_jobs, d_bases, njobs, max_rows);
  else
    encode_group_kernel<1><<<grid, kEncThreads, smem, st>>>(d_jobs, d_bases, njobs, max_rows);
  return cudaGetLastError();
}

cudaError_t launch_encode_f16(const DevGraph& g, const DevPlan& p, const float* A, int M, int K, int h,
                              void* a_hi, void* a_lo, int32_t* a_exp, cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  if (rows > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto* hi = static_cast<__half*>(a_hi);
  auto* lo = static_cast<__half*>(a_lo);
  if (encode_f16_chunked(g)) {  // high mean degree: the K-chunked form (the B staging has cleared a_exp)
    const dim3 grid(static_cast<unsigned>(enc_row_blocks(rows, K)), static_cast<unsigned>(enc_k_chunks(K)));
    const long long chunks = rows * (K / 8);
    if ((chunks + 255) / 256 > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaError_t e = launch(encode_f16_sum_kernel, grid, kEncThreads, 0, st, g, p, A, M, K, h,
                           static_cast<uint16_t*>(a_hi), static_cast<uint16_t*>(a_lo),
                           reinterpret_cast<uint32_t*>(a_exp));
    if (e != cudaSuccess) return e;
    e = launch(encode_f16_exp_kernel, dim3(static_cast<unsigned>((rows + 255) / 256)), 256, 0, st, p, h, a_exp);
    if (e != cudaSuccess) return e;
    return launch(encode_f16_rescale_kernel, dim3(static_cast<unsigned>((chunks + 255) / 256)), 256, 0, st, p, K, h, hi,
                  lo, a_exp);
  }
  const bool wide = K > 256 * 8 * kF16Keep;
  return launch(wide ? encode_f16_kernel<512> : encode_f16_kernel<256>, dim3(static_cast<unsigned>(rows)),
                wide ? 512 : 256, 0, st, g, p, A, M, K, h, hi, lo, a_exp);
}

cudaError_t launch_colmax(const float* B, int K, int N, uint32_t* bmax, uint32_t* cleared, long long clear,
                          cudaStream_t st, bool early, int ldb) {
  return launch(b_colmax_kernel, dim3((N + 31) / 32, kColSplit), 256, 0, st, B, K, N, ldb ? ldb : N, bmax, cleared,
                clear, early);
}

cudaError_t launch_b_f16(const DevGraph& g, int h, const float* B, int K, int N, void* b_hi, void* b_lo,
                         uint32_t* b_max, int32_t* b_exp, int32_t* a_exp, cudaStream_t st, bool early, int ldb) {
  if (K == 0 || N == 0) return cudaSuccess;
  const long long rows = a_exp && encode_f16_chunked(g) ? static_cast<long long>(g.num_cells) * h : 0;
  const cudaError_t e = launch_colmax(B, K, N, b_max, reinterpret_cast<uint32_t*>(a_exp), rows, st, early, ldb);
  if (e != cudaSuccess) return e;
  return launch(b_split_f16_kernel, dim3((N + kTile - 1) / kTile, (K + kTile - 1) / kTile), 256, 0, st, B, K, N,
                ldb ? ldb : N, b_max, static_cast<__half*>(b_hi), static_cast<__half*>(b_lo), b_exp);
}

cudaError_t launch_encode_parts(const DevGraph& g, const DevPlan& p, const float* A, int M, int K, int h,
                                void* const a[3], cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>(enc_row_blocks(rows, K)), static_cast<unsigned>(enc_k_chunks(K)));
  return launch(encode_parts_kernel, grid, kEncThreads, 0, st, g, p, A, M, K, h, static_cast<__nv_bfloat16*>(a[0]),
                static_cast<__nv_bfloat16*>(a[1]), static_cast<__nv_bfloat16*>(a[2]));
}

cudaError_t launch_b_parts(const DevPlan& p, const float* B, int K, int N, void* const b[3], cudaStream_t st,
                           bool early, int ldb) {
  if (K == 0 || N == 0) return cudaSuccess;
  dim3 grid((N + kTile - 1) / kTile, (K + kTile - 1) / kTile);
  return launch(b_parts_kernel, grid, 256, 0, st, p, B, K, N, ldb ? ldb : N, static_cast<__nv_bfloat16*>(b[0]),
                static_cast<__nv_bfloat16*>(b[1]), static_cast<__nv_bfloat16*>(b[2]), early);
}

cudaError_t launch_encode_f32_flagged(const DevGraph& g, const DevPlan& p, const float* A, int M, int K, int h,
                                      float* out, cudaStream_t st) {
  const long long rows = static_cast<long long>(g.num_cells) * h;
  if (rows == 0 || K == 0) return cudaSuccess;
  const long long rb = enc_row_blocks(rows, K), blocks = rb * enc_k_chunks(K);
  const unsigned grid = static_cast<unsigned>(std::min<long long>(blocks, 8LL * num_sms()));
  return launch(encode_f32_flagged_kernel, dim3(grid), kEncThreads, 0, st, g, p, A, M, K, h, out, rb, blocks);
}

cudaError_t launch_b_split(const float* B, int K, int N, void* b_hi, void* b_lo, cudaStream_t st, bool early,
                           int ldb) {
  if (K == 0 || N == 0) return cudaSuccess;
  dim3 grid((N + kTile - 1) / kTile, (K + kTile - 1) / kTile);
  return launch(b_split_kernel, grid, 256, 0, st, B, K, N, ldb ? ldb : N, static_cast<__nv_bfloat16*>(b_hi),
                static_cast<__nv_bfloat16*>(b_lo), early);
}

}  // namespace bpx

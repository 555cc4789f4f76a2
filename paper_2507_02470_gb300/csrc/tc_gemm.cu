// BF16 x BF16 -> FP32 GEMM on the 5th-generation tensor cores (tcgen05) of sm_103a.
//
// One CTA of 128 threads computes a 128 x BN tile of C = A B^T:
//   - warp 0 / lane 0 streams 128 x 64 tiles of A and BN x 64 tiles of B into a ring of
//     kStages shared-memory stages with the tensor-memory-access engine (TMA, 128-byte
//     swizzle, zero fill past the tensor edges), each stage guarded by a "full" mbarrier
//     that counts the bytes in flight;
//   - warp 1 / lane 0 issues tcgen05.mma (M = 128, N = BN, K = 16 per instruction, four per
//     stage) into an FP32 accumulator in tensor memory (TMEM), and releases each stage with
//     tcgen05.commit on its "empty" mbarrier once the MMAs that read it have finished;
//   - after the last stage a commit on the "done" mbarrier hands the accumulator to all four
//     warps, which read it back with tcgen05.ld (warp w owns TMEM lanes 32w..32w+31, i.e.
//     rows 32w.. of the tile) and store FP32 rows to global memory.
// Every mbarrier wait is bounded: when a wait gives up the kernel records an error code in
// g_tc_error, stops issuing work, still commits the done barrier so the other warps are not
// left waiting, frees its TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace hprqp {
namespace tc {
namespace {

constexpr int kBM = 128;                       // tile rows = TMEM lanes
constexpr int kBK = 64;                        // K per stage: one 128-byte swizzle row of BF16
constexpr uint32_t kATile = kBM * kBK * 2;     // bytes of one A stage

__device__ int g_tc_error;

template <int BN, int STAGES>
constexpr uint32_t smem_bytes() {
  return 1024 + STAGES * (kATile + (uint32_t)BN * kBK * 2);
}

// Epilogues: what becomes of 32 consecutive columns of one accumulator row.  row < M and col < N
// hold for the first column; columns from N on are not to be stored.
struct EpiStore {   // C[row][col..] of the K-split `split`
  float* C;
  int64_t ldc, split_stride;
  int vec;          // rows are 16-byte aligned
  static constexpr int kStages = 4, kBlocks = 1;   // a long K loop: deep ring, one CTA per SM
  struct Row {};
  __device__ __forceinline__ Row row(int) const { return Row(); }
  __device__ __forceinline__ void operator()(const Row&, int split, int row, int col, int N,
                                             const uint32_t (&r)[32]) const {
    float* d0 = C + (int64_t)split * split_stride + (int64_t)row * ldc + col;
    if (vec && col + 32 <= N) {
      float4* d = reinterpret_cast<float4*>(d0);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        d[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                           __uint_as_float(r[4 * j + 3]));
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (col + j < N) d0[j] = __uint_as_float(r[j]);
    }
  }
};

// The exact FP64 value of an FP32 one, and min(max(z, lo), hi), on the integer pipe: on GB300 the
// conversion and the FP64 min/max issue on the FP64 pipe (1.7 lanes/clk/SM).  Zeros, subnormals,
// infinities and NaN take the instructions, in functions of their own: inlined, the compiler runs
// them for every element and selects (measured: the decoder at 444 us instead of its rate below).
__device__ __noinline__ double widen_rare(uint32_t b) { return (double)__uint_as_float(b); }
__device__ __noinline__ double clip_rare(double z, double lo, double hi) { return fmin(fmax(z, lo), hi); }
__device__ __forceinline__ double widen(uint32_t b) {
  const uint32_t e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return widen_rare(b);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
// monotone map of the non-NaN doubles onto signed integers, and back
__device__ __forceinline__ long long order(double a) {
  const long long b = __double_as_longlong(a);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
// (by halves: masking the sign of the whole word is compiled to an FP64 absolute value)
__device__ __forceinline__ bool is_nan(double a) {
  const unsigned h = (unsigned)__double2hiint(a) & 0x7fffffffu;
  return h + (__double2loint(a) != 0 ? 1u : 0u) > 0x7ff00000u;
}

// Z[col][row] = clip(mu[row] + alpha acc, lo[row], hi[row]) in FP64: the decoder of the learned start.
// A warp's 32 lanes hold 32 consecutive rows of one column, so the stores of Z are coalesced without
// a transpose and the FP32 product never goes to memory.  One FP64 operation per element (19 SM
// cycles per warp) bounds it at 72 us for 150,000 x 256, beside the 45 us that writing Z's
// 307 MB takes; three CTAs per SM overlap the FP64 epilogue of one with the short K loops of the
// others.  150,000 x 256, K = 256: 155 us, against 309 us for a separate decoder kernel behind a
// 100 us product.
struct EpiDecode {
  double alpha;
  const double *mu, *lo, *hi;
  double* Z;
  int64_t ldz;
  static constexpr int kStages = 2, kBlocks = 3;
  struct Row {
    double mu;
    long long lo, hi;   // order() of the bounds
    bool rare;          // a bound is NaN
  };
  __device__ __forceinline__ Row row(int i) const {
    return Row{mu[i], order(lo[i]), order(hi[i]), is_nan(lo[i]) || is_nan(hi[i])};
  }
  __device__ __forceinline__ void operator()(const Row& q, int, int row, int col, int N,
                                             const uint32_t (&r)[32]) const {
    double* d = Z + (int64_t)col * ldz + row;
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col + j < N) {
        const double z = fma(alpha, widen(r[j]), q.mu);
        if (q.rare || is_nan(z)) {
          d[j * ldz] = clip_rare(z, lo[row], hi[row]);
        } else {
          long long k = order(z);
          k = k < q.lo ? q.lo : k;
          k = k > q.hi ? q.hi : k;
          d[j * ldz] = __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
        }
      }
  }
};

template <int BN, class Epi>
__global__ void __launch_bounds__(128, Epi::kBlocks)
    k_gemm_bf16(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const Epi epi, int M,
                int N, int kb_total, int kb_per) {
  static_assert(BN == 64 || BN == 128 || BN == 256, "TMEM columns must be a power of two >= 32");
  static_assert(BN * Epi::kBlocks <= 512, "the resident CTAs share 512 TMEM columns");
  constexpr int kStages = Epi::kStages;
  constexpr uint32_t kBTile = (uint32_t)BN * kBK * 2;
  __shared__ __align__(8) uint64_t bar_full[kStages];
  __shared__ __align__(8) uint64_t bar_empty[kStages];
  __shared__ __align__(8) uint64_t bar_done;
  __shared__ uint32_t tmem_slot;
  extern __shared__ uint8_t dsm[];
  const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;   // stages start on 1024-byte boundaries

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
  const int kb0 = blockIdx.z * kb_per;
  const int nkb = min(kb0 + kb_per, kb_total) - kb0;        // >= 1 (host)

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0 && lane == 0) {
    // producer: stage s of round r waits for the MMAs of round r-1 to release it
    for (int i = 0; i < nkb; ++i) {
      const int s = i % kStages;
      const uint32_t ph = (uint32_t)(i / kStages) & 1u;
      if (!mbar_wait(smem_u32(&bar_empty[s]), ph ^ 1u, &g_tc_error, 1)) break;
      const uint32_t fb = smem_u32(&bar_full[s]);
      mbar_expect_tx(fb, kATile + kBTile);
      const int kx = (kb0 + i) * kBK;   // multiple of 64 elements: 16-byte aligned
      tma_load_2d(base + s * kATile, &ta, fb, kx, m0);
      tma_load_2d(base + kStages * kATile + s * kBTile, &tb, fb, kx, n0);
    }
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t idesc = idesc_bf16(kBM, BN);
    for (int i = 0; i < nkb; ++i) {
      const int s = i % kStages;
      const uint32_t ph = (uint32_t)(i / kStages) & 1u;
      if (!mbar_wait(smem_u32(&bar_full[s]), ph, &g_tc_error, 2)) break;
      tc_fence_after();
      const uint64_t ad = sdesc_sw128(base + s * kATile);
      const uint64_t bd = sdesc_sw128(base + kStages * kATile + s * kBTile);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk)   // +32 bytes along K inside the swizzle row
        mma_bf16(tmem, ad + 2 * kk, bd + 2 * kk, idesc, (i > 0 || kk > 0) ? 1u : 0u);
      mma_commit(smem_u32(&bar_empty[s]));
    }
    mma_commit(smem_u32(&bar_done));    // arrives when every MMA issued above has completed
  }
  __syncwarp();

  // epilogue: TMEM lane (32 warp + lane) holds row m0 + 32 warp + lane of the tile
  const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_done), 0, &g_tc_error, 3));
  tc_fence_after();
  if (ok) {
    const int row = m0 + warp * 32 + lane;
    typename Epi::Row q = {};
    if (row < M) q = epi.row(row);
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
      const int col = n0 + c0;
      if (row < M && col < N) epi(q, (int)blockIdx.z, row, col, N, r);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
  }
}

// C[i][j] = sum_s work[s][i][j], s = 0..S-1 in order
__global__ void k_splitk_sum(const float* __restrict__ work, int S, int64_t M, int64_t N, float* __restrict__ C,
                             int64_t ldc) {
  const int64_t total = M * N, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += stride) {
    float acc = 0.f;
    for (int s = 0; s < S; ++s) acc += work[(int64_t)s * total + e];
    C[(e / N) * ldc + (e % N)] = acc;
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder(cudaError_t* err) {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static cudaError_t e0 = cudaSuccess;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    e0 = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
    if (e0 == cudaSuccess && q != cudaDriverEntryPointSuccess) e0 = cudaErrorSymbolNotFound;
    if (e0 == cudaSuccess) fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  *err = e0;
  return fn;
}


// ------------------------------------------------------------------------------------ products of the network
// A layer's product with everything that follows it, in one launch: the S K-splits of a 128 x BN tile
// are one thread-block cluster.  Each CTA leaves its FP32 partial tile in its own shared memory (the ring
// is free by then); after a cluster barrier CTA z adds rows [z R, (z + 1) R) of all S partials, read through
// distributed shared memory in split order (the sums of k_splitk_sum, bit for bit), and applies the
// epilogue.  The layers' products are 5 to 9 us each and their followers (split sum, bias, ReLU and BF16
// conversion, transposed copy) as much again in launches: a training step of 512-1024-1024-257 at batch 256
// took 28 launches and 203 us, with this form, the joined kernels of learn.cu and programmatic dependent
// launches 12 launches and 131 us (a cluster launch alone costs about 5 us, most of which these hide).
struct EpiLayer {
  const float* bias;        // HIDDEN, FINAL: per row
  const uint16_t* mask;     // MASK: BF16, M x N, ldmask
  int64_t ldmask;
  uint16_t* outT;           // HIDDEN, MASK: BF16, M x N, ldT
  int64_t ldT;
  uint16_t* outB;           // ... and transposed, N x M, ldB
  int64_t ldB;
  float* out;               // FINAL: transposed, N x M, ldo; PLAIN: M x N, ldo
  int64_t ldo;
};

__device__ __forceinline__ uint32_t cluster_rank_addr(uint32_t addr, uint32_t rank) {
  uint32_t to;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(addr), "r"(rank));
  return to;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <int BN, int MODE>
__global__ void __launch_bounds__(128, 1)
    k_gemm_layer(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, const EpiLayer e, int M,
                 int N, int kb_total, int kb_per) {
  constexpr int kStages = EpiStore::kStages;
  constexpr int kLd = BN + 4;   // row stride of the partial tile: float4 stores of 8 neighbouring rows hit all banks
  constexpr uint32_t kBTile = (uint32_t)BN * kBK * 2;
  static_assert(kBM * kLd * 4 <= kStages * (kATile + kBTile), "the partial tile takes the place of the ring");
  __shared__ __align__(8) uint64_t bar_full[kStages];
  __shared__ __align__(8) uint64_t bar_empty[kStages];
  __shared__ __align__(8) uint64_t bar_done;
  __shared__ uint32_t tmem_slot;
  extern __shared__ uint8_t dsm[];
  const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
  const int kb0 = blockIdx.z * kb_per;
  const int nkb = min(kb0 + kb_per, kb_total) - kb0;        // >= 1 (host)
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  pdl_wait();   // the set-up above overlaps the end of the kernel before
  if (warp == 0 && lane == 0) {
    for (int i = 0; i < nkb; ++i) {
      const int s = i % kStages;
      const uint32_t ph = (uint32_t)(i / kStages) & 1u;
      if (!mbar_wait(smem_u32(&bar_empty[s]), ph ^ 1u, &g_tc_error, 1)) break;
      const uint32_t fb = smem_u32(&bar_full[s]);
      mbar_expect_tx(fb, kATile + kBTile);
      const int kx = (kb0 + i) * kBK;   // multiple of 64 elements: 16-byte aligned
      tma_load_2d(base + s * kATile, &ta, fb, kx, m0);
      tma_load_2d(base + kStages * kATile + s * kBTile, &tb, fb, kx, n0);
    }
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t idesc = idesc_bf16(kBM, BN);
    for (int i = 0; i < nkb; ++i) {
      const int s = i % kStages;
      const uint32_t ph = (uint32_t)(i / kStages) & 1u;
      if (!mbar_wait(smem_u32(&bar_full[s]), ph, &g_tc_error, 2)) break;
      tc_fence_after();
      const uint64_t ad = sdesc_sw128(base + s * kATile);
      const uint64_t bd = sdesc_sw128(base + kStages * kATile + s * kBTile);
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk)
        mma_bf16(tmem, ad + 2 * kk, bd + 2 * kk, idesc, (i > 0 || kk > 0) ? 1u : 0u);
      mma_commit(smem_u32(&bar_empty[s]));
    }
    mma_commit(smem_u32(&bar_done));
  }
  __syncwarp();
  const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_done), 0, &g_tc_error, 3));
  tc_fence_after();
  // every product of this CTA has ended, so no copy or MMA touches the ring any more
  __syncthreads();
  float* tile = reinterpret_cast<float*>(dsm + (base - smem_u32(dsm)));
  if (ok) {
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
      float4* d = reinterpret_cast<float4*>(tile + (warp * 32 + lane) * kLd + c0);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        d[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                           __uint_as_float(r[4 * j + 3]));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
  }
  cluster_sync();
  // rows of this CTA, in 4 x 4 pieces per thread
  const int S = (int)gridDim.z, R = ((kBM + S - 1) / S + 3) / 4 * 4;
  const int r0 = (int)blockIdx.z * R, rows = min(R, kBM - r0);
  for (int u = threadIdx.x; u < rows / 4 * (BN / 4); u += 128) {
    const int rr = r0 + u / (BN / 4) * 4, cc = u % (BN / 4) * 4;
    float v[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i][j] = 0.f;
    for (int s0 = 0; s0 < S; s0 += 4) {   // four peers' loads in flight, added in split order
      float4 q[4][4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t peer = cluster_rank_addr(smem_u32(tile + rr * kLd + cc), (uint32_t)min(s0 + s, S - 1));
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(q[s][i].x), "=f"(q[s][i].y), "=f"(q[s][i].z), "=f"(q[s][i].w)
                       : "r"(peer + (uint32_t)(i * kLd * 4)));
      }
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (s0 + s < S) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i][0] += q[s][i].x;
            v[i][1] += q[s][i].y;
            v[i][2] += q[s][i].z;
            v[i][3] += q[s][i].w;
          }
        }
    }
    const int m = m0 + rr, n = n0 + cc;
    if (m >= M || n >= N) continue;
    const int mi = min(4, M - m), ni = min(4, N - n);
    if constexpr (MODE == LAYER_PLAIN) {
      for (int i = 0; i < mi; ++i) {
        float* d = e.out + (int64_t)(m + i) * e.ldo + n;
        for (int j = 0; j < ni; ++j) d[j] = v[i][j];
      }
      continue;
    }
    if constexpr (MODE == LAYER_FINAL) {
      for (int j = 0; j < ni; ++j)
        for (int i = 0; i < mi; ++i) e.out[(int64_t)(n + j) * e.ldo + m + i] = v[i][j] + e.bias[m + i];
      continue;
    }
    uint16_t h[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float b = MODE == LAYER_HIDDEN && i < mi ? e.bias[m + i] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float x = v[i][j];
        if (MODE == LAYER_HIDDEN) {
          x = fmaxf(x + b, 0.f);
        } else {
          const bool in = i < mi && j < ni;
          const uint16_t k = in ? e.mask[(int64_t)(m + i) * e.ldmask + n + j] : (uint16_t)0;
          x = (k & 0x8000u) == 0 && (k & 0x7fffu) != 0 && (k & 0x7fffu) <= 0x7f80u ? x : 0.f;   // mask > 0
        }
        h[i][j] = __bfloat16_as_ushort(__float2bfloat16_rn(x));
      }
    }
    // leading dimensions are multiples of 8 and the arrays 256-byte aligned: 8-byte stores of four
    for (int i = 0; i < mi; ++i) {
      uint16_t* d = e.outT + (int64_t)(m + i) * e.ldT + n;
      if (ni == 4) *reinterpret_cast<uint2*>(d) = make_uint2(h[i][0] | (h[i][1] << 16), h[i][2] | (h[i][3] << 16));
      else
        for (int j = 0; j < ni; ++j) d[j] = h[i][j];
    }
    for (int j = 0; j < ni; ++j) {
      uint16_t* d = e.outB + (int64_t)(n + j) * e.ldB + m;
      if (mi == 4) *reinterpret_cast<uint2*>(d) = make_uint2(h[0][j] | (h[1][j] << 16), h[2][j] | (h[3][j] << 16));
      else
        for (int i = 0; i < mi; ++i) d[i] = h[i][j];
    }
  }
  cluster_sync();   // no CTA ends while a peer reads its tile
}

}  // namespace

// 2-D map over a rows x cols BF16 matrix with leading dimension ld; boxes of 64 x box_rows
cudaError_t make_map(CUtensorMap* map, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  cudaError_t e;
  auto fn = encoder(&e);
  if (!fn) return e;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

namespace {

template <int BN, class Epi>
cudaError_t launch(const CUtensorMap& ta, const CUtensorMap& tb, const Epi& epi, int64_t M, int64_t N, int kb_total,
                   int kb_per, int splits, cudaStream_t s) {
  constexpr uint32_t bytes = smem_bytes<BN, Epi::kStages>();
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_gemm_bf16<BN, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  });
  if (attr != cudaSuccess) return attr;
  dim3 grid((unsigned)((M + kBM - 1) / kBM), (unsigned)((N + BN - 1) / BN), (unsigned)splits);
  k_gemm_bf16<BN, Epi><<<grid, 128, bytes, s>>>(ta, tb, epi, (int)M, (int)N, kb_total, kb_per);
  return cudaGetLastError();
}

// Lets the kernel take its shared memory and clusters of 16
template <int BN, int MODE>
cudaError_t layer_setup() {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(k_gemm_layer<BN, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_bytes<BN, EpiStore::kStages>());
    if (attr == cudaSuccess)
      attr = cudaFuncSetAttribute(k_gemm_layer<BN, MODE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  return attr;
}

template <int BN, int MODE>
cudaError_t launch_layer(const CUtensorMap& ta, const CUtensorMap& tb, const EpiLayer& epi, int64_t M, int64_t N,
                         int kb_total, int kb_per, int splits, cudaStream_t s) {
  constexpr uint32_t bytes = smem_bytes<BN, EpiStore::kStages>();
  const cudaError_t attr = layer_setup<BN, MODE>();
  if (attr != cudaSuccess) return attr;
  return launch_kernel(true, splits, k_gemm_layer<BN, MODE>,
                       dim3((unsigned)((M + kBM - 1) / kBM), (unsigned)((N + BN - 1) / BN), (unsigned)splits), dim3(128),
                       bytes, s, ta, tb, epi, (int)M, (int)N, kb_total, kb_per);
}

// The operand checks that every product shares; what is wrong, or null.
const char* check_operands(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb) {
  if (!A || !B) return "A or B is null";
  if (lda < K || ldb < K) return "lda and ldb must be >= K";
  if (lda % 8 || ldb % 8) return "lda and ldb must be multiples of 8 (16-byte rows)";
  if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return "A and B must be 16-byte aligned";
  return nullptr;
}

}  // namespace

cudaError_t gemm_bf16(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                      float* C, int64_t ldc, int splits, float* work, cudaStream_t stream, const char** why) {
  auto bad = [why](const char* w) {
    if (why) *why = w;
    return cudaErrorInvalidValue;
  };
  if (M < 0 || N < 0 || K < 0) return bad("negative size");
  if (M == 0 || N == 0) return cudaSuccess;
  if (M >= (1ll << 31) || N > 65535ll * 64 || K >= (1ll << 31)) return bad("size out of range");
  if (!C || ldc < N) return bad("C is null or ldc < N");
  if (K == 0) {
    for (int64_t i = 0; i < M; ++i) {   // rows may be strided: one memset per row
      cudaError_t e = cudaMemsetAsync(C + i * ldc, 0, (size_t)N * sizeof(float), stream);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (const char* w = check_operands(M, N, K, A, lda, B, ldb)) return bad(w);
  const int kb_total = (int)((K + kBK - 1) / kBK);
  splits = std::max(1, std::min(splits, kb_total));
  const int kb_per = (kb_total + splits - 1) / splits;
  splits = (kb_total + kb_per - 1) / kb_per;   // no empty split
  if (splits > 1 && !work) return bad("splits > 1 needs a work buffer of splits*M*N floats");
  if (splits > 65535) return bad("too many splits");
  // tile width: 256 columns (128 x 256 accumulator, 256 TMEM columns) when N is wide enough
  // to keep many tiles, else 128 or 64
  const int BN = N <= 64 ? 64 : N < 512 ? 128 : 256;
  CUtensorMap ta, tb;
  cudaError_t e;
  if ((e = make_map(&ta, A, M, K, lda, kBM)) != cudaSuccess) return e;
  if ((e = make_map(&tb, B, N, K, ldb, BN)) != cudaSuccess) return e;
  float* out = splits > 1 ? work : C;
  const int64_t ld = splits > 1 ? N : ldc;
  const int vec = ((reinterpret_cast<uintptr_t>(out) & 15) == 0 && ld % 4 == 0) ? 1 : 0;
  const EpiStore epi{out, ld, M * N, vec};
  e = BN == 64    ? launch<64>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream)
      : BN == 128 ? launch<128>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream)
                  : launch<256>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream);
  if (e != cudaSuccess || splits == 1) return e;
  const int64_t total = M * N;
  const int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  k_splitk_sum<<<blocks, 256, 0, stream>>>(work, splits, M, N, C, ldc);
  return cudaGetLastError();
}

cudaError_t gemm_decode(int64_t D, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                        double alpha, const double* mu, const double* lo, const double* hi, double* Z, int64_t ldz,
                        cudaStream_t stream, const char** why) {
  auto bad = [why](const char* w) {
    if (why) *why = w;
    return cudaErrorInvalidValue;
  };
  if (D < 1 || N < 1 || K < 1 || D >= (1ll << 31) || N > 65535ll * 64 || K >= (1ll << 31)) return bad("size out of range");
  if (const char* w = check_operands(D, N, K, A, lda, B, ldb)) return bad(w);
  // the tile width of gemm_bf16 up to 128 columns (256 would leave room for two CTAs per SM only)
  const int BN = N <= 64 ? 64 : 128;
  const int kb = (int)((K + kBK - 1) / kBK);
  CUtensorMap ta, tb;
  cudaError_t e;
  if ((e = make_map(&ta, A, D, K, lda, kBM)) != cudaSuccess) return e;
  if ((e = make_map(&tb, B, N, K, ldb, BN)) != cudaSuccess) return e;
  const EpiDecode epi{alpha, mu, lo, hi, Z, ldz};
  return BN == 64 ? launch<64>(ta, tb, epi, D, N, kb, kb, 1, stream) : launch<128>(ta, tb, epi, D, N, kb, kb, 1, stream);
}

int layer_cluster() {
  // asked of the form with the most shared memory and registers; a single block always fits
  constexpr int BN = 256;
  const auto k = k_gemm_layer<BN, LAYER_MASK>;
  int most = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = smem_bytes<BN, EpiStore::kStages>();
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = at[0].val.clusterDim.y = 1;
  int c = layer_setup<BN, LAYER_MASK>() == cudaSuccess ? kLayerSplits : 1;
  for (; c > 1; c /= 2) {
    at[0].val.clusterDim.z = (unsigned)c;
    cfg.gridDim = dim3(1, 1, (unsigned)c);
    if (cudaOccupancyMaxActiveClusters(&most, k, &cfg) == cudaSuccess && most >= 1) break;
    cudaGetLastError();
  }
  return c;
}

int layer_splits(int64_t K, int splits) {
  const int kb_total = (int)((K + kBK - 1) / kBK);
  splits = std::max(1, std::min(splits, kb_total));
  const int kb_per = (kb_total + splits - 1) / splits;
  return (kb_total + kb_per - 1) / kb_per;
}

cudaError_t gemm_layer(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                       int splits, const Layer& l, cudaStream_t stream, const char** why) {
  auto bad = [why](const char* w) {
    if (why) *why = w;
    return cudaErrorInvalidValue;
  };
  if (M < 1 || N < 1 || K < 1 || M >= (1ll << 31) || N > 65535ll * 64 || K >= (1ll << 31)) return bad("size out of range");
  if (const char* w = check_operands(M, N, K, A, lda, B, ldb)) return bad(w);
  const int kb_total = (int)((K + kBK - 1) / kBK);
  splits = layer_splits(K, splits);
  if (splits > kLayerSplits) return bad("too many splits for a cluster");
  const int kb_per = (kb_total + splits - 1) / splits;
  const int BN = N <= 64 ? 64 : N < 512 ? 128 : 256;   // the tile rule of gemm_bf16
  CUtensorMap ta, tb;
  cudaError_t e;
  if ((e = make_map(&ta, A, M, K, lda, kBM)) != cudaSuccess) return e;
  if ((e = make_map(&tb, B, N, K, ldb, BN)) != cudaSuccess) return e;
  const EpiLayer epi{l.bias, l.mask, l.ldmask, l.outT, l.ldT, l.outB, l.ldB, l.out, l.ldo};
  auto go = [&](auto mode) {
    constexpr int m = decltype(mode)::value;
    return BN == 64    ? launch_layer<64, m>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream)
           : BN == 128 ? launch_layer<128, m>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream)
                       : launch_layer<256, m>(ta, tb, epi, M, N, kb_total, kb_per, splits, stream);
  };
  switch (l.mode) {
    case LAYER_HIDDEN: return go(std::integral_constant<int, LAYER_HIDDEN>());
    case LAYER_MASK: return go(std::integral_constant<int, LAYER_MASK>());
    case LAYER_FINAL: return go(std::integral_constant<int, LAYER_FINAL>());
    default: return go(std::integral_constant<int, LAYER_PLAIN>());
  }
}

int gemm_error_flag() {
  int v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)) != cudaSuccess) return -1;
  if (v) cudaMemcpyToSymbol(g_tc_error, &z, sizeof(int));
  return v;
}

}  // namespace tc
}  // namespace hprqp

// The QAP-relaxation operator of Sec. 4.5 on the tensor cores, at FP64 accuracy:
//
//   Q vec(X) = vec(Ahat X Bhat - S X - X T),   X = reshape(x, d, d) column-major.
//
// GB300 issues one FP64 warp instruction per 16 to 19 SM cycles (1.06 TFLOP/s on the chip); the tensor
// cores multiply BF16 at 1.8 PFLOP/s with FP32 sums.  Each operand is therefore cut into seven signed
// digits of eight bits, relative to the largest magnitude of its row (for the right operand: of its
// column), the digits' products are summed exactly, and only the recombination rounds (the splitting of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication", 2012, with the
// sums in integers):
//   * an entry v of a row whose largest exponent is e is the integer q = round(v 2^(1077 - e)), |q| <= 2^55,
//     q = sum_i d_i 256^(6-i), d_i in [-128, 128]: a BF16 value holds a digit exactly;
//   * P_s = sum over i + j = s and over 64 values of k of d_i(A) d_j(B) is at most 7 * 64 * 2^14 < 2^23, so the
//     FP32 accumulators (one 64-column block of tensor memory per s) are exact; s = 0 .. 7 are kept (34 digit
//     products);
//   * the P_s are joined in two 64-bit integers (s < 4 and s >= 4), chunks of k added there, so the result does
//     not depend on any order; the last step is one FP64 rounding of the exact sum.
// Accuracy, element by element.  Let a be the power of two at or below the largest magnitude of a left operand's row
// and b that of a right operand's column.  An entry is off by at most 2^-55 a (half a unit of q), so a term of
// a product by less than 1.02 2^-53 a b, the dropped digit products (5 * 2^46 units of 2^-108 a b) among it, and
// an element of k terms by less than 1.02 k 2^-53 a b.  An FP64 sum of the terms may be off by k 2^-53
// (|A| |B|)_ij.  So where |(A B)_ij| >= 1.02 a b the digits are no worse, whatever the data; where it is smaller (a
// row's or column's few large entries meet small ones, or the sum cancels) the element is formed anew, in
// FP64, by the kernel that joins it (dot8).  T1 is held to this element by element; the three products of the result
// together, as their one FP64 sum would be.  Rows and columns that are not finite take the same way, so that NaN
// and infinities come out as FP64 gives them.  Share of elements formed anew on the iterates of the
// relaxation (d = 16 to 128, 1 to 400 steps): none of Q w and Q w_{1/2}, 0.1 to 0.5 of Q xbar (tests only).
// In the 2-norm the digits are closer than the FP64 contraction (relative to a long double product: 8e-17
// against 6e-16 at d = 96).
//
// One product is five kernels: k_slice_x (digits of X by rows and by columns), k_fix on Ahat X, S X and X T at
// once, k_slice_t1 (joins Ahat X, digits by rows), k_fix on T1 Bhat, k_join.  A CTA of k_fix owns a 128 x 64
// tile of one product and one or several chunks of 64 k's; a chunk's digits of both operands (172 KB) are
// fetched with 14 TMA loads behind one mbarrier and multiplied by 136 tcgen05.mma.
// us per product before a pass, FP64 contractions (qap.cu) / this path: d = 9: 49 / 43, 32: 85 / 43, 64: 162 / 49,
// 128: 186 / 53, 256: 189 / 58, 400: 728 / 175; at d = 256 the two k_fix take 13 us each.  Below d = 8 one
// FP64 tile is as fast.  With every element formed anew (rows and columns over 20 orders of magnitude) a product takes
// 21 us more at d = 64, 40 at 128, 98 at 256: no longer than the contractions.
#include <algorithm>
#include <cfloat>
#include <vector>

#include "qap_tc.cuh"
#include "tc_ptx.cuh"

namespace hprqp {
namespace {

using tc::smem_u32;

constexpr int kDig = 7;            // digits of an operand
constexpr int kSum = 8;            // digit sums kept
constexpr int kBM = 128, kBN = 64, kBK = 64;
constexpr int kGroups = 4;          // partial sums per product at most
constexpr uint32_t kABytes = kBM * kBK * 2, kBBytes = kBN * kBK * 2;
constexpr uint32_t kFixSmem = 1024 + kDig * (kABytes + kBBytes);

// ------------------------------------------------------------------------------------ digits
// biased exponent of v (2047: not finite; 1 for subnormals, which share its unit; 0: v is 0)
__device__ __forceinline__ int exponent(double v) {
  const unsigned mag = (unsigned)__double2hiint(v) & 0x7fffffffu;
  return mag >> 20 ? (int)(mag >> 20) : (mag | (unsigned)__double2loint(v)) != 0u;
}

// 2^(e - 1057): a row's scale; 0 for a row of zeros; NaN for a row that is not finite, so that its products are NaN
__device__ __forceinline__ double row_scale(int e) {
  if (e == 0) return 0.0;
  return e == 2047 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(1.0, e - 1057);
}

// round(v 2^(1077 - e)) for a finite v of exponent <= e
__device__ __forceinline__ long long fixed(double v, int e) {
  const int ev = exponent(v);
  if (ev == 0 || ev == 2047 || e == 2047) return 0;
  const unsigned hi = (unsigned)__double2hiint(v), top = (hi & 0x7ff00000u) ? 0x100000u : 0u;
  const long long man = ((long long)((hi & 0xfffffu) | top) << 32) | (unsigned)__double2loint(v);
  const int sh = e - ev - 2;   // man 2^(2 - (e - ev))
  long long q;
  if (sh <= 0) q = man << -sh;
  else q = sh > 54 ? 0 : (man + (1ll << (sh - 1))) >> sh;
  return (hi >> 31) ? -q : q;
}

// BF16 bits of an integer in [-128, 128] (exact): through the FP32 number 1.5 2^23 + d
__device__ __forceinline__ unsigned digit_bits(int d) {
  return __float_as_uint(__uint_as_float(0x4B400000u + (unsigned)d) - 12582912.0f) >> 16;
}

// Stores the digits of two neighbouring entries: out[digit * plane + at] as pairs
__device__ __forceinline__ void put_digits(uint32_t* out, size_t plane, size_t at, long long qa, long long qb) {
#pragma unroll
  for (int i = kDig - 1; i >= 0; i--) {
    int a = (int)qa, b = (int)qb;
    if (i > 0) {
      a = (int)(signed char)(qa & 255);
      b = (int)(signed char)(qb & 255);
      qa = (qa - a) >> 8;
      qb = (qb - b) >> 8;
    }
    out[i * plane + at] = digit_bits(a) | (digit_bits(b) << 16);
  }
}

// Eight rows of a matrix whose element (row, k) is val(row, k), with the rows' elements far apart and neighbouring
// rows' next to each other (a column-major matrix by rows): exponents, scales and digits.  1024 threads, so that
// d = 256 (32 blocks) has two values per thread to wait for.
constexpr int kFarThreads = 1024;
template <class F>
__device__ void slice_far(F val, int r0, int d, int kp, size_t plane, uint32_t* out, double* scale) {
  __shared__ int top[8];
  __shared__ long long tile[8][4 * kBK + 1];
  const int t = threadIdx.x, i = t & 7, g = t >> 3, warp = t >> 5, lane = t & 31;
  if (t < 8) top[t] = 0;
  __syncthreads();
  int e = 0;
  if (r0 + i < d)
    for (int k = g; k < d; k += 128) e = max(e, exponent(val(r0 + i, k)));
  atomicMax(&top[i], e);
  __syncthreads();
  if (t < 8 && r0 + t < d) scale[r0 + t] = row_scale(top[t]);
  for (int k0 = 0; k0 < kp; k0 += 4 * kBK) {
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int k = g + 128 * q;
      tile[i][k] = r0 + i < d && k0 + k < d ? fixed(val(r0 + i, k0 + k), top[i]) : 0;
    }
    __syncthreads();
    const int row = warp & 7, k = (warp >> 3) * kBK + 2 * lane;   // a warp: one row, 64 of the k's
    if (r0 + row < d && k0 + k < kp)
      put_digits(out, plane, ((size_t)(r0 + row) * kp + k0 + k) / 2, tile[row][k], tile[row][k + 1]);
    __syncthreads();
  }
}

// The same for rows that are contiguous: one warp per row.
__device__ void slice_near(const double* src, int64_t ld, int r, int d, int kp, size_t plane, uint32_t* out,
                           double* scale) {
  if (r >= d) return;
  const int lane = threadIdx.x & 31;
  const double* v = src + (size_t)r * ld;
  int e = 0;
  for (int k = lane; k < d; k += 32) e = max(e, exponent(v[k]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  if (lane == 0) scale[r] = row_scale(e);
  for (int k = 2 * lane; k < kp; k += 64)
    put_digits(out, plane, ((size_t)r * kp + k) / 2, k < d ? fixed(v[k], e) : 0, k + 1 < d ? fixed(v[k + 1], e) : 0);
}

// digits of contiguous rows (the stored matrices, at create)
__global__ void __launch_bounds__(256) k_slice_rows(const double* src, int d, int kp, size_t plane, uint32_t* out,
                                                    double* scale) {
  slice_near(src, d, blockIdx.x * 8 + (threadIdx.x >> 5), d, kp, plane, out, scale);
}

// digits of X by rows (the first blocks, eight rows each) and by columns (32 each)
__global__ void __launch_bounds__(kFarThreads) k_slice_x(const double* x, QapTcDev q) {
  tc::pdl_wait();
  const int half = (q.d + 7) / 8;
  if ((int)blockIdx.x < half)
    slice_far([&](int i, int k) { return x[(size_t)k * q.d + i]; }, (int)blockIdx.x * 8, q.d, q.kp, q.plane, q.dig[kXRow],
              q.scale[kXRow]);
  else
    slice_near(x, q.d, ((int)blockIdx.x - half) * 32 + (threadIdx.x >> 5), q.d, q.kp, q.plane, q.dig[kXCol], q.scale[kXCol]);
}

// ------------------------------------------------------------------------------------ products
// biased exponent of |v| by its upper half (0 for subnormals too)
__device__ __forceinline__ int field(double v) { return (int)(((unsigned)__double2hiint(v) >> 20) & 0x7ffu); }

// element (i, j) of product `prod`, from its partial sums; size: field() of its row's and its column's scale, summed
__device__ __forceinline__ double join(const QapTcDev& q, int prod, int a, int b, int i, int j, int& size) {
  const size_t dd = (size_t)q.d * q.d;
  const long long* p = q.part + (size_t)prod * q.groups * 2 * dd + (size_t)j * q.d + i;
  long long h[kGroups], l[kGroups];   // all loads in flight
#pragma unroll
  for (int g = 0; g < kGroups; g++) {
    h[g] = g < q.groups ? __ldcg(p + 2 * g * dd) : 0;
    l[g] = g < q.groups ? __ldcg(p + (2 * g + 1) * dd) : 0;
  }
  const long long hi = (h[0] + h[1]) + (h[2] + h[3]), lo = (l[0] + l[1]) + (l[2] + l[3]);
  // |hi| < 2^45 per chunk of k: exact in FP64 up to 2^8 chunks (d = 16,384), rounded once beyond, like the result.
  // |lo| < 2^47 per chunk: from 2^6 chunks on it may round too, by less than 2^-53 of it, where an element that
  // is kept is 2^68 at least.
  // The smaller scale first: a product in FP64's range does not overflow on the way to it.
  const double v = fma((double)hi, 4294967296.0, (double)lo), sa = q.scale[a][i], sb = q.scale[b][j];
  size = field(sa) + field(sb);
  return sa < sb ? v * sa * sb : v * sb * sa;
}
// Whether a finite sum of up to three products, the largest of exponent field `top`, reaches the sum of their 1.02 a b,
// by exponents alone (FP64 operations on every element took 5 us of a product at d = 256): a b is at most
// 2^(size + 68 - 2046), three times 1.02 of it less than four.
__device__ __forceinline__ bool reaches(int top, int size) { return top < 2047 && top >= size + 68 + 2 - 1023; }
// 1.02 a b (a is 2^34 of the row's scale); 0 for a row or column of zeros
__device__ __forceinline__ double least(const QapTcDev& q, int a, int b, int i, int j) {
  return 1.02 * (17179869184.0 * q.scale[a][i]) * (17179869184.0 * q.scale[b][j]);
}

// For each lane with bad set: term(k, src) summed over k < d in FP64, src the lane whose element it is; returned in
// that lane (others: `keep`).  Eight lanes an element, four elements of the warp at a time, two running sums a lane
// of eight loads in flight: a fixed order.  All lanes call it.
template <class F>
__device__ __forceinline__ double dot8(bool bad, double keep, int d, F term) {
  const unsigned all = 0xffffffffu, mask = __ballot_sync(all, bad);
  const int lane = threadIdx.x & 31, l = lane & 7, grp = lane >> 3, rank = __popc(mask & ((1u << lane) - 1u));
  unsigned left = mask;
  for (int round = 0; left; round++) {
    int src = -1;   // the element of this group of lanes
#pragma unroll
    for (int g = 0; g < 4; g++) {
      if (g == grp && left) src = __ffs(left) - 1;
      left &= left - 1u;
    }
    double s0 = 0.0, s1 = 0.0;
    if (src >= 0) {
      int k = l;
#pragma unroll 4
      for (; k + 8 < d; k += 16) {
        s0 = term(s0, k, src);
        s1 = term(s1, k + 8, src);
      }
      if (k < d) s0 = term(s0, k, src);
    }
    double s = s0 + s1;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(all, s, o);
    const double got = __shfl_sync(all, s, 8 * (rank & 3));
    if (bad && rank >> 2 == round) keep = got;
  }
  return keep;
}

// T1 = Ahat X (kept in t1, column-major) and its digits by rows
__global__ void __launch_bounds__(kFarThreads) k_slice_t1(QapTcDev q, const double* x) {
  tc::pdl_wait();
  const int r0 = blockIdx.x * 8, i = threadIdx.x & 7;
  const int kw = (threadIdx.x >> 5) * 4, kl = (threadIdx.x & 31) >> 3;   // a warp: eight rows of four columns
  constexpr int kStep = kFarThreads / 8;
  for (int c0 = kw; c0 < q.d; c0 += 32 * kStep) {
    unsigned bad = 0u;   // by step
    for (int t = 0; t < 32 && c0 + t * kStep < q.d; t++) {
      const int k = c0 + t * kStep + kl;
      if (r0 + i >= q.d || k >= q.d) continue;
      int size;
      const double v = join(q, 0, kAhat, kXCol, r0 + i, k, size);
      q.t1[(size_t)k * q.d + r0 + i] = v;
      if (!reaches(field(v), size) && !(fabs(v) >= least(q, kAhat, kXCol, r0 + i, k) && fabs(v) <= DBL_MAX)) bad |= 1u << t;
    }
    unsigned any = __reduce_or_sync(0xffffffffu, bad);
    for (; any; any &= any - 1u) {
      const int t = __ffs(any) - 1, k0 = c0 + t * kStep;
      const bool mine = (bad >> t) & 1u;
      const double v = dot8(mine, 0.0, q.d, [&](double s, int l, int src) {
        return fma(q.mats[(size_t)(r0 + (src & 7)) * q.d + l], x[(size_t)(k0 + (src >> 3)) * q.d + l], s);
      });
      if (mine) q.t1[(size_t)(k0 + kl) * q.d + r0 + i] = v;
    }
  }
  __syncthreads();
  slice_far([&](int r, int k) { return q.t1[(size_t)k * q.d + r]; }, r0, q.d, q.kp, q.plane, q.dig[kT1], q.scale[kT1]);
}

// out = T1 Bhat - S X - X T
__global__ void __launch_bounds__(256) k_join(QapTcDev q, const double* x, double* out) {
  tc::pdl_wait();
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x, e0 = e - (threadIdx.x & 31), dd = (int64_t)q.d * q.d;
  const bool in = e < dd;
  double v = 0.0;
  bool bad = false;
  if (in) {
    const int i = (int)(e % q.d), j = (int)(e / q.d);
    int sa, sb, sc;
    const double a = join(q, 3, kT1, kBhat, i, j, sa), b = join(q, 1, kS, kXCol, i, j, sb),
                 c = join(q, 2, kXRow, kT, i, j, sc);
    v = a - b - c;
    if (!reaches(max(field(a), max(field(b), field(c))), max(sa, max(sb, sc)))) {
      const double most = fabs(a) + fabs(b) + fabs(c);
      bad = !(most >= least(q, kT1, kBhat, i, j) + least(q, kS, kXCol, i, j) + least(q, kXRow, kT, i, j) && most <= DBL_MAX);
    }
  }
  v = dot8(bad, v, q.d, [&](double s, int t, int src) {
    const int i = (int)((e0 + src) % q.d);
    const size_t j = (size_t)((e0 + src) / q.d) * q.d, k = (size_t)t * q.d + i;
    s = fma(q.t1[k], q.mats[dd + j + t], s);
    s = fma(-q.mats[2 * dd + (size_t)i * q.d + t], x[j + t], s);
    return fma(-x[k], q.mats[3 * dd + j + t], s);
  });
  if (in) out[e] = v;
}

struct Maps {
  CUtensorMap a[3], b[3];
};

// Digit products of up to three matrix products A B^T (rows of digits of both): partials of product first + p
__global__ void __launch_bounds__(128, 1) k_fix(const __grid_constant__ Maps maps, QapTcDev q, int first) {
  __shared__ __align__(8) uint64_t bar_full, bar_done;
  __shared__ uint32_t tmem_slot;
  extern __shared__ uint8_t dsm[];
  const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = (q.d + kBM - 1) / kBM, nt = (q.d + kBN - 1) / kBN;
  int id = blockIdx.x;
  const int m0 = (id % mt) * kBM, n0 = (id / mt % nt) * kBN;
  id /= mt * nt;
  const int group = id % q.groups, prod = id / q.groups;
  const uint32_t full = smem_u32(&bar_full), done = smem_u32(&bar_done);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    tc::mbar_init(full, 1);
    tc::mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  tc::pdl_wait();   // the set-up above overlaps the end of the kernel before
  const size_t dd = (size_t)q.d * q.d;
  long long* part = q.part + ((size_t)(first + prod) * q.groups + group) * 2 * dd;
  bool ok = true;
  for (int c = group, it = 0; c * kBK < q.kp && ok; c += q.groups, it++) {
    const uint32_t ph = (uint32_t)it & 1u;
    if (threadIdx.x == 0) {
      tc::mbar_expect_tx(full, kDig * (kABytes + kBBytes));
      for (int s = 0; s < kDig; s++) {   // x = c 64 elements: 16-byte aligned
        tc::tma_load_2d(base + s * kABytes, &maps.a[prod], full, c * kBK, s * q.dp + m0);
        tc::tma_load_2d(base + kDig * kABytes + s * kBBytes, &maps.b[prod], full, c * kBK, s * q.dp + n0);
      }
    }
    if (threadIdx.x == 32) {
      // a wait that gives up has recorded its error; a second one lets the copies in flight end (read from memory: the
      // launches of a captured graph keep their arguments)
      const uint32_t polls = (uint32_t)__ldcg(q.err + 1);
      if (tc::mbar_wait(full, ph, q.err, 1, polls ? polls : tc::kSpin) || tc::mbar_wait(full, ph, q.err, 1)) {
        tc::tc_fence_after();
        constexpr uint32_t idesc = tc::idesc_bf16(kBM, kBN);
        for (int s = 0; s < kSum; s++) {
          uint32_t add = 0;
          for (int i = s < kDig ? 0 : s - kDig + 1; i <= s && i < kDig; i++) {
            const uint64_t ad = tc::sdesc_sw128(base + i * kABytes);
            const uint64_t bd = tc::sdesc_sw128(base + kDig * kABytes + (s - i) * kBBytes);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; kk++) {
              tc::mma_bf16(tmem + s * kBN, ad + 2 * kk, bd + 2 * kk, idesc, add);
              add = 1;
            }
          }
        }
      }
      tc::mma_commit(done);
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, tc::mbar_wait(done, ph, q.err, 2));
    tc::tc_fence_after();
    if (ok) {
      const int i = m0 + warp * 32 + lane;
#pragma unroll 1
      for (int c0 = 0; c0 < kBN; c0 += 32) {
        // (loops over the sums that are not unrolled: the code is run once, and fetching it would bound it)
#pragma unroll 1
        for (int half = 0; half < 2; half++) {
          long long v[32];
#pragma unroll
          for (int j = 0; j < 32; j++) v[j] = 0;
#pragma unroll 1
          for (int s = half * 4; s < half * 4 + 4; s++) {
            uint32_t r[32];
            tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(s * kBN + c0), r);
#pragma unroll
            for (int j = 0; j < 32; j++) v[j] = v[j] * 256 + (long long)__float2int_rn(__uint_as_float(r[j]));
          }
          if (i < q.d) {
            long long* h = part + (half ? dd : 0) + (size_t)(n0 + c0) * q.d + i;
#pragma unroll
            for (int j = 0; j < 32; j++, h += q.d)
              if (n0 + c0 + j < q.d) *h = it ? *h + v[j] : v[j];
          }
        }
      }
    }
    // the next chunk overwrites the operands and the sums
    tc::tc_fence_before();
    ok = __syncthreads_and(ok);
    tc::tc_fence_after();
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

}  // namespace

struct QapTc {
  QapTcDev dev;
  Maps one, two;   // the products Ahat X, S X, X T, and T1 Bhat
};

void qap_tc_free(QapTc* t) { delete t; }
int* qap_tc_error(const QapTc* t) { return t->dev.err; }

size_t qap_tc_bytes(int64_t d, size_t (&part)[5]) {
  const int64_t dp = (d + kBM - 1) / kBM * kBM, kp = (d + kBK - 1) / kBK * kBK;
  const int64_t groups = std::min<int64_t>(kp / kBK, kGroups);
  part[0] = (size_t)kDig * dp * kp * 2 * kTcMats;        // digits
  part[1] = (size_t)kTcMats * d * sizeof(double);        // scales
  part[2] = (size_t)4 * groups * 2 * d * d * sizeof(long long);
  part[3] = (size_t)d * d * sizeof(double);              // T1
  part[4] = 256;                                         // error word
  size_t sum = 0;
  for (size_t& b : part) {
    b = (b + 1023) / 1024 * 1024;
    sum += b;
  }
  return sum;
}

cudaError_t qap_tc_create(QapTc** out, int64_t d, const double* mats, void* mem, cudaStream_t s) {
  size_t part[5];
  const size_t bytes = qap_tc_bytes(d, part);
  QapTc* t = new QapTc();
  QapTcDev& q = t->dev;
  q.d = (int)d;
  q.mats = mats;
  q.dp = (int)((d + kBM - 1) / kBM * kBM);
  q.kp = (int)((d + kBK - 1) / kBK * kBK);
  q.groups = std::min(q.kp / kBK, kGroups);
  q.plane = (size_t)q.dp * q.kp / 2;
  uint8_t* m = static_cast<uint8_t*>(mem);
  for (int k = 0; k < kTcMats; k++) {
    q.dig[k] = reinterpret_cast<uint32_t*>(m) + (size_t)k * kDig * q.plane;
    q.scale[k] = reinterpret_cast<double*>(m + part[0]) + (size_t)k * d;
  }
  q.part = reinterpret_cast<long long*>(m + part[0] + part[1]);
  q.t1 = reinterpret_cast<double*>(m + part[0] + part[1] + part[2]);
  q.err = reinterpret_cast<int*>(m + part[0] + part[1] + part[2] + part[3]);
  cudaError_t e = cudaMemsetAsync(mem, 0, bytes, s);   // also the digits of the padding rows and columns
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fix, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFixSmem);
  // symmetric matrices: rows and columns alike
  const int which[4] = {kAhat, kBhat, kS, kT};
  for (int k = 0; k < 4 && e == cudaSuccess; k++) {
    k_slice_rows<<<(q.d + 7) / 8, 256, 0, s>>>(mats + (size_t)k * d * d, q.d, q.kp, q.plane, q.dig[which[k]], q.scale[which[k]]);
    e = cudaGetLastError();
  }
  auto map = [&](CUtensorMap* c, int k, int rows) {
    if (e == cudaSuccess) e = tc::make_map(c, q.dig[k], (int64_t)kDig * q.dp, q.kp, q.kp, rows);
  };
  const int a[4] = {kAhat, kS, kXRow, kT1}, b[4] = {kXCol, kXCol, kT, kBhat};
  for (int k = 0; k < 4; k++) {
    Maps& M = k < 3 ? t->one : t->two;
    map(&M.a[k % 3], a[k], kBM);
    map(&M.b[k % 3], b[k], kBN);
  }
  if (e != cudaSuccess) {
    delete t;
    return e;
  }
  *out = t;
  return cudaSuccess;
}

cudaError_t qap_tc_apply(const QapTc* t, const double* x, double* out, bool pdl, cudaStream_t s) {
  const QapTcDev& q = t->dev;
  const int rows = (q.d + 7) / 8, tiles = ((q.d + kBM - 1) / kBM) * ((q.d + kBN - 1) / kBN);
  const dim3 far(kFarThreads), fix(128), flat(256);
  cudaError_t e = tc::launch_kernel(false, 1, k_slice_x, dim3(rows + (q.d + 31) / 32), far, 0, s, x, q);
  if (e == cudaSuccess) e = tc::launch_kernel(pdl, 1, k_fix, dim3(3 * tiles * q.groups), fix, kFixSmem, s, t->one, q, 0);
  if (e == cudaSuccess) e = tc::launch_kernel(pdl, 1, k_slice_t1, dim3(rows), far, 0, s, q, x);
  if (e == cudaSuccess) e = tc::launch_kernel(pdl, 1, k_fix, dim3(tiles * q.groups), fix, kFixSmem, s, t->two, q, 3);
  if (e == cudaSuccess)
    e = tc::launch_kernel(pdl, 1, k_join, dim3((unsigned)(((int64_t)q.d * q.d + 255) / 256)), flat, 0, s, q, x, out);
  return e;
}

}  // namespace hprqp

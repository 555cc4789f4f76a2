// Resident form of the single-instance solver for problems whose state fits the SMs' shared
// memory: many inner steps of Algorithm 4 in one cooperative launch.
//
// A small or mid-sized problem's step as separate kernels is latency: four to six launches, each
// walking row pointer -> index -> gathered value through L2, with the vectors of its epilogue behind
// them (30 us a step at n = 1000, 40 us at n = 1e5).  Here block b owns the rows [b rn, (b+1) rn) of
// the n-vectors and [b rm, (b+1) rm) of the m-vectors for the whole solve.  Its part of the state and
// of the matrices lies in shared memory; only the vectors that the products gather from
// (wbar_{1/2}, v, ybar, w, and the factor products t) go through L2, each followed by a grid
// barrier.  A plain step is E (elementwise) | Q wbar_{1/2}, v | A v, ybar | A^T ybar, w | Q w, E of the
// next step: four barriers, two more when Q has a factor product to form first.  Without rows of A a
// step is E | Q wbar_{1/2} with the one barrier between them, and wbar_{1/2} lies in two vectors in turn: a
// block that is done with its products stores the next step's while others still gather this one's, and
// the barrier keeps it from getting further ahead.  The arithmetic per
// row is that of the fused passes of kernels.cuh; a step that evaluates R~ or the stopping rule takes
// the unfused form, like there.  Every block sums the blocks' partial results itself, in block order,
// and runs the controller on its own copy: no broadcast, and the same decisions everywhere.
//
// Two ways for the gathered vectors to travel (the template parameter CL):
//   * up to 16 blocks (n up to a few thousand) form one thread-block cluster.  Every block holds a copy
//     of the gathered vectors in its shared memory; a block stores its rows into all copies through
//     distributed shared memory, and the barrier is the cluster's (690 cycles, 1700 with writes to
//     global memory before it).  A gather is a local shared-memory read (30 cycles, 300 from L2).
//   * larger problems use up to one block per SM and vectors in L2.  The barrier is a counter: one
//     release-add per block, one thread per block polls with acquire loads.  On 152 blocks that is 2640
//     cycles; flags read by every block took 8000, and a fence per polling thread more.  Every wait
//     is bounded (ResRun::spin polls); a block whose wait gives up sets the error flag and leaves, the others follow at their
//     next barrier, and the host reports HPRQP_TIMEOUT.
// FP64 (measured): a dependent FMA takes 64 cycles, as long as its issue slot, so four warps fill an
// SM's FP64 pipe; a division takes 640.
#define HPRQP_COHERENT 1
#include <algorithm>
#include <cstring>

#include "kernels.cuh"
#include "resident.cuh"

namespace hprqp {
namespace {

constexpr int kTerm = 16;              // sums of one reduction: 12 end-of-step, 4 of the y-step

// rows of the shared-memory state, rn values each
enum { SX, SX0, SW, SW0, SQW, SQW0, SATY, SATY0, SXB, SXH, SWH, SWB, SQWB, SATYB, SC, SL, SU, kStateN };
static_assert(kStateN == kResStateN, "the host sizes the state");
enum { MY, MY0, MYB, ML, MU, kStateM };
static_assert(kStateM == kResStateM, "the host sizes the state");

struct Mat {           // a matrix as this block reads it: row i at rp[i], entries indexed globally
  const int* rp;
  const int* ci;
  const double* v;
};
struct Dense {
  const double* col;   // entry (r, own column c) at col[r * ldc + c]
  int64_t ldc;
  const double* row;   // entry (own row r - row0, j) at row[(r - row0) * n + j]
};

// scalars of the running step (the controller moves C on to the next step in the background)
struct Step {
  double ha, hb, fha, fhb, sigma, isigma, c1, c2, s, slA, islA, tau;
  int mode, rtest, ttest;
};

struct Block {
  Ctrl C;
  Step st[2];   // of the running step and of the next one, in turn
  Mat A, AT, Qc, thin, fac[kMaxFac], fact[kMaxFac];
  Dense dn[kMaxDense];
  const double* diag;
  const double* dia[kMaxDia];   // dia[k][j] = Q[j][j + off_k]
  double part[32];
  double tot[kTerm];
  int bad;
};

// What the row sums need of a block, passed by value (the whole context would go through local memory)
template <bool CL>
struct Team {
  int tid, T, B;
  double* scratch;
  __device__ __forceinline__ double ld(const double* q) const { return CL ? *q : __ldcg(q); }
  // *q = val in every block's copy
  __device__ __forceinline__ void put(double* q, double val) const {
    if (!CL) {
      *q = val;
      return;
    }
    const unsigned at = (unsigned)__cvta_generic_to_shared(q);
    for (int k = 0; k < B; k++) {
      unsigned to;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(k));
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(val) : "memory");
    }
  }
};

template <bool CL>
struct Ctx {
  const Args& a;
  const ResPlan& p;
  const ResRun& r;
  Block& S;
  double* sm;        // dynamic shared memory
  int b, tid, T;
  int j0, nr, i0, mr;
  unsigned epoch;
  int slot;          // which of the two partial buffers the running reduction uses
  // the gathered vectors: wbar_{1/2}; v, then w (or wbar, or the restart difference); xbar; ybar; t
  double *wh, *v, *w, *xb, *yb, *t1, *t2, *part;

  __device__ __forceinline__ double* n_row(int k) const { return sm + (size_t)k * p.rn; }
  __device__ __forceinline__ double* m_row(int k) const { return sm + (size_t)kStateN * p.rn + (size_t)k * p.rm; }
  __device__ __forceinline__ double* rs0() const { return sm + p.o_rs; }
  __device__ __forceinline__ double* rs1() const { return sm + p.o_rs + p.rs_len; }
  __device__ __forceinline__ double* scratch() const { return sm + p.o_scratch; }   // 4 T values
  __device__ __forceinline__ Team<CL> team() const { return Team<CL>{tid, T, p.B, scratch()}; }
  __device__ __forceinline__ double ld(const double* q) const { return team().ld(q); }
  __device__ __forceinline__ void put(double* q, double val) const { team().put(q, val); }
};

// All blocks have stored what they wrote before it, once it returns true.  Meanwhile, the last warp of
// the block runs `work`.
template <bool CL, class F>
__device__ __forceinline__ bool all_sync(Ctx<CL>& x, F work) {
  if (CL) {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    if (x.tid >= x.T - 32) work();
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    __syncthreads();
    return true;
  }
  x.epoch += (unsigned)x.p.B;
  __syncthreads();
  int bad = 0;
  if (x.tid >= x.T - 32) work();
  if (x.tid == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(x.r.flags) : "memory");
    unsigned v;
    for (unsigned i = 0;; ++i) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(x.r.flags) : "memory");
      if ((int)(v - x.epoch) >= 0) break;
      if (i >= x.r.spin || ((i & 1023u) == 1023u && *(volatile int*)x.r.err)) {
        atomicExch(x.r.err, 1);
        bad = 1;
        break;
      }
    }
  }
  return __syncthreads_or(bad) == 0;
}
template <bool CL>
__device__ bool all_sync(Ctx<CL>& x) {
  return all_sync(x, [] {});
}

// The sum (MX: the maximum of non-negative values) of v[0 .. len) by one warp, len a multiple of 32, in
// lane 0.  Four running sums, so that four additions are in flight (64 cycles each).
template <bool MX>
__device__ __forceinline__ double warp_total(const double* v, int len) {
  auto op = [](double a, double b) { return MX ? imax(a, b) : a + b; };
  const int lane = threadIdx.x & 31;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int i = lane;
  for (; i + 96 < len; i += 128)
#pragma unroll
    for (int q = 0; q < 4; q++) s[q] = op(s[q], v[i + 32 * q]);
  for (; i < len; i += 32) s[0] = op(s[0], v[i]);
  double t = op(op(s[0], s[1]), op(s[2], s[3]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t = op(t, __shfl_down_sync(0xffffffffu, t, o));
  return t;
}

// Where row sums go: the block's own buffers, or every block's copy of t
struct Own {
  double *o0, *o1;
  bool add;
  template <bool CL>
  __device__ __forceinline__ void operator()(const Team<CL>&, int rr, int v, double s) const {
    double* o = (v ? o1 : o0) + rr;
    *o = add ? *o + s : s;
  }
};
struct Everywhere {
  double *o0, *o1;
  template <bool CL>
  __device__ __forceinline__ void operator()(const Team<CL>& c, int rr, int v, double s) const {
    c.put((v ? o1 : o0) + rr, s);
  }
};

// Sums of the rows r0 + rr, rr < nr, with G lanes per row.
template <bool CL, int G, class Out>
__device__ __forceinline__ void row_lanes(const Team<CL> c, const Mat M, int r0, int nr, const double* x0,
                                          const double* x1, const Out out) {
  const int lane = c.tid % G, ng = c.T / G;
  for (int base = 0; base < nr; base += ng) {
    const int rr = base + c.tid / G;
    if (base + (c.tid & ~31) / G >= nr) return;   // the whole warp: its additions would hold up the others'

    double s0 = 0.0, s1 = 0.0;
    if (rr < nr) {
      const int e = M.rp[r0 + rr + 1];
      int k = M.rp[r0 + rr] + lane;
      for (; k + 3 * G < e; k += 4 * G) {
        const int j0 = M.ci[k], j1 = M.ci[k + G], j2 = M.ci[k + 2 * G], j3 = M.ci[k + 3 * G];
        const double a0 = c.ld(x0 + j0), a1 = c.ld(x0 + j1), a2 = c.ld(x0 + j2), a3 = c.ld(x0 + j3);
        const double v0 = M.v[k], v1 = M.v[k + G], v2 = M.v[k + 2 * G], v3 = M.v[k + 3 * G];
        s0 = fma(v0, a0, s0);
        s0 = fma(v1, a1, s0);
        s0 = fma(v2, a2, s0);
        s0 = fma(v3, a3, s0);
        if (x1) {
          s1 = fma(v0, c.ld(x1 + j0), s1);
          s1 = fma(v1, c.ld(x1 + j1), s1);
          s1 = fma(v2, c.ld(x1 + j2), s1);
          s1 = fma(v3, c.ld(x1 + j3), s1);
        }
      }
      if (k < e) {   // the remaining 1-3 entries: all loads first
        const bool h1 = k + G < e, h2 = k + 2 * G < e;
        const int j0 = M.ci[k], j1 = h1 ? M.ci[k + G] : j0, j2 = h2 ? M.ci[k + 2 * G] : j0;
        const double a0 = c.ld(x0 + j0), a1 = c.ld(x0 + j1), a2 = c.ld(x0 + j2);
        const double v0 = M.v[k], v1 = h1 ? M.v[k + G] : 0.0, v2 = h2 ? M.v[k + 2 * G] : 0.0;
        s0 = fma(v0, a0, s0);
        if (h1) s0 = fma(v1, a1, s0);
        if (h2) s0 = fma(v2, a2, s0);
        if (x1) {
          s1 = fma(v0, c.ld(x1 + j0), s1);
          if (h1) s1 = fma(v1, c.ld(x1 + j1), s1);
          if (h2) s1 = fma(v2, c.ld(x1 + j2), s1);
        }
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      s0 += __shfl_down_sync(0xffffffffu, s0, o, G);
      if (x1) s1 += __shfl_down_sync(0xffffffffu, s1, o, G);
    }
    if (lane == 0 && rr < nr) {
      out(c, rr, 0, s0);
      if (x1) out(c, rr, 1, s1);
    }
  }
}

// out(rr, 0, .) (and out(rr, 1, .) for a second vector) = sums of the rows r0 + rr, rr < nr, of M with the
// vectors x0, x1; G lanes per row, or the whole block for each row (G = 0: few long rows).
template <bool CL, class Out>
__device__ __noinline__ void row_sums(const Team<CL> c, const Mat M, int r0, int nr, int G, const double* x0,
                                      const double* x1, const Out out) {
  switch (G) {
    case 1: row_lanes<CL, 1>(c, M, r0, nr, x0, x1, out); return;
    case 2: row_lanes<CL, 2>(c, M, r0, nr, x0, x1, out); return;
    case 4: row_lanes<CL, 4>(c, M, r0, nr, x0, x1, out); return;
    case 8: row_lanes<CL, 8>(c, M, r0, nr, x0, x1, out); return;
    case 16: row_lanes<CL, 16>(c, M, r0, nr, x0, x1, out); return;
    case 32: row_lanes<CL, 32>(c, M, r0, nr, x0, x1, out); return;
    default: break;
  }
  double* red = c.scratch;
  for (int rr = 0; rr < nr; rr++) {
    const int b = M.rp[r0 + rr], e = M.rp[r0 + rr + 1];
    double s0 = 0.0, s1 = 0.0;
    for (int k = b + c.tid; k < e; k += 4 * c.T) {   // four entries' loads at once
      double v[4], a0[4], a1[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int i = k + q * c.T, j = i < e ? M.ci[i] : 0;
        v[q] = i < e ? M.v[i] : 0.0;
        a0[q] = i < e ? c.ld(x0 + j) : 0.0;
        a1[q] = x1 && i < e ? c.ld(x1 + j) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (k + q * c.T < e) {
          s0 = fma(v[q], a0[q], s0);
          if (x1) s1 = fma(v[q], a1[q], s1);
        }
    }
    red[c.tid] = s0;
    if (x1) red[c.T + c.tid] = s1;
    __syncthreads();
    if (c.tid < (x1 ? 64 : 32)) {
      const double s = warp_total<false>(red + (c.tid >> 5) * c.T, c.T);
      if ((c.tid & 31) == 0) out(c, rr, c.tid >> 5, s);
    }
    __syncthreads();
  }
}

// The part of t = B x and F x that this block owns (t1: of the second vector x1, when given); step:
// thin factors are left out (their products are formed in q_sums).
template <bool CL>
__device__ void factor_rows(const Ctx<CL>& c, const double* x0, const double* x1, double* t0, double* t1, bool step) {
  const QDev& Q = c.a.Q;
  const int f0 = c.b * c.p.rp;
  for (int f = 0; f < Q.nfac; f++) {
    if (step && Q.inl[f]) continue;
    const int lo = (int)Q.toff[f], hi = lo + (int)Q.fac[f].rows;
    const int q0 = max(f0, lo), q1 = min(f0 + c.p.rp, hi);
    if (q0 < q1) row_sums(c.team(), c.S.fac[f], q0 - lo, q1 - q0, c.p.gP, x0, x1, Everywhere{t0 + q0, t1 + q0});
  }
  if (!Q.ndense) return;
  const int nfac_rows = (int)Q.toff[Q.nfac];
  const int d0 = nfac_rows + c.b * c.p.rd, d1 = min((int)Q.tfd, d0 + c.p.rd);
  const int n = (int)Q.n;
  double* red = c.scratch();
  for (int r = d0; r < d1; r += 2) {   // two rows at a time share the loads of x
    const double* Fr[2] = {nullptr, nullptr};
    for (int q = 0; q < 2; q++) {
      const int rq = min(r + q, d1 - 1);
      int g = 0;
      while (g + 1 < Q.ndense && rq >= (int)Q.toff[Q.nfac + g + 1]) g++;
      const int own0 = max(d0, (int)Q.toff[Q.nfac + g]);   // first own row of this term
      Fr[q] = c.S.dn[g].row + (size_t)(rq - own0) * n;
    }
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int v = 0; v < (x1 ? 2 : 1); v++) {
      const double* x = v ? x1 : x0;
      double sa = 0.0, sb = 0.0;
#pragma unroll 4
      for (int j = c.tid; j < n; j += c.T) {
        const double xv = c.ld(x + j);
        sa = fma(Fr[0][j], xv, sa);
        sb = fma(Fr[1][j], xv, sb);
      }
      s[2 * v] = sa;
      s[2 * v + 1] = sb;
    }
#pragma unroll
    for (int q = 0; q < 4; q++)
      if (q < 2 || x1) red[q * c.T + c.tid] = s[q];
    __syncthreads();
    if (c.tid < (x1 ? 128 : 64)) {
      const int q = c.tid >> 5, rq = r + (q & 1);
      const double w = warp_total<false>(red + q * c.T, c.T);
      if ((c.tid & 31) == 0 && rq < d1) c.put((q < 2 ? t0 : t1) + rq, w);
    }
    __syncthreads();
  }
}

// rs0 (rs1) = everything of (Q x0)_j ((Q x1)_j) for the own rows but the diagonal and the bands: explicit
// CSR, the thin factors' explicit B^T B, B^T t of the other sparse factors, F^T t of the dense ones.
// Ends with a barrier of the block.
template <bool CL>
__device__ void q_sums(const Ctx<CL>& c, const double* x0, const double* x1, const double* t0, const double* t1,
                       bool factors) {
  const QDev& Q = c.a.Q;
  double *o0 = c.rs0(), *o1 = c.rs1();
  bool add = false;
  if (Q.csr.rows) {
    row_sums(c.team(), c.S.Qc, c.j0, c.nr, c.p.gQ, x0, x1, Own{o0, o1, false});
    add = true;
  }
  if (Q.thin.rows && factors) {
    if (add) __syncthreads();
    row_sums(c.team(), c.S.thin, c.j0, c.nr, c.p.gT, x0, x1, Own{o0, o1, add});
    add = true;
  }
  for (int f = 0; f < Q.nfac && factors; f++) {
    if (Q.inl[f]) continue;
    if (add) __syncthreads();
    row_sums(c.team(), c.S.fact[f], c.j0, c.nr, c.p.gF, t0 + Q.toff[f], x1 ? t1 + Q.toff[f] : nullptr, Own{o0, o1, add});
    add = true;
  }
  if (!add) {
    for (int rr = c.tid; rr < c.nr; rr += c.T) {
      o0[rr] = 0.0;
      if (x1) o1[rr] = 0.0;
    }
  }
  __syncthreads();
  if (!factors) return;
  for (int g = 0; g < Q.ndense; g++) {
    const Dense D = c.S.dn[g];
    const int p = (int)Q.dense_p[g], cw = c.p.cw;   // cw columns (a power of two) by T / cw groups of rows
    const int col = c.tid & (cw - 1), grp = c.tid / cw, ng = c.T / cw;
    double* red = c.scratch();
    for (int v = 0; v < (x1 ? 2 : 1); v++) {
      const double* t = (v ? t1 : t0) + Q.toff[Q.nfac + g];
      double* out = v ? o1 : o0;
      for (int base = 0; base < c.nr; base += cw) {
        const int cc = base + col;
        double s = 0.0;
        double* ts = red + c.T;   // 3 T values of t at a time, read by every group of rows
        for (int q0 = 0; q0 < p; q0 += 3 * c.T) {
          const int q1 = min(3 * c.T, p - q0);
          for (int i = c.tid; i < q1; i += c.T) ts[i] = c.ld(t + q0 + i);
          __syncthreads();
          if (cc < c.nr) {
#pragma unroll 4
            for (int r = grp; r < q1; r += ng) s = fma(D.col[(q0 + r) * D.ldc + cc], ts[r], s);
          }
          if (q0 + q1 < p) __syncthreads();
        }
        red[c.tid] = s;
        __syncthreads();
        if (c.tid < cw && cc < c.nr) {
          double w = out[cc];
          for (int q = 0; q < ng; q++) w += red[q * cw + c.tid];
          out[cc] = w;
        }
        __syncthreads();
      }
    }
  }
}

// the diagonal and the bands of (Q x)_j
template <bool CL>
__device__ __forceinline__ double q_bands(const Ctx<CL>& c, int j, const double* x) {
  auto get = [&](int i) { return c.ld(x + i); };
  const QDev& Q = c.a.Q;
  const int n = (int)Q.n;
  double acc = 0.0;
  if (Q.diag) acc = c.S.diag[j] * get(j);
  for (int k = 0; k < Q.ndia; k++) {
    const int o = Q.dia_off[k];
    const double* d = c.S.dia[k];
    if (o == 0) {
      acc = fma(d[j], get(j), acc);
    } else {
      // past either end of the band: operands selected, so that a warp issues the same two FMAs
      const bool up = j + o < n, dn = j - o >= 0;
      const double du = up ? d[j] : 0.0, xu = up ? get(j + o) : 0.0;
      const double dd = dn ? d[j - o] : 0.0, xd = dn ? get(j - o) : 0.0;
      acc = fma(du, xu, acc);
      acc = fma(dd, xd, acc);
    }
  }
  return acc;
}

// This block's part of the sums of v[k], k < NT (a maximum where maxmask has bit k), into the partials at
// slot position at + k; terms outside `want` are left alone.  rows: only threads below it have added anything.
// The threads' values go through shared memory and one warp adds those of one term: rows / 32 + 5 FP64
// instructions a term, where shuffles by every warp would issue 5 rows / 32.
template <bool CL, int NT>
__device__ void block_part(const Ctx<CL>& c, const double (&v)[NT], unsigned want, unsigned maxmask, int at, int rows) {
  double* red = c.scratch();
  const int len = min(c.T, (rows + 31) & ~31), most = len > 0 ? 4 * c.T / len : NT;   // terms that fit the scratch
  unsigned left = want;
  while (left) {
    unsigned now = 0u;   // the next `most` terms
    for (int q = 0; q < most && (left & ~now); q++) now |= (left & ~now) & (~(left & ~now) + 1u);
    int n = 0;
#pragma unroll
    for (int k = 0; k < NT; k++)
      if ((now >> k) & 1u) {
        if (c.tid < len) red[n * len + c.tid] = v[k];
        n++;
      }
    __syncthreads();
    for (int q = c.tid >> 5; q < n; q += c.T >> 5) {
      int k = __ffs(now) - 1;
      unsigned rest = now;
      for (int i = 0; i < q; i++) {
        rest &= rest - 1u;
        k = __ffs(rest) - 1;
      }
      const double s = (maxmask >> k) & 1u ? warp_total<true>(red + q * len, len) : warp_total<false>(red + q * len, len);
      if ((c.tid & 31) == 0) c.put(c.part + (c.slot * c.p.B + c.b) * kTerm + at + k, s);
    }
    left &= ~now;
    __syncthreads();
  }
}
// After a grid barrier: every block adds the blocks' partials in block order.  The next reduction
// uses the other buffer, so that no block overwrites what another still reads.
template <bool CL>
__device__ void all_parts(Ctx<CL>& c, unsigned want, unsigned maxmask) {
  const int k = c.tid >> 5, lane = c.tid & 31, nw = c.T >> 5;
  for (int q = k; q < kTerm; q += nw) {
    if (!((want >> q) & 1u)) {
      if (lane == 0) c.S.tot[q] = 0.0;
      continue;
    }
    const bool mx = (maxmask >> q) & 1u;
    double s = 0.0;
    for (int b = lane; b < c.p.B; b += 32) {
      const double t = c.ld(c.part + (c.slot * c.p.B + b) * kTerm + q);
      s = mx ? imax(s, t) : s + t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_down_sync(0xffffffffu, s, o);
      s = mx ? imax(s, t) : s + t;
    }
    if (lane == 0) c.S.tot[q] = s;
  }
  c.slot ^= 1;
  __syncthreads();
}

// copies of this block's part of the matrices
template <bool CL>
__device__ void stage_mat(const Ctx<CL>& c, Mat& out, const Csr& M, const ResPlan::M& pm, int r0, int nr) {
  const int b = nr > 0 ? M.rp[r0] : 0, e = nr > 0 ? M.rp[r0 + nr] : 0;
  const int* ci = M.ci;
  const double* v = M.v;
  const int* rp = M.rp;
  if (pm.o_v >= 0) {
    double* dv = c.sm + pm.o_v;
    int* di = reinterpret_cast<int*>(c.sm + pm.o_ci);
    int* dr = reinterpret_cast<int*>(c.sm + pm.o_rp);
    for (int k = b + c.tid; k < e; k += c.T) {
      dv[k - b] = M.v[k];
      di[k - b] = M.ci[k];
    }
    for (int i = c.tid; i <= nr; i += c.T) dr[i] = M.rp[r0 + i] - b;   // local entry numbers
    v = dv;
    ci = di;
    rp = dr - r0;
  }
  if (c.tid == 0) out = Mat{rp, ci, v};
}

template <bool CL>
__device__ void stage(Ctx<CL>& c) {
  const Args& a = c.a;
  const QDev& Q = a.Q;
  const ResPlan& p = c.p;
  Block& S = c.S;
  if (a.m > 0) {
    stage_mat(c, S.A, a.A, p.A, c.i0, c.mr);
    stage_mat(c, S.AT, a.AT, p.AT, c.j0, c.nr);
  }
  if (Q.csr.rows) stage_mat(c, S.Qc, Q.csr, p.Qc, c.j0, c.nr);
  if (Q.thin.rows) stage_mat(c, S.thin, Q.thin, p.thin, c.j0, c.nr);
  for (int f = 0; f < Q.nfac; f++) {
    stage_mat(c, S.fact[f], Q.fact[f], p.fact[f], c.j0, c.nr);
    const int lo = (int)Q.toff[f], q0 = max(c.b * p.rp, lo),
              q1 = min(c.b * p.rp + p.rp, lo + (int)Q.fac[f].rows);
    stage_mat(c, S.fac[f], Q.fac[f], p.fac[f], q0 < q1 ? q0 - lo : 0, max(0, q1 - q0));
  }
  const int n = (int)a.n;
  if (c.tid == 0) S.diag = Q.diag;
  if (Q.diag && p.o_diag >= 0) {
    for (int i = c.tid; i < c.nr; i += c.T) c.sm[p.o_diag + i] = Q.diag[c.j0 + i];
    if (c.tid == 0) S.diag = c.sm + p.o_diag - c.j0;
  }
  for (int k = 0; k < Q.ndia; k++) {
    const double* src = Q.dia + (size_t)k * n;
    const int o = Q.dia_off[k];
    if (p.o_dia[k] >= 0) {   // rows j0 - o .. j0 + nr
      double* d = c.sm + p.o_dia[k];
      for (int i = c.tid; i < c.nr + o; i += c.T) {
        const int j = c.j0 - o + i;
        d[i] = j >= 0 && j < n ? src[j] : 0.0;
      }
      src = d + o - c.j0;
    }
    if (c.tid == 0) S.dia[k] = src;
  }
  const int nfac_rows = Q.ndense ? (int)Q.toff[Q.nfac] : 0;
  for (int g = 0; g < Q.ndense; g++) {
    const double* F = Q.dense[g];
    const int P = (int)Q.dense_p[g], lo = (int)Q.toff[Q.nfac + g];
    const int q0 = max(nfac_rows + c.b * p.rd, lo), q1 = min(nfac_rows + (c.b + 1) * p.rd, lo + P);
    Dense D;
    D.col = F + c.j0;
    D.ldc = n;
    D.row = F + (size_t)max(0, min(q0 - lo, P - 1)) * n;
    if (p.o_dcol[g] >= 0) {
      double* d = c.sm + p.o_dcol[g];
      for (int i = c.tid; i < P * c.nr; i += c.T) d[(i / c.nr) * p.rn + i % c.nr] = F[(size_t)(i / c.nr) * n + c.j0 + i % c.nr];
      D.col = d;
      D.ldc = p.rn;
    }
    if (p.o_drow[g] >= 0 && q0 < q1) {
      double* d = c.sm + p.o_drow[g];
      const double* src = F + (size_t)(q0 - lo) * n;
      for (int i = c.tid; i < (q1 - q0) * n; i += c.T) d[i] = src[i];
      D.row = d;
    }
    if (c.tid == 0) S.dn[g] = D;
  }
  __syncthreads();
}

template <bool CL>
__device__ __forceinline__ void init_ctx(Ctx<CL>& c) {
  const Vec& V = c.a.V;
  const int n = (int)c.a.n, m = (int)c.a.m, tl = (int)c.a.Q.tlen;
  if (CL) {   // the block's copies
    double* q = c.sm + c.p.o_vec;
    c.wh = q;
    c.v = c.w = q + n;
    c.xb = q + 2 * n;
    c.yb = q + 3 * n;   // 2 m: the power method alternates between two vectors
    c.t1 = q + 3 * n + 2 * m;
    c.t2 = c.t1 + 2 * tl;
    c.part = c.t2 + tl;
  } else {
    c.wh = V.wh;
    c.v = V.v;
    c.w = V.w;   // also wbar of a step with a test (V.w itself is stored at the end)
    c.xb = V.xb;
    c.yb = V.yb;
    c.t1 = V.t1;
    c.t2 = V.t2;
    c.part = c.r.part;
  }
  c.j0 = min((int)c.a.n, c.b * c.p.rn);
  c.nr = min((int)c.a.n - c.j0, c.p.rn);
  c.i0 = min((int)c.a.m, c.b * c.p.rm);
  c.mr = min((int)c.a.m - c.i0, c.p.rm);
}

// E: the pending Halpern or restart update of (x, w_Q, Q w, A^* y) and eqs. (3.1)-(3.3) on the own rows,
// wbar_{1/2} into the gathered vector `half`
template <bool CL>
__device__ void elementwise(const Ctx<CL>& c, const Step& st, double* half) {
  const int mode = st.mode, ttest = st.ttest;
  const double ha = st.ha, hb = st.hb;
  const Args& a = c.a;
  const Vec& V = a.V;
  const bool HA = a.m > 0;
  for (int i = c.tid; i < c.nr; i += c.T) {
    const int j = c.j0 + i;
    double *X = c.n_row(SX) + i, *W = c.n_row(SW) + i, *QW = c.n_row(SQW) + i, *AY = c.n_row(SATY) + i;
    double x = *X, w = *W, qw = *QW, aty = HA ? *AY : 0.0;
    if (mode == 1) {
      x = fma(hb, fma(2.0, c.n_row(SXB)[i], -x), ha * c.n_row(SX0)[i]);
      w = fma(hb, fma(2.0, c.n_row(SWB)[i], -w), ha * c.n_row(SW0)[i]);
      qw = fma(hb, fma(2.0, c.n_row(SQWB)[i], -qw), ha * c.n_row(SQW0)[i]);
      if (HA) aty = fma(hb, fma(2.0, c.n_row(SATYB)[i], -aty), ha * c.n_row(SATY0)[i]);
    } else if (mode == 2) {
      x = c.n_row(SX0)[i] = c.n_row(SXB)[i];
      w = c.n_row(SW0)[i] = c.n_row(SWB)[i];
      qw = c.n_row(SQW0)[i] = c.n_row(SQWB)[i];
      if (HA) aty = c.n_row(SATY0)[i] = c.n_row(SATYB)[i];
    }
    *X = x;
    *W = w;
    *QW = qw;
    if (HA) *AY = aty;
    double g = -c.n_row(SC)[i] - qw;
    if (HA) g += aty;
    const double rz = fma(st.sigma, g, x);
    const double xbar = prox_phi(a.phi, rz, c.n_row(SL)[i], c.n_row(SU)[i], st.tau);
    const double xh = fma(2.0, xbar, -x), wh = fma(st.c2, xh, st.c1 * w);
    c.n_row(SXB)[i] = xbar;
    c.n_row(SXH)[i] = xh;
    c.n_row(SWH)[i] = wh;
    if (!HA) c.n_row(SWB)[i] = wh;
    c.put(half + j, wh);
    if (ttest) {
      c.put(c.xb + j, xbar);
      V.zb[j] = (xbar - rz) * st.isigma;
    }
  }
}

__device__ __forceinline__ Step step_of(const Ctrl& C) {
  Step s;
  s.ha = C.ha;
  s.hb = C.hb;
  s.fha = C.fha;
  s.fhb = C.fhb;
  s.sigma = C.sigma;
  s.isigma = C.inv_sigma;
  s.c1 = C.c1;
  s.c2 = C.c2;
  s.s = C.s;
  s.slA = C.slA;
  s.islA = C.inv_slA;
  s.tau = C.tau;
  s.mode = C.mode;
  s.rtest = C.rtest;
  s.ttest = C.ttest;
  return s;
}

// controller() for a step without a test, by one warp, and the scalars of the next step
__device__ __forceinline__ void advance_plain(Ctrl& C, const Step& now, Step& next, int lane) {
  const long long k = C.k + 1, t = C.t + 1;
  const double i = C.halpern_total ? (double)k : (double)t;
  const double fha = 1.0 / (i + 2.0);
  const int rtest = !C.restart_off && (t == 0 || (k + 1) % C.restart_every == 0);
  const int ttest = (k + 1) % C.check_every == 0 || k + 1 >= C.max_iter;
  __syncwarp();
  if (lane != 0) return;
  C.ha = now.fha;   // the weights of the step after this one, set when this one began
  C.hb = now.fhb;
  C.fha = fha;
  C.fhb = 1.0 - fha;
  C.mode = 1;
  C.t = t;
  C.k = k;
  C.rtest = rtest;
  C.ttest = ttest;
  next = now;
  next.ha = now.fha;
  next.hb = now.fhb;
  next.fha = fha;
  next.fhb = 1.0 - fha;
  next.mode = 1;
  next.rtest = rtest;
  next.ttest = ttest;
}

// theta~ of eq. (3.11) and Algorithm 5, after a step whose test asked for a restart; false: a wait gave up
template <bool CL>
__device__ bool restart_pass(Ctx<CL>& c) {
  const Args& a = c.a;
  const QDev& Q = a.Q;
  const bool HA = a.m > 0;
  double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (HA) {
    for (int i = c.tid; i < c.nr; i += c.T) c.put(c.v + c.j0 + i, c.n_row(SATYB)[i] - c.n_row(SATY0)[i]);
    if (!all_sync(c)) return false;
    if (Q.nfac || Q.ndense) {
      // <d, Q d> of the factor terms is ||t||^2: of the own rows, as soon as this block has formed them
      factor_rows(c, c.v, nullptr, c.t2, c.t2, false);
      __syncthreads();
      const int nf = Q.nfac ? (int)(Q.toff[Q.nfac - 1] + Q.fac[Q.nfac - 1].rows) : 0;
      for (int q = c.b * c.p.rp + c.tid; q < min(nf, (c.b + 1) * c.p.rp); q += c.T) s[4] = fma(c.ld(c.t2 + q), c.ld(c.t2 + q), s[4]);
      for (int q = nf + c.b * c.p.rd + c.tid; q < min((int)Q.tfd, nf + (c.b + 1) * c.p.rd); q += c.T)
        s[4] = fma(c.ld(c.t2 + q), c.ld(c.t2 + q), s[4]);
    }
    q_sums(c, c.v, nullptr, c.t2, nullptr, false);
  }
  for (int i = c.tid; i < c.nr; i += c.T) {
    const int j = c.j0 + i;
    const double dx = c.n_row(SXB)[i] - c.n_row(SX0)[i];
    const double dw = c.n_row(SWB)[i] - c.n_row(SW0)[i];
    const double qdw = c.n_row(SQWB)[i] - c.n_row(SQW0)[i];
    s[3] = fma(dx, dx, s[3]);
    s[1] = fma(dw, qdw, s[1]);
    if (HA) {
      const double d = c.n_row(SATYB)[i] - c.n_row(SATY0)[i];
      const double qd = c.rs0()[i] + q_bands(c, j, c.v);
      s[2] = fma(qdw, d, s[2]);
      s[4] = fma(d, qd, s[4]);
    }
  }
  for (int i = c.tid; i < c.mr; i += c.T) {
    const double dy = c.m_row(MYB)[i] - c.m_row(MY0)[i];
    s[0] = fma(dy, dy, s[0]);
  }
  __syncthreads();
  block_part(c, s, 0x1fu, 0u, 0, max(max(c.nr, c.mr), max(c.p.rp, c.p.rd)));
  if (!all_sync(c)) return false;
  all_parts(c, 0x1fu, 0u);
  if (c.tid < 32) {
    const double* t = c.S.tot;
    algorithm5(c.S.C, t[0], t[1], t[2], t[3], t[4]);
  }
  return true;
}

template <bool CL, int MT>
__global__ void __launch_bounds__(MT, 1)
    k_resident(const __grid_constant__ Args a, const __grid_constant__ ResPlan p, const ResRun r) {
  extern __shared__ __align__(16) double sm[];
  __shared__ Block S;
  Ctx<CL> c{a, p, r, S, sm, (int)blockIdx.x, (int)threadIdx.x, (int)blockDim.x};
  init_ctx(c);
  const Vec& V = a.V;
  const QDev& Q = a.Q;
  const bool HA = a.m > 0;
  const bool pre = p.pre != 0;
  {
    const int* src = reinterpret_cast<const int*>(a.C);
    int* dst = reinterpret_cast<int*>(&S.C);
    for (int i = c.tid; i < (int)(sizeof(Ctrl) / sizeof(int)); i += c.T) dst[i] = src[i];
  }
  double* const nv[] = {V.x, V.x0, V.w, V.w0, V.Qw, V.Qw0, V.ATy, V.ATy0, V.xb, V.xh, V.wh, V.wb, V.Qwb, V.ATyb};
  for (int i = c.tid; i < c.nr; i += c.T) {
    const int j = c.j0 + i;
#pragma unroll
    for (int k = 0; k <= SATYB; k++) c.n_row(k)[i] = nv[k][j];
    c.n_row(SC)[i] = V.c[j];
    c.n_row(SL)[i] = V.L[j];
    c.n_row(SU)[i] = V.U[j];
  }
  for (int i = c.tid; i < c.mr; i += c.T) {
    const int q = c.i0 + i;
    c.m_row(MY)[i] = V.y[q];
    c.m_row(MY0)[i] = V.y0[q];
    c.m_row(MYB)[i] = V.yb[q];
    c.m_row(ML)[i] = V.l[q];
    c.m_row(MU)[i] = V.u[q];
  }
  stage(c);
  if (S.C.done) return;
  if (CL) all_sync(c);   // a block's shared memory may be written once it runs
  if (c.tid == 0) S.st[1] = step_of(S.C);
  __syncthreads();
  // wbar_{1/2} of step `it` as the products gather it: with m = 0 no barrier lies between them and E of the next
  // step, which stores into the other vector (v, unused then)
  // (in the cluster form v = wh + n: an offset, so that the loads stay shared-memory loads; a choice of two pointers
  // made them generic, 0.4 us of a 15 us step at n = 1000)
  auto half = [&](long long it) {
    const bool first = HA || (it & 1);
    if constexpr (CL) return c.wh + (first ? 0 : (int)a.n);
    else return first ? c.wh : c.v;
  };
  elementwise(c, S.st[1], half(1));
  bool ok = true;
  for (long long it = 1;; it++) {
    // E of this step is done
    const Step& st = S.st[it & 1];
    Step& next = S.st[(it + 1) & 1];
    const bool rtest = st.rtest, ttest = st.ttest;
    const bool plain = !rtest && !ttest;
    const bool fused = plain && HA && it < r.steps;
    const double* x1 = ttest ? c.xb : nullptr;
    const double* wh = half(it);
    // a plain step takes no decision: the controller moves on to the next step meanwhile
    if (!(ok = all_sync(c, [&] { if (plain) advance_plain(S.C, st, next, c.tid & 31); }))) break;
    if (pre) {
      factor_rows(c, wh, x1, c.t1, c.t1 + Q.tlen, true);
      if (!(ok = all_sync(c))) break;
    }
    // Q wbar_{1/2} (and Q xbar), v
    q_sums(c, wh, x1, c.t1, c.t1 + Q.tlen, true);
    for (int i = c.tid; i < c.nr; i += c.T) {
      const int j = c.j0 + i;
      const double qwh = c.rs0()[i] + q_bands(c, j, wh);
      if (HA) c.put(c.v + j, fma(st.sigma, c.n_row(SQW)[i] - qwh, c.n_row(SXH)[i]));
      else c.n_row(SQWB)[i] = qwh;
      if (rtest) V.Qwh[j] = qwh;
      if (ttest) V.Qxb[j] = c.rs1()[i] + q_bands(c, j, c.xb);
    }
    if (HA) {
      if (!(ok = all_sync(c))) break;
      // A v (and A xbar), y-step of eq. (3.5)
      row_sums(c.team(), S.A, c.i0, c.mr, p.gA, c.v, x1, Own{c.rs0(), c.rs1(), false});
      __syncthreads();
      double e[4] = {0.0, 0.0, 0.0, 0.0};
      for (int i = c.tid; i < c.mr; i += c.T) {
        double *Y = c.m_row(MY) + i, *Y0 = c.m_row(MY0) + i, *YB = c.m_row(MYB) + i;
        double y = *Y;
        if (st.mode == 1) y = fma(st.hb, fma(2.0, *YB, -y), st.ha * *Y0);
        else if (st.mode == 2) y = *Y0 = *YB;
        *Y = y;
        const double lo = c.m_row(ML)[i], hi = c.m_row(MU)[i];
        const double ry = fma(-st.slA, y, c.rs0()[i]);
        const double yb = (iclamp(ry, lo, hi) - ry) * st.islA;
        *YB = yb;
        c.put(c.yb + c.i0 + i, yb);
        if (rtest) e[0] = fma(y - yb, y - yb, e[0]);
        if (ttest) {
          const double ax = c.rs1()[i], sc = V.ise ? V.ise[c.i0 + i] : 1.0;
          e[1] = imax(e[1], iabs(ax - iclamp(ax, lo, hi)) * sc);
          e[2] = imax(e[2], iabs(ax) * sc);
          if (igt0(yb)) e[3] += lo * yb;
          else if (ilt0(yb)) e[3] += hi * yb;
        }
      }
      if (!plain) block_part(c, e, (rtest ? 1u : 0u) | (ttest ? 14u : 0u), 6u, kWL, c.mr);
      if (!(ok = all_sync(c))) break;
      // A^T ybar, wbar; fused: the next Halpern update of (A^* y, w)
      row_sums(c.team(), S.AT, c.j0, c.nr, p.gAT, c.yb, nullptr, Own{c.rs0(), nullptr, false});
      __syncthreads();
      for (int i = c.tid; i < c.nr; i += c.T) {
        const double r0 = c.rs0()[i], aty = c.n_row(SATY)[i];
        const double wb = fma(st.s, r0 - aty, c.n_row(SWH)[i]);
        if (fused) {
          c.n_row(SATY)[i] = fma(st.fhb, fma(2.0, r0, -aty), st.fha * c.n_row(SATY0)[i]);
          const double w = fma(st.fhb, fma(2.0, wb, -c.n_row(SW)[i]), st.fha * c.n_row(SW0)[i]);
          c.n_row(SW)[i] = w;
          c.put(c.w + c.j0 + i, w);
        } else {
          c.n_row(SATYB)[i] = r0;
          c.n_row(SWB)[i] = wb;
          c.put(c.w + c.j0 + i, wb);
        }
      }
      if (!(ok = all_sync(c))) break;
      if (pre) {
        factor_rows(c, c.w, nullptr, c.t2, c.t2, true);
        if (!(ok = all_sync(c))) break;
      }
      q_sums(c, c.w, nullptr, c.t2, nullptr, true);
      for (int i = c.tid; i < c.nr; i += c.T) {
        const int j = c.j0 + i;
        const double q = c.rs0()[i] + q_bands(c, j, c.w);
        if (!fused) {
          c.n_row(SQWB)[i] = q;
          continue;
        }
        // the next step's Halpern update of x and eqs. (3.1)-(3.3)
        c.n_row(SQW)[i] = q;
        const double x = fma(st.fhb, c.n_row(SXH)[i], st.fha * c.n_row(SX0)[i]);
        const double g = -c.n_row(SC)[i] - q + c.n_row(SATY)[i];
        const double rz = fma(st.sigma, g, x);
        const double xbar = prox_phi(a.phi, rz, c.n_row(SL)[i], c.n_row(SU)[i], st.tau);
        const double xh = fma(2.0, xbar, -x), wh = fma(st.c2, xh, st.c1 * c.n_row(SW)[i]);
        c.n_row(SX)[i] = x;
        c.n_row(SXB)[i] = xbar;
        c.n_row(SXH)[i] = xh;
        c.n_row(SWH)[i] = wh;
        c.put(c.wh + j, wh);
        if (S.C.ttest) {
          c.put(c.xb + j, xbar);
          V.zb[j] = (xbar - rz) * st.isigma;
        }
      }
    }
    if (!plain) {
      // R~ of eq. (2.12) and the stopping rule of Sec. 4.1, on every block alike
      double e[kWL];
#pragma unroll
      for (int k = 0; k < kWL; k++) e[k] = 0.0;
      for (int i = c.tid; i < c.nr; i += c.T) {
        const int j = c.j0 + i;
        const double xb = c.n_row(SXB)[i], qwb = c.n_row(SQWB)[i], atyb = HA ? c.n_row(SATYB)[i] : 0.0;
        if (rtest) {
          const double dx = c.n_row(SX)[i] - xb, qdw = c.n_row(SQW)[i] - qwb;
          const double ady = HA ? c.n_row(SATY)[i] - atyb : 0.0;
          e[0] = fma(dx, dx, e[0]);
          e[1] = fma(c.n_row(SW)[i] - c.n_row(SWB)[i], qdw, e[1]);
          if (HA) {
            e[2] = fma(qdw, ady, e[2]);
            e[3] = fma(ady, V.Qwh[j] - qwb, e[3]);
          }
          e[4] = fma(dx, ady - qdw, e[4]);
        }
        if (ttest) {
          const double qxb = V.Qxb[j], cj = c.n_row(SC)[i], sc = V.isd ? V.isd[j] : 1.0, zb = V.zb[j];
          e[5] = imax(e[5], iabs(atyb - qxb + zb - cj) * sc);
          e[6] = imax(e[6], iabs(atyb) * sc);
          e[7] = imax(e[7], iabs(qxb) * sc);
          e[8] = fma(xb, qxb, e[8]);
          e[9] = fma(cj, xb, e[9]);
          if (a.phi != PHI_BOX) e[10] += iabs(xb);
          e[11] += conj_phi_term(a.phi, zb, c.n_row(SL)[i], c.n_row(SU)[i], S.C.lambda);
        }
      }
      __syncthreads();
      const unsigned want = (rtest ? 0x1fu : 0u) | (ttest ? 0xfe0u : 0u);
      const unsigned wanty = HA ? (rtest ? 1u : 0u) | (ttest ? 14u : 0u) : 0u;
      block_part(c, e, want, kEndMax, 0, c.nr);
      if (!(ok = all_sync(c))) break;
      all_parts(c, want | (wanty << kWL), kEndMax | (6u << kWL));
      if (c.tid == 0) controller(S.C, S.tot, S.tot + kWL, c.b == 0 ? a.hist : nullptr);
      __syncthreads();
      if (S.C.restart_pending && !S.C.done) {
        if (!(ok = restart_pass(c))) break;
      }
    }
    __syncthreads();
    if (S.C.done || it >= r.steps) break;
    if (!plain) {
      if (c.tid == 0) next = step_of(S.C);
      __syncthreads();
    }
    if (!fused) elementwise(c, next, half(it + 1));
  }
  // no block still gathers from the vectors that are stored below (or from a copy in a block that ends)
  if (!ok || !all_sync(c)) return;
  // the state for hprqp_get and for a later launch (which applies the pending update, C.mode)
  for (int i = c.tid; i < c.nr; i += c.T) {
    const int j = c.j0 + i;
#pragma unroll
    for (int k = 0; k <= SATYB; k++) nv[k][j] = c.n_row(k)[i];
  }
  for (int i = c.tid; i < c.mr; i += c.T) {
    V.y[c.i0 + i] = c.m_row(MY)[i];
    V.y0[c.i0 + i] = c.m_row(MY0)[i];
    V.yb[c.i0 + i] = c.m_row(MYB)[i];
  }
  if (c.b == 0) {
    __syncthreads();
    int* dst = reinterpret_cast<int*>(a.C);
    const int* src = reinterpret_cast<const int*>(&S.C);
    for (int i = c.tid; i < (int)(sizeof(Ctrl) / sizeof(int)); i += c.T) dst[i] = src[i];
  }
}

// Both power methods of Sec. 4.1 (on A A^* and on Q, whichever `which` asks for: bits 0 and 1) side by side in one
// launch; each iteration folds the normalisation of the one before into its products, as in kernels.cuh.
template <bool CL, int MT>
__global__ void __launch_bounds__(MT, 1)
    k_resident_power(const __grid_constant__ Args a, const __grid_constant__ ResPlan p, const ResRun r, int which,
                     ResPower pw) {
  extern __shared__ __align__(16) double sm[];
  __shared__ Block S;
  __shared__ double lam[2], scale[2];
  __shared__ long long its[2];
  __shared__ int on[2];
  Ctx<CL> c{a, p, r, S, sm, (int)blockIdx.x, (int)threadIdx.x, (int)blockDim.x};
  init_ctx(c);
  stage(c);
  // the vectors on R^m (two), R^n (two) and A^T v
  double *va = CL ? c.yb : pw.va, *wa = CL ? c.yb + a.m : pw.wa;
  double *vq = CL ? c.wh : a.V.pv, *wq = CL ? c.v : a.V.pw, *u = CL ? c.xb : pw.u;
  if (CL) all_sync(c);   // a block's shared memory may be written once it runs
  auto start = [](int i) { return 0.5 + (double)((uint32_t)((uint64_t)(i + 1) * 2654435761u)) / 4294967296.0; };
  for (int i = c.tid; i < c.mr && (which & 1); i += c.T) c.put(va + c.i0 + i, start(c.i0 + i));
  for (int i = c.tid; i < c.nr && (which & 2); i += c.T) c.put(vq + c.j0 + i, start(c.j0 + i));
  if (c.tid < 2) {
    lam[c.tid] = 0.0;
    its[c.tid] = 0;
    on[c.tid] = (which >> c.tid) & 1;
    scale[c.tid] = pw.scale[c.tid];
  }
  __syncthreads();
  const bool pre = p.pre != 0;
  if (!all_sync(c)) return;
  for (;;) {   // the vectors that this iteration gathers from were stored before the last barrier
    const bool doA = on[0], doQ = on[1];
    if (!doA && !doQ) break;
    if (doA) row_sums(c.team(), S.AT, c.j0, c.nr, p.gAT, va, nullptr, Own{c.rs0(), nullptr, false});
    __syncthreads();
    for (int i = c.tid; i < c.nr && doA; i += c.T) c.put(u + c.j0 + i, c.rs0()[i]);
    if (doQ && pre) factor_rows(c, vq, nullptr, c.t1, c.t1, true);
    if (doA || (doQ && pre)) {
      if (!all_sync(c)) return;
    }
    double e[4] = {0.0, 0.0, 0.0, 0.0};
    if (doA) {
      row_sums(c.team(), S.A, c.i0, c.mr, p.gA, u, nullptr, Own{c.rs0(), nullptr, false});
      __syncthreads();
      for (int i = c.tid; i < c.mr; i += c.T) {
        const double w = scale[0] * c.rs0()[i];
        c.put(wa + c.i0 + i, w);
        e[0] = fma(scale[0] * c.ld(va + c.i0 + i), w, e[0]);
        e[1] = fma(w, w, e[1]);
      }
      __syncthreads();
    }
    if (doQ) {
      q_sums(c, vq, nullptr, c.t1, nullptr, true);
      for (int i = c.tid; i < c.nr; i += c.T) {
        const int j = c.j0 + i;
        const double w = scale[1] * (c.rs0()[i] + q_bands(c, j, vq));
        c.put(wq + j, w);
        e[2] = fma(scale[1] * c.ld(vq + j), w, e[2]);
        e[3] = fma(w, w, e[3]);
      }
      __syncthreads();
    }
    const unsigned want = (doA ? 3u : 0u) | (doQ ? 12u : 0u);
    block_part(c, e, want, 0u, 0, max(c.nr, c.mr));
    if (!all_sync(c)) return;
    all_parts(c, want, 0u);
    if ((c.tid == 0 && doA) || (c.tid == 32 && doQ)) {
      // Rayleigh quotient of the unit vector, Sec. 4.1
      const int q = c.tid >> 5;
      const double lnew = S.tot[2 * q], nw = sqrt(S.tot[2 * q + 1]);
      if (nw == 0.0 || !isfinite(nw)) {
        lam[q] = 0.0;
        on[q] = 0;
      } else {
        const bool conv = its[q] > 0 && fabs(lnew - lam[q]) <= pw.tol * fabs(lnew);
        lam[q] = lnew;
        scale[q] = 1.0 / nw;
        its[q]++;
        if (conv || its[q] >= pw.max_iter) on[q] = 0;
      }
    }
    __syncthreads();
    double* t = va;
    va = wa;
    wa = t;
    t = vq;
    vq = wq;
    wq = t;
  }
  if (CL) all_sync(c);   // no block ends while another may store into its copies
  if (c.b == 0 && c.tid < 2) r.lam[c.tid] = lam[c.tid];
}

}  // namespace

namespace {

using Kernel = void (*)(Args, ResPlan, ResRun);
using PowerKernel = void (*)(Args, ResPlan, ResRun, int, ResPower);
// up to 512 threads the compiler has 128 registers a thread, above 64
Kernel solve_kernel(const ResPlan& p) {
  return p.cluster ? k_resident<true, 512> : p.T > 512 ? k_resident<false, kResThreads> : k_resident<false, 512>;
}
PowerKernel power_kernel(const ResPlan& p) {
  return p.cluster ? k_resident_power<true, 512>
                   : p.T > 512 ? k_resident_power<false, kResThreads> : k_resident_power<false, 512>;
}

// Lets kernel k take any plan's shared memory and cluster.  The limits belong to the kernel, not to a launch: they are
// set to the same values every time, so that handles with other plans may launch k from other threads meanwhile.
cudaError_t setup(const ResPlan& p, const void* k) {
  cudaError_t e = shared_memory_limit(k);
  if (e == cudaSuccess && p.cluster) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

// The launch of a plan: one cluster, or a cooperative grid
struct Launch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  Launch(const ResPlan& p, cudaStream_t s) {
    cfg.gridDim = dim3(p.B);
    cfg.blockDim = dim3(p.T);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    if (p.cluster) {
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)p.B;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

bool fits(const ResPlan& p, const void* k, int sms) {
  if (setup(p, k) != cudaSuccess) return false;
  int most = 0;
  if (p.cluster) {
    Launch l(p, nullptr);
    return cudaOccupancyMaxActiveClusters(&most, k, &l.cfg) == cudaSuccess && most >= 1;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&most, k, p.T, p.smem) == cudaSuccess && most * sms >= p.B;
}

}  // namespace

size_t resident_static_smem() {
  size_t most = 0;
  for (const void* k : {(const void*)k_resident<true, 512>, (const void*)k_resident<false, 512>,
                        (const void*)k_resident<false, kResThreads>, (const void*)k_resident_power<true, 512>,
                        (const void*)k_resident_power<false, 512>, (const void*)k_resident_power<false, kResThreads>}) {
    cudaFuncAttributes f;
    if (cudaFuncGetAttributes(&f, k) != cudaSuccess) {
      cudaGetLastError();
      return 1 << 20;
    }
    most = std::max(most, f.sharedSizeBytes);
  }
  return most;
}

bool resident_fits(const ResPlan& p, int sms) {
  const bool ok = fits(p, (const void*)solve_kernel(p), sms) && fits(p, (const void*)power_kernel(p), sms);
  if (!ok) cudaGetLastError();
  return ok;
}

cudaError_t launch_resident(const Args& a, const ResPlan& p, const ResRun& r, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(r.flags, 0, 2 * sizeof(unsigned), s);   // the counter and the error word
  if (e == cudaSuccess) e = setup(p, (const void*)solve_kernel(p));
  if (e != cudaSuccess) return e;
  Launch l(p, s);
  return cudaLaunchKernelEx(&l.cfg, solve_kernel(p), a, p, r);
}

cudaError_t launch_resident_power(const Args& a, const ResPlan& p, const ResRun& r, int which, const ResPower& pw,
                                  cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(r.flags, 0, 2 * sizeof(unsigned), s);
  if (e == cudaSuccess) e = setup(p, (const void*)power_kernel(p));
  if (e != cudaSuccess) return e;
  Launch l(p, s);
  return cudaLaunchKernelEx(&l.cfg, power_kernel(p), a, p, r, which, pw);
}

}  // namespace hprqp

// Launch plan of the resident solver (resident.cu): how a problem is split over the blocks and what
// each block keeps in shared memory.
#pragma once
#include "solver.cuh"

namespace hprqp {

constexpr int kResThreads = 1024;   // most threads of a block
constexpr int kResStateN = 17;      // doubles of state per own row of R^n
constexpr int kResStateM = 5;       // ... of R^m

struct ResPlan {
  int B = 0, T = 0;          // blocks (0: the problem does not run resident) and threads per block
  int cluster = 0;           // the blocks form one thread-block cluster and hold copies of the gathered vectors
  int rn = 0, rm = 0;        // rows of the n- and m-vectors per block
  int rp = 0, rd = 0;        // rows of the sparse and dense factors per block
  int gQ = 1, gT = 1, gF = 1, gA = 1, gAT = 1, gP = 1;   // lanes per row of Q, thin, B^T, A, A^T, B (0: the block)
  int cw = 32;               // columns of a dense factor that a block handles at once
  int pre = 0;               // the step forms factor products before its Q passes
  int rs_len = 0;            // rows of the row-sum buffers
  int o_rs = 0, o_scratch = 0, o_vec = 0;
  // shared-memory copies: offsets in doubles, -1: read from global memory
  struct M {
    int o_v = -1, o_ci = -1, o_rp = -1;
  };
  M A, AT, Qc, thin, fac[kMaxFac], fact[kMaxFac];
  int o_diag = -1;
  int o_dia[kMaxDia] = {-1, -1, -1, -1, -1, -1, -1, -1};
  int o_dcol[kMaxDense] = {-1, -1, -1, -1}, o_drow[kMaxDense] = {-1, -1, -1, -1};
  size_t smem = 0;           // dynamic shared memory of a block
};

constexpr unsigned kResSpin = 1u << 22;   // polls of one wait, unless asked otherwise (a few seconds; each is a round trip to L2)

// Per launch: at most `steps` inner steps; flags: the barrier's counter, followed by the error word; part:
// 2 x B x 16 partial sums; lam: 2 results of the power methods; spin: polls of one wait of the grid barrier.
struct ResRun {
  long long steps = 0;
  unsigned spin = kResSpin;
  unsigned* flags = nullptr;
  int* err = nullptr;
  double* part = nullptr;
  double* lam = nullptr;
};

// The power methods: vectors of the one on A A^* (the one on Q uses pv and pw), 1 / ||start|| of both
struct ResPower {
  double *va = nullptr, *wa = nullptr, *u = nullptr;
  double scale[2] = {0.0, 0.0};
  double tol = 0.0;
  long long max_iter = 0;
};

size_t resident_static_smem();
// Whether the plan's blocks can be resident at once
bool resident_fits(const ResPlan& p, int sms);
cudaError_t launch_resident(const Args& a, const ResPlan& p, const ResRun& r, cudaStream_t s);
cudaError_t launch_resident_power(const Args& a, const ResPlan& p, const ResRun& r, int which, const ResPower& pw,
                                  cudaStream_t s);

}  // namespace hprqp

// The QAP operator on the tensor cores (qap_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hprqp {

// operands cut into digits: the stored matrices, X by rows and by columns, T1 = Ahat X by rows
enum { kAhat = 0, kBhat = 1, kS = 2, kT = 3, kXRow = 4, kXCol = 5, kT1 = 6, kTcMats = 7 };

struct QapTcDev {
  int d, dp, kp;              // size; rows of a digit plane (a multiple of 128), columns (of 64)
  int groups;                 // partial sums per product: chunks of 64 k's are dealt to them in turn
  size_t plane;               // pairs of digits per plane
  const double* mats;         // Ahat, Bhat, S, T
  uint32_t* dig[kTcMats];     // seven planes each, most significant first
  double* scale[kTcMats];     // 2^(exponent - 34) of every row
  long long* part;            // [product][group][high, low][column][row]
  double* t1;
  int* err;                   // [0] set by a bounded wait that gave up; [1] polls of a wait for operands (0: kSpin)
};

struct QapTc;
// device memory that a handle provides for size d; part: its pieces
size_t qap_tc_bytes(int64_t d, size_t (&part)[5]);
// mats: Ahat, Bhat, S, T on the device (read by every product); mem: qap_tc_bytes(d) bytes, 1024-byte aligned
cudaError_t qap_tc_create(QapTc** out, int64_t d, const double* mats, void* mem, cudaStream_t s);
void qap_tc_free(QapTc* t);
int* qap_tc_error(const QapTc* t);   // device words: QapTcDev::err
// out = vec(Ahat X Bhat - S X - X T): five kernels; pdl: the last four as programmatic dependent launches
cudaError_t qap_tc_apply(const QapTc* t, const double* x, double* out, bool pdl, cudaStream_t s);
constexpr int kQapTcKernels = 5;

}  // namespace hprqp

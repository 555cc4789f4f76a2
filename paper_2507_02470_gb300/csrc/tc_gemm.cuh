// BF16 tensor-core GEMM for the learned warm start: C = A * B^T with A (M x K) and B (N x K)
// both row-major with K contiguous ("K-major"), BF16 inputs, FP32 accumulation in tensor
// memory, FP32 output.  Every product of the warm-start network (forward and backward), the
// feature projection and the decoder is written in this one form by choosing which stored
// layout (batch-major or feature-major) plays A and which plays B.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace hprqp {
namespace tc {

// Launches C = A B^T (split along K into `splits` parts summed in a fixed order when
// splits > 1, using `work` of splits * M * N floats).  A: M x K with leading dimension lda
// (elements), B: N x K with ldb, C: M x N with ldc.  Requirements checked here: lda, ldb
// multiples of 8 (16-byte rows), A and B 16-byte aligned, lda >= K, ldb >= K, ldc >= N.
// Rows and columns past M, N, K are read as zeros by the copy engine and never written.
// Returns cudaSuccess or the first failing runtime/driver call as a cudaError_t;
// cudaErrorInvalidValue for bad arguments (message in *why when why != nullptr).
cudaError_t gemm_bf16(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                      float* C, int64_t ldc, int splits, float* work, cudaStream_t stream, const char** why);

// Z[n][i] = clip(mu[i] + alpha (A B^T)[i][n], lo[i], hi[i]) in FP64 for A (D x K) and B (N x K) as
// above, in one launch: the FP32 product stays in tensor memory.  Z is N x D with leading dimension ldz.
cudaError_t gemm_decode(int64_t D, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                        double alpha, const double* mu, const double* lo, const double* hi, double* Z, int64_t ldz,
                        cudaStream_t stream, const char** why);

// What follows a layer's product acc (M features x N members), in the same launch:
//   HIDDEN  v = bf16(relu(acc + bias)) -> outT (M x ldT) and outB (N x ldB)
//   MASK    v = bf16(acc where mask > 0, else 0) -> outT, outB   (mask: BF16, M x ldmask)
//   FINAL   out[n][m] = acc + bias (N x ldo)
//   PLAIN   out[m][n] = acc (M x ldo)
// outT and outB rows are 8-byte aligned.
enum LayerMode { LAYER_HIDDEN = 0, LAYER_MASK = 1, LAYER_FINAL = 2, LAYER_PLAIN = 3 };
struct Layer {
  int mode = LAYER_PLAIN;
  const float* bias = nullptr;
  const uint16_t* mask = nullptr;
  int64_t ldmask = 0;
  uint16_t* outT = nullptr;
  int64_t ldT = 0;
  uint16_t* outB = nullptr;
  int64_t ldB = 0;
  float* out = nullptr;
  int64_t ldo = 0;
};
constexpr int kLayerSplits = 16;              // K-splits of a tile: CTAs of one cluster
int layer_splits(int64_t K, int splits);      // the splits that a request for `splits` comes to
// The most K-splits of a layer that the current device can hold as one cluster: kLayerSplits, or the largest power
// of two below it for which it has a group of that many SMs
int layer_cluster();
cudaError_t gemm_layer(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, const void* B, int64_t ldb,
                       int splits, const Layer& l, cudaStream_t stream, const char** why);

// Reads and clears the device flag that a GEMM kernel sets when one of its bounded waits
// gave up (0: none; 1 producer, 2 MMA issuer, 3 epilogue).  Synchronises the device.
int gemm_error_flag();

}  // namespace tc
}  // namespace hprqp

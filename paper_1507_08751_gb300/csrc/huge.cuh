// Shared by the kernels of blocks wider than 256: the subspace iteration
// (k_block_huge.cu) and the certificate (k_cert_tc.cu).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "internal.h"

namespace msllr {

constexpr int kHP = 32;          // subspace width
constexpr int kHK = 16;          // most Ritz pairs kept per block
constexpr int kCertLevels = 8;   // squarings of the certificate, at most

enum : int { kHsSkip = 1, kHsIter = 2 };                 // HugeBlock::status
enum : int { kCertOpen = 0, kCertYes = 1, kCertNo = 2 };  // HugeBlock::cert

// per-block state of the wide path
struct HugeBlock {
  float trace;   // trace(G) (>= lambda_max)
  float gF;      // ||G||_F
  float c;       // certificate bound
  float theta[kHK];
  int status;    // kHs*
  int ku;        // kept Ritz pairs
  int k;         // pairs above tau
  int conv;      // Rayleigh-Ritz residual test passed
  int orth_fail; // a CholQR factorisation broke down (basis restarted)
  int cert;      // kCert*
  int arrived;   // CTAs of the running certificate level that are done
  double fro[kCertLevels + 1];  // F-norm of each level
  double err[kCertLevels + 1];  // bound of each level's rounding
};

// tile (i, j), i >= j, of position t in the row-by-row lower triangle
__device__ __forceinline__ void tile_of(int t, int* ta, int* tc) {
  int i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while (((i + 1) * (i + 2)) / 2 <= t) ++i;
  while ((i * (i + 1)) / 2 > t) --i;
  *ta = i;
  *tc = t - (i * (i + 1)) / 2;
}

// Certificate workspace per block (bytes of one of the two FP16 matrices,
// F-norm partials) and its launches: form plus kCertLevels squarings.
size_t cert_matrix_bytes(int nn);
size_t cert_fpart_count(int nn);
cudaError_t configure_cert();
cudaError_t launch_cert(const float* G, const float* U, const float* Wh, void* Ma, void* Mb,
                        double* fpart, HugeBlock* hb, int nn, int B, int* err, cudaStream_t st,
                        Prof* prof);

}  // namespace msllr

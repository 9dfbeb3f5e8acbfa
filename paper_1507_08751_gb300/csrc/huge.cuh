// Shared by the kernels of blocks wider than 256: Gram and rebuild
// (k_block_huge.cu), subspace iteration (k_subspace.cu) and certificate
// (k_cert_tc.cu; its bound also by k_eig.cu).
#pragma once

#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
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
  int conv;      // Rayleigh-Ritz residual test passed
  int stop;      // further rounds would not bring the pairs to convergence
  float worst;   // largest residual of the pairs relative to its bar
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

// The bound the certificate has to prove: ||P G P||_2 < c shows, by Cauchy
// interlacing, that G has at most ku eigenvalues above c (and the ku Ritz
// values above tau^2 are lower bounds of ku eigenvalues), so exactly the kept
// pairs lie above tau^2.  c = tau^2 less the rounding of forming X = P G P
// entry by entry as G - U What^T - What U^T: 2 ku multiply-adds, so an entry
// errs by at most ku eps (|G| + 2 |U| |What|^T) of it.  gnorm bounds the
// spectral norm of |G|: ||G||_F, its trace, or its largest row sum; that of
// |U| |What|^T is at most sqrt(ku) ||What||_F, wsum = ||What||_F^2.  The
// certificate accounts for its own rounding.
__host__ __device__ __forceinline__ float cert_bound(float thr, float gnorm, int ku, float wsum) {
  const float xf = gnorm + 2.f * sqrtf((float)ku) * sqrtf(wsum);
  return thr - 1.1f * FLT_EPSILON * (float)(2 * ku + 4) * xf;
}

// deterministic pseudo-random value in [-1, 1)
__device__ __forceinline__ float huge_hash(uint32_t a, uint32_t b) {
  uint32_t h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (float)(h >> 8) * (2.f / 16777216.f) - 1.f;
}

// How the subspace iteration of blocks of order np (a multiple of 64), B of
// them in a job, runs on a device of `sms` multiprocessors whose clusters hold
// up to `widest` CTAs (16, or 8 where the device has no room for 16).  The
// cluster size sets the order of the sums, so it depends on the job alone and
// not on how many jobs share the launch: a batched job then sums as its solo
// run does.
constexpr int kSMaxRows = 128;    // rows per CTA of the one-launch kernel, at most
constexpr int kSPhaseRows = 512;  // rows per CTA of the phase kernels, at most
struct SubspacePlan {
  int cluster;  // CTAs per block; 0: the device cannot run blocks this wide
  bool phases;  // a launch per phase instead of one for every step
};
inline SubspacePlan subspace_plan(int np, int B, int sms, int widest) {
  // 8 CTAs per block up to 512 wide, 16 above (32 to 128 rows a CTA), where a
  // lone block's latency counts; 8 up to 1024 wide when the blocks fill the
  // chip anyway (64 blocks of 1024: 3.4 -> 2.3 ms)
  const bool few = np <= 512 || (16 * B > sms && np <= 8 * kSMaxRows);
  const int cl = few || widest < 16 ? 8 : 16;
  if (np / cl <= kSMaxRows) return {cl, false};
  return {np / cl <= kSPhaseRows ? cl : 0, true};
}

// Subspace iteration and Rayleigh-Ritz (k_subspace.cu): kernel attributes and
// the launches (first: steps of the first round; W: workspace, np x kHP).
cudaError_t configure_subspace();
// The launches cover B blocks of jobs with `job_blocks` blocks each; W is used
// only where subspace_phases(np).
bool subspace_phases(int np);
cudaError_t launch_subspace(const float* G, float* V, float* W, float* U, float* GU, int nn, int np,
                            float thr, int first, HugeBlock* hb, int B, int job_blocks, cudaStream_t st,
                            Prof* prof);

// Certificate workspace per block (F-norm partials; Ma and Mb hold np x np FP16
// each) and its launches: form plus kCertLevels squarings.  Mb may be G's own
// space: only the forming launch, which writes Ma, reads G.
size_t cert_fpart_count(int nn);
cudaError_t configure_cert();
cudaError_t launch_cert(const float* G, const float* U, const float* Wh, void* Ma, void* Mb,
                        double* fpart, HugeBlock* hb, int nn, int B, int* err, cudaStream_t st,
                        Prof* prof);

}  // namespace msllr

// Certified top eigenpairs of a block's Gram matrix G = C^T C without a full
// tridiagonalisation, for the block SVT (eq:svt): SVT needs only the
// eigenpairs with lambda > tau^2.
//
//  1. Lanczos with full reorthogonalisation (Golub & Van Loan, Sec. 10.1)
//     builds an orthonormal Q_J and the tridiagonal T_J = Q_J^T G Q_J.  The
//     start vector is either pseudo-random or the sum of the previous
//     iteration's Ritz vectors (warm start).  On breakdown the process is
//     continued from a random vector orthogonal to Q_J.
//  2. Ritz pairs of T_J above 0.95 tau^2: Sturm-count multisection and
//     inverse iteration on T_J (symeig.cuh), U = Q_J Y.
//  3. Explicit residuals: W = G U, B = U^T W, rho = ||W - U diag(B)||_F.
//  4. Certificate: with P = I - U U^T, every eigenvalue of G lies within
//     2 rho of an eigenvalue of diag(B) (+) (P G P restricted to range P)
//     (Weyl, block form in the basis [U, U_perp]).  If the Cholesky of
//     (tau^2 - 2 rho - margins) I - P G P succeeds, no eigenvalue of G
//     outside span(U) exceeds tau^2, so the eigenpairs above tau^2 are the
//     Ritz pairs above tau^2 (up to pairs within 2 rho of tau^2, whose
//     thresholded contribution is below rho / tau).
// If any step fails (too many pairs, no convergence, certificate refused),
// the caller falls back to the Householder path.
#pragma once

#include <float.h>

#include "common.cuh"
#include "regchol.cuh"
#include "symeig.cuh"

namespace msllr {

constexpr int kLzMaxJ = 32;  // Lanczos steps
// A coupling beta below this fraction of the norm bound counts as a breakdown
// and is set to zero, which moves G by as much: the rounding level of G q (a
// few eps).  At 1e-5 the neglected coupling showed in the result: blocks of rank
// three (5, 3 and 2 tau) came out up to 8e-5 tau off, 4e-6 tau now.  A breakdown
// that goes unnoticed does no harm: the next direction is rounding, made
// orthogonal like any other.
constexpr float kLzBreak = 3e-7f;
// Ritz pairs kept (above 0.95 tau^2): 8 for blocks up to 64 wide, 16 above,
// where the alternative, a Householder reduction, takes some 0.3 ms (256 wide)
constexpr int lz_maxk(int nmax) { return nmax > 64 ? 16 : 8; }

// FP32 flops of the eigen-solve steps, each counted at its algorithmic cost
// (a multiply-add is 2 flops); the kernels add them up per block so that the
// ALU roofline follows the steps that actually ran.
__device__ __forceinline__ double fl_symv(int n) { return 2.0 * n * n; }
__device__ __forceinline__ double fl_chol(int n) { return (double)n * n * n / 3.0; }
// J Lanczos steps (matrix-vector product plus two Gram-Schmidt passes over
// j + 1 vectors), U = Q_J Y, W = G U for 8 vectors, B = U^T W
__device__ __forceinline__ double fl_lanczos(int n, int J, int ku) {
  return 2.0 * n * n * J + 4.0 * n * J * (J + 1) + 2.0 * n * J * ku + 2.0 * n * n * ((ku + 7) & ~7) + 16.0 * n * ku;
}
// the rank-2k deflation G - U What^T - What U^T on the lower triangle
__device__ __forceinline__ double fl_deflate(int n, int ku) { return 2.0 * ku * n * n; }
// Householder tridiagonalisation, back-transformation of k eigenvectors
__device__ __forceinline__ double fl_householder(int n, int k) {
  return 4.0 * n * n * n / 3.0 + 2.0 * n * n * k;
}

// leading dimension of the Lanczos basis in shared memory
__host__ __device__ constexpr int lz_ldq(int n) { return n + 1; }

// shared scratch (floats) of the certificate step of lanczos_candidates
__host__ __device__ constexpr int lz_cert_floats(int nmax, int nt) {
  return 2 * lz_maxk(nmax) * nmax + regchol_scratch_floats(nmax, nt);
}

// Shared-memory scratch of the Lanczos path.
struct LzScratch {
  float* x;      // [n] current Lanczos vector q_j
  float* w;      // [n] G q_j, then the next residual
  float* alpha;  // [kLzMaxJ]
  float* beta;   // [kLzMaxJ]
  float* h;      // [2 * kLzMaxJ + 8] projection coefficients (two passes)
  float* ty;     // [jcap * K] eigenvectors of T_J (row i, column q), K = lz_maxk
  float* lu;     // [4 * jcap * K] inverse-iteration LU factors
  float* Bm;     // [K * K] U^T G U
  int jcap;      // row capacity of ty / lu (>= Lanczos steps)
};

// floats of LzScratch for a given n capacity and J capacity
__host__ __device__ constexpr int lz_scratch_floats(int nmax, int jcap) {
  return 2 * nmax + 2 * kLzMaxJ + (2 * kLzMaxJ + 8) + 5 * jcap * lz_maxk(nmax) +
         lz_maxk(nmax) * lz_maxk(nmax);
}

template <int NT>
__device__ void lz_bind(LzScratch& z, float* base, int nmax, int jcap) {
  z.x = base;
  z.w = z.x + nmax;
  z.alpha = z.w + nmax;
  z.beta = z.alpha + kLzMaxJ;
  z.h = z.beta + kLzMaxJ;
  z.ty = z.h + 2 * kLzMaxJ + 8;
  const int K = lz_maxk(nmax);
  z.lu = z.ty + jcap * K;
  z.Bm = z.lu + 4 * jcap * K;
  z.jcap = jcap;
}

__device__ __forceinline__ float lz_hash(uint32_t seed, int i) {
  uint32_t h = seed * 0x9E3779B9u + (uint32_t)i * 0x85EBCA6Bu + 0x27D4EB2Fu;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (float)(h >> 8) * (2.f / 16777216.f) - 1.f;
}

// Ritz values of T_J above thr (descending, at most K) into lam and their
// vectors into z.ty, a warp per pair: count and multisection on Sturm counts
// (32 points a round), then two steps of inverse iteration in its lane 0 (the
// approximate division only perturbs the factors by an ulp or two, which the
// second step corrects).
// Returns the count (above K: nothing else is set).  Uses s.d, s.e2, s.lam,
// s.shf, s.clus (J entries) and s.red.
template <int NT, int K>
__device__ __forceinline__ int lz_ritz(int J, float thr, const LzScratch& z, EigScratch& s) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *d = s.d, *e2 = s.e2, *lam = s.lam, *shf = s.shf;
  int* clus = s.clus;
  __syncthreads();
  // norm and bounds, in every warp (J <= 32)
  const float ai = lane < J ? z.alpha[lane] : 0.f;
  const float bi = lane < J - 1 ? z.beta[lane] : 0.f;
  const float bm = __shfl_up_sync(0xffffffffu, bi, 1);
  const float rad = fabsf(bi) + (lane > 0 ? fabsf(bm) : 0.f);
  const float gup = warp_max(lane < J ? ai + rad : -FLT_MAX);
  const float tn = warp_max(lane < J ? fabsf(ai) + rad : -FLT_MAX);
  const float pivmin = FLT_MIN * fmaxf(1.f, warp_max(bi * bi));
  if (warp == 0 && lane < J) {
    d[lane] = ai;
    e2[lane] = bi * bi;
  }
  __syncthreads();
  const int k = J - sturm_below(d, e2, J, thr, pivmin);
  if (k <= 0 || k > K) return k < 0 ? 0 : k;
  for (int q = warp; q < k; q += NW) {
    const int target = J - 1 - q;  // ascending index of the eigenvalue sought
    float lo = thr, hi = gup + 4.f * FLT_EPSILON * fmaxf(fabsf(gup), tn) + pivmin;
    const float tol = 2.f * FLT_EPSILON * tn;
    for (int round = 0; round < 64; ++round) {
      if (!(hi - lo > fmaxf(tol, 2.f * FLT_EPSILON * fmaxf(fabsf(lo), fabsf(hi))))) break;
      const float x = lo + (hi - lo) * ((float)(lane + 1) / 33.f);
      const unsigned above =
          __ballot_sync(0xffffffffu, sturm_below(d, e2, J, x, pivmin) > target);
      // counts grow with x: the first point above the target brackets it
      float nlo = lo, nhi = hi;
      if (above == 0u) {
        nlo = __shfl_sync(0xffffffffu, x, 31);
      } else {
        const int f = __ffs(above) - 1;
        nhi = __shfl_sync(0xffffffffu, x, f);
        if (f > 0) nlo = __shfl_sync(0xffffffffu, x, f - 1);
      }
      lo = fminf(nlo, nhi);
      hi = nhi;
    }
    if (lane == 0) lam[q] = 0.5f * (lo + hi);
  }
  __syncthreads();
  // inverse-iteration shifts kept apart, clusters of close eigenvalues
  if (tid == 0) {
    shf[0] = lam[0];
    clus[0] = 0;
    for (int j = 1; j < k; ++j) {
      shf[j] = fminf(lam[j], shf[j - 1] - 10.f * FLT_EPSILON * tn);
      clus[j] = (lam[j - 1] - lam[j] <= 1e-3f * tn) ? clus[j - 1] : j;
    }
  }
  __syncthreads();
  bool grouped = false;
  for (int j = 1; j < k; ++j) grouped = grouped || clus[j] != j;
  const float tiny = FLT_EPSILON * tn;
  constexpr int PQ = (K + NW - 1) / NW;  // pairs per warp, at most
  unsigned pbits[PQ] = {};
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
    for (int w = 0; w < PQ; ++w) {
    const int q = warp + w * NW;
    float* dd = z.lu + q;
    float* du = dd + z.jcap * K;
    float* du2 = du + z.jcap * K;
    float* dl = du2 + z.jcap * K;
    float* y = z.ty + q;
    unsigned bits = pbits[w];
    // deterministic pseudo-random start vector of size ~eps |T|
    if (pass == 0 && q < k && lane < J) y[lane * K] = tiny * lz_hash(977u + q, lane);
    if (pass == 1 && q < k && lane < J) y[lane * K] *= tiny;
    __syncwarp();
    if (q < k && lane == 0) {
      if (pass == 0) {
        // pivoted LU of T - shift I, tiny pivots replaced by +-tiny
        const float shift = shf[q];
        float di = d[0] - shift, ui = J > 1 ? z.beta[0] : 0.f;
        for (int i = 0; i < J - 1; ++i) {
          const float li = z.beta[i], dn = d[i + 1] - shift, un = i < J - 2 ? z.beta[i + 1] : 0.f;
          float f, p;
          if (fabsf(di) >= fabsf(li)) {
            p = (di == 0.f) ? tiny : di;
            f = __fdividef(li, p);
            du[i * K] = ui;
            du2[i * K] = 0.f;
            di = dn - f * ui;
            ui = un;
          } else {
            f = __fdividef(di, li);
            p = li;
            du[i * K] = dn;
            du2[i * K] = un;
            di = ui - f * dn;
            ui = -f * un;
            bits |= 1u << i;
          }
          dl[i * K] = f;
          // (the reciprocal pivot: the solves multiply)
          dd[i * K] = __fdividef(1.f, fabsf(p) < tiny ? (p < 0.f ? -tiny : tiny) : p);
        }
        dd[(J - 1) * K] = __fdividef(1.f, fabsf(di) < tiny ? (di < 0.f ? -tiny : tiny) : di);
      }
      float a = y[0];
      for (int i = 0; i < J - 1; ++i) {
        const float b = y[(i + 1) * K], f = dl[i * K];
        if ((bits >> i) & 1u) {
          y[i * K] = b;
          a = a - f * b;
        } else {
          y[i * K] = a;
          a = b - f * a;
        }
      }
      float y1 = a * dd[(J - 1) * K], y2 = 0.f;
      y[(J - 1) * K] = y1;
      for (int i = J - 2; i >= 0; --i) {
        const float u2 = i < J - 2 ? du2[i * K] : 0.f;
        const float v = (y[i * K] - du[i * K] * y1 - u2 * y2) * dd[i * K];
        y[i * K] = v;
        y2 = y1;
        y1 = v;
      }
    }
    pbits[w] = bits;
    __syncwarp();
    if (q < k) {
      // unit length (a lane per entry)
      const float v = lane < J ? y[lane * K] : 0.f;
      const float ss = warp_sum(v * v);
      if (lane < J) y[lane * K] = v * (ss > 0.f ? rsqrtf(ss) : 0.f);
    }
    }
    __syncthreads();
    if (grouped) {
      cluster_mgs<NT>(z.ty, K, J, k, clus, s.red);
      __syncthreads();
    }
  }
  return k;
}

// the sum over a warp's lanes of eight values (one per row of the warp): row
// 4 bit4 + 2 bit3 + bit2 of the lane, in all four lanes that agree on them
__device__ __forceinline__ float sum8(float p[8], int lane) {
#pragma unroll
  for (int o = 16, h = 4; o >= 4; o >>= 1, h >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float keep = up ? p[i + h] : p[i], give = up ? p[i] : p[i + h];
      p[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  p[0] += __shfl_xor_sync(0xffffffffu, p[0], 2);
  p[0] += __shfl_xor_sync(0xffffffffu, p[0], 1);
  return p[0];
}

// The Gram matrix of a narrow block (order n <= NMAX) in the registers of a
// CTA of NMAX / 16 warps: warp w holds rows 16 w .., lane l the columns l,
// l + 32.  A product is 16 NMAX / 32 multiply-adds per thread and a
// 16-shuffle multi-reduction; from shared memory with a thread or two per row
// it took ten times as long (2.8k -> 0.25k cycles at n = 64).
template <int NT, int NMAX>
struct SmallGram {
  static constexpr int RW = 16, NC = NMAX >= 32 ? NMAX / 32 : 1, NW = NT / 32;
  static_assert(NW * RW == NMAX, "16 rows per warp");
  float A[RW][NC];
  int n, lane, warp;
  template <class S>
  __device__ __forceinline__ void load(S G, int n_) {
    n = n_;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int r = RW * warp + i, c = lane + 32 * k;
        const int hi = max(r, c), lo = min(r, c);
        A[i][k] = hi < n ? G.at(hi, lo) : 0.f;
      }
  }
  // the sums over the lanes of the warp's 16 row values: row 8 bit4 + 4 bit3
  // + 2 bit2 + bit1 of the lane
  __device__ __forceinline__ float sum16(float p[RW]) const {
#pragma unroll
    for (int o = 16, h = 8; o >= 2; o >>= 1, h >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < h; ++i) {
        const float keep = up ? p[i + h] : p[i], give = up ? p[i] : p[i + h];
        p[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    return p[0] + __shfl_xor_sync(0xffffffffu, p[0], 1);
  }
  __device__ __forceinline__ int sum_row() const {
    return RW * warp + ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 +
           ((lane >> 1) & 1);
  }
  // y (n shared entries) = A x, x in registers (entry lane + 32 k, zero from n
  // on); the caller's barrier publishes y
  __device__ __forceinline__ void mul(const float x[NC], float* y) const {
    float p[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) p[i] = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
      for (int i = 0; i < RW; ++i) p[i] = fmaf(A[i][k], x[k], p[i]);
    const float t = sum16(p);
    const int r = sum_row();
    if ((lane & 1) == 0 && r < n) y[r] = t;
  }
  // entries of a shared n-vector for mul
  __device__ __forceinline__ void vec(const float* x, float v[NC]) const {
#pragma unroll
    for (int k = 0; k < NC; ++k) v[k] = lane + 32 * k < n ? x[lane + 32 * k] : 0.f;
  }
  // Gershgorin bound max_i sum_j |A_ij| of the warp's rows (every lane)
  __device__ __forceinline__ float row_bound() const {
    float p[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      p[i] = 0.f;
#pragma unroll
      for (int k = 0; k < NC; ++k) p[i] += fabsf(A[i][k]);
    }
    return warp_max(sum16(p));
  }
  // dot product of two n-vectors, the same in every warp
  __device__ __forceinline__ float dot(const float* x, const float* y) const {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int c = lane + 32 * k;
      if (c < n) t = fmaf(x[c], y[c], t);
    }
    return warp_sum(t);
  }
};

// w <- (I - Q Q^T) w twice over nq basis vectors (vector i at Q + i ldq), all
// in the calling warp: w in registers, eight basis vectors at a time with one
// multi-reduction.  Every warp of the CTA does the same, so no barrier is
// needed.  Adds the coefficients of vector nq - 1 to *alpha; returns |w|^2.
template <int NT, int NMAX>
__device__ __forceinline__ float lz_project(const SmallGram<NT, NMAX>& g,
                                            float w[SmallGram<NT, NMAX>::NC], const float* Q,
                                            int ldq, int nq, float* alpha) {
  constexpr int NC = SmallGram<NT, NMAX>::NC;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
    for (int i0 = 0; i0 < nq; i0 += 8) {
      float q[8][NC], p[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        p[u] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          q[u][k] = (i0 + u < nq && g.lane + 32 * k < g.n) ? Q[(i0 + u) * ldq + g.lane + 32 * k] : 0.f;
          p[u] = fmaf(q[u][k], w[k], p[u]);
        }
      }
      const float t = sum8(p, g.lane);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float h = __shfl_sync(0xffffffffu, t, u << 2);
        if (i0 + u == nq - 1) *alpha += h;
#pragma unroll
        for (int k = 0; k < NC; ++k) w[k] = fmaf(-h, q[u][k], w[k]);
      }
    }
  }
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < NC; ++k) t = fmaf(w[k], w[k], t);
  return warp_sum(t);
}

// Steps 1-3 of the Lanczos path of a narrow block and the set-up of step 4.
//  g   G in registers.
//  Q   shared scratch of jmax vectors, ldq apart (every warp writes the same
//      values and each lane reads only its own entries of it).
//  U   receives the kept Ritz vectors (lz_maxk(NMAX) * n shared floats,
//      column-major).
//  gbound: an upper bound of ||G||_2.
//  panel: lz_cert_floats(NMAX, NT) floats of 16-byte aligned shared scratch
//      for the certificate (apart from Q and U).
// On success returns k >= 0 (pairs above thr) with s.lam[0..k), the vectors
// in U's columns 0..k-1 (U holds ku >= k kept pairs, *ku_out = ku), U and
// What = W - U sym(B) / 2 staged column-major at panel and panel + K n8 (n8 =
// roundup(n, 8), K = lz_maxk(NMAX)) and the certificate shift in *c0_out:
// the pairs are certified iff
//   regchol_pd<NT, NMAX>(G, n, *c0_out, true, panel, panel + K n8, ku,
//                        panel + 2 K n8, red)
// holds.  Returns -1 when the caller must fall back.  *J_out: steps run.
template <int NT, int NMAX>
__device__ int lanczos_candidates(const SmallGram<NT, NMAX>& g, float thr, float gbound, float* Q,
                                  int ldq, int jmax, float* U, uint32_t seed, EigScratch& s,
                                  LzScratch& z, float* panel, int* ku_out, float* c0_out, int slot,
                                  int* J_out) {
  constexpr int NW = NT / 32, K = lz_maxk(NMAX);
  const int tid = threadIdx.x, lane = g.lane, warp = g.warp, n = g.n;
  PHASE_INIT();
  const float thr_keep = 0.95f * thr;  // pairs kept in U (deflated)
  // the vectors of a step live in every warp's registers (entry lane + 32 k);
  // only G q passes through shared memory, two buffers in turn
  constexpr int NC = SmallGram<NT, NMAX>::NC;
  float q[NC], w[NC];
  auto store_q = [&](int j) {
#pragma unroll
    for (int k = 0; k < NC; ++k)
      if (lane + 32 * k < n) Q[j * ldq + lane + 32 * k] = q[k];
  };
  {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      q[k] = lane + 32 * k < n ? 1e-3f * lz_hash(seed, lane + 32 * k) : 0.f;
      t = fmaf(q[k], q[k], t);
    }
    const float inrm = 1.f / sqrtf(warp_sum(t));
#pragma unroll
    for (int k = 0; k < NC; ++k) q[k] *= inrm;
    store_q(0);
  }
  const int jmin = min(jmax, 8);
  int J = 0, k = -1;
  uint32_t restart = 1;
  PHASE(slot, 6);
  for (int j = 0; j < jmax; ++j) {
    // w = G q_j, then w <- w - Q_j Q_j^T w twice: alpha_j is the q_j
    // coefficient of the two passes, beta_j = ||w|| (full reorthogonalisation)
    float* y = (j & 1) ? z.w : z.x;
    g.mul(q, y);
    __syncthreads();
    g.vec(y, w);
    PHASE(slot, 7);
    float al = 0.f;
    float b = sqrtf(lz_project(g, w, Q, ldq, j + 1, &al));
    PHASE(slot, 9);
    if (tid == 0) {
      z.alpha[j] = al;
      z.beta[j] = b;
    }
    J = j + 1;
    if (J == n) break;  // Q spans everything: T_J is similar to G
    if (J < jmax) {
      if (!(b > kLzBreak * gbound)) {
        // breakdown: an invariant subspace was found; continue from a random
        // direction orthogonal to it
#pragma unroll
        for (int c = 0; c < NC; ++c)
          w[c] = lane + 32 * c < n ? lz_hash(seed + 7919u * restart, lane + 32 * c) : 0.f;
        ++restart;
        const float bn = sqrtf(lz_project(g, w, Q, ldq, j + 1, &al));
        if (!(bn > 0.f)) break;
        if (tid == 0) z.beta[j] = 0.f;
        b = bn;
      }
      const float ib = 1.f / b;
#pragma unroll
      for (int c = 0; c < NC; ++c) q[c] = w[c] * ib;
      store_q(j + 1);
    }
    PHASE(slot, 10);
    if (J >= jmin && ((J - jmin) % 4 == 0 || J == jmax)) {
      // converged when every kept Ritz pair has |beta_J * y_{J-1}| small
      k = lz_ritz<NT, K>(J, thr_keep, z, s);
      PHASE(slot, 11);
      if (k > K) {
        *J_out = J;
        return -1;
      }
      bool conv = true;
      const float bJ = z.beta[J - 1];
      for (int q = 0; q < k; ++q)
        if (fabsf(bJ * z.ty[(J - 1) * K + q]) > 1e-5f * fmaxf(s.lam[0], thr)) conv = false;
      if (conv) break;
      k = -1;
    }
  }
  *J_out = J;
  if (k < 0) {
    k = lz_ritz<NT, K>(J, thr_keep, z, s);
    // pairs that jmax < n steps did not settle are not taken: the certificate
    // below admits any residual that leaves lambda_max(P G P) below tau^2 -
    // 2 rho, up to some per cent of tau^2
    if (k > K || (J == jmax && J < n && k > 0)) return -1;
  }
  const int ku = k, n8 = (n + 7) & ~7;
  float* U8 = panel;
  float* W8 = panel + K * n8;
  // U = Q_J Y; W = G U
  for (int e = tid; e < ku * n8; e += NT) {
    const int q = e / n8, r = e - q * n8;
    float v = 0.f;
    if (r < n) {
      for (int j = 0; j < J; ++j) v = fmaf(Q[j * ldq + r], z.ty[j * K + q], v);
      U[q * n + r] = v;
    }
    U8[e] = v;
    W8[e] = 0.f;
  }
  __syncthreads();
  PHASE(slot, 12);
  for (int p = 0; p < ku; ++p) {
    g.vec(U8 + p * n8, q);
    g.mul(q, W8 + p * n8);
  }
  __syncthreads();
  // B = U^T W, residuals |W_q - B_qq U_q|^2: a warp per row of B
  for (int p = warp; p < ku; p += NW) {
    float bpp = 0.f;
    for (int q = 0; q < ku; ++q) {
      const float t = g.dot(U8 + p * n8, W8 + q * n8);
      if (q == p) bpp = t;
      if (lane == 0) z.Bm[p * K + q] = t;
    }
    float rr = 0.f;
    for (int r = lane; r < n; r += 32) {
      const float d = W8[p * n8 + r] - bpp * U8[p * n8 + r];
      rr = fmaf(d, d, rr);
    }
    rr = warp_sum(rr);
    if (lane == 0) z.h[p] = rr;
  }
  __syncthreads();
  PHASE(slot, 13);
  // kept pairs: Rayleigh quotients, count above thr; pairs above thr first
  float rho = 0.f;
  int kk = 0;
  for (int q = 0; q < ku; ++q) {
    rho += z.h[q];
    const float th = z.Bm[q * K + q];
    kk += th > thr;
    if (q > 0 && th > thr && !(z.Bm[(q - 1) * K + (q - 1)] > thr)) return -1;
  }
  rho = sqrtf(rho);
  const float c0 = thr - 2.f * rho - 8.f * (float)(ku + 1) * FLT_EPSILON * gbound;
  if (!(c0 > 0.f)) return -1;
  if (tid < ku) s.lam[tid] = z.Bm[tid * K + tid];
  // What = W - U sym(B) / 2 in place: a thread owns a row
  for (int r = tid; r < n; r += NT) {
    float u[K];
#pragma unroll
    for (int p = 0; p < K; ++p) u[p] = p < ku ? U8[p * n8 + r] : 0.f;
    for (int q = 0; q < ku; ++q) {
      float w = W8[q * n8 + r];
#pragma unroll
      for (int p = 0; p < K; ++p)
        if (p < ku) w = fmaf(-0.25f * (z.Bm[p * K + q] + z.Bm[q * K + p]), u[p], w);
      W8[q * n8 + r] = w;
    }
  }
  __syncthreads();
  PHASE(slot, 11);
  *ku_out = ku;
  *c0_out = c0;
  return kk;
}

}  // namespace msllr

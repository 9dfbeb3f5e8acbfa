// Subspace iteration and Rayleigh-Ritz of blocks wider than 256.  Up to 2048
// wide one thread-block cluster per block does every step of every round in
// one launch; above, where 16 SMs would be too few for G V, a step is a
// grid-wide G V launch and a cluster launch for the rest.
//
// Per step X = G V + mu V, then V = orth(X) by shifted CholQR and plain CholQR
// passes (Fukaya, Kannan, Nakatsukasa, Yamamoto, Yanagisawa, SIAM J. Sci.
// Comput. 2020); mu = 1e-4 ||G||_F (a shift of G) keeps X of full rank when G
// is numerically of rank below kHP.  Per round a Rayleigh-Ritz test.  What
// bounds a block of this size is latency,
// not arithmetic: a step's product is n^2 kHP multiply-adds (0.4 us of the
// whole GPU at n = 1024), its orthonormalisation three dependent 32 x 32
// factorisations.  As launches a step took 130 us at n = 1024 (five launches
// whose CTAs each summed all partials and factored with one thread per
// column in shared memory); here the CTAs of the cluster own np / CL rows
// each, the partial 32 x 32 products are summed over distributed shared
// memory behind hardware cluster barriers, every CTA factors the same sum in
// one warp's registers, and the rows never leave shared memory inside a
// step.
//
//   G V     8 x 8 register tiles over 64-column chunks of G and V (cp.async,
//           three stages), the chunk's columns split over the warps; V comes
//           from L2
//   X^T X   4 x 4 register tiles, rows split four ways
//   R       Cholesky in one warp: lane i holds row i
//   X R^-1  a warp per four rows: lane t holds column t
//   T = V^T G V: parallel two-sided Jacobi on 32 x 32 (Golub & Van Loan,
//           Sec. 8.5): 16 disjoint pairs a round, a thread per 2 x 2 block
//
// All arrays have np = nn rounded up to 64 rows; the padding is zero.
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "huge.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace msllr {

namespace {

constexpr int kSNT = 256;      // threads per CTA
constexpr int kSNW = kSNT / 32;
constexpr int kSKC = 64;       // columns of G per stage
constexpr int kSStages = 3;
constexpr int kSLdG = kSKC + 4;  // row stride of a G chunk (floats): 8 rows on distinct banks
constexpr int kSLd = 36;       // row stride of X and W
constexpr int kSM = kHP * 33;
static_assert(kSMaxRows == 2 * 64, "two 64-row halves of 8 x 8 register tiles");

// floats of one pipeline stage; between products the stages' space holds the
// split sums of the products
__host__ __device__ constexpr int sub_stage_floats(int rp) { return rp * kSLdG + kSKC * kHP; }
__host__ __device__ constexpr int sub_pipe_floats(int rp) {
  // (above kSMaxRows rows G V comes from elsewhere: the products' sums only)
  return rp > kSMaxRows ? kSNT / 64 * kHP * kHP
         : kSStages * sub_stage_floats(rp) > kSNW / 2 * 64 * kHP ? kSStages * sub_stage_floats(rp)
                                                                 : kSNW / 2 * 64 * kHP;
}
size_t sub_smem_bytes(int rp) {
  return sizeof(float) *
         (size_t)(sub_pipe_floats(rp) + 2 * rp * kSLd + kHP * kHP + 3 * kSM + kHK * kHK);
}
// subspace_more_kernel: the phases' arrays, or G V of 64 rows and its result
size_t sub_more_bytes(int rp) {
  const size_t gv = sizeof(float) * (size_t)(sub_pipe_floats(64) + 64 * kSLd);
  return gv > sub_smem_bytes(rp) ? gv : sub_smem_bytes(rp);
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Ws = rows [r0, r0 + rp) of G V.  A warp covers 64 rows x 32 columns with
// 8 x 8 register tiles (lane: rows lr + 8 i, columns 8 lc ..), which balances
// its shared-memory reads (16 x 128 bits per 4 columns of G) with its 256
// multiply-adds; the warps of a row half split each chunk's columns, and
// their sums are added pairwise in a fixed order.  MANY: compact code for
// launches that fill the chip (its instruction fetch limits the unrolled form
// there: 16 blocks 512 wide 6 % slower; a lone 1024-wide block is 3 % faster
// with it).
template <bool MANY>
__device__ void sub_gv(const float* __restrict__ Gr, const float* V, int np, int rp, float* pipe,
                       float* Ws) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int halves = rp > 64 ? 2 : 1, ns = kSNW / halves;
  const int half = warp / ns, split = warp - half * ns;
  const int lr = lane >> 2, lc = lane & 3;
  const int row0 = 64 * half, rows = min(64, rp - row0);
  const int sf = sub_stage_floats(rp), nch = np / kSKC;
  auto load = [&](int c) {
    float* st = pipe + (c % kSStages) * sf;
    const float* g = Gr + c * kSKC;
    for (int e = tid; e < rp * (kSKC / 4); e += kSNT) {
      const int r = e / (kSKC / 4), q = e % (kSKC / 4);
      cp16(st + r * kSLdG + 4 * q, g + (size_t)r * np + 4 * q);
    }
#pragma unroll
    for (int e = 4 * tid; e < kSKC * kHP; e += 4 * kSNT)
      cp16(st + rp * kSLdG + e, V + (size_t)c * kSKC * kHP + e);
  };
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  for (int c = 0; c < kSStages - 1; ++c) {
    if (c < nch) load(c);
    cp_commit();
  }
  for (int c = 0; c < nch; ++c) {
    cp_wait<kSStages - 2>();
    __syncthreads();
    if (c + kSStages - 1 < nch) load(c + kSStages - 1);
    cp_commit();
    const float* Gs = pipe + (c % kSStages) * sf;
    const float* Vs = Gs + rp * kSLdG;
    for (int k4 = split; k4 < kSKC / 4; k4 += ns) {
      const float* gp = Gs + (row0 + lr) * kSLdG + 4 * k4;
#pragma unroll(MANY ? 1 : 2)
      for (int k2 = 0; k2 < 4; k2 += 2) {
        float2 g[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // (rows past the end read other shared memory; their sums are not stored)
          g[i] = *reinterpret_cast<const float2*>(gp + 8 * i * kSLdG + k2);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float* vr = Vs + (4 * k4 + k2 + k) * kHP + 8 * lc;
          const float4 v0 = *reinterpret_cast<const float4*>(vr);
          const float4 v1 = *reinterpret_cast<const float4*>(vr + 4);
          const float vv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float gk = k == 0 ? g[i].x : g[i].y;
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(gk, vv[j], acc[i][j]);
          }
        }
      }
    }
  }
  cp_wait<0>();
  // pairwise sums of the splits through shared memory
  for (int o = ns >> 1; o > 0; o >>= 1) {
    __syncthreads();
    float* slot = pipe + (size_t)(half * (ns >> 1) + (split & (o - 1))) * 64 * kHP + 4 * lane;
    if (split >= o && split < 2 * o) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        *reinterpret_cast<float4*>(slot + i * 256) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(slot + i * 256 + 128) =
            make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
      }
    }
    __syncthreads();
    if (split < o) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(slot + i * 256);
        const float4 y = *reinterpret_cast<const float4*>(slot + i * 256 + 128);
        acc[i][0] += x.x;
        acc[i][1] += x.y;
        acc[i][2] += x.z;
        acc[i][3] += x.w;
        acc[i][4] += y.x;
        acc[i][5] += y.y;
        acc[i][6] += y.z;
        acc[i][7] += y.w;
      }
    }
  }
  if (split == 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (lr + 8 * i < rows) {
        float* d = Ws + (row0 + lr + 8 * i) * kSLd + 8 * lc;
        *reinterpret_cast<float4*>(d) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(d + 4) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
      }
  }
  __syncthreads();
}

// P (32 x 32, row-major) = A^T B over rp rows (row stride kSLd); `tmp`: 4 x
// 1024 floats.
__device__ void sub_atb(const float* A, const float* B, int rp, float* tmp, float* P) {
  const int tid = threadIdx.x, q = tid >> 6, t = tid & 63;
  const int a0 = 4 * (t >> 3), b0 = 4 * (t & 7);
  float acc[4][4] = {};
  for (int r = q; r < rp; r += kSNT / 64) {
    const float4 x = *reinterpret_cast<const float4*>(A + r * kSLd + a0);
    const float4 y = *reinterpret_cast<const float4*>(B + r * kSLd + b0);
    const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xv[i], yv[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4*>(tmp + q * (kHP * kHP) + (a0 + i) * kHP + b0) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  __syncthreads();
#pragma unroll
  for (int e = tid; e < kHP * kHP; e += kSNT) {
    float v = tmp[e];
#pragma unroll
    for (int s = 1; s < kSNT / 64; ++s) v += tmp[s * kHP * kHP + e];
    P[e] = v;
  }
}

// Sm (32 x 33, in every CTA) = the sum of P over the cluster's CTAs: each CTA
// sums one slice (a lane per rank, shuffle tree) and stores it to all.
// Contains two cluster barriers.
__device__ void sub_cluster_sum(const cg::cluster_group& cl, float* P, float* Sm) {
  cl.sync();
  const int tid = threadIdx.x, n = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  if (tid < kHP * kHP / 4) {
    // n = 8 or 16 lanes share a slice entry of four floats
    const int r = tid & (n - 1), e = 4 * (rank * (kHP * kHP / 4 / n) + tid / n);
    float4 v = *reinterpret_cast<const float4*>(cl.map_shared_rank(P, r) + e);
    for (int o = 1; o < n; o <<= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      v.z += __shfl_xor_sync(0xffffffffu, v.z, o);
      v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
    }
    float* d = cl.map_shared_rank(Sm, r) + (e >> 5) * 33 + (e & 31);
    d[0] = v.x;
    d[1] = v.y;
    d[2] = v.z;
    d[3] = v.w;
  }
  cl.sync();
}

// 1 / sqrt(x) by the approximation and one Newton step
__device__ __forceinline__ float sub_rsqrt(float x) {
  const float r = rsqrtf(x);
  return r * fmaf(-0.5f * x * r, r, 1.5f);
}

// Warp 0: Sm + rel_shift trace(Sm) I = R^T R (R upper, row j at Rm + 33 j, zero below the
// diagonal; rinv[j] = 1 / R_jj).  Returns false in every thread on a
// non-positive or non-finite pivot.
__device__ bool sub_chol(const float* Sm, float rel_shift, float* Rm, float* rinv) {
  const int tid = threadIdx.x, lane = tid & 31;
  bool ok = true;
  if (tid < 32) {
    float a[kHP], myinv = 0.f;
    const float shift = rel_shift > 0.f ? rel_shift * warp_sum(Sm[lane * 33 + lane]) : 0.f;
#pragma unroll
    for (int j = 0; j < kHP; ++j) a[j] = Sm[lane * 33 + j] + (j == lane ? shift : 0.f);
#pragma unroll
    for (int j = 0; j < kHP; ++j) {
      const float d = __shfl_sync(0xffffffffu, a[j], j);
      ok = ok && d > 0.f && d <= FLT_MAX;
      const float inv = sub_rsqrt(d);
      if (lane == j) myinv = inv;
      a[j] *= inv;  // lane j: d / sqrt(d) = R_jj
#pragma unroll
      for (int t = j + 1; t < kHP; ++t)
        a[t] = fmaf(-a[j], __shfl_sync(0xffffffffu, a[j], t), a[t]);
    }
#pragma unroll
    for (int j = 0; j < kHP; ++j) Rm[j * 33 + lane] = lane >= j ? a[j] : 0.f;
    rinv[lane] = myinv;
  }
  return __syncthreads_and(ok);
}

// X <- X R^{-1}, rp rows: a warp per four rows, lane t holds column t.
__device__ void sub_solve(float* X, int rp, const float* Rm, const float* rinv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r0 = 4 * warp; r0 < rp; r0 += 4 * kSNW) {
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = X[(r0 + i) * kSLd + lane];
#pragma unroll 8
    for (int j = 0; j < kHP; ++j) {
      const float rj = Rm[j * 33 + lane], ij = rinv[j];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float x = __shfl_sync(0xffffffffu, v[i], j) * ij;
        v[i] = lane == j ? x : fmaf(-x, rj, v[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) X[(r0 + i) * kSLd + lane] = v[i];
  }
  __syncthreads();
}

// Eigen-decomposition of the symmetric A (32 x 33, entries scaled to about
// 1): on return the eigenvalues stand on A's diagonal and the eigenvectors in
// the columns of Q.  Parallel two-sided Jacobi, 16 disjoint pairs a round:
// half of warp 0 forms the rotations, then thread (bi, bj) applies both
// rotations of its 2 x 2 block and rotates its part of Q.
// Converged when every off-diagonal entry is below 3e-7 of the geometric
// mean of its diagonal entries (or of `floor_`), a few ulp.
__device__ void sub_jacobi(float* A, float* Q, float floor_, float2* cs) {
  const int tid = threadIdx.x;
  for (int e = tid; e < kHP * kHP; e += kSNT) Q[(e >> 5) * 33 + (e & 31)] = (e >> 5) == (e & 31);
  __syncthreads();
  const int bi = (tid >> 4) & 15, bj = tid & 15;
  // pair i of round rd (round robin): column 31 stays, the others turn
  auto pair = [](int rd, int i, int& p, int& q) {
    p = rd + i;
    if (p >= 31) p -= 31;
    q = i == 0 ? 31 : rd - i;
    if (q < 0) q += 31;
  };
  for (int sweep = 0; sweep < 12; ++sweep) {
    bool any = false;
    for (int rd = 0; rd < 31; ++rd) {
      int pj, qj;
      pair(rd, bj, pj, qj);
      if (tid < 16) {
        // the rotation that zeroes a_pq: cos 2 phi = |D| / q, sin 2 phi =
        // 2 a_pq sign(D) / q, q = sqrt(D^2 + 4 a_pq^2), |phi| <= pi / 4
        const float app = A[pj * 33 + pj], aqq = A[qj * 33 + qj], apq = A[pj * 33 + qj];
        float c = 1.f, s = 0.f;
        if (apq * apq > 9e-14f * fmaxf(fabsf(app * aqq), floor_ * floor_)) {
          const float d = aqq - app, g = 2.f * apq;
          const float r = sub_rsqrt(fmaf(d, d, g * g));
          const float c2 = fmaf(0.5f * fabsf(d), r, 0.5f);
          const float rc = sub_rsqrt(c2);
          c = c2 * rc;
          s = copysignf(0.5f, d) * g * r * rc;
          any = true;
        }
        cs[tid] = make_float2(c, s);
      }
      __syncthreads();
      const float2 rj = cs[bj];
      const float cj = rj.x, sj = rj.y;
      {
        int pi, qi;
        pair(rd, bi, pi, qi);
        const float2 ri = cs[bi];
        const float ci = ri.x, si = ri.y;
        const float b00 = A[pi * 33 + pj], b01 = A[pi * 33 + qj];
        const float b10 = A[qi * 33 + pj], b11 = A[qi * 33 + qj];
        const float x0 = ci * b00 - si * b10, x1 = ci * b01 - si * b11;
        const float y0 = si * b00 + ci * b10, y1 = si * b01 + ci * b11;
        const bool own = bi == bj && si != 0.f;
        A[pi * 33 + pj] = cj * x0 - sj * x1;
        A[pi * 33 + qj] = own ? 0.f : sj * x0 + cj * x1;
        A[qi * 33 + pj] = own ? 0.f : cj * y0 - sj * y1;
        A[qi * 33 + qj] = sj * y0 + cj * y1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float* row = Q + (bi + 16 * h) * 33;
          const float vp = row[pj], vq = row[qj];
          row[pj] = cj * vp - sj * vq;
          row[qj] = sj * vp + cj * vq;
        }
      }
      __syncthreads();
    }
    if (!__syncthreads_or(any)) break;
  }
}

// The shared memory of a CTA that owns rp rows.
struct SubSmem {
  float *pipe, *Xs, *Ws, *P, *Sm, *Rm, *Qm, *Bm;
  __device__ SubSmem(float* sm, int rp) {
    pipe = sm;
    Xs = pipe + sub_pipe_floats(rp);
    Ws = Xs + rp * kSLd;
    P = Ws + rp * kSLd;  // this CTA's partial sum
    Sm = P + kHP * kHP;
    Rm = Sm + kSM;
    Qm = Rm + kSM;
    Bm = Qm + kSM;  // kHK x kHK
  }
};

// Xs = orth(Ws + mu Xs) by `passes` CholQR passes, the first one shifted.
// False (in every CTA) when a factorisation breaks down: Xs is then a fresh
// start basis.
__device__ bool sub_orth(const cg::cluster_group& cl, const SubSmem& m, int rp, int r0, int nn, int b,
                         float mu, int passes) {
  const int tid = threadIdx.x;
  for (int e = tid; e < rp * kHP; e += kSNT) {
    const int o = (e >> 5) * kSLd + (e & 31);
    m.Xs[o] = fmaf(mu, m.Xs[o], m.Ws[o]);
  }
  __syncthreads();
  __shared__ float rinv[kHP];
  for (int pass = 1; pass <= passes; ++pass) {
    sub_atb(m.Xs, m.Xs, rp, m.pipe, m.P);
    sub_cluster_sum(cl, m.P, m.Sm);
    const float shift =
        pass == 1 ? 11.f * (float)((double)nn * kHP + kHP * (kHP + 1)) * FLT_EPSILON : 0.f;
    // the same sum in every CTA: all of them fail or none
    if (!sub_chol(m.Sm, shift, m.Rm, rinv)) {
      for (int e = tid; e < rp * kHP; e += kSNT) {
        const int r = r0 + (e >> 5), c = e & 31;
        m.Xs[(e >> 5) * kSLd + c] =
            r < nn ? huge_hash((uint32_t)r + 977u * b, (uint32_t)c + 0xB0Bu) : 0.f;
      }
      __syncthreads();
      return false;
    }
    sub_solve(m.Xs, rp, m.Rm, rinv);
  }
  return true;
}

// Rounds of a block: `first`, 4 and 8 steps for every block, then up to
// kSMoreRounds of 8 for blocks whose pairs have not converged but will at the
// rate seen so far.  128 further steps bring the residual of a pair down by a
// factor of 1000 where the eigenvalue below the basis is 0.95 of the pair's;
// what is slower is counted as uncertified.
constexpr int kSRounds = 3;
constexpr int kSMoreRounds = 16;
static_assert((kSMoreRounds & (kSMoreRounds - 1)) == 0, "a power of two (sub_ritz)");

// Rayleigh-Ritz with V in Xs and G V in Ws: T = V^T G V, its eigenpairs above
// thr (at most kHK, largest first), the Ritz vectors U = V Q, G U, B = U^T G
// U, the residuals and What = G U - U sym(B) / 2 (into GU).  Overwrites Xs.
// Returns true (in every CTA) when the pairs have converged.  `t`: the block's
// previous test on entry, this one on return.
struct SubTest {
  float worst;  // largest residual relative to its bar (0: no test yet)
  int ku;       // pairs
  bool stop;    // no further rounds: they would not bring it to convergence
};
__device__ bool sub_ritz(const cg::cluster_group& cl, const SubSmem& m, int rp, float* Ub, float* GUb,
                         float thr, HugeBlock& h, SubTest& t) {
  const int tid = threadIdx.x, CL = (int)cl.num_blocks();
  __shared__ float rq[2 * kHK], red[kSNW][2 * kHK];
  __shared__ float2 cs[16];
  __shared__ int sel[kHK], nabove;
  __shared__ float qn[kHP];
  float *Xs = m.Xs, *Ws = m.Ws, *P = m.P, *Sm = m.Sm, *Rm = m.Rm, *Qm = m.Qm, *Bm = m.Bm;
  const float gF = h.gF;
  sub_atb(Xs, Ws, rp, m.pipe, P);
  sub_cluster_sum(cl, P, Sm);
  // scaled by its trace (a sum of Rayleigh quotients of a Gram matrix), so
  // that the rotations' squares stay in range
  const float tr = warp_sum(Sm[(tid & 31) * 33 + (tid & 31)]);
  const float isc = tr > 0.f ? 1.f / tr : 1.f;
  for (int e = tid; e < kHP * kHP; e += kSNT) {
    const int i = e >> 5, j = e & 31;
    Rm[i * 33 + j] = 0.5f * (Sm[i * 33 + j] + Sm[j * 33 + i]) * isc;
  }
  __syncthreads();
  sub_jacobi(Rm, Qm, 1e-2f * thr * isc, cs);
  // the pairs above tau^2, largest first, at most kHK
  if (tid < 32) {
    const float th = Rm[tid * 33 + tid] * (tr > 0.f ? tr : 1.f);
    int rk = 0;
    for (int j = 0; j < kHP; ++j) {
      const float o = __shfl_sync(0xffffffffu, th, j);
      rk += o > th || (o == th && j < tid);
    }
    const unsigned above = __ballot_sync(0xffffffffu, th > thr);
    if (th > thr && rk < kHK) sel[rk] = tid;
    // some two hundred rotations leave the columns of Q 1e-6 off unit length
    float n2 = 0.f;
#pragma unroll 8
    for (int a = 0; a < kHP; ++a) n2 = fmaf(Qm[a * 33 + tid], Qm[a * 33 + tid], n2);
    qn[tid] = fmaf(-0.5f, n2, 1.5f);
    if (tid == 0) nabove = __popc(above);
  }
  __syncthreads();
  const int ku = min(nabove, kHK);
  // U = V Q and G U = W Q, over V's rows in Xs: entries 0 .. 15 U, 16 .. 31 G
  // U (the 16 threads of a row are in one warp)
  {
    const int q = tid & 15;
    const int cq = q < ku ? sel[q] : 0;
    const float cn = qn[cq];
    for (int r = tid >> 4; r < rp; r += kSNT / 16) {
      float u = 0.f, g = 0.f;
#pragma unroll
      for (int a = 0; a < kHP; a += 4) {
        const float4 x = *reinterpret_cast<const float4*>(Xs + r * kSLd + a);
        const float4 w = *reinterpret_cast<const float4*>(Ws + r * kSLd + a);
        const float xv[4] = {x.x, x.y, x.z, x.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float qv = Qm[(a + i) * 33 + cq];
          u = fmaf(xv[i], qv, u);
          g = fmaf(wv[i], qv, g);
        }
      }
      __syncwarp();
      Xs[r * kSLd + q] = q < ku ? u * cn : 0.f;
      Xs[r * kSLd + kHK + q] = q < ku ? g * cn : 0.f;
    }
  }
  __syncthreads();
  // B = U^T G U: partial sums in rank order
  if (tid < kHK * kHK) {
    const int p = tid >> 4, q = tid & 15;
    float t = 0.f;
#pragma unroll 4
    for (int r = 0; r < rp; ++r) t = fmaf(Xs[r * kSLd + p], Xs[r * kSLd + kHK + q], t);
    P[tid] = t;
  }
  cl.sync();
  if (tid < kHK * kHK) {
    float s = 0.f;
#pragma unroll 8
    for (int c = 0; c < CL; ++c) s += cl.map_shared_rank(P, c)[tid];
    Bm[tid] = s;
  }
  __syncthreads();
  // residuals |G u_q - theta_q u_q|^2 and What = G U - U sym(B) / 2, |What_q|^2
  {
    const int q = tid & 15, rr = tid >> 4;
    float ra = 0.f, wa = 0.f;
    for (int r = rr; r < rp; r += kSNT / 16) {
      const float u = Xs[r * kSLd + q], g = Xs[r * kSLd + kHK + q];
      float wh = g;
      for (int p = 0; p < ku; ++p)
        wh = fmaf(-0.25f * (Bm[p * kHK + q] + Bm[q * kHK + p]), Xs[r * kSLd + p], wh);
      if (q < ku) {
        const float res = g - Bm[q * kHK + q] * u;
        ra = fmaf(res, res, ra);
        wa = fmaf(wh, wh, wa);
      }
      Ub[(size_t)r * kHK + q] = u;
      GUb[(size_t)r * kHK + q] = q < ku ? wh : 0.f;
    }
    ra += __shfl_xor_sync(0xffffffffu, ra, 16);
    wa += __shfl_xor_sync(0xffffffffu, wa, 16);
    if ((tid & 31) < 16) {
      red[tid >> 5][q] = ra;
      red[tid >> 5][kHK + q] = wa;
    }
  }
  __syncthreads();
  // (the B partials in P's first 256 entries may still be read)
  float* P2 = P + kHK * kHK;
  if (tid < 2 * kHK) {
    float t = 0.f;
    for (int w = 0; w < kSNW; ++w) t += red[w][tid];
    P2[tid] = t;
  }
  cl.sync();
  if (tid < 2 * kHK) {
    float t = 0.f;
#pragma unroll 8
    for (int c = 0; c < CL; ++c) t += cl.map_shared_rank(P2, c)[tid];
    rq[tid] = t;
  }
  __syncthreads();
  // converged: every kept pair's residual is small against tau^2, or at the
  // rounding level of G V (set by the largest eigenvalue).  Pairs just above
  // tau converge slowly; they need this accuracy all the same, since the
  // consensus step carries their error into every scale.
  bool conv = true;
  float th0 = 0.f, wsum = 0.f;
  for (int q = 0; q < ku; ++q) {
    th0 = fmaxf(th0, Bm[q * kHK + q]);
    wsum += rq[kHK + q];
  }
  const float bar = fmaxf(3e-4f * thr, 4e-6f * th0);
  float worst = 0.f;
  for (int q = 0; q < ku; ++q) {
    const float res = sqrtf(rq[q]);
    if (res > bar) conv = false;
    worst = fmaxf(worst, res);
  }
  worst /= bar;
  // more than kHK Ritz values above tau^2 are never certified; and at the rate
  // of the last eight steps kSMoreRounds rounds of eight have to be enough (a
  // new pair has no rate yet)
  bool stop = nabove > kHK;
  if (ku == t.ku && t.worst > 0.f) {
    float rate = worst / t.worst;
#pragma unroll
    for (int i = 1; i < kSMoreRounds; i *= 2) rate *= rate;
    stop = stop || worst * rate > 1.f;
  }
  t = SubTest{worst, ku, stop};
  if (cl.block_rank() == 0 && tid == 0) {
    for (int q = 0; q < ku; ++q) h.theta[q] = Bm[q * kHK + q];
    h.c = cert_bound(thr, gF, ku, wsum);
    h.ku = ku;
    h.conv = conv;
    h.worst = worst;
    h.stop = stop;
  }
  cl.sync();  // the partial sums have been read
  return conv;
}

__device__ __forceinline__ bool sub_active(const HugeBlock& h) {
  return h.status == kHsIter && !h.conv && !h.orth_fail;
}

// The further rounds of a lone block; false when a factorisation broke down.
// Not inlined: as more turns of the loop below they cost every block 0.8 %
// (1024 wide: 383 us instead of 377 without a further round).
__device__ __noinline__ bool sub_further(const float* Gr, float* Vb, float* Ub, float* GUb, int nn, int np,
                                         float thr, int rp, int r0, int b, float* sm, HugeBlock& h,
                                         SubTest t) {
  const cg::cluster_group cl = cg::this_cluster();
  const SubSmem m(sm, rp);
  const int tid = threadIdx.x;
  const float mu = 1e-4f * h.gF;
  for (int rd = 0; rd < kSMoreRounds && !t.stop; ++rd) {
    for (int st = 0; st <= 8; ++st) {
      sub_gv<false>(Gr, Vb, np, rp, m.pipe, m.Ws);
      if (st < 8) {
        const bool ok = sub_orth(cl, m, rp, r0, nn, b, mu, st + 1 < 8 ? 2 : 3);
        for (int e = tid; e < rp * kHP; e += kSNT)
          Vb[(size_t)r0 * kHP + e] = m.Xs[(e >> 5) * kSLd + (e & 31)];
        cl.sync();  // the new V is visible to the cluster
        if (!ok) return false;
      } else {
        if (sub_ritz(cl, m, rp, Ub, GUb, thr, h, t)) return true;
        for (int e = tid; e < rp * kHP; e += kSNT)
          m.Xs[(e >> 5) * kSLd + (e & 31)] = Vb[(size_t)r0 * kHP + e];
        __syncthreads();
      }
    }
  }
  return true;
}

// Every step of every round for the blocks of a scale, a cluster per block.
template <bool MANY>
__global__ void __launch_bounds__(kSNT)
subspace_cluster_kernel(const float* __restrict__ G, float* V, float* __restrict__ U,
                        float* __restrict__ GU, int nn, int np, float thr, int first,
                        HugeBlock* __restrict__ hb) {
  extern __shared__ __align__(16) float sm[];
  const cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int b = blockIdx.x / CL, tid = threadIdx.x;
  const int rp = np / CL, r0 = rank * rp;
  HugeBlock& h = hb[b];
  if (h.status != kHsIter) return;  // the whole cluster leaves
  const SubSmem m(sm, rp);
  const float* Gr = G + (size_t)b * np * np + (size_t)r0 * np;
  float* Vb = V + (size_t)b * np * kHP;
  const size_t uo = ((size_t)b * np + r0) * kHK;
  const float mu = 1e-4f * h.gF;
  for (int e = tid; e < rp * kHP; e += kSNT) m.Xs[(e >> 5) * kSLd + (e & 31)] = Vb[(size_t)r0 * kHP + e];
  __syncthreads();
  const int rounds[kSRounds] = {first, 4, 8};
  bool failed = false, conv = false;
  SubTest t{0.f, -1, false};
  int more = kSMoreRounds;
  for (int rd = 0; rd < kSRounds && !conv && !failed; ++rd) {
    for (int st = 0; st < rounds[rd] && !failed; ++st) {
      sub_gv<MANY>(Gr, Vb, np, rp, m.pipe, m.Ws);
      // the third pass brings V to working precision for the Ritz problem;
      // between steps a well-conditioned basis of the same span is enough
      failed = !sub_orth(cl, m, rp, r0, nn, b, mu, st + 1 < rounds[rd] ? 2 : 3);
      for (int e = tid; e < rp * kHP; e += kSNT)
        Vb[(size_t)r0 * kHP + e] = m.Xs[(e >> 5) * kSLd + (e & 31)];
      cl.sync();  // the new V is visible to the cluster
    }
    if (failed) break;
    sub_gv<MANY>(Gr, Vb, np, rp, m.pipe, m.Ws);
    conv = sub_ritz(cl, m, rp, U + uo, GU + uo, thr, h, t);
    if (!conv) {
      for (int e = tid; e < rp * kHP; e += kSNT)
        m.Xs[(e >> 5) * kSLd + (e & 31)] = Vb[(size_t)r0 * kHP + e];
      __syncthreads();
      // the last round again: here the call below would take the kernel from
      // 128 registers to 221 (one CTA per SM, 16 blocks of 512: 279 -> 428 us)
      if (MANY && rd == kSRounds - 1 && !t.stop && more-- > 0) --rd;
    }
  }
  if constexpr (!MANY) {
    if (!conv && !failed && !t.stop)
      failed = !sub_further(Gr, Vb, U + uo, GU + uo, nn, np, thr, rp, r0, b, sm, h, t);
  }
  if (failed && rank == 0 && tid == 0) h.orth_fail = 1;
  cl.sync();  // no CTA leaves while others read its shared memory
}

// Wider blocks, a launch per phase.  W = G V, 64 rows a CTA.
__global__ void __launch_bounds__(kSNT)
subspace_gv_kernel(const float* __restrict__ G, const float* __restrict__ V, float* __restrict__ W,
                   int np, const HugeBlock* __restrict__ hb) {
  extern __shared__ __align__(16) float sm[];
  const int b = blockIdx.y, r0 = blockIdx.x * 64, tid = threadIdx.x;
  if (!sub_active(hb[b])) return;
  float* Ws = sm + sub_pipe_floats(64);
  sub_gv<true>(G + (size_t)b * np * np + (size_t)r0 * np, V + (size_t)b * np * kHP, np, 64, sm, Ws);
  float* Wb = W + ((size_t)b * np + r0) * kHP;
  for (int e = tid; e < 64 * kHP; e += kSNT) Wb[e] = Ws[(e >> 5) * kSLd + (e & 31)];
}

// V = orth(W + mu V) (passes > 0), or the Rayleigh-Ritz test on V and W
// (passes = 0), for the rows at Vr, Wr of a CTA.  False when the
// orthonormalisation broke down or the pairs have not converged.
__device__ bool sub_phase(const cg::cluster_group& cl, const SubSmem& m, int rp, int r0, float* Vr,
                          const float* Wr, float* Ub, float* GUb, int nn, int b, float thr, int passes,
                          HugeBlock& h, SubTest& t) {
  const int tid = threadIdx.x;
  for (int e = tid; e < rp * kHP; e += kSNT) {
    const int o = (e >> 5) * kSLd + (e & 31);
    m.Xs[o] = Vr[e];
    m.Ws[o] = Wr[e];
  }
  __syncthreads();
  if (passes == 0) return sub_ritz(cl, m, rp, Ub, GUb, thr, h, t);
  const bool ok = sub_orth(cl, m, rp, r0, nn, b, 1e-4f * h.gF, passes);
  for (int e = tid; e < rp * kHP; e += kSNT) Vr[e] = m.Xs[(e >> 5) * kSLd + (e & 31)];
  cl.sync();  // the new V is visible to the cluster
  return ok;
}

// One phase of the blocks that have not converged, a cluster per block.
__global__ void __launch_bounds__(kSNT)
subspace_phase_kernel(float* V, const float* W, float* __restrict__ U, float* __restrict__ GU, int nn,
                      int np, float thr, int passes, HugeBlock* __restrict__ hb) {
  extern __shared__ __align__(16) float sm[];
  const cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int b = blockIdx.x / CL;
  const int rp = np / CL, r0 = rank * rp;
  HugeBlock& h = hb[b];
  // (the state is written only after a later cluster barrier)
  if (!sub_active(h)) return;
  const size_t vo = ((size_t)b * np + r0) * kHP, uo = ((size_t)b * np + r0) * kHK;
  SubTest t{h.worst, h.ku, false};
  const bool ok = sub_phase(cl, SubSmem(sm, rp), rp, r0, V + vo, W + vo, U + uo, GU + uo, nn, b, thr,
                            passes, h, t);
  if (passes > 0 && !ok && rank == 0 && threadIdx.x == 0) h.orth_fail = 1;
  cl.sync();  // no CTA leaves while others read its shared memory
}

// The further rounds of a block, all steps in its cluster: G V of a CTA's rows
// by 64 at a time (its scratch lies over the phases' arrays).  16 SMs read G
// several times slower than the grid-wide launch, but blocks that get here
// are rare and a launch with none of them costs its launch only.
__global__ void __launch_bounds__(kSNT)
subspace_more_kernel(const float* __restrict__ G, float* V, float* W, float* __restrict__ U,
                     float* __restrict__ GU, int nn, int np, float thr, HugeBlock* __restrict__ hb) {
  extern __shared__ __align__(16) float sm[];
  const cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int b = blockIdx.x / CL, tid = threadIdx.x;
  const int rp = np / CL, r0 = rank * rp;
  HugeBlock& h = hb[b];
  // (the state is written only after a later cluster barrier)
  if (!sub_active(h) || h.stop) return;
  const SubSmem m(sm, rp);
  const float* Gr = G + (size_t)b * np * np + (size_t)r0 * np;
  const float* Vb = V + (size_t)b * np * kHP;
  const size_t vo = ((size_t)b * np + r0) * kHP, uo = ((size_t)b * np + r0) * kHK;
  float* Wc = sm + sub_pipe_floats(64);
  bool ok = true, conv = false;
  SubTest t{h.worst, h.ku, false};
  for (int rd = 0; rd < kSMoreRounds && ok && !conv && !t.stop; ++rd) {
    for (int st = 0; st <= 8 && ok; ++st) {
      for (int c = 0; c < rp; c += 64) {
        const int rows = min(64, rp - c);
        sub_gv<true>(Gr + (size_t)c * np, Vb, np, rows, sm, Wc);
        for (int e = tid; e < rows * kHP; e += kSNT)
          W[vo + (size_t)c * kHP + e] = Wc[(e >> 5) * kSLd + (e & 31)];
        __syncthreads();
      }
      const int passes = st < 8 ? (st + 1 < 8 ? 2 : 3) : 0;
      const bool r = sub_phase(cl, m, rp, r0, V + vo, W + vo, U + uo, GU + uo, nn, b, thr, passes, h,
                               t);
      if (passes > 0) ok = r;
      else conv = r;
    }
  }
  if (!ok && rank == 0 && tid == 0) h.orth_fail = 1;
  cl.sync();  // no CTA leaves while others read its shared memory
}

// the widest cluster the device runs at the largest shared-memory size
int widest_cluster() {
  static const int w = [] {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kSNT);
    cfg.dynamicSmemBytes = sub_smem_bytes(kSPhaseRows);
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, subspace_phase_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    return n > 0 ? 16 : 8;
  }();
  return w;
}

template <class K>
cudaError_t sub_attributes(K k, int rows) {
  if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sub_smem_bytes(rows)))
    return e;
  return cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

template <class K, class... A>
cudaError_t sub_launch(K k, int CL, int B, size_t bytes, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL * B);
  cfg.blockDim = dim3(kSNT);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace

// (any number of blocks: the plans differ up to 1024 wide only, in one launch)
bool subspace_phases(int np) { return subspace_plan(np, 1, sm_count(), widest_cluster()).phases; }

cudaError_t configure_subspace() {
  if (cudaError_t e = sub_attributes(subspace_cluster_kernel<false>, kSMaxRows)) return e;
  if (cudaError_t e = sub_attributes(subspace_cluster_kernel<true>, kSMaxRows)) return e;
  if (cudaError_t e = sub_attributes(subspace_phase_kernel, kSPhaseRows)) return e;
  if (cudaError_t e = sub_attributes(subspace_more_kernel, kSPhaseRows)) return e;
  if (cudaError_t e = cudaFuncSetAttribute(subspace_gv_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sub_smem_bytes(64)))
    return e;
  widest_cluster();  // cached outside any stream capture
  return cudaSuccess;
}

cudaError_t launch_subspace(const float* G, float* V, float* W, float* U, float* GU, int nn, int np,
                            float thr, int first, HugeBlock* hb, int B, int job_blocks, cudaStream_t st,
                            Prof* prof) {
  auto timed = [&](auto&& launch) -> cudaError_t {
    if (prof)
      if (cudaError_t e = prof->before(st, KK_SUBSPACE)) return e;
    if (cudaError_t e = launch()) return e;
    return prof ? prof->after(st) : cudaSuccess;
  };
  const bool many = 16 * B > sm_count();  // (the code's form: the same sums)
  const SubspacePlan plan = subspace_plan(np, job_blocks, sm_count(), widest_cluster());
  const int CL = plan.cluster;
  if (CL == 0) return cudaErrorNotSupported;
  const size_t bytes = sub_smem_bytes(np / CL);
  if (!plan.phases)
    return timed([&] {
      return many ? sub_launch(subspace_cluster_kernel<true>, CL, B, bytes, st, G, V, U, GU, nn, np,
                               thr, first, hb)
                  : sub_launch(subspace_cluster_kernel<false>, CL, B, bytes, st, G, V, U, GU, nn, np,
                               thr, first, hb);
    });
  auto gv = [&] {
    subspace_gv_kernel<<<dim3(np / 64, B), kSNT, sub_smem_bytes(64), st>>>(G, V, W, np, hb);
    return cudaGetLastError();
  };
  const int rounds[kSRounds] = {first, 4, 8};
  for (int r = 0; r < kSRounds; ++r) {
    for (int i = 0; i <= rounds[r]; ++i) {
      if (cudaError_t e = timed(gv)) return e;
      const int passes = i < rounds[r] ? (i + 1 < rounds[r] ? 2 : 3) : 0;
      if (cudaError_t e = timed([&] {
            return sub_launch(subspace_phase_kernel, CL, B, bytes, st, V, W, U, GU, nn, np, thr,
                              passes, hb);
          }))
        return e;
    }
  }
  return timed([&] {
    return sub_launch(subspace_more_kernel, CL, B, sub_more_bytes(np / CL), st, G, V, W, U, GU, nn, np,
                      thr, hb);
  });
}

}  // namespace msllr

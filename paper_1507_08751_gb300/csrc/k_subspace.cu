// Subspace iteration and Rayleigh-Ritz of blocks 257 .. 2048 wide: one
// thread-block cluster per block does every step of every round in one
// launch (the wider blocks keep a launch per step, k_block_huge.cu).
//
// Per step X = G V + mu V, then V = orth(X) by shifted CholQR and two plain
// CholQR passes (the method and mu are those of huge_orth_sweep_kernel); per
// round a Rayleigh-Ritz test.  What bounds a block of this size is latency,
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
//   G V     4 x 4 register tiles over 32-column chunks of G and V (cp.async,
//           three stages), the chunk's columns split over the thread groups
//           that the row count leaves idle; V comes from L2
//   X^T X   4 x 4 register tiles, rows split four ways
//   R       Cholesky in one warp: lane i holds row i
//   X R^-1  a warp per row (eight at a time): lane t holds column t
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

constexpr int kSNT = 256;   // threads per CTA
constexpr int kSKC = 32;    // columns of G per stage
constexpr int kSStages = 3;
constexpr int kSLdG = 36;   // row stride of a G chunk (floats; 16-byte rows, distinct banks)
constexpr int kSLd = 36;    // row stride of X and W
constexpr int kSM = kHP * 33;
constexpr int kSMaxRows = 128;  // rows per CTA: 32 groups of 4 x 4 register tiles

// floats of one pipeline stage, and of the region that the stages share with
// the split sums (used when no copy is in flight)
__host__ __device__ constexpr int sub_stage_floats(int rp) { return rp * kSLdG + kSKC * kHP; }
__host__ __device__ constexpr int sub_pipe_floats(int rp) {
  return kSStages * sub_stage_floats(rp) > 4 * kHP * kHP ? kSStages * sub_stage_floats(rp)
                                                          : 4 * kHP * kHP;
}
size_t sub_smem_bytes(int rp) {
  return sizeof(float) *
         (size_t)(sub_pipe_floats(rp) + 2 * rp * kSLd + 2 * kHP * kHP + 3 * kSM + kHK * kHK);
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

// Ws = rows [r0, r0 + rp) of G V.
__device__ void sub_gv(const float* __restrict__ Gr, const float* V, int np, int rp, float* pipe,
                       float* Ws) {
  const int tid = threadIdx.x;
  const int RG = rp >> 2, cgp = tid & 7, rest = tid >> 3;
  const int split = rest / RG, rg = rest - split * RG;
  const int ns = (kSNT / 8) / RG;  // groups that share a chunk's columns
  const bool on = split < ns;
  const int sf = sub_stage_floats(rp), nch = np / kSKC;
  auto load = [&](int c) {
    float* st = pipe + (c % kSStages) * sf;
    const float* g = Gr + c * kSKC;
    for (int e = tid; e < rp * 8; e += kSNT) {
      const int r = e >> 3, q = e & 7;
      cp16(st + r * kSLdG + 4 * q, g + (size_t)r * np + 4 * q);
    }
    cp16(st + rp * kSLdG + 4 * tid, V + (size_t)c * kSKC * kHP + 4 * tid);
  };
  static_assert(kSKC * kHP == 4 * kSNT, "one 16-byte copy of V per thread");
  float acc[4][4] = {};
  for (int c = 0; c < kSStages - 1; ++c) {
    if (c < nch) load(c);
    cp_commit();
  }
  for (int c = 0; c < nch; ++c) {
    cp_wait<kSStages - 2>();
    __syncthreads();
    if (c + kSStages - 1 < nch) load(c + kSStages - 1);
    cp_commit();
    if (on) {
      const float* Gs = pipe + (c % kSStages) * sf;
      const float* Vs = Gs + rp * kSLdG;
      for (int k4 = split; k4 < kSKC / 4; k4 += ns) {
        float4 g[4], v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          g[i] = *reinterpret_cast<const float4*>(Gs + (rg + i * RG) * kSLdG + 4 * k4);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          v[k] = *reinterpret_cast<const float4*>(Vs + (4 * k4 + k) * kHP + 4 * cgp);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float gk[4] = {g[i].x, g[i].y, g[i].z, g[i].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            acc[i][0] = fmaf(gk[k], v[k].x, acc[i][0]);
            acc[i][1] = fmaf(gk[k], v[k].y, acc[i][1]);
            acc[i][2] = fmaf(gk[k], v[k].z, acc[i][2]);
            acc[i][3] = fmaf(gk[k], v[k].w, acc[i][3]);
          }
        }
      }
    }
  }
  cp_wait<0>();
  // the groups' sums are added in group order
  for (int s = 0; s < ns; ++s) {
    __syncthreads();
    if (on && split == s) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float4* d = reinterpret_cast<float4*>(Ws + (rg + i * RG) * kSLd + 4 * cgp);
        float4 t = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        if (s > 0) {
          const float4 o = *d;
          t = make_float4(o.x + t.x, o.y + t.y, o.z + t.z, o.w + t.w);
        }
        *d = t;
      }
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
  for (int r = q; r < rp; r += 4) {
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
  const float4 s0 = reinterpret_cast<const float4*>(tmp)[tid];
  const float4 s1 = reinterpret_cast<const float4*>(tmp + kHP * kHP)[tid];
  const float4 s2 = reinterpret_cast<const float4*>(tmp + 2 * kHP * kHP)[tid];
  const float4 s3 = reinterpret_cast<const float4*>(tmp + 3 * kHP * kHP)[tid];
  reinterpret_cast<float4*>(P)[tid] =
      make_float4((s0.x + s1.x) + (s2.x + s3.x), (s0.y + s1.y) + (s2.y + s3.y),
                  (s0.z + s1.z) + (s2.z + s3.z), (s0.w + s1.w) + (s2.w + s3.w));
}

// Sm (32 x 33) = the sum of P over the cluster's CTAs, in rank order (the
// same in every CTA).  Contains the cluster barrier that publishes P.
__device__ void sub_cluster_sum(const cg::cluster_group& cl, float* P, float* Sm) {
  cl.sync();
  const int tid = threadIdx.x, n = (int)cl.num_blocks();
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int r = 0; r < n; ++r) {
    const float4 v = reinterpret_cast<const float4*>(cl.map_shared_rank(P, r))[tid];
    s.x += v.x;
    s.y += v.y;
    s.z += v.z;
    s.w += v.w;
  }
  float* d = Sm + (tid >> 3) * 33 + 4 * (tid & 7);
  d[0] = s.x;
  d[1] = s.y;
  d[2] = s.z;
  d[3] = s.w;
  __syncthreads();
}

// Warp 0: Sm + shift I = R^T R (R upper, row j at Rm + 33 j, zero below the
// diagonal; rinv[j] = 1 / R_jj).  Returns false in every thread on a
// non-positive or non-finite pivot.
__device__ bool sub_chol(const float* Sm, float shift, float* Rm, float* rinv) {
  const int tid = threadIdx.x, lane = tid & 31;
  bool ok = true;
  if (tid < 32) {
    float a[kHP];
#pragma unroll
    for (int j = 0; j < kHP; ++j) a[j] = Sm[lane * 33 + j] + (j == lane ? shift : 0.f);
#pragma unroll
    for (int j = 0; j < kHP; ++j) {
      const float d = __shfl_sync(0xffffffffu, a[j], j);
      ok = ok && d > 0.f && d <= FLT_MAX;
      const float r = sqrtf(d), inv = 1.f / r;
      a[j] = lane == j ? r : a[j] * inv;
      if (lane == j) rinv[j] = inv;
#pragma unroll
      for (int t = j + 1; t < kHP; ++t)
        a[t] = fmaf(-a[j], __shfl_sync(0xffffffffu, a[j], t), a[t]);
    }
#pragma unroll
    for (int j = 0; j < kHP; ++j) Rm[j * 33 + lane] = lane >= j ? a[j] : 0.f;
  }
  return __syncthreads_and(ok);
}

// X <- X R^{-1}, rp rows.
__device__ void sub_solve(float* X, int rp, const float* Rm, const float* rinv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r0 = 8 * warp; r0 < rp; r0 += kSNT / 4) {
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = r0 + i < rp ? X[(r0 + i) * kSLd + lane] : 0.f;
#pragma unroll 8
    for (int j = 0; j < kHP; ++j) {
      const float rj = Rm[j * 33 + lane], ij = rinv[j];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x = __shfl_sync(0xffffffffu, v[i], j) * ij;
        v[i] = lane == j ? x : fmaf(-x, rj, v[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (r0 + i < rp) X[(r0 + i) * kSLd + lane] = v[i];
  }
  __syncthreads();
}

// Eigen-decomposition of the symmetric A (32 x 33): A becomes diagonal, the
// columns of Q the eigenvectors.  Off-diagonal entries below 3e-8 of the
// geometric mean of their diagonal entries (or of `floor`) stay.
__device__ void sub_jacobi(float* A, float* Q, float floor_, float* cs, int* flag) {
  const int tid = threadIdx.x;
  for (int e = tid; e < kHP * kHP; e += kSNT) Q[(e >> 5) * 33 + (e & 31)] = (e >> 5) == (e & 31);
  const int bi = tid >> 4, bj = tid & 15;
  // pair i of round rd (round robin): column 31 stays, the others turn
  auto pair = [](int rd, int i, int& p, int& q) {
    p = rd + i;
    if (p >= 31) p -= 31;
    q = i == 0 ? 31 : rd - i;
    if (q < 0) q += 31;
  };
  for (int sweep = 0; sweep < 12; ++sweep) {
    if (tid == 0) *flag = 0;
    __syncthreads();
    for (int rd = 0; rd < 31; ++rd) {
      if (tid < 16) {
        int p, q;
        pair(rd, tid, p, q);
        const float app = A[p * 33 + p], aqq = A[q * 33 + q];
        const float apq = 0.5f * (A[p * 33 + q] + A[q * 33 + p]);
        float c = 1.f, s = 0.f;
        const float lim = 3e-8f * fmaxf(sqrtf(fabsf(app)) * sqrtf(fabsf(aqq)), floor_);
        if (fabsf(apq) > lim) {
          const float tau = (aqq - app) / (2.f * apq);
          const float t = copysignf(1.f, tau) / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f)));
          c = 1.f / sqrtf(fmaf(t, t, 1.f));
          s = t * c;
          *flag = 1;
        }
        cs[2 * tid] = c;
        cs[2 * tid + 1] = s;
      }
      __syncthreads();
      int pi, qi, pj, qj;
      pair(rd, bi, pi, qi);
      pair(rd, bj, pj, qj);
      const float ci = cs[2 * bi], si = cs[2 * bi + 1], cj = cs[2 * bj], sj = cs[2 * bj + 1];
      const float b00 = A[pi * 33 + pj], b01 = A[pi * 33 + qj];
      const float b10 = A[qi * 33 + pj], b11 = A[qi * 33 + qj];
      const float x0 = ci * b00 - si * b10, x1 = ci * b01 - si * b11;
      const float y0 = si * b00 + ci * b10, y1 = si * b01 + ci * b11;
      float n01 = sj * x0 + cj * x1, n10 = cj * y0 - sj * y1;
      if (bi == bj && si != 0.f) n01 = n10 = 0.f;
      A[pi * 33 + pj] = cj * x0 - sj * x1;
      A[pi * 33 + qj] = n01;
      A[qi * 33 + pj] = n10;
      A[qi * 33 + qj] = sj * y0 + cj * y1;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float* row = Q + (bi + 16 * h) * 33;
        const float vp = row[pj], vq = row[qj];
        row[pj] = cj * vp - sj * vq;
        row[qj] = sj * vp + cj * vq;
      }
      __syncthreads();
    }
    if (!*flag) break;
    __syncthreads();
  }
  __syncthreads();
}

// `first`: steps of the first round (later rounds: 4 and 8).
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
  float* pipe = sm;
  float* Xs = pipe + sub_pipe_floats(rp);
  float* Ws = Xs + rp * kSLd;
  float* Sp = Ws + rp * kSLd;  // two 32 x 32 partial sums, used in turn
  float* Sm = Sp + 2 * kHP * kHP;
  float* Rm = Sm + kSM;
  float* Qm = Rm + kSM;
  float* Bm = Qm + kSM;  // kHK x kHK
  __shared__ float rinv[kHP], cs[32], rq[2 * kHK], red[kSNT / 32][2 * kHK];
  __shared__ int flag, sel[kHK], ku_s;
  const float* Gr = G + (size_t)b * np * np + (size_t)r0 * np;
  float* Vb = V + (size_t)b * np * kHP;
  const float gF = h.gF, mu = 1e-4f * gF;
  for (int e = tid; e < rp * kHP; e += kSNT) Xs[(e >> 5) * kSLd + (e & 31)] = Vb[(size_t)r0 * kHP + e];
  __syncthreads();
  int turn = 0;
  auto part = [&]() {
    float* p = Sp + turn * kHP * kHP;
    turn ^= 1;
    return p;
  };
  const int rounds[3] = {first, 4, 8};
  bool failed = false, conv = false;
  for (int rd = 0; rd < 3 && !conv && !failed; ++rd) {
    for (int st = 0; st < rounds[rd] && !failed; ++st) {
      sub_gv(Gr, Vb, np, rp, pipe, Ws);
      for (int e = tid; e < rp * kHP; e += kSNT) {
        const int o = (e >> 5) * kSLd + (e & 31);
        Xs[o] = fmaf(mu, Xs[o], Ws[o]);
      }
      __syncthreads();
      for (int pass = 1; pass <= 3; ++pass) {
        float* P = part();
        sub_atb(Xs, Xs, rp, pipe, P);
        sub_cluster_sum(cl, P, Sm);
        float shift = 0.f;
        if (pass == 1) {
          float tr = 0.f;
          for (int i = 0; i < kHP; ++i) tr += Sm[i * 33 + i];
          shift = 11.f * (float)((double)nn * kHP + kHP * (kHP + 1)) * FLT_EPSILON * tr;
        }
        // the same sum in every CTA: all of them fail or none
        if (!sub_chol(Sm, shift, Rm, rinv)) {
          failed = true;
          break;
        }
        sub_solve(Xs, rp, Rm, rinv);
      }
      if (failed)
        for (int e = tid; e < rp * kHP; e += kSNT) {
          const int r = r0 + (e >> 5), c = e & 31;
          Xs[(e >> 5) * kSLd + c] =
              r < nn ? huge_hash((uint32_t)r + 977u * b, (uint32_t)c + 0xB0Bu) : 0.f;
        }
      __syncthreads();
      for (int e = tid; e < rp * kHP; e += kSNT) Vb[(size_t)r0 * kHP + e] = Xs[(e >> 5) * kSLd + (e & 31)];
      cl.sync();  // the new V is visible to the cluster
    }
    if (failed) break;
    // Rayleigh-Ritz on T = V^T G V
    sub_gv(Gr, Vb, np, rp, pipe, Ws);
    {
      float* P = part();
      sub_atb(Xs, Ws, rp, pipe, P);
      sub_cluster_sum(cl, P, Sm);
    }
    for (int e = tid; e < kHP * kHP; e += kSNT) {
      const int i = e >> 5, j = e & 31;
      Rm[i * 33 + j] = 0.5f * (Sm[i * 33 + j] + Sm[j * 33 + i]);
    }
    __syncthreads();
    sub_jacobi(Rm, Qm, 1e-2f * thr, cs, &flag);
    // the pairs above tau^2, largest first, at most kHK
    if (tid < 32) {
      const float th = Rm[tid * 33 + tid];
      int rk = 0;
      for (int j = 0; j < kHP; ++j) {
        const float o = __shfl_sync(0xffffffffu, th, j);
        rk += o > th || (o == th && j < tid);
      }
      const unsigned above = __ballot_sync(0xffffffffu, th > thr);
      if (th > thr && rk < kHK) sel[rk] = tid;
      if (tid == 0) ku_s = min(__popc(above), kHK);
    }
    __syncthreads();
    const int ku = ku_s;
    // U = V Q and G U in the pipeline's space (row stride 2 kHK); V stays,
    // it is the next round's start
    float* Us = pipe;
    for (int e = tid; e < rp * kHK; e += kSNT) {
      const int r = e >> 4, q = e & 15;
      float u = 0.f, g = 0.f;
      if (q < ku) {
        const int cq = sel[q];
#pragma unroll 8
        for (int a = 0; a < kHP; ++a) {
          const float w = Qm[a * 33 + cq];
          u = fmaf(Xs[r * kSLd + a], w, u);
          g = fmaf(Ws[r * kSLd + a], w, g);
        }
      }
      Us[r * 2 * kHK + q] = u;
      Us[r * 2 * kHK + kHK + q] = g;
    }
    __syncthreads();
    // B = U^T G U: partial sums in rank order
    {
      float* P = part();
      const int p = tid >> 4, q = tid & 15;
      float t = 0.f;
      for (int r = 0; r < rp; ++r) t = fmaf(Us[r * 2 * kHK + p], Us[r * 2 * kHK + kHK + q], t);
      P[tid] = t;
      cl.sync();
      float s = 0.f;
      for (int c = 0; c < CL; ++c) s += cl.map_shared_rank(P, c)[tid];
      Bm[tid] = s;
    }
    __syncthreads();
    // residuals |G u_q - theta_q u_q|^2 and What = G U - U sym(B) / 2, |What_q|^2
    {
      const int q = tid & 15, rr = tid >> 4;
      float ra = 0.f, wa = 0.f;
      for (int r = rr; r < rp; r += kSNT / 16) {
        const float u = Us[r * 2 * kHK + q], g = Us[r * 2 * kHK + kHK + q];
        float wh = g;
        for (int p = 0; p < ku; ++p)
          wh = fmaf(-0.25f * (Bm[p * kHK + q] + Bm[q * kHK + p]), Us[r * 2 * kHK + p], wh);
        if (q < ku) {
          const float res = g - Bm[q * kHK + q] * u;
          ra = fmaf(res, res, ra);
          wa = fmaf(wh, wh, wa);
        }
        U[((size_t)b * np + r0 + r) * kHK + q] = u;
        GU[((size_t)b * np + r0 + r) * kHK + q] = q < ku ? wh : 0.f;
      }
      ra += __shfl_xor_sync(0xffffffffu, ra, 16);
      wa += __shfl_xor_sync(0xffffffffu, wa, 16);
      if ((tid & 31) < 16) {
        red[tid >> 5][q] = ra;
        red[tid >> 5][kHK + q] = wa;
      }
    }
    __syncthreads();
    float* P = part();
    if (tid < 2 * kHK) {
      float t = 0.f;
      for (int w = 0; w < kSNT / 32; ++w) t += red[w][tid];
      P[tid] = t;
    }
    cl.sync();
    if (tid < 2 * kHK) {
      float t = 0.f;
      for (int c = 0; c < CL; ++c) t += cl.map_shared_rank(P, c)[tid];
      rq[tid] = t;
    }
    __syncthreads();
    // converged: see huge_rr_kernel (the same test)
    conv = true;
    float th0 = 0.f, wsum = 0.f;
    for (int q = 0; q < ku; ++q) {
      th0 = fmaxf(th0, Bm[q * kHK + q]);
      wsum += rq[kHK + q];
    }
    for (int q = 0; q < ku; ++q)
      if (sqrtf(rq[q]) > fmaxf(3e-4f * thr, 4e-6f * th0)) conv = false;
    if (rank == 0 && tid == 0) {
      int k = 0;
      for (int q = 0; q < ku; ++q) {
        const float th = Bm[q * kHK + q];
        h.theta[q] = th;
        k += th > thr;
      }
      h.c = cert_bound(thr, gF, ku, wsum);
      h.ku = ku;
      h.k = k;
      h.conv = conv;
    }
    __syncthreads();
  }
  if (failed && rank == 0 && tid == 0) h.orth_fail = 1;
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
    cfg.dynamicSmemBytes = sub_smem_bytes(kSMaxRows);
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, subspace_cluster_kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    return n > 0 ? 16 : 8;
  }();
  return w;
}

// CTAs per block: 8 up to 512 wide, 16 above (32 to 128 rows a CTA)
int cluster_size(int np) { return np <= 512 ? 8 : widest_cluster(); }

}  // namespace

cudaError_t configure_subspace() {
  if (cudaError_t e = cudaFuncSetAttribute(subspace_cluster_kernel,
                                           cudaFuncAttributeNonPortableClusterSizeAllowed, 1))
    return e;
  if (cudaError_t e = cudaFuncSetAttribute(subspace_cluster_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)sub_smem_bytes(kSMaxRows)))
    return e;
  widest_cluster();
  return cudaSuccess;
}

bool subspace_cluster_path(int np) { return np / cluster_size(np) <= kSMaxRows; }

cudaError_t launch_subspace(const float* G, float* V, float* U, float* GU, int nn, int np, float thr,
                            int first, HugeBlock* hb, int B, cudaStream_t st) {
  const int CL = cluster_size(np);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL * B);
  cfg.blockDim = dim3(kSNT);
  cfg.dynamicSmemBytes = sub_smem_bytes(np / CL);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, subspace_cluster_kernel, G, V, U, GU, nn, np, thr, first, hb);
}

}  // namespace msllr

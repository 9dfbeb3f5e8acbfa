// Householder path of blocks up to 256 wide on the wide-block route (eq:svt,
// Sec. 8): the eigenpairs of G above tau^2 for the blocks whose certified
// Lanczos path did not settle (more than 16 pairs, slow convergence, or a
// spectrum that crowds below tau^2), and for every block when the shortcuts
// are off.  Tridiagonalisation (Golub & Van Loan, Sec. 8.3), Sturm
// multisection (symeig.cuh), inverse iteration, back-transformation.
//
// The whole symmetric G stays in registers: a cluster of two CTAs (one up to
// 128 wide) holds 128 rows per CTA, a thread 8 rows x 8 columns (warp: 8
// rows; lane: every 32nd column).  A step is a matrix-vector product out of
// registers with a 9-shuffle multi-reduction, a rank-2 update, and two
// cluster barriers (the product and the next row are exchanged over
// distributed shared memory).  What bounds a step is that chain of latencies,
// about 1 us; with the packed G in the shared memory of one CTA and a thread
// per row a step took 12 us at 256 wide (3.0 ms per block).  Inverse
// iteration runs a lane per eigenvalue with its LU factors in shared memory,
// the back-transformation a warp per vector with the vector in registers and
// the reflectors streamed from the block's (no longer needed) G storage.
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "lanczos.cuh"
#include "symeig.cuh"

namespace cg = cooperative_groups;

namespace msllr {

namespace {

constexpr int kTNT = 512;   // threads per CTA
constexpr int kTNW = kTNT / 32;
constexpr int kTRows = 128;  // rows per CTA
constexpr int kTMax = 256;
constexpr int kTB = 32;      // eigenvectors per inverse-iteration batch

// shared floats: two row buffers, the product, EigScratch (9 NMAX + 4 NT +
// 64), LU factors and vectors of a batch, its pivot bits
constexpr int kTSmemFloats = 3 * kTMax + 9 * kTMax + 4 * kTNT + 64 + 5 * kTMax * kTB + 8 * kTB;

// Two steps of inverse iteration on T (s.d, s.e, order n) for the k shifts
// s.shf: eigenvectors into Y (row i at Y + i ldy), orthonormalised inside
// clusters.  Warp 0 solves, lane q for target q0 + q, factors at [i][q].
__device__ void tri_vectors(int n, int k, float tnorm, EigScratch& s, float* buf, float* Y, int ldy) {
  const int tid = threadIdx.x;
  const float tiny = FLT_EPSILON * tnorm;
  float* dd = buf + tid;  // (lanes of warp 0)
  float* du = dd + kTMax * kTB;
  float* du2 = du + kTMax * kTB;
  float* dl = du2 + kTMax * kTB;
  float* y = dl + kTMax * kTB;
  unsigned* piv = reinterpret_cast<unsigned*>(buf + 5 * kTMax * kTB) + tid;
  for (int pass = 0; pass < 2; ++pass) {
    for (int q0 = 0; q0 < k; q0 += kTB) {
      const int q = q0 + tid;
      if (tid < kTB && q < k) {
        if (pass == 0 || k > kTB) {
          // pivoted LU of T - shift I, tiny pivots replaced by +-tiny
          const float shift = s.shf[q];
          float di = s.d[0] - shift, ui = n > 1 ? s.e[0] : 0.f;
          unsigned bits = 0u;
          for (int i = 0; i < n - 1; ++i) {
            // row i: (di, ui, u2i); row i + 1: (li, dn, un)
            const float li = s.e[i], dn = s.d[i + 1] - shift, un = i < n - 2 ? s.e[i + 1] : 0.f;
            float f;
            if (fabsf(di) >= fabsf(li)) {
              const float dv = (di == 0.f) ? tiny : di;
              f = li / dv;
              dd[i * kTB] = dv;
              du[i * kTB] = ui;
              du2[i * kTB] = 0.f;
              di = dn - f * ui;
              ui = un;
            } else {
              f = di / li;
              dd[i * kTB] = li;
              du[i * kTB] = dn;
              du2[i * kTB] = un;
              di = ui - f * dn;
              ui = -f * un;
              bits |= 1u << (i & 31);
            }
            dl[i * kTB] = f;
            const float p = dd[i * kTB];
            if (fabsf(p) < tiny) dd[i * kTB] = p < 0.f ? -tiny : tiny;
            if ((i & 31) == 31) {
              piv[(i >> 5) * kTB] = bits;
              bits = 0u;
            }
          }
          if ((n - 1) & 31) piv[((n - 1) >> 5) * kTB] = bits;
          dd[(n - 1) * kTB] = fabsf(di) < tiny ? (di < 0.f ? -tiny : tiny) : di;
        }
        if (pass == 0) {
          // deterministic pseudo-random start vector of size ~eps |T|
          uint32_t h = 0x9E3779B9u * (uint32_t)(q + 1);
          for (int i = 0; i < n; ++i) {
            h ^= h << 13;
            h ^= h >> 17;
            h ^= h << 5;
            y[i * kTB] = tiny * ((float)(h >> 8) * (2.f / 16777216.f) - 1.f + 1e-3f);
          }
        } else {
          for (int i = 0; i < n; ++i) y[i * kTB] = Y[(size_t)i * ldy + q] * tiny;
        }
        float a = y[0];
        for (int i = 0; i < n - 1; ++i) {
          const float b = y[(i + 1) * kTB], f = dl[i * kTB];
          if ((piv[(i >> 5) * kTB] >> (i & 31)) & 1u) {
            y[i * kTB] = b;
            a = a - f * b;
          } else {
            y[i * kTB] = a;
            a = b - f * a;
          }
        }
        float y1 = a / dd[(n - 1) * kTB], y2 = 0.f, ss = y1 * y1;
        y[(n - 1) * kTB] = y1;
        for (int i = n - 2; i >= 0; --i) {
          const float u2 = i < n - 2 ? du2[i * kTB] : 0.f;
          const float v = (y[i * kTB] - du[i * kTB] * y1 - u2 * y2) / dd[i * kTB];
          y[i * kTB] = v;
          y2 = y1;
          y1 = v;
          ss = fmaf(v, v, ss);
        }
        const float inv = ss > 0.f && ss <= FLT_MAX ? rsqrtf(ss) : 0.f;
        if (inv > 0.f) {
          for (int i = 0; i < n; ++i) Y[(size_t)i * ldy + q] = y[i * kTB] * inv;
        } else {
          // the squares left the FP32 range: scale by the largest entry first
          float mx = 0.f;
          for (int i = 0; i < n; ++i) mx = fmaxf(mx, fabsf(y[i * kTB]));
          const float im = mx > 0.f ? 1.f / mx : 0.f;
          float s2 = 0.f;
          for (int i = 0; i < n; ++i) s2 = fmaf(y[i * kTB] * im, y[i * kTB] * im, s2);
          const float i2 = s2 > 0.f ? im * rsqrtf(s2) : 0.f;
          for (int i = 0; i < n; ++i) Y[(size_t)i * ldy + q] = y[i * kTB] * i2;
        }
      }
      __syncwarp();
    }
    __syncthreads();
    cluster_mgs<kTNT>(Y, ldy, n, k, s.clus, s.red);
    __syncthreads();
  }
}

// CL: CTAs per block, NC = 4 CL columns per lane
template <int CL>
__global__ void __launch_bounds__(kTNT)
tridiag_kernel(ScaleLaunch a, float* __restrict__ Gall, BigWorkspace ws, int nblocks) {
  extern __shared__ __align__(16) float sm[];
  constexpr int NC = 4 * CL;
  const cg::cluster_group cl = cg::this_cluster();
  const int rank = CL > 1 ? (int)cl.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.m >= a.n ? a.n : a.m;
  float* xb[2] = {sm, sm + kTMax};
  float* ps = sm + 2 * kTMax;
  EigScratch s;
  s.d = ps + kTMax;
  s.e = s.d + kTMax;
  s.e2 = s.e + kTMax;
  s.beta = s.e2 + kTMax;
  s.vbuf = s.beta + kTMax;
  s.pbuf = s.vbuf + kTMax;
  s.lam = s.pbuf + kTMax;
  s.shf = s.lam + kTMax;
  s.clus = reinterpret_cast<int*>(s.shf + kTMax);
  s.lo = reinterpret_cast<float*>(s.clus + kTMax);
  s.hi = s.lo + kTNT;
  s.xs = s.hi + kTNT;
  s.cnt = reinterpret_cast<int*>(s.xs + kTNT);
  s.red = reinterpret_cast<float*>(s.cnt + kTNT);
  float* lubuf = s.red + 64;
  auto barrier = [&] {
    if constexpr (CL > 1) cl.sync();
    else __syncthreads();
  };
  auto other = [&](float* p) -> float* {
    if constexpr (CL > 1) return cl.map_shared_rank(p, rank ^ 1);
    else return p;
  };
  float* xo[2] = {other(xb[0]), other(xb[1])};
  float* po = other(ps);
  const int r0 = kTRows * rank + 8 * warp;
  // most launches find nothing to do
  bool any = false;
  for (int b = blockIdx.x / CL; b < nblocks && !any; b += gridDim.x / CL) any = ws.k[b] < 0;
  if (!any) return;
  barrier();  // (k is written below)
  for (int b = blockIdx.x / CL; b < nblocks; b += gridDim.x / CL) {
    const bool todo = ws.k[b] < 0;
    barrier();  // (k is written below)
    if (!todo) continue;
    float* G = Gall + (size_t)b * n * n;
    // scale by a power of two: the largest diagonal entry comes to [1, 2)
    float gd = 0.f;
    for (int i = tid; i < n; i += kTNT) gd = fmaxf(gd, G[((size_t)i * (i + 1)) / 2 + i]);
    gd = block_max<kTNT>(gd, s.red);
    int ex = 0;
    if (gd > 0.f) ex = ilogbf(gd);
    float A[8][NC];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int r = r0 + i, c = lane + 32 * k;
        const int hi = max(r, c), lo = min(r, c);
        A[i][k] = hi < n ? scalbnf(G[(size_t)hi * (hi + 1) / 2 + lo], -ex) : 0.f;
      }
    // row 0 (and, for the last diagonal entry, row n - 1) to both CTAs
    if (r0 == 0) {
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        xb[0][lane + 32 * k] = A[0][k];
        if (CL > 1) xo[0][lane + 32 * k] = A[0][k];
      }
    }
    barrier();  // G has been read, row 0 is there
    for (int j = 0; j < n - 2; ++j) {
      const float* x = xb[j & 1];
      const int k0 = (j + 1) >> 5;  // columns below 32 k0 are done
      float v[NC], sq = 0.f;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int c = lane + 32 * k;
        v[k] = (k >= k0 && c > j + 1) ? x[c] : 0.f;
        sq = fmaf(v[k], v[k], sq);
      }
      const float sigma = warp_sum(sq);
      const float x0 = x[j + 1];
      float bt = 0.f, ej = x0, v0 = 0.f;
      // entries below 2^-40 of the largest diagonal entry count as zero
      const bool refl = sigma > 8.3e-25f;
      if (refl) {
        const float xn = sqrtf(fmaf(x0, x0, sigma));
        ej = x0 >= 0.f ? -xn : xn;
        v0 = x0 - ej;
        bt = 2.f / fmaf(v0, v0, sigma);
#pragma unroll
        for (int k = 0; k < NC; ++k)
          if (lane + 32 * k == j + 1) v[k] = v0;
        // p = A v on the warp's rows; the eight sums of a warp by halving:
        // lane bits 4, 3, 2 pick the row
        if (r0 + 7 > j) {
          float p[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) p[i] = 0.f;
#pragma unroll
          for (int k = 0; k < NC; ++k)
            if (k >= k0) {
#pragma unroll
              for (int i = 0; i < 8; ++i) p[i] = fmaf(A[i][k], v[k], p[i]);
            }
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
          const int r = r0 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
          if ((lane & 3) == 0) ps[r] = p[0];
          if (CL > 1 && (lane & 3) == 1) po[r] = p[0];
        }
        if (rank == 0 && warp == kTNW - 1) {
          // the reflector, for the back-transformation
#pragma unroll
          for (int k = 0; k < NC; ++k)
            if (lane + 32 * k < n) G[(size_t)j * n + lane + 32 * k] = v[k];
        }
        barrier();
        float w[NC], dot = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          const int c = lane + 32 * k;
          w[k] = (k >= k0 && c > j && c < n) ? ps[c] : 0.f;
          dot = fmaf(v[k], w[k], dot);
        }
        const float K = 0.5f * bt * bt * warp_sum(dot);
#pragma unroll
        for (int k = 0; k < NC; ++k) w[k] = fmaf(-K, v[k], bt * w[k]);
        if (r0 + 7 > j) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = r0 + i;
            const float vr = r == j + 1 ? v0 : (r > j + 1 ? x[r] : 0.f);
            const float wr = r > j && r < n ? fmaf(-K, vr, bt * ps[r]) : 0.f;
#pragma unroll
            for (int k = 0; k < NC; ++k)
              if (k >= k0) A[i][k] = fmaf(-wr, v[k], fmaf(-vr, w[k], A[i][k]));
          }
        }
      }
      if (rank == 0 && tid == 0) {
        s.d[j] = x[j];
        s.e[j] = ej;
        s.beta[j] = bt;
      }
      // row j + 1 to both CTAs
      const int nr = j + 1 - r0;
      if (nr >= 0 && nr < 8) {
        float* xn0 = xb[(j + 1) & 1];
        float* xn1 = xo[(j + 1) & 1];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i == nr) {
#pragma unroll
            for (int k = 0; k < NC; ++k)
              if (k >= k0) {
                xn0[lane + 32 * k] = A[i][k];
                if (CL > 1) xn1[lane + 32 * k] = A[i][k];
              }
          }
      }
      barrier();
    }
    // the last diagonal entry, from the thread that holds it
    {
      const int nr = n - 1 - r0, kc = (n - 1) >> 5;
      if (nr >= 0 && nr < 8 && lane == ((n - 1) & 31)) {
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int k = 0; k < NC; ++k)
            if (i == nr && k == kc) t = A[i][k];
        if (rank == 0) s.d[n - 1] = t;
        else *other(s.d + n - 1) = t;
      }
      if (rank == 0 && tid == 0 && n >= 2) {
        const float* x = xb[(n - 2) & 1];
        s.d[n - 2] = x[n - 2];
        s.e[n - 2] = x[n - 1];
      }
    }
    barrier();
    if (rank != 0) continue;
    float* Y = ws.Y + (size_t)b * ws.ystride;
    const float thr = a.tau * a.tau;
    float tn = 0.f;
    const int k = top_eigenvalues<kTNT>(n, scalbnf(thr, -ex), s, &tn);
    if (k > 0) {
      tri_vectors(n, k, tn, s, lubuf, Y, n);
      // back-transformation v = H_0 (H_1 (... H_{n-3} y)), a warp per vector,
      // the next reflector's loads in flight; then V_f = V diag(sqrt(f)),
      // f = 1 - tau / sigma
      for (int q = warp; q < k; q += kTNW) {
        float y[NC], vn[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int i = lane + 32 * c;
          y[c] = i < n ? Y[(size_t)i * n + q] : 0.f;
          vn[c] = (n >= 3 && i < n) ? G[(size_t)(n - 3) * n + i] : 0.f;
        }
        for (int j = n - 3; j >= 0; --j) {
          float v[NC], dot = 0.f;
          const float bt = s.beta[j];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const int i = lane + 32 * c;
            v[c] = bt != 0.f ? vn[c] : 0.f;
            vn[c] = (j > 0 && i < n) ? G[(size_t)(j - 1) * n + i] : 0.f;
            dot = fmaf(v[c], y[c], dot);
          }
          dot = warp_sum(dot) * bt;
#pragma unroll
          for (int c = 0; c < NC; ++c) y[c] = fmaf(-dot, v[c], y[c]);
        }
        const float sig = sqrtf(scalbnf(s.lam[q], ex));
        const float f = sqrtf(fmaxf(1.f - a.tau / sig, 0.f));
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int i = lane + 32 * c;
          if (i < n) Y[(size_t)i * n + q] = y[c] * f;
        }
      }
    }
    __syncthreads();
    if (tid == 0) {
      ws.k[b] = k;
      if (a.rank_out) a.rank_out[b] = k;
      if (a.cnt) {
        if (k == 0) atomicAdd(a.cnt + 1, 1ull);
        atomicAdd(a.cnt + 3, 1ull);
        atomicAdd(a.cnt + 6, (unsigned long long)fl_householder(n, k));
      }
      if (a.nuc_acc && k > 0) {
        double t = 0.0;
        for (int q = 0; q < k; ++q)
          t += (double)fmaxf(sqrtf(scalbnf(s.lam[q], ex)) - a.tau, 0.f);
        atomicAdd(a.nuc_acc, t);
      }
    }
    __syncthreads();
  }
  // (nothing of another CTA's shared memory is used after the loop's barriers)
}

}  // namespace

cudaError_t configure_tridiag() {
  const int bytes = (int)sizeof(float) * kTSmemFloats;
  if (cudaError_t e = cudaFuncSetAttribute(tridiag_kernel<1>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes))
    return e;
  return cudaFuncSetAttribute(tridiag_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_tridiag(const ScaleLaunch& s, const BigWorkspace& ws, int nblocks, int groups,
                           cudaStream_t st) {
  const int n = s.m < s.n ? s.m : s.n;
  const size_t bytes = sizeof(float) * kTSmemFloats;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  const int CL = n <= kTRows ? 1 : 2;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL * groups);
  cfg.blockDim = dim3(kTNT);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (CL == 1) return cudaLaunchKernelEx(&cfg, tridiag_kernel<1>, s, ws.G, ws, nblocks);
  return cudaLaunchKernelEx(&cfg, tridiag_kernel<2>, s, ws.G, ws, nblocks);
}

}  // namespace msllr

// Block SVT (eq:svt, eq:bsvt) for blocks wider than 256 (256 < min(m, n) <=
// MSLLR_MAX_BLOCK_WIDTH), e.g. the full-matrix scale of a 1024 x 1024 job or
// the 1024 x 1024 blocks of an 8192 x 8192 one.  A block of that width does
// not fit one CTA, so every phase is spread over many CTAs and the blocks of
// a scale go through each launch together:
//   1. Gram: G_b = C_b^T C_b, 64x64 tiles of the lower triangle split over
//      row chunks; the partial sums are added in a fixed order and G_b is
//      stored as a full square (both triangles);
//   2. subspace iteration on G_b with a basis of kHP = 32 columns kept from
//      the previous call (warm start), in one cluster launch up to 2048 wide
//      (k_subspace.cu): W = G V, then W + mu V is orthonormalised by a shifted
//      CholQR pass and one more, two before a test;
//   3. Rayleigh-Ritz on V^T G V (32 x 32, parallel Jacobi) for the pairs above
//      tau^2, their residuals and a convergence test; unconverged blocks get
//      further rounds of steps;
//   4. certificate: ||P G P||_2 < tau^2 with P = I - U U^T over the kept
//      Ritz vectors, by repeated squaring on the tensor cores
//      (k_cert_tc.cu); by Cauchy interlacing G then has no eigenvalue above
//      tau^2 besides the kept ones;
//   5. rebuild: Z'_b = (C_b V_f) V_f^T with V_f = U diag(sqrt(1 - tau/sigma))
//      over the pairs above tau, scattered through Shift_{-s}, with the fused
//      dual update W' = 2 Z' - A of eq:admm.
// A block whose pairs do not converge in every round run, or whose certificate
// fails, keeps its Ritz pairs and is counted.
#include <float.h>
#include <math.h>

#include "../../include/msllr.h"
#include "common.cuh"
#include "huge.cuh"
#include "internal.h"

namespace msllr {

namespace {

constexpr int kHT = 64;          // Gram tile
constexpr int kHThreads = 256;   // tile kernels

struct HugeDims {
  int mm, nn, nblocks, T, ntiles, chunk_rows, chunks;
};

HugeDims huge_dims(int M, int N, int m, int n) {
  HugeDims d;
  d.mm = m >= n ? m : n;
  d.nn = m >= n ? n : m;
  d.nblocks = (M / m) * (N / n);
  d.T = (d.nn + kHT - 1) / kHT;
  d.ntiles = d.T * (d.T + 1) / 2;
  // row chunks: enough CTAs for two waves of 5 per SM, chunks of >= 256 rows
  d.chunk_rows = 256;
  const long long waves = 10LL * sm_count();
  while (d.chunk_rows < d.mm &&
         (long long)d.ntiles * d.nblocks * ((d.mm + 2 * d.chunk_rows - 1) / (2 * d.chunk_rows)) >= waves)
    d.chunk_rows *= 2;
  d.chunks = (d.mm + d.chunk_rows - 1) / d.chunk_rows;
  return d;
}


__device__ __forceinline__ size_t huge_off(const BlockGeom& g, int i, int c) {
  return g.transposed() ? g.offset(c, i) : g.offset(i, c);
}

__device__ __forceinline__ float huge_load(const ScaleLaunch& a, size_t off) {
  float v = a.A1[off];
  if (a.A2) v += a.A2[off];
  return v;
}

// ---------------------------------------------------------------------------
// 1. Gram partial sums: tile t of the lower triangle over one row chunk.
// ---------------------------------------------------------------------------
template <bool ST>
__global__ void __launch_bounds__(kHThreads, 4)
huge_gram_kernel(ScaleLaunch a, float* __restrict__ part, int chunk_rows, int chunks) {
  __shared__ __align__(16) float As[32][kHT + 4];
  __shared__ __align__(16) float Bs[32][kHT + 4];
  const int t = blockIdx.x, chunk = blockIdx.y, b = blockIdx.z;
  int ta, tc;
  tile_of(t, &ta, &tc);
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const int a0 = ta * kHT, c0 = tc * kHT;
  const int r_begin = chunk * chunk_rows;
  const int r_end = min(mm, r_begin + chunk_rows);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
  for (int r0 = r_begin; r0 < r_end; r0 += 32) {
#pragma unroll
    for (int j = 0; j < (32 * kHT) / kHThreads; ++j) {
      const int e = tid + j * kHThreads;
      const int rr = e / kHT, cc = e - rr * kHT;
      const int i = r0 + rr;
      float va = 0.f, vb = 0.f;
      if (i < r_end) {
        if (a0 + cc < nn) va = huge_load(a, huge_off(g, i, a0 + cc));
        if (c0 + cc < nn) vb = (ta == tc) ? va : huge_load(a, huge_off(g, i, c0 + cc));
      }
      As[rr][cc] = va;
      Bs[rr][cc] = vb;
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[rr][ty * 4]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[rr][tx * 4]);
      const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(av[x], bv[y], acc[x][y]);
    }
    __syncthreads();
  }
  const int ntiles = gridDim.x;
  float* dst = part + (((size_t)b * chunks + chunk) * ntiles + t) * (kHT * kHT);
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) dst[(ty * 4 + x) * kHT + tx * 4 + y] = acc[x][y];
}

// Sum of the chunk partials in chunk order; G_b written as a full square of
// order np (nn rounded up to the tile; the tiles are zero beyond nn), and per
// tile: the diagonal sum and the sum of squares (off-diagonal tiles twice).
// The mirrored tile goes through shared memory, so that both triangles are
// written as row segments (1024 wide: 15 -> 10 us).  The CTA that finishes
// a block last adds the tile sums in tile order to trace(G) and ||G||_F,
// takes the zero-rank shortcut trace(G) <= tau^2 (the trace bounds
// lambda_max) and resets the block's state (a launch of its own before).
__global__ void __launch_bounds__(kHThreads)
huge_gram_finish_kernel(const float* __restrict__ part, float* __restrict__ G, float* tstat, int np,
                        int chunks, HugeBlock* __restrict__ hb, int* __restrict__ arrived, float thr) {
  __shared__ __align__(16) float Ts[kHT][kHT + 4];
  __shared__ double red[2][kHThreads / 32];
  __shared__ int slast;
  const int t = blockIdx.x, b = blockIdx.y, ntiles = gridDim.x;
  int ta, tc;
  tile_of(t, &ta, &tc);
  const int tid = threadIdx.x;
  float* Gb = G + (size_t)b * np * np;
  const float4* src = reinterpret_cast<const float4*>(part + ((size_t)b * chunks * ntiles + t) * (kHT * kHT));
  const size_t cstep = (size_t)ntiles * (kHT * kHT / 4);
  constexpr int PER = kHT * kHT / 4 / kHThreads;
  float4 s[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) s[j] = src[tid + j * kHThreads];
  for (int c = 1; c < chunks; ++c) {
    float4 v[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) v[j] = src[c * cstep + tid + j * kHThreads];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      s[j].x += v[j].x;
      s[j].y += v[j].y;
      s[j].z += v[j].z;
      s[j].w += v[j].w;
    }
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = tid + j * kHThreads, x = e / (kHT / 4), y = 4 * (e % (kHT / 4));
    *reinterpret_cast<float4*>(&Ts[x][y]) = s[j];
  }
  __syncthreads();
  float dsum = 0.f, sq = 0.f;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = tid + j * kHThreads, x = e / (kHT / 4), y = 4 * (e % (kHT / 4));
    float v[4] = {s[j].x, s[j].y, s[j].z, s[j].w};
    if (ta == tc) {
      // diagonal tile: the lower half is authoritative
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (y + i > x) v[i] = Ts[y + i][x];
        sq += v[i] * v[i];
        if (y + i == x) dsum += v[i];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) sq += 2.f * v[i] * v[i];
      // mirrored tile: row y of it is column y of this one
      *reinterpret_cast<float4*>(Gb + (size_t)(tc * kHT + x) * np + ta * kHT + y) =
          make_float4(Ts[y][x], Ts[y + 1][x], Ts[y + 2][x], Ts[y + 3][x]);
    }
    *reinterpret_cast<float4*>(Gb + (size_t)(ta * kHT + x) * np + tc * kHT + y) =
        make_float4(v[0], v[1], v[2], v[3]);
  }
  dsum = warp_sum(dsum);
  sq = warp_sum(sq);
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = dsum;
    red[1][tid >> 5] = sq;
  }
  __syncthreads();
  float* ts = tstat + (size_t)b * ntiles * 2;
  if (tid == 0) {
    double d = 0.0, q = 0.0;
    for (int w = 0; w < kHThreads / 32; ++w) {
      d += red[0][w];
      q += red[1][w];
    }
    ts[2 * t] = (float)d;
    ts[2 * t + 1] = (float)q;
    __threadfence();
    slast = atomicAdd(arrived + b, 1) == ntiles - 1;
  }
  __syncthreads();
  if (!slast) return;
  __threadfence();
  double d = 0.0, q = 0.0;
  for (int i = tid; i < ntiles; i += kHThreads) {
    d += (double)__ldcg(ts + 2 * i);
    q += (double)__ldcg(ts + 2 * i + 1);
  }
  d = warp_sum_d(d);
  q = warp_sum_d(q);
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = d;
    red[1][tid >> 5] = q;
  }
  __syncthreads();
  if (tid == 0) {
    double dt = 0.0, qt = 0.0;
    for (int w = 0; w < kHThreads / 32; ++w) {
      dt += red[0][w];
      qt += red[1][w];
    }
    arrived[b] = 0;  // for the next call
    HugeBlock& h = hb[b];
    h.trace = (float)dt;
    h.gF = (float)sqrt(qt);
    h.status = (h.trace <= thr) ? kHsSkip : kHsIter;
    h.ku = 0;
    h.conv = 0;
    h.stop = 0;
    h.worst = 0.f;
    h.cert = kCertOpen;
    h.arrived = 0;
    h.orth_fail = 0;
    h.c = 0.f;
  }
}

// Start basis: deterministic pseudo-random columns (any full-rank start
// serves subspace iteration), the same for every block (rows r of a block
// at V + (b np + r) kHP, zero beyond nn), so that a block's start does not depend on its
// index.
__global__ void huge_init_basis_kernel(float* __restrict__ V, size_t total, int nn, int np) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)((e / kHP) % np);
    V[e] = r < nn ? huge_hash((uint32_t)r, (uint32_t)(e % kHP) + 0x51EDu) : 0.f;
  }
}

// ---------------------------------------------------------------------------
// 5. The outcome: Z' = sum over the pairs above tau of (1 - tau / sigma) (C u)
// u^T and W' = 2 Z' - A; blocks without such pairs get Z' = 0, W' = -A.  A
// CTA takes kHRebRows rows of C: every thread forms the partial products of
// its columns for all rows (one read of U serves all of them), the CTA sums
// them, and every thread rebuilds its columns.  Pairs go in groups of eight
// (one group for most blocks); the rows are read once per group and once
// more, from cache, for the output.  With a warp per four rows and 32 CTAs at
// 1024 rows, and V_f scaled by a one-CTA launch before it, this took 85 + 13
// us at 1024 x 1024.  The CTA of the first rows also reports the block.
// ---------------------------------------------------------------------------
constexpr int kHRebRows = 8;
constexpr int kHRebPairs = 8;
template <bool ST>
__global__ void __launch_bounds__(kHThreads)
huge_rebuild_kernel(ScaleLaunch a, const float* __restrict__ U, int np,
                    const HugeBlock* __restrict__ hb) {
  constexpr int R = kHRebRows, Q = kHRebPairs, NW = kHThreads / 32;
  __shared__ __align__(16) float Ps[NW][R * Q];
  __shared__ __align__(16) float Pf[kHK / Q][R * Q];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const HugeBlock& h = hb[b];
  const float thr = a.tau * a.tau;
  const int ku = h.status == kHsIter ? h.ku : 0;
  int k = 0, kend = 0;  // pairs above tau, end of their range
  for (int q = 0; q < ku; ++q)
    if (h.theta[q] > thr) {
      ++k;
      kend = q + 1;
    }
  if (blockIdx.x == 0 && tid == 0) {
    const bool skipped = h.status == kHsSkip;
    // certified: no other eigenvalue above tau^2, and the pairs kept have
    // small residuals (the certificate alone says nothing about them)
    const bool cert = skipped || (h.status == kHsIter && h.cert == kCertYes && h.conv);
    if (a.rank_out) a.rank_out[b] = k;
    if (a.cnt) {
      if (skipped) atomicAdd(a.cnt, 1ull);
      if (k == 0) atomicAdd(a.cnt + 1, 1ull);
      if (cert && !skipped) atomicAdd(a.cnt + 2, 1ull);
      if (!cert) atomicAdd(a.cnt + 4, 1ull);
    }
    if (a.nuc_acc && k > 0) {
      double t = 0.0;
      for (int q = 0; q < ku; ++q)
        if (h.theta[q] > thr) t += (double)fmaxf(sqrtf(h.theta[q]) - a.tau, 0.f);
      atomicAdd(a.nuc_acc, t);
    }
  }
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const int i0 = blockIdx.x * R;
  const float* Ub = U + (size_t)b * np * kHK;
  const int groups = (kend + Q - 1) / Q;
  for (int gq = 0; gq < groups; ++gq) {
    float acc[R * Q];
#pragma unroll
    for (int e = 0; e < R * Q; ++e) acc[e] = 0.f;
    for (int c = tid; c < nn; c += kHThreads) {
      float av[R];
#pragma unroll
      for (int r = 0; r < R; ++r) av[r] = i0 + r < mm ? huge_load(a, huge_off(g, i0 + r, c)) : 0.f;
      const float4* u4 = reinterpret_cast<const float4*>(Ub + (size_t)c * kHK + gq * Q);
      const float4 u0 = u4[0], u1 = u4[1];
      const float u[Q] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[r * Q + q] = fmaf(av[r], u[q], acc[r * Q + q]);
    }
    // the warp's sums of the 64 products by halving: lane l ends with the
    // products 2 l and 2 l + 1
    static_assert(R * Q == 64, "two products per lane");
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int e = 0; e < 2 * o; ++e) {
        const float keep = up ? acc[e + 2 * o] : acc[e], give = up ? acc[e] : acc[e + 2 * o];
        acc[e] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    }
    __syncthreads();
    Ps[warp][2 * lane] = acc[0];
    Ps[warp][2 * lane + 1] = acc[1];
    __syncthreads();
    if (tid < R * Q) {
      float t = 0.f;
      for (int w = 0; w < NW; ++w) t += Ps[w][tid];
      // f = 1 - tau / sigma for the pairs above tau, else 0
      const int q = gq * Q + tid % Q;
      const float th = q < ku ? h.theta[q] : 0.f;
      Pf[gq][tid] = th > thr ? t * fmaxf(1.f - a.tau / sqrtf(th), 0.f) : 0.f;
    }
  }
  __syncthreads();
  for (int c = tid; c < nn; c += kHThreads) {
    float z[R];
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = 0.f;
    for (int gq = 0; gq < groups; ++gq) {
      const float4* u4 = reinterpret_cast<const float4*>(Ub + (size_t)c * kHK + gq * Q);
      const float4 u0 = u4[0], u1 = u4[1];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 p0 = *reinterpret_cast<const float4*>(&Pf[gq][r * Q]);
        const float4 p1 = *reinterpret_cast<const float4*>(&Pf[gq][r * Q + 4]);
        z[r] = fmaf(p0.x, u0.x, z[r]);
        z[r] = fmaf(p0.y, u0.y, z[r]);
        z[r] = fmaf(p0.z, u0.z, z[r]);
        z[r] = fmaf(p0.w, u0.w, z[r]);
        z[r] = fmaf(p1.x, u1.x, z[r]);
        z[r] = fmaf(p1.y, u1.y, z[r]);
        z[r] = fmaf(p1.z, u1.z, z[r]);
        z[r] = fmaf(p1.w, u1.w, z[r]);
      }
    }
    // (all loads before the stores: Zout may be A1)
    float av[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
      av[r] = (a.Wout && i0 + r < mm) ? huge_load(a, huge_off(g, i0 + r, c)) : 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (i0 + r < mm) {
        const size_t off = huge_off(g, i0 + r, c);
        a.Zout[off] = z[r];
        if (a.Wout) a.Wout[off] = 2.f * z[r] - av[r];
      }
    }
  }
}


}  // namespace

static char* halign(char* p) { return (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255); }

size_t huge_workspace_bytes(int M, int N, int m, int n) {
  const HugeDims d = huge_dims(M, N, m, n);
  const size_t B = (size_t)d.nblocks, np = (size_t)d.T * kHT;
  size_t bytes = 0;
  bytes += sizeof(float) * B * d.chunks * d.ntiles * kHT * kHT;  // Gram partials
  bytes += sizeof(float) * B * np * np;                          // G
  bytes += sizeof(double) * B * cert_fpart_count(d.nn);
  bytes += 2 * sizeof(float) * B * d.ntiles;                     // tile sums
  bytes += (subspace_phases((int)np) ? 2 : 1) * sizeof(float) * B * np * kHP;  // V, W
  bytes += 2 * sizeof(float) * B * np * kHK;                     // U, What
  bytes += sizeof(HugeBlock) * B + sizeof(int) * B;
  bytes += 16 * 256;
  return bytes;
}

BigWorkspace carve_huge_workspace(void* base, int M, int N, int m, int n) {
  BigWorkspace w{};
  if (!base) return w;
  const HugeDims d = huge_dims(M, N, m, n);
  const size_t B = (size_t)d.nblocks, np = (size_t)d.T * kHT;
  char* p = halign((char*)base);
  auto take = [&](size_t bytes) {
    char* q = p;
    p = halign(p + bytes);
    return q;
  };
  w.part = (float*)take(sizeof(float) * B * d.chunks * d.ntiles * kHT * kHT);
  w.G = (float*)take(sizeof(float) * B * np * np);
  // the certificate matrices take no room of their own: the first lies over
  // the Gram partials, which are summed by then (np (np + 64) / 2 floats per
  // chunk), the second over G, which forming the first reads last
  w.Ma = w.part;
  w.Mb = w.G;
  w.fpart = (double*)take(sizeof(double) * B * cert_fpart_count(d.nn));
  w.tstat = (float*)take(2 * sizeof(float) * B * d.ntiles);
  w.V = (float*)take(sizeof(float) * B * np * kHP);
  if (subspace_phases((int)np)) w.Wv = (float*)take(sizeof(float) * B * np * kHP);
  w.U = (float*)take(sizeof(float) * B * np * kHK);
  w.GU = (float*)take(sizeof(float) * B * np * kHK);
  w.hb = take(sizeof(HugeBlock) * B);
  w.k = (int*)take(sizeof(int) * B);
  return w;
}

// Start basis of every block (start of a decomposition, or a fresh call).
cudaError_t reset_huge_basis(const BigWorkspace& w, int M, int N, int m, int n, cudaStream_t st) {
  if (!w.V) return cudaSuccess;
  const HugeDims d = huge_dims(M, N, m, n);
  const size_t total = (size_t)d.nblocks * d.T * kHT * kHP;
  const int grid = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  huge_init_basis_kernel<<<grid, 256, 0, st>>>(w.V, total, d.nn, d.T * kHT);
  if (cudaError_t e = cudaGetLastError()) return e;
  // the Gram kernels' arrival counters
  return cudaMemsetAsync(w.k, 0, sizeof(int) * (size_t)d.nblocks, st);
}

cudaError_t launch_huge(const ScaleLaunch& s, const BigWorkspace& ws, cudaStream_t st, Prof* prof,
                        cudaEvent_t after_gram) {
  const HugeDims d = huge_dims(s.M, s.N, s.m, s.n);
  if (d.nn > MSLLR_MAX_BLOCK_WIDTH || !ws.V) return cudaErrorInvalidValue;
#define PROF_BEFORE(kind) \
  if (prof)               \
    if (cudaError_t e_ = prof->before(st, kind)) return e_;
#define PROF_AFTER() \
  if (prof)          \
    if (cudaError_t e_ = prof->after(st)) return e_;
  HugeBlock* hb = (HugeBlock*)ws.hb;
  const float thr = s.tau * s.tau;
  const int B = d.nblocks, nn = d.nn, np = d.T * kHT;
  PROF_BEFORE(KK_GRAM)
  if (gram_tc_eligible(s) && !gram_fp32_forced()) {
    // tensor-core Gram (k_gram_tc.cu), partial sums in the same 64 x 64 tile
    // layout and chunks, reduced below
    if (cudaError_t e_ = launch_gram_tc(s, nullptr, ws.part, d.chunks, B, d.ntiles, d.chunk_rows,
                                        1, st))
      return e_;
  } else if (s.fw || s.rows)
    huge_gram_kernel<true><<<dim3(d.ntiles, d.chunks, B), kHThreads, 0, st>>>(s, ws.part, d.chunk_rows,
                                                                              d.chunks);
  else
    huge_gram_kernel<false><<<dim3(d.ntiles, d.chunks, B), kHThreads, 0, st>>>(s, ws.part, d.chunk_rows,
                                                                               d.chunks);
  PROF_AFTER()
  PROF_BEFORE(KK_GRAM_REDUCE)
  huge_gram_finish_kernel<<<dim3(d.ntiles, B), kHThreads, 0, st>>>(ws.part, ws.G, ws.tstat, np,
                                                                   d.chunks, hb, ws.k, thr);
  PROF_AFTER()
  if (after_gram)
    if (cudaError_t e_ = cudaEventRecord(after_gram, st)) return e_;
  // subspace iteration: a first round (short when the grid does not move and
  // the basis carries over from the previous call), a second round for the
  // blocks whose Ritz residuals are still large
  const bool full = (s.m == launch_rows(s) && s.n == s.N);
  const bool warm = s.warm_start && (full || !s.shift);
  const int job_blocks = (launch_rows(s) / s.m) * (s.N / s.n);
  if (cudaError_t e_ = launch_subspace(ws.G, ws.V, ws.Wv, ws.U, ws.GU, nn, np, thr, warm ? 2 : 6,
                                       hb, B, job_blocks, st, prof))
    return e_;
  if (cudaError_t e_ = launch_cert(ws.G, ws.U, ws.GU, ws.Ma, ws.Mb, ws.fpart, hb, nn, B, s.err, st,
                                   prof))
    return e_;
  PROF_BEFORE(KK_REBUILD)
  const dim3 rgrid((d.mm + kHRebRows - 1) / kHRebRows, B);
  if (s.fw || s.rows) huge_rebuild_kernel<true><<<rgrid, kHThreads, 0, st>>>(s, ws.U, np, hb);
  else huge_rebuild_kernel<false><<<rgrid, kHThreads, 0, st>>>(s, ws.U, np, hb);
  PROF_AFTER()
#undef PROF_BEFORE
#undef PROF_AFTER
  return cudaGetLastError();
}

}  // namespace msllr

// Block SVT for wide blocks (64 < min(m, n) <= 256, or m*n > 8192), which
// includes the full-matrix scale of eq:bsvt.  Phases per scale:
//   1. gram_tiles: G_b = C_b^T C_b for every block, tiled 64x64 over the
//      lower triangle and split over row chunks (partial sums reduced in a
//      fixed order, so results are deterministic), stored packed;
//   2. eig (k_eig.cu): a cluster per block -- skip bound (Sec. 8), certified
//      zero rank or certified Lanczos eigenpairs of G_b, output V_b
//      diag(sqrt(f));
//   3. tridiag (k_tridiag.cu): the Householder path for the blocks step 2
//      could not certify;
//   4. rebuild: Z'_b = (C_b V_f) V_f^T, scattered through Shift_{-s}, with
//      the fused dual update W' = 2 Z' - A of eq:admm (warp per row for
//      ranks up to 8, row slabs above).
#include <math.h>
#include <stdlib.h>

#include "common.cuh"
#include "huge.cuh"
#include "internal.h"
#include "lanczos.cuh"
#include "symeig.cuh"

namespace msllr {

namespace {

constexpr int kTile = 64;       // Gram tile
constexpr int kChunk = 256;     // rows of C per Gram partial sum
constexpr int kGramThreads = 256;
constexpr int kEigMax = 256;
constexpr int kRebThreads = 256;
constexpr int kRebElems = 4096;  // rows-per-slab * nn
constexpr int kKC = 16;          // eigenvectors per rebuild step

struct BigDims {
  int mm, nn, nblocks, nbn, T, ntiles, chunks;
};

BigDims big_dims(int M, int N, int m, int n) {
  BigDims d;
  d.mm = m >= n ? m : n;
  d.nn = m >= n ? n : m;
  d.nbn = N / n;
  d.nblocks = (M / m) * (N / n);
  d.T = (d.nn + kTile - 1) / kTile;
  d.ntiles = d.T * (d.T + 1) / 2;
  d.chunks = (d.mm + kChunk - 1) / kChunk;
  return d;
}


// element (i, c) of C (mm x nn) -> global offset
__device__ __forceinline__ size_t c_offset(const BlockGeom& g, int i, int c) {
  return g.transposed() ? g.offset(c, i) : g.offset(i, c);
}

__device__ __forceinline__ float load_a(const ScaleLaunch& a, size_t off) {
  float v = a.A1[off];
  if (a.A2) v += a.A2[off];
  return v;
}

template <bool ST>
__global__ void __launch_bounds__(kGramThreads, 5)
gram_tiles_kernel(ScaleLaunch a, float* __restrict__ G, float* __restrict__ part, int chunks) {
  __shared__ __align__(16) float As[32][kTile + 4];
  __shared__ __align__(16) float Bs[32][kTile + 4];
  const int t = blockIdx.x, chunk = blockIdx.y, b = blockIdx.z;
  int ta = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while (((ta + 1) * (ta + 2)) / 2 <= t) ++ta;
  while ((ta * (ta + 1)) / 2 > t) --ta;
  const int tc = t - (ta * (ta + 1)) / 2;
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const int a0 = ta * kTile, c0 = tc * kTile;
  const int r_begin = chunk * kChunk;
  const int r_end = min(mm, r_begin + kChunk);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
  const bool has2 = a.A2 != nullptr, dg = ta == tc;
  constexpr int kPer = (32 * kTile) / kGramThreads;
  for (int r0 = r_begin; r0 < r_end; r0 += 32) {
    // predicated loads, all in flight before the sums are formed
    float xa[kPer], ya[kPer], xb[kPer], yb[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int e = tid + j * kGramThreads;
      const int rr = e / kTile, cc = e - rr * kTile;
      const int i = r0 + rr;
      const bool in = i < r_end, ina = in && a0 + cc < nn, inb = in && !dg && c0 + cc < nn;
      const size_t oa = c_offset(g, ina ? i : r_begin, ina ? a0 + cc : 0);
      const size_t ob = c_offset(g, inb ? i : r_begin, inb ? c0 + cc : 0);
      xa[j] = ina ? __ldg(a.A1 + oa) : 0.f;
      ya[j] = (ina && has2) ? __ldg(a.A2 + oa) : 0.f;
      xb[j] = inb ? __ldg(a.A1 + ob) : 0.f;
      yb[j] = (inb && has2) ? __ldg(a.A2 + ob) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int e = tid + j * kGramThreads;
      const int rr = e / kTile, cc = e - rr * kTile;
      const float va = xa[j] + ya[j];
      As[rr][cc] = va;
      Bs[rr][cc] = dg ? va : xb[j] + yb[j];
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
  if (chunks == 1) {
    float* Gb = G + (size_t)b * nn * nn;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int i = a0 + ty * 4 + x;
      if (i >= nn) continue;
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int j = c0 + tx * 4 + y;
        if (j <= i) Gb[(size_t)i * (i + 1) / 2 + j] = acc[x][y];
      }
    }
  } else {
    const int ntiles = gridDim.x;
    float* dst = part + (((size_t)b * chunks + chunk) * ntiles + t) * (kTile * kTile);
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) dst[(ty * 4 + x) * kTile + tx * 4 + y] = acc[x][y];
  }
}

__global__ void __launch_bounds__(256)
gram_reduce_kernel(const float* __restrict__ part, float* __restrict__ G, int nn, int ntiles,
                   int chunks) {
  const int t = blockIdx.x, b = blockIdx.y;
  int ta = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while (((ta + 1) * (ta + 2)) / 2 <= t) ++ta;
  while ((ta * (ta + 1)) / 2 > t) --ta;
  const int tc = t - (ta * (ta + 1)) / 2;
  const int per = (kTile * kTile) / gridDim.z;
  const int e0 = blockIdx.z * per;
  for (int e = e0 + threadIdx.x; e < e0 + per; e += blockDim.x) {
    const int x = e / kTile, y = e - x * kTile;
    const int i = ta * kTile + x, j = tc * kTile + y;
    if (i >= nn || j >= nn) continue;
    float s = 0.f;
    for (int c = 0; c < chunks; ++c)
      s += part[(((size_t)b * chunks + c) * ntiles + t) * (kTile * kTile) + e];
    if (j <= i) G[(size_t)b * nn * nn + (size_t)i * (i + 1) / 2 + j] = s;
  }
}

// Z' = (C V_f) V_f^T, W' = 2 Z' - A for blocks of rank k <= kRowK: one warp
// per row of C, a lane per 32nd column.  Row i: P = C_i V_f by lane partial
// sums and k warp reductions, Z'_i = P V_f^T; V_f (transposed) is staged once
// per CTA.  Every load of C and store of Z', W' is a warp-wide row segment.
constexpr int kRowK = 8;
constexpr int kRowsPerCta = 32;  // 8 warps x 4 rows: one wave at 4 CTAs per SM
// ST: spatio-temporal blocks; the 2-D instantiation knows fw = 0 at compile
// time, which keeps its index arithmetic in registers.
template <bool ST>
__global__ void __launch_bounds__(kRebThreads, 4)
rebuild_rows_kernel(ScaleLaunch a, const float* __restrict__ Yall, size_t ystride,
                    const int* __restrict__ kin) {
  __shared__ float Vt[kRowK * kEigMax];
  const int b = blockIdx.y;
  const int k = kin[b];
  if (k > kRowK) return;  // rebuild_kernel takes the block
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* Yb = Yall + (size_t)b * ystride;
  for (int i = tid; i < nn; i += kRebThreads)
    for (int q = 0; q < k; ++q) Vt[q * nn + i] = Yb[(size_t)i * nn + q];
  __syncthreads();
  constexpr int RPW = kRowsPerCta / (kRebThreads / 32);
  constexpr int CPL = kEigMax / 32;  // columns per lane
  const int row0 = blockIdx.x * kRowsPerCta + warp * RPW;
  // the next row's inputs are loaded while the current row is finished
  float nx[CPL];
#pragma unroll
  for (int t = 0; t < CPL; ++t) {
    const int c = lane + 32 * t;
    nx[t] = (row0 < mm && c < nn) ? load_a(a, c_offset(g, row0, c)) : 0.f;
  }
  for (int rr = 0; rr < RPW; ++rr) {
    const int i = row0 + rr;
    if (i >= mm) break;
    float av[CPL];
#pragma unroll
    for (int t = 0; t < CPL; ++t) {
      av[t] = nx[t];
      const int c = lane + 32 * t;
      nx[t] = (rr + 1 < RPW && i + 1 < mm && c < nn) ? load_a(a, c_offset(g, i + 1, c)) : 0.f;
    }
    float P[kRowK];
#pragma unroll
    for (int q = 0; q < kRowK; ++q) {
      P[q] = 0.f;
      if (q < k) {
#pragma unroll
        for (int t = 0; t < kEigMax / 32; ++t) {
          const int c = lane + 32 * t;
          if (c < nn) P[q] = fmaf(av[t], Vt[q * nn + c], P[q]);
        }
        P[q] = warp_sum(P[q]);
      }
    }
#pragma unroll
    for (int t = 0; t < kEigMax / 32; ++t) {
      const int c = lane + 32 * t;
      if (c < nn) {
        float z = 0.f;
#pragma unroll
        for (int q = 0; q < kRowK; ++q)
          if (q < k) z = fmaf(P[q], Vt[q * nn + c], z);
        const size_t off = c_offset(g, i, c);
        a.Zout[off] = z;
        if (a.Wout) a.Wout[off] = 2.f * z - av[t];
      }
    }
  }
}

// Z' = (C V_f) V_f^T for a slab of `rs` rows of C, W' = 2 Z' - A: blocks of
// rank above kRowK (Lanczos keeps up to 16 pairs, Householder any).  The CTAs
// stride over the (slab, block) items, so that a launch with nothing to do
// holds few SMs.
template <bool ST>
__device__ __forceinline__ void rebuild_slab(const ScaleLaunch& a, const float* __restrict__ Yall,
                                             size_t ystride, const int* __restrict__ kin, int rs,
                                             int slab, int b) {
  extern __shared__ float sm[];
  const int tid = threadIdx.x;
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const int r0 = slab * rs;
  const int rows = min(rs, mm - r0);
  const int k = kin[b];
  float* Cs = sm;                          // rows x nn
  float* Vs = Cs + rs * nn;                // kKC x (nn + 1): V_f chunk, transposed
  float* Ps = Vs + kKC * (nn + 1);         // rows x kKC
  const int ldv = nn + 1;
  const int nel = rows * nn;
#pragma unroll 4
  for (int e = tid; e < nel; e += kRebThreads) {
    const int i = e / nn, c = e - i * nn;
    Cs[e] = load_a(a, c_offset(g, r0 + i, c));
  }
  __syncthreads();
  constexpr int EL = kRebElems / kRebThreads;
  float acc[EL];
#pragma unroll
  for (int t = 0; t < EL; ++t) acc[t] = 0.f;
  const float* Yb = Yall + (size_t)b * ystride;
  for (int q0 = 0; q0 < k; q0 += kKC) {
    const int kc = min(kKC, k - q0);
    for (int e = tid; e < nn * kKC; e += kRebThreads) {
      const int i = e / kKC, j = e - i * kKC;
      Vs[j * ldv + i] = j < kc ? Yb[(size_t)i * nn + q0 + j] : 0.f;
    }
    __syncthreads();
    for (int e = tid; e < rows * kKC; e += kRebThreads) {
      const int i = e / kKC, j = e - i * kKC;
      const float* crow = Cs + i * nn;
      const float* vrow = Vs + j * ldv;
      float t0 = 0.f, t1 = 0.f, t2 = 0.f, t3 = 0.f;
      int c = 0;
      for (; c + 3 < nn; c += 4) {
        t0 = fmaf(crow[c], vrow[c], t0);
        t1 = fmaf(crow[c + 1], vrow[c + 1], t1);
        t2 = fmaf(crow[c + 2], vrow[c + 2], t2);
        t3 = fmaf(crow[c + 3], vrow[c + 3], t3);
      }
      for (; c < nn; ++c) t0 = fmaf(crow[c], vrow[c], t0);
      Ps[e] = (t0 + t1) + (t2 + t3);
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < EL; ++t) {
      const int e = tid + t * kRebThreads;
      if (e < nel) {
        const int i = e / nn, c = e - i * nn;
        float z = acc[t];
#pragma unroll
        for (int j = 0; j < kKC; ++j) z = fmaf(Ps[i * kKC + j], Vs[j * ldv + c], z);
        acc[t] = z;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int t = 0; t < EL; ++t) {
    const int e = tid + t * kRebThreads;
    if (e < nel) {
      const int i = e / nn, c = e - i * nn;
      const size_t off = c_offset(g, r0 + i, c);
      a.Zout[off] = acc[t];
      if (a.Wout) a.Wout[off] = 2.f * acc[t] - Cs[e];
    }
  }
}

template <bool ST>
__global__ void __launch_bounds__(kRebThreads)
rebuild_kernel(ScaleLaunch a, const float* __restrict__ Yall, size_t ystride,
               const int* __restrict__ kin, int rs, int slabs, int nblocks) {
  for (int w = blockIdx.x; w < slabs * nblocks; w += gridDim.x) {
    const int b = w / slabs;
    if (kin[b] <= kRowK) continue;  // rebuild_rows_kernel took the block
    rebuild_slab<ST>(a, Yall, ystride, kin, rs, w - b * slabs, b);
    __syncthreads();
  }
}

}  // namespace

// the thresholded eigenvectors of a block: nn x k, k <= nn
static size_t y_stride(int nn) { return ((size_t)nn * nn + 63) & ~(size_t)63; }

size_t big_workspace_bytes(int M, int N, int m, int n) {
  if (choose_path(m, n) == ScalePath::Huge) return huge_workspace_bytes(M, N, m, n);
  if (choose_path(m, n) != ScalePath::Big) return 0;
  const BigDims d = big_dims(M, N, m, n);
  size_t bytes = 0;
  bytes += sizeof(float) * (size_t)d.nblocks * d.nn * d.nn;  // G
  if (d.chunks > 1) bytes += sizeof(float) * (size_t)d.nblocks * d.chunks * d.ntiles * kTile * kTile;
  bytes += sizeof(float) * (size_t)d.nblocks * y_stride(d.nn);  // Y
  bytes += sizeof(int) * (size_t)d.nblocks;                      // k
  bytes += sizeof(float) * (size_t)d.nblocks * kBigWarm * d.nn;   // warm
  bytes += sizeof(int) * (size_t)d.nblocks;                      // kwarm
  bytes += 8 * 256;  // alignment slack for the carve below
  return bytes;
}

static char* align256(char* p) {
  return (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
}

BigWorkspace carve_big_workspace(void* base, int M, int N, int m, int n) {
  BigWorkspace w{};
  if (choose_path(m, n) == ScalePath::Huge) return carve_huge_workspace(base, M, N, m, n);
  if (!base || choose_path(m, n) != ScalePath::Big) return w;
  const BigDims d = big_dims(M, N, m, n);
  char* p = align256((char*)base);
  w.G = (float*)p;
  p = align256(p + sizeof(float) * (size_t)d.nblocks * d.nn * d.nn);
  if (d.chunks > 1) {
    w.part = (float*)p;
    p = align256(p + sizeof(float) * (size_t)d.nblocks * d.chunks * d.ntiles * kTile * kTile);
  }
  w.ystride = y_stride(d.nn);
  w.Y = (float*)p;
  p = align256(p + sizeof(float) * (size_t)d.nblocks * w.ystride);
  w.k = (int*)p;
  p = align256(p + sizeof(int) * (size_t)d.nblocks);
  w.warm = (float*)p;
  p = align256(p + sizeof(float) * (size_t)d.nblocks * kBigWarm * d.nn);
  w.kwarm = (int*)p;
  return w;
}

cudaError_t reset_warm_start(const BigWorkspace& w, int M, int N, int m, int n, cudaStream_t st) {
  if (choose_path(m, n) == ScalePath::Huge) return reset_huge_basis(w, M, N, m, n, st);
  if (!w.kwarm) return cudaSuccess;
  const BigDims d = big_dims(M, N, m, n);
  return cudaMemsetAsync(w.kwarm, 0, sizeof(int) * (size_t)d.nblocks, st);
}

// The FP32 CUDA-core Gram instead of the tensor-core one (MSLLR_GRAM_FP32=1;
// for comparisons), read once.
bool gram_fp32_forced() {
  static const bool v = [] {
    const char* e = getenv("MSLLR_GRAM_FP32");
    return e && e[0] && e[0] != '0';
  }();
  return v;
}

cudaError_t configure_big_kernels() {
  sm_count();  // cache the SM count outside any stream capture
  gram_fp32_forced();
  if (cudaError_t e0 = configure_gram_tc()) return e0;
  if (cudaError_t e1 = configure_cert()) return e1;
  if (cudaError_t e2 = configure_subspace()) return e2;
  if (cudaError_t e4 = configure_eig()) return e4;
  if (cudaError_t e3 = configure_tridiag()) return e3;
  cudaError_t e = cudaFuncSetAttribute(rebuild_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           100 * 1024);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(rebuild_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              100 * 1024);
}

// `after_gram` (optional) is recorded on `st` once the Gram kernels are
// enqueued, so that other streams can wait for the Gram phase to finish.
cudaError_t launch_big(const ScaleLaunch& s, const BigWorkspace& ws, cudaStream_t st, Prof* prof,
                       cudaEvent_t after_gram) {
  const BigDims d = big_dims(s.M, s.N, s.m, s.n);
  if (d.nn > kEigMax) return cudaErrorInvalidValue;
#define PROF_BEFORE(kind) \
  if (prof)               \
    if (cudaError_t e_ = prof->before(st, kind)) return e_;
#define PROF_AFTER() \
  if (prof)          \
    if (cudaError_t e_ = prof->after(st)) return e_;
  PROF_BEFORE(KK_GRAM)
  const dim3 ggrid(d.ntiles, d.chunks, d.nblocks);
  if (gram_tc_eligible(s) && !gram_fp32_forced()) {
    if (cudaError_t e_ = launch_gram_tc(s, ws.G, ws.part, d.chunks, d.nblocks, d.ntiles, kChunk,
                                        0, st))
      return e_;
  } else if (s.fw || s.rows) {
    gram_tiles_kernel<true><<<ggrid, kGramThreads, 0, st>>>(s, ws.G, ws.part, d.chunks);
  } else {
    gram_tiles_kernel<false><<<ggrid, kGramThreads, 0, st>>>(s, ws.G, ws.part, d.chunks);
  }
  PROF_AFTER()
  if (d.chunks > 1) {
    PROF_BEFORE(KK_GRAM_REDUCE)
    gram_reduce_kernel<<<dim3(d.ntiles, d.nblocks, 16), 256, 0, st>>>(ws.part, ws.G, d.nn,
                                                                      d.ntiles, d.chunks);
    PROF_AFTER()
  }
  if (after_gram)
    if (cudaError_t e_ = cudaEventRecord(after_gram, st)) return e_;
  PROF_BEFORE(KK_EIG)
  if (cudaError_t e_ = launch_eig(s, ws, d.nblocks, st)) return e_;
  PROF_AFTER()
  PROF_BEFORE(KK_EIG_FALLBACK)
  // up to 64 CTAs stride over the blocks: enough for scales where many blocks
  // need the Householder path, few idle SMs where almost none do
  const int fb_groups = s.skip_bound ? (d.nblocks < 32 ? d.nblocks : 32) : d.nblocks;
  if (cudaError_t e_ = launch_tridiag(s, ws, d.nblocks, fb_groups, st)) return e_;
  PROF_AFTER()
  const int rs = kRebElems / d.nn;
  const int slabs = (d.mm + rs - 1) / rs;
  const size_t smem = sizeof(float) * ((size_t)rs * d.nn + (size_t)(d.nn + 1) * kKC + (size_t)rs * kKC);
  PROF_BEFORE(KK_REBUILD)
  const dim3 rgrid((d.mm + kRowsPerCta - 1) / kRowsPerCta, d.nblocks);
  if (s.fw || s.rows) rebuild_rows_kernel<true><<<rgrid, kRebThreads, 0, st>>>(s, ws.Y, ws.ystride, ws.k);
  else rebuild_rows_kernel<false><<<rgrid, kRebThreads, 0, st>>>(s, ws.Y, ws.ystride, ws.k);
  PROF_AFTER()
  PROF_BEFORE(KK_REBUILD)
  const int slab_items = slabs * d.nblocks;
  const int nsm = sm_count();
  const int reb_grid = s.skip_bound ? (slab_items < nsm ? slab_items : nsm) : slab_items;
  if (s.fw || s.rows)
    rebuild_kernel<true><<<reb_grid, kRebThreads, smem, st>>>(s, ws.Y, ws.ystride, ws.k, rs, slabs,
                                                             d.nblocks);
  else
    rebuild_kernel<false><<<reb_grid, kRebThreads, smem, st>>>(s, ws.Y, ws.ystride, ws.k, rs, slabs,
                                                      d.nblocks);
  PROF_AFTER()
#undef PROF_BEFORE
#undef PROF_AFTER
  return cudaGetLastError();
}

}  // namespace msllr

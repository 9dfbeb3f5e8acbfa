// Certificate of blocks wider than 256 (Sec. 8): a proof that the deflated
// Gram matrix X = P G P has ||X||_2 < c, so that by Cauchy interlacing G has
// no eigenvalue above c besides the kept Ritz pairs.
//
// Repeated squaring on the 5th-generation tensor cores.  With M_0 = X / c
// rounded to FP16 and M_k = fl16(M_{k-1} M_{k-1}^T) (FP32 accumulation),
//   ||X / c||_2 <= ||M_0||_2 + e_0,   ||M_{k-1}||_2^2 <= ||M_k||_2 + e_k,
//   ||M_k||_2 <= ||M_k||_F,
// so the F-norm of level k bounds ||X||_2 through k square roots: a bound by
// the power sum (sum_i lambda_i^p)^{1/p} with p = 2^{k+1}, which exceeds
// lambda_max by at most the factor n^{1/p} (1.4 % at n = 1024, k = 8).  Most
// blocks are settled at k = 3 or 4, and the remaining launches return at
// once.  The error terms are worst-case bounds from the norms computed on
// the way:
//   rounding to FP16   2^-11 ||.||_F + n 2^-25  (normal + subnormal entries;
//     round to nearest errs by 2^-11 / (1 + 2^-11) at most, which leaves 2^-22
//     for the FP32 scaling by 1 / c)
//   accumulation       (n / 16 + 8) 2^-22 ||M_{k-1}||_F^2: every addition of
//     the running FP32 sum (one per 16-wide MMA step) errs by at most 2^-22
//     of sum_l |m_il m_jl| <= |m_i| |m_j| (truncating adders included; the
//     tensor core's adder is not documented: this is an assumption)
// They cost 0.5-1 % of c at n = 512-1024.
//
// Why not a Cholesky factorisation of c I - X: that is n/64 dependent panels
// of dependent columns (two launches per panel), and its backward-error
// margin is larger at these widths (1.8 % of c at n = 1024); the squarings are plain
// symmetric matrix products with no dependences inside a launch.
//
// power_kernel: one CTA per 128 x 128 tile of the lower triangle of
// M M^T (the mirrored tile is written from the same accumulator), operands
// staged by TMA (128-byte swizzle, three stages of 64 columns, 2 CTAs per
// SM), tcgen05.mma.kind::f16 issued by one thread, accumulator in TMEM.
// M is symmetric up to rounding and M M^T is formed, so both operands are
// row tiles of the same K-major array.
#include <cuda.h>
#include <cuda_fp16.h>
#include <math.h>

#include "common.cuh"
#include "huge.cuh"
#include "internal.h"

namespace msllr {

namespace {

constexpr int kCT = 128;                          // output tile
constexpr int kCK = 64;                           // columns per stage (128 bytes)
constexpr int kCStages = 3;
constexpr int kCTileBytes = kCT * kCK * 2;        // one operand tile: 16 KB
constexpr int kCStageBytes = 2 * kCTileBytes;
constexpr int kCThreads = 192;                    // producer, MMA and four epilogue warps
constexpr int kCSmem = 1024 + kCStages * kCStageBytes + 256;
constexpr uint32_t kCTmemCols = 128;
constexpr int kCPolls = 1 << 20;

__device__ __forceinline__ uint32_t c_smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool c_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kCPolls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (i >= 64) __nanosleep(64);
  }
  return false;
}

// K-major operand with the 128-byte swizzle: 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t c_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// kind::f16, D FP32, A and B FP16, both K-major, M = N = 128
constexpr uint32_t kCIdesc = (1u << 4) | ((uint32_t)(kCT >> 3) << 17) | ((uint32_t)(kCT >> 4) << 24);

__device__ __forceinline__ void c_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(d), "l"(ad), "l"(bd), "r"(kCIdesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void c_tma(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x,
                                      int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4, %5}], [%2];"
      :
      : "r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// Level `level` of block h is complete with squared F-norm f2: extend the
// chain of bounds and settle the block where possible.  n: matrix order
// (padding adds zeros only).
__device__ void settle_level(HugeBlock& h, int level, double f2, int n) {
  // partial sums ran in FP32 (128 terms): far inside the factor below
  const double F = sqrt(f2) * 1.0001;
  const double u16 = 1.0 / 2048.0, sub = n * 2.98023224e-8;
  const double prev = level > 0 ? h.fro[level - 1] * (1.0 + u16) + sub : 0.0;
  h.fro[level] = F;
  h.err[level] = u16 * F + sub + (level > 0 ? (n / 16 + 8) * 2.384185791e-7 * prev * prev : 0.0);
  // the F-norm of the computed (FP32) matrix of this level, its accumulation
  // error included, bounds the product of the level below
  double x = level > 0 ? F + (h.err[level] - u16 * F - sub) : F;
  for (int k = level - 1; k >= 0; --k) x = sqrt(x) + h.err[k];
  if (x < 1.0) h.cert = kCertYes;
  // ||M||_2 >= ||M||_F / sqrt(n): no further level can bring the bound below 1
  else if (!(F < 1.01 * sqrt((double)n))) h.cert = kCertNo;
}

// The squared F-norm partials of one level: every CTA stores its own, the
// last one to arrive adds them in tile order and settles the level.
__device__ void finish_level(HugeBlock& h, double* fp, int ntiles, int tile, double part, int level,
                             int n, int nthreads, double* sred, int* slast) {
  const int tid = threadIdx.x;
  if (tid == 0) {
    fp[tile] = part;
    __threadfence();
    *slast = atomicAdd(&h.arrived, 1) == ntiles - 1;
  }
  __syncthreads();
  if (!*slast) return;
  __threadfence();
  double t = 0.0;
  for (int i = tid; i < ntiles; i += nthreads) t += __ldcg(fp + i);
  t = warp_sum_d(t);
  if ((tid & 31) == 0) sred[tid >> 5] = t;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < nthreads / 32; ++w) s += sred[w];
    h.arrived = 0;
    settle_level(h, level, s, n);
  }
}

// M_0 = fl16(X / c), X = G - U What^T - What U^T = P G P, 64 x 64 tiles of
// the lower triangle and their mirror images; rows and columns beyond nn
// (up to np, a multiple of 64) are zero.
constexpr int kFT = 64;
constexpr int kFThreads = 256;
__global__ void __launch_bounds__(kFThreads)
cert_form_kernel(const float* __restrict__ G, const float* __restrict__ U,
                 const float* __restrict__ Wh, __half* __restrict__ M0, int nn, int np,
                 double* __restrict__ fpart, HugeBlock* __restrict__ hb) {
  // U and What of the tile's rows and columns, pair by pair
  __shared__ __align__(16) float Ui[kHK][kFT], Wi[kHK][kFT], Uj[kHK][kFT], Wj[kHK][kFT];
  __shared__ __align__(8) __half Xs[kFT][kFT + 4];
  __shared__ double sred[kFThreads / 32];
  __shared__ int slast;
  const int t = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  HugeBlock& h = hb[b];
  if (h.status != kHsIter) return;
  const float c = h.c;
  if (!(c > 0.f)) {
    if (t == 0 && tid == 0) h.cert = kCertNo;
    return;
  }
  const float ic = 1.f / c;
  const int ku = h.ku;
  int ta, tc;
  tile_of(t, &ta, &tc);
  const float* Ub = U + (size_t)b * np * kHK;
  const float* Wb = Wh + (size_t)b * np * kHK;
  if (ku > 0) {
    for (int e = tid; e < kFT * kHK; e += kFThreads) {
      const int x = e / kHK, q = e - x * kHK;
      Ui[q][x] = Ub[(size_t)(ta * kFT + x) * kHK + q];
      Wi[q][x] = Wb[(size_t)(ta * kFT + x) * kHK + q];
      Uj[q][x] = Ub[(size_t)(tc * kFT + x) * kHK + q];
      Wj[q][x] = Wb[(size_t)(tc * kFT + x) * kHK + q];
    }
    __syncthreads();
  }
  const float* Gb = G + (size_t)b * np * np;
  __half* Mb = M0 + (size_t)b * np * np;
  // a 4 x 4 register tile per thread: rows x0 .., columns y0 ..
  const int x0 = 4 * (tid >> 4), y0 = 4 * (tid & 15);
  float v[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 g4 = *reinterpret_cast<const float4*>(Gb + (size_t)(ta * kFT + x0 + i) * np + tc * kFT + y0);
    v[i][0] = g4.x;
    v[i][1] = g4.y;
    v[i][2] = g4.z;
    v[i][3] = g4.w;
  }
  for (int q = 0; q < ku; ++q) {
    const float4 ui = *reinterpret_cast<const float4*>(&Ui[q][x0]);
    const float4 wi = *reinterpret_cast<const float4*>(&Wi[q][x0]);
    const float4 uj = *reinterpret_cast<const float4*>(&Uj[q][y0]);
    const float4 wj = *reinterpret_cast<const float4*>(&Wj[q][y0]);
    const float uiv[4] = {ui.x, ui.y, ui.z, ui.w}, wiv[4] = {wi.x, wi.y, wi.z, wi.w};
    const float ujv[4] = {uj.x, uj.y, uj.z, uj.w}, wjv[4] = {wj.x, wj.y, wj.z, wj.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[i][j] = fmaf(-wiv[i], ujv[j], fmaf(-uiv[i], wjv[j], v[i][j]));
  }
  float f2 = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    union {
      __half h[4];
      uint2 u;
    } o;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float x = v[i][j] * ic;
      f2 = fmaf(x, x, f2);
      o.h[j] = __float2half_rn(x);
      Xs[y0 + j][x0 + i] = o.h[j];
    }
    *reinterpret_cast<uint2*>(Mb + (size_t)(ta * kFT + x0 + i) * np + tc * kFT + y0) = o.u;
  }
  __syncthreads();
  if (ta != tc) {
    // the mirrored tile, in row segments
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<uint2*>(Mb + (size_t)(tc * kFT + x0 + i) * np + ta * kFT + y0) =
          *reinterpret_cast<const uint2*>(&Xs[x0 + i][y0]);
  }
  f2 = warp_sum(f2);
  if ((tid & 31) == 0) sred[tid >> 5] = (double)f2;
  __syncthreads();
  double part = 0.0;
  if (tid == 0) {
    for (int w = 0; w < kFThreads / 32; ++w) part += sred[w];
    if (ta != tc) part *= 2.0;
  }
  __syncthreads();
  finish_level(h, fpart + (size_t)b * gridDim.x, gridDim.x, t, part, 0, nn, kFThreads, sred, &slast);
}

__global__ void __launch_bounds__(kCThreads, 2)
power_kernel(const __grid_constant__ CUtensorMap map, __half* __restrict__ out, int nn, int np,
             int level, double* __restrict__ fpart, HugeBlock* __restrict__ hb, int* err) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ double sred[kCThreads / 32];
  __shared__ int slast;
  const int t = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  HugeBlock& h = hb[b];
  if (h.status != kHsIter || h.cert != kCertOpen) return;
  int ti, tj;
  tile_of(t, &ti, &tj);
  const bool diag = ti == tj;
  const int ksteps = np / kCK;
  const uint32_t base = (c_smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + kCStages * kCStageBytes;  // full[], empty[], done, then the TMEM slot
  const uint32_t bar_done = bars + 16 * kCStages, slot = bar_done + 8;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
                 "r"(kCTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < 2 * kCStages + 1; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8 * s) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  uint32_t tmem;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem) : "r"(slot));

  bool ok = true;
  if (tid == 0) {
    // producer: A rows of tile row ti, B rows of tile row tj (the same tile
    // on the diagonal)
    int k = 0;
    for (; k < ksteps; ++k) {
      const int s = k % kCStages, round = k / kCStages;
      if (round > 0 && !c_wait(bars + 8 * (kCStages + s), (round - 1) & 1)) {
        ok = false;
        break;
      }
      const uint32_t full = bars + 8 * s, st = base + s * kCStageBytes;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full),
                   "r"(diag ? kCTileBytes : kCStageBytes)
                   : "memory");
      c_tma(st, &map, full, k * kCK, ti * kCT, b);
      if (!diag) c_tma(st + kCTileBytes, &map, full, k * kCK, tj * kCT, b);
    }
    // a wait ran out: the copies in flight land before the CTA leaves
    if (!ok)
      for (int q = k > kCStages ? k - kCStages : 0; q < k; ++q)
        c_wait(bars + 8 * (q % kCStages), (q / kCStages) & 1);
  } else if (warp == 1 && lane == 0) {
    for (int k = 0; k < ksteps; ++k) {
      const int s = k % kCStages, round = k / kCStages;
      if (!c_wait(bars + 8 * s, round & 1)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t st = base + s * kCStageBytes;
      const uint32_t sb = diag ? st : st + kCTileBytes;
#pragma unroll
      for (int kk = 0; kk < kCK / 16; ++kk)
        c_mma(tmem, c_desc(st + 32 * kk), c_desc(sb + 32 * kk), (k > 0 || kk > 0) ? 1u : 0u);
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              bars + 8 * (kCStages + s))
          : "memory");
    }
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_done)
        : "memory");
    ok = c_wait(bar_done, 0) && ok;
  }
  ok = __syncthreads_and(ok);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  float f2 = 0.f;
  if (ok && warp >= 2) {
    const int quad = warp & 3;  // TMEM lanes 32 quad ..
    const int i = ti * kCT + 32 * quad + lane;
    __half* Ob = out + (size_t)b * np * np;
    const uint32_t taddr = tmem + ((uint32_t)(32 * quad) << 16);
#pragma unroll 1
    for (int c = 0; c < kCT; c += 32) {
      uint32_t v[32];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
          "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
          "%28, %29, %30, %31}, [%32];\n\t"
          "tcgen05.wait::ld.sync.aligned;"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
            "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
            "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
            "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
            "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
            "=r"(v[31])
          : "r"(taddr + (uint32_t)c)
          : "memory");
      uint32_t p[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const float x = __uint_as_float(v[2 * e]), y = __uint_as_float(v[2 * e + 1]);
        f2 = fmaf(x, x, fmaf(y, y, f2));
        const __half2 hh = __floats2half2_rn(x, y);
        p[e] = *reinterpret_cast<const uint32_t*>(&hh);
      }
      const int j = tj * kCT + c;
      if (i < np && j < np) {
        // a row segment of 32 entries, and its mirror image
        uint4* dst = reinterpret_cast<uint4*>(Ob + (size_t)i * np + j);
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[e] = make_uint4(p[4 * e], p[4 * e + 1], p[4 * e + 2], p[4 * e + 3]);
        if (!diag) {
#pragma unroll
          for (int e = 0; e < 32; ++e)
            Ob[(size_t)(j + e) * np + i] =
                __ushort_as_half((unsigned short)(p[e >> 1] >> (16 * (e & 1))));
        }
      }
    }
  } else if (!ok && tid == 0 && err) {
    atomicOr(err, 1);
  }
  f2 = warp_sum(f2);
  if (lane == 0) sred[warp] = (double)f2;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kCTmemCols)
                 : "memory");
  double part = 0.0;
  if (tid == 0) {
    for (int w = 2; w < kCThreads / 32; ++w) part += sred[w];
    if (!diag) part *= 2.0;
    if (!ok) part = (double)INFINITY;  // the level settles as not certified
  }
  __syncthreads();
  finish_level(h, fpart + (size_t)b * gridDim.x, gridDim.x, t, part, level, nn, kCThreads, sred,
               &slast);
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                 const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                 const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// the driver's tensor-map encoder, looked up once per process
EncodeTiled encode_tiled() {
  static const EncodeTiled f = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult r;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return (EncodeTiled)p;
  }();
  return f;
}

cudaError_t cert_map(CUtensorMap* map, __half* M, int np, int B) {
  EncodeTiled enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)np, (cuuint64_t)np, (cuuint64_t)B};
  const cuuint64_t strides[2] = {(cuuint64_t)np * 2, (cuuint64_t)np * np * 2};
  const cuuint32_t box[3] = {kCK, kCT, 1}, one[3] = {1, 1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, M, dims, strides, box, one,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

size_t cert_fpart_count(int nn) {
  const size_t t = ((size_t)nn + kFT - 1) / kFT;
  return t * (t + 1) / 2;
}

cudaError_t configure_cert() {
  encode_tiled();
  return cudaFuncSetAttribute(power_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCSmem);
}

cudaError_t launch_cert(const float* G, const float* U, const float* Wh, void* Ma, void* Mb,
                        double* fpart, HugeBlock* hb, int nn, int B, int* err, cudaStream_t st,
                        Prof* prof) {
  const int np = (nn + 63) & ~63, tf = np / kFT, tc = (np + kCT - 1) / kCT;
  __half* m[2] = {(__half*)Ma, (__half*)Mb};
  CUtensorMap maps[2];
  for (int i = 0; i < 2; ++i)
    if (cudaError_t e = cert_map(&maps[i], m[i], np, B)) return e;
  if (prof)
    if (cudaError_t e = prof->before(st, KK_CERT)) return e;
  cert_form_kernel<<<dim3(tf * (tf + 1) / 2, B), kFThreads, 0, st>>>(G, U, Wh, m[0], nn, np, fpart,
                                                                     hb);
  if (prof)
    if (cudaError_t e = prof->after(st)) return e;
  for (int k = 1; k <= kCertLevels; ++k) {
    if (prof)
      if (cudaError_t e = prof->before(st, KK_CERT)) return e;
    power_kernel<<<dim3(tc * (tc + 1) / 2, B), kCThreads, kCSmem, st>>>(
        maps[(k - 1) & 1], m[k & 1], nn, np, k, fpart, hb, err);
    if (prof)
      if (cudaError_t e = prof->after(st)) return e;
  }
  return cudaGetLastError();
}

}  // namespace msllr

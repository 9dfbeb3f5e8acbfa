// Eigenpairs above tau^2 of the Gram matrices of blocks up to 256 wide on the
// wide-block route (eq:svt, Sec. 8), one cluster per block: the bounds that
// skip a block, Lanczos with full reorthogonalisation for the pairs (the
// steps of lanczos.cuh), and a certificate that no further eigenvalue lies
// above tau^2.  Blocks that this does not settle get ws.k = -1 and go to
// k_tridiag.cu.
//
// The whole symmetric G stays in registers: a cluster of two CTAs (one up to
// 128 wide) holds 128 rows per CTA, a thread 8 rows x 8 columns (warp: 8
// rows; lane: every 32nd column), so G x is 64 multiply-adds per thread, a
// 9-shuffle multi-reduction and one cluster barrier that exchanges the
// halves over distributed shared memory; the vector work of a Lanczos step is
// done by both CTAs alike.  The certificate squares the (deflated) matrix,
// rounded to FP16, on the tensor cores as k_cert_tc.cu does, with the same
// bounds; here both operands stay in shared memory and a CTA forms its 128
// rows of every level (tcgen05.mma M = 128, N = 256 out of one 128-byte
// swizzled copy of the matrix), which the CTAs exchange.
//
// What bounds it is the chain of dependent steps in a block.  In one CTA
// with the packed G in shared memory a Lanczos step took 9.9k cycles and a
// Cholesky certificate 135k (256 wide).
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "huge.cuh"
#include "internal.h"
#include "lanczos.cuh"
#include "symeig.cuh"

namespace cg = cooperative_groups;

namespace msllr {

cudaError_t set_phase_buffer_big(unsigned long long* p) {
  return cudaMemcpyToSymbol(g_phase_acc, &p, sizeof(p));
}

namespace {

constexpr int kENT = 512;    // threads per CTA
constexpr int kENW = kENT / 32;
constexpr int kERows = 128;  // rows per CTA
constexpr int kEMax = 256;
constexpr int kEK = lz_maxk(kEMax);  // Ritz pairs kept
constexpr int kEPolls = 1 << 20;

// dynamic shared memory: the FP16 matrix (its space first holds the Lanczos
// basis), Ritz vectors U and W = G U, Lanczos and eigenvalue scratch
__host__ __device__ constexpr int eig_matrix_bytes(int CL) { return CL * kERows * CL * kERows * 2; }
__host__ __device__ constexpr int eig_front_bytes(int CL) {
  return eig_matrix_bytes(CL) > kLzMaxJ * kERows * CL * 4 ? eig_matrix_bytes(CL)
                                                          : kLzMaxJ * kERows * CL * 4;
}
__host__ __device__ constexpr int eig_smem_bytes(int CL) {
  return 1024 + eig_front_bytes(CL) +
         4 * (2 * kEK * kERows * CL + 3 * kEMax + lz_scratch_floats(kEMax, kLzMaxJ) +
              6 * 64 + 4 * kENT + 64 + 4 * 64);
}

__device__ __forceinline__ uint32_t e_smem(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool e_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kEPolls; ++i) {
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
__device__ __forceinline__ uint64_t e_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// The distributed matrix of one block.
template <int CL>
struct RegGram {
  static constexpr int NC = 4 * CL, NV = kERows * CL;  // columns per lane, vector length
  float A[8][NC];
  int rank, lane, warp, r0;

  __device__ __forceinline__ void barrier() const {
    if constexpr (CL > 1) cg::this_cluster().sync();
    else __syncthreads();
  }
  template <class T>
  __device__ __forceinline__ T* other(T* p) const {
    if constexpr (CL > 1) return cg::this_cluster().map_shared_rank(p, rank ^ 1);
    else return p;
  }
  // y (its NV entries in both CTAs) = A x or |A| x; x is read before the
  // caller's next barrier().  The caller's barrier publishes y.
  template <bool ABS>
  __device__ __forceinline__ void mul(const float* x, float* y) const {
    float p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const float v = x[lane + 32 * k];
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = fmaf(ABS ? fabsf(A[i][k]) : A[i][k], v, p[i]);
    }
    const float t = sum8(p, lane);
    const int r = r0 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    if ((lane & 3) == 0) y[r] = t;
    if (CL > 1 && (lane & 3) == 1) other(y)[r] = t;
  }
  // sum over all entries of two vectors' products, the same in every warp
  __device__ __forceinline__ float dot(const float* x, const float* y) const {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) t = fmaf(x[lane + 32 * k], y[lane + 32 * k], t);
    return warp_sum(t);
  }
};

// w <- (I - Q Q^T) w twice over nq basis vectors (length NV each); h1, h2
// receive the passes' coefficients; returns |w|^2 (the same in every warp).
template <int CL>
__device__ __forceinline__ float eig_project(const RegGram<CL>& g, float* w, const float* Q, int nq, float* h1,
                             float* h2) {
  constexpr int NV = RegGram<CL>::NV;
  const int tid = threadIdx.x;
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    float* h = pass == 0 ? h1 : h2;
    for (int i = g.warp; i < nq; i += kENW) {
      const float t = g.dot(Q + i * NV, w);
      if (g.lane == 0) h[i] = t;
    }
    __syncthreads();
    if (tid < NV) {
      float v0 = w[tid], v1 = 0.f, v2 = 0.f, v3 = 0.f;
      int i = 0;
      for (; i + 3 < nq; i += 4) {
        v0 = fmaf(-h[i], Q[i * NV + tid], v0);
        v1 = fmaf(-h[i + 1], Q[(i + 1) * NV + tid], v1);
        v2 = fmaf(-h[i + 2], Q[(i + 2) * NV + tid], v2);
        v3 = fmaf(-h[i + 3], Q[(i + 3) * NV + tid], v3);
      }
      for (; i < nq; ++i) v0 = fmaf(-h[i], Q[i * NV + tid], v0);
      w[tid] = (v0 + v1) + (v2 + v3);
    }
    __syncthreads();
  }
  return g.dot(w, w);
}

// Certificate ||X||_2 < c for the X whose FP16 rounding of X / c the CTAs
// hold (own rows written and fenced, squared F-norm part f2 of the own rows
// before rounding): repeated squaring, see k_cert_tc.cu for the bounds.
// `fx`: four shared floats, `bar`: shared mbarrier, `phase`: its parity.
template <int CL>
__device__ __forceinline__ bool eig_power_cert(const RegGram<CL>& g, unsigned char* M, uint32_t tmem, uint32_t bar,
                               uint32_t& phase, float f2, int n, float* fx, float* red, int* err) {
  constexpr int NV = RegGram<CL>::NV, PANEL = NV * 128;  // 64 columns of all rows
  constexpr int CG = NV / 4;                              // columns per warp group of the epilogue
  const int tid = threadIdx.x, lane = g.lane, warp = g.warp;
  // own rows to the other CTA
  if constexpr (CL > 1) {
    __syncthreads();
    unsigned char* Mo = g.other(M);
    for (int e = tid; e < NV / 64 * kERows * 8; e += kENT) {
      const int p = e / (kERows * 8), o = p * PANEL + g.rank * kERows * 128 + (e - p * kERows * 8) * 16;
      *reinterpret_cast<uint4*>(Mo + o) = *reinterpret_cast<const uint4*>(M + o);
    }
  }
  float fro[kCertLevels + 1], er[kCertLevels + 1];
  const float u16 = 1.f / 2048.f, sub = (float)n * 2.98023224e-8f;
  for (int level = 0;; ++level) {
    // F-norm of the level (of the FP32 values), both CTAs' parts
    const float t = block_sum<kENT>(f2, red);
    if (tid == 0) {
      fx[2 * (level & 1) + g.rank] = t;
      if (CL > 1) g.other(fx)[2 * (level & 1) + g.rank] = t;
    }
    asm volatile("fence.proxy.async;" ::: "memory");
    g.barrier();  // the level's matrix and norm parts are in both CTAs
    float ff = fx[2 * (level & 1)];
    if (CL > 1) ff += fx[2 * (level & 1) + 1];
    const float F = sqrtf(ff) * 1.0001f;
    float acc = 0.f;
    if (level > 0) {
      float prev = 0.f;
#pragma unroll
      for (int k = 0; k < kCertLevels; ++k)
        if (k == level - 1) prev = fro[k] * (1.f + u16) + sub;
      acc = (float)(n / 16 + 8) * 2.384186e-7f * prev * prev;
    }
    float x = F + acc;
#pragma unroll
    for (int k = kCertLevels; k >= 0; --k) {
      if (k == level) {
        fro[k] = F;
        er[k] = u16 * F + sub + acc;
      } else if (k < level) {
        x = sqrtf(x) * 1.000001f + er[k];
      }
    }
    if (x < 1.f) return true;
    // ||M||_2 >= ||M||_F / sqrt(n): no further level can settle it
    if (level == kCertLevels || !(F < 1.01f * sqrtf((float)n))) return false;
    // the next level: this CTA's 128 rows of M M^T
    if (tid == 0) {
      asm volatile("fence.proxy.async;" ::: "memory");
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      constexpr uint32_t idesc =
          (1u << 4) | ((uint32_t)(NV >> 3) << 17) | ((uint32_t)(kERows >> 4) << 24);
      const uint32_t base = e_smem(M);
#pragma unroll 1
      for (int p = 0; p < NV / 64; ++p) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t ad = e_desc(base + p * PANEL + g.rank * kERows * 128 + 32 * kk);
          const uint64_t bd = e_desc(base + p * PANEL + 32 * kk);
          const uint32_t accum = (p > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n\t.reg .pred p;\n\t"
              "setp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
              :
              : "r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
              : "memory");
        }
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
          : "memory");
    }
    bool ok = e_wait(bar, phase);
    phase ^= 1u;
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    g.barrier();  // both CTAs have read the level
    f2 = 0.f;
    if (ok) {
      const int quad = warp & 3, cg0 = CG * (warp >> 2);
      const int r = g.rank * kERows + 32 * quad + lane;
      unsigned char* Mo = g.other(M);
#pragma unroll 1
      for (int c = 0; c < CG; c += 32) {
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
            : "r"(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(cg0 + c))
            : "memory");
        const int col = cg0 + c;
        const int o = (col >> 6) * PANEL + r * 128, ch = (col & 63) >> 3;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          uint32_t p[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float a = __uint_as_float(v[8 * e + 2 * i]), b = __uint_as_float(v[8 * e + 2 * i + 1]);
            f2 = fmaf(a, a, fmaf(b, b, f2));
            const __half2 hh = __floats2half2_rn(a, b);
            p[i] = *reinterpret_cast<const uint32_t*>(&hh);
          }
          const uint4 u = make_uint4(p[0], p[1], p[2], p[3]);
          const int oo = o + (((ch + e) ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(M + oo) = u;
          if (CL > 1) *reinterpret_cast<uint4*>(Mo + oo) = u;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    } else {
      f2 = INFINITY;  // the level settles as not certified, in both CTAs
      if (tid == 0 && err) atomicOr(err, 1);
    }
  }
}

// Power steps route only: a block whose Rayleigh quotient comes this close
// to tau^2 goes straight to Lanczos (its zero-rank certificate would most
// likely fail).
constexpr float kZeroTry = 0.85f;

template <int CL>
__global__ void __launch_bounds__(kENT, 1)
eig_cluster_kernel(ScaleLaunch a, const float* __restrict__ Gall, BigWorkspace ws) {
  extern __shared__ unsigned char smraw[];
  constexpr int NT = kENT, NV = RegGram<CL>::NV, NC = RegGram<CL>::NC, K = kEK;
  __shared__ __align__(8) uint64_t bar_s;
  __shared__ uint32_t tmem_s;
  __shared__ float fx[4];
  const int b = blockIdx.x / CL, tid = threadIdx.x;
  const int n = a.m >= a.n ? a.n : a.m;
  const float* Gg = Gall + (size_t)b * n * n;
  unsigned char* M = smraw + ((1024u - (e_smem(smraw) & 1023u)) & 1023u);
  float* Q = reinterpret_cast<float*>(M);
  float* U = reinterpret_cast<float*>(M + eig_front_bytes(CL));  // U[q NV + r]
  float* W = U + K * NV;
  float* xv = W + K * NV;
  // G x, two buffers in turn: the next product's remote writes then need no
  // barrier of their own
  float* wb[2] = {xv + kEMax, xv + 2 * kEMax};
  int turn = 0;
  LzScratch z;
  lz_bind<NT>(z, xv + 3 * kEMax, kEMax, kLzMaxJ);
  EigScratch s;
  s.d = xv + 3 * kEMax + lz_scratch_floats(kEMax, kLzMaxJ);
  s.e = s.d + 64;
  s.e2 = s.e + 64;
  s.lam = s.e2 + 64;
  s.shf = s.lam + 64;
  s.clus = reinterpret_cast<int*>(s.shf + 64);
  s.lo = reinterpret_cast<float*>(s.clus + 64);
  s.hi = s.lo + NT;
  s.xs = s.hi + NT;
  s.cnt = reinterpret_cast<int*>(s.xs + NT);
  s.red = reinterpret_cast<float*>(s.cnt + NT);
  PHASE_INIT();
  RegGram<CL> g;
  g.rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  g.lane = tid & 31;
  g.warp = tid >> 5;
  g.r0 = kERows * g.rank + 8 * g.warp;
  const int lane = g.lane, warp = g.warp;
  const uint32_t bar = e_smem(&bar_s);
  constexpr uint32_t kCols = NV;  // TMEM columns: the FP32 accumulator
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     e_smem(&tmem_s)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the packed triangle through shared memory (rows and columns of it are
  // read on distinct banks: the triangular numbers are a permutation mod 32)
  {
    float* T = reinterpret_cast<float*>(M);
    const int ntri = n * (n + 1) / 2;
    if ((ntri & 3) == 0 && ((reinterpret_cast<uintptr_t>(Gg) & 15) == 0)) {
      const float4* src = reinterpret_cast<const float4*>(Gg);
      float4* dst = reinterpret_cast<float4*>(T);
#pragma unroll 4
      for (int e = tid; e < ntri / 4; e += NT) dst[e] = __ldg(src + e);
    } else {
#pragma unroll 4
      for (int e = tid; e < ntri; e += NT) T[e] = __ldg(Gg + e);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const int r = g.r0 + i, c = lane + 32 * k;
        const int hi = max(r, c), lo = min(r, c);
        g.A[i][k] = hi < n ? T[hi * (hi + 1) / 2 + lo] : 0.f;
      }
  }
  float tr = 0.f;
  for (int i = tid; i < n; i += NT) tr += reinterpret_cast<const float*>(M)[i * (i + 1) / 2 + i];
  tr = block_sum<NT>(tr, s.red);
  for (int e = tid; e < kEMax; e += NT) xv[e] = 1.f;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  g.barrier();  // (also: the other CTA runs before its memory is written)
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_s;
  uint32_t phase = 0u;
  PHASE(3, 0);
  const float thr = a.tau * a.tau;
  // trace and Gershgorin bounds of lambda_max(G)
  auto next = [&] {
    turn ^= 1;
    return wb[turn];
  };
  float rs = 0.f;
  {
    float* wv = next();
    g.template mul<true>(xv, wv);
    g.barrier();
    for (int e = tid; e < n; e += NT) rs = fmaxf(rs, wv[e]);
  }
  rs = block_max<NT>(rs, s.red);
  const float gbound = fminf(tr, rs);
  double fl = n + fl_symv(n);
  const bool full = (a.m == launch_rows(a) && a.n == a.N);
  const int kwarm = (a.warm_start && (full || !a.shift)) ? min(ws.kwarm[b], kBigWarm) : 0;
  const float* warm = ws.warm + (size_t)b * kBigWarm * n;
  bool skipped = false, lanczos_ok = false;
  int k = -1, ku = 0;
  // FP16 of the register matrix / c into the own rows of M; the thread's part
  // of the squared F-norm
  auto stage = [&](float c) {
    const float ic = 1.f / c;
    float f2 = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = g.r0 + i;
#pragma unroll
      for (int kk = 0; kk < NC; ++kk) {
        const int col = lane + 32 * kk;
        const float v = g.A[i][kk] * ic;
        f2 = fmaf(v, v, f2);
        *reinterpret_cast<__half*>(M + (col >> 6) * (NV * 128) + r * 128 +
                                   ((((col & 63) >> 3) ^ (r & 7)) << 4) + (col & 7) * 2) =
            __float2half_rn(v);
      }
    }
    return f2;
  };
  if (a.skip_bound) {
    if (gbound <= thr) {
      skipped = true;
      k = 0;
    } else if (kwarm == 0) {
      // up to three power steps from a pseudo-random vector
      for (int e = tid; e < kEMax; e += NT) xv[e] = e < n ? lz_hash(0xC0FFEEu, e) + 1.5f : 0.f;
      __syncthreads();
      float nrm = sqrtf(g.dot(xv, xv)), rq = 0.f;
      int steps = 0;
      for (int it = 0; it < 3; ++it) {
        steps = it + 1;
        __syncthreads();
        if (tid < NV) xv[tid] /= nrm;
        __syncthreads();
        float* wv = next();
        g.template mul<false>(xv, wv);
        g.barrier();
        rq = g.dot(xv, wv);
        nrm = sqrtf(g.dot(wv, wv));
        if (rq > kZeroTry * thr || !(nrm > 0.f)) break;
        __syncthreads();
        if (tid < NV) xv[tid] = wv[tid];
      }
      fl += steps * (fl_symv(n) + 4.0 * n);
      PHASE(3, 6);
      // certified lambda_max(G) < tau^2
      if (rq <= kZeroTry * thr) {
        const float f2 = stage(thr);
        if (eig_power_cert<CL>(g, M, tmem, bar, phase, f2, n, fx, s.red, a.err)) {
          skipped = true;
          k = 0;
        }
        PHASE(3, 7);
      }
      g.barrier();
    }
    if (k < 0) {
      // Lanczos, see lanczos.cuh
      const float thr_keep = 0.95f * thr;
      const uint32_t seed = 0x1234567u + 977u * job_block(a, b);
      if (tid < NV) {
        float v = 0.f;
        if (tid < n) {
          for (int i = 0; i < kwarm; ++i) v += warm[(size_t)i * n + tid] * (1.f + 0.25f * i);
          v += 1e-3f * lz_hash(seed, tid);
        }
        xv[tid] = v;
      }
      __syncthreads();
      const float inrm = 1.f / sqrtf(g.dot(xv, xv));
      if (tid < NV) Q[tid] = xv[tid] * inrm;
      g.barrier();
      const int jmax = min(n, kLzMaxJ), jmin = min(jmax, kwarm > 0 ? kwarm + 3 : 8);
      int J = 0, kr = -1;
      uint32_t restart = 1;
      bool many = false;
      PHASE(4, 6);
      for (int j = 0; j < jmax; ++j) {
        float* wv = next();
        g.template mul<false>(Q + j * NV, wv);
        g.barrier();
        PHASE(4, 7);
        float bt = sqrtf(eig_project<CL>(g, wv, Q, j + 1, z.h, z.h + kLzMaxJ));
        if (tid == 0) {
          z.alpha[j] = z.h[j] + z.h[kLzMaxJ + j];
          z.beta[j] = bt;
        }
        PHASE(4, 9);
        J = j + 1;
        if (J == n) break;  // Q spans everything: T_J is similar to G
        if (J < jmax) {
          if (!(bt > kLzBreak * gbound)) {
            // breakdown: an invariant subspace was found; continue from a
            // random direction orthogonal to it
            __syncthreads();
            if (tid < NV) wv[tid] = tid < n ? lz_hash(seed + 7919u * restart, tid) : 0.f;
            ++restart;
            __syncthreads();
            const float bn = sqrtf(eig_project<CL>(g, wv, Q, j + 1, z.h, z.h + kLzMaxJ));
            if (!(bn > 0.f)) break;
            if (tid == 0) z.beta[j] = 0.f;
            bt = bn;
          }
          const float ib = 1.f / bt;
          __syncthreads();
          if (tid < NV) Q[(j + 1) * NV + tid] = wv[tid] * ib;
          __syncthreads();
        }
        PHASE(4, 10);
        if (J >= jmin && ((J - jmin) % 4 == 0 || J == jmax)) {
          // converged when every kept Ritz pair has |beta_J y_{J-1}| small
          kr = lz_ritz<NT, K>(J, thr_keep, z, s);
          PHASE(4, 11);
          if (kr > K) {
            many = true;
            break;
          }
          bool conv = true;
          const float bJ = z.beta[J - 1];
          // (many pairs: each adds its share of the error)
          const float tol = kr > 8 ? 1e-6f : 1e-5f;
          for (int q = 0; q < kr; ++q)
            if (fabsf(bJ * z.ty[(J - 1) * K + q]) > tol * fmaxf(s.lam[0], thr)) conv = false;
          if (conv) break;
          kr = -1;
        }
      }
      __syncthreads();
      if (kr < 0 && !many) {
        kr = lz_ritz<NT, K>(J, thr_keep, z, s);
        // pairs that jmax steps did not settle go to the Householder path
        // (the certificate alone admits a residual of some per cent of tau^2)
        many = kr > K || (J == jmax && J < n && kr > 0);
      }
      fl += fl_lanczos(n, J, many ? 0 : kr);
      PHASE(3, 1);
      if (!many) {
        ku = kr;
        // U = Q_J Y, W = G U
        for (int e = tid; e < ku * NV; e += NT) {
          const int q = e / NV, r = e - q * NV;
          float v = 0.f;
          for (int j = 0; j < J; ++j) v = fmaf(Q[j * NV + r], z.ty[j * K + q], v);
          U[e] = v;
        }
        g.barrier();  // (W of both CTAs is free)
        for (int q = 0; q < ku; ++q) g.template mul<false>(U + q * NV, W + q * NV);
        g.barrier();
        PHASE(4, 12);
        // B = U^T W, residuals |W_q - B_qq U_q|^2: a warp per row of B
        for (int p = warp; p < ku; p += kENW) {
          float bpp = 0.f;
          for (int q = 0; q < ku; ++q) {
            const float t = g.dot(U + p * NV, W + q * NV);
            if (q == p) bpp = t;
            if (lane == 0) z.Bm[p * K + q] = t;
          }
          float rr = 0.f;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const int e = p * NV + lane + 32 * c;
            const float d = W[e] - bpp * U[e];
            rr = fmaf(d, d, rr);
          }
          rr = warp_sum(rr);
          if (lane == 0) z.h[p] = rr;
        }
        __syncthreads();
        // kept pairs: Rayleigh quotients, count above thr; pairs above thr
        // first
        float rho = 0.f, wsum = 0.f;
        int kk = 0;
        bool ordered = true;
        for (int q = 0; q < ku; ++q) {
          rho += z.h[q];
          const float th = z.Bm[q * K + q];
          wsum = fmaf(0.25f * th, th, wsum);
          kk += th > thr;
          if (q > 0 && th > thr && !(z.Bm[(q - 1) * K + (q - 1)] > thr)) ordered = false;
        }
        rho = sqrtf(rho);
        // the pairs above tau^2 may be off by 2 rho (see lanczos.cuh).  gbound is
        // the trace or the largest row sum; What_q = W_q - U sym(B)_q / 2 has
        // half of W_q's part along U and the rest, so ||What||_F^2 <= sum
        // theta_q^2 / 4 + rho^2
        const float c0 = cert_bound(thr, gbound, ku, fmaf(rho, rho, wsum)) - 2.f * rho;
        if (ordered && c0 > 0.f) {
          // What = W - U sym(B) / 2 in place (a thread owns a row), then A <-
          // P G P = A - U What^T - What U^T
          if (tid < NV) {
            float u[K];
#pragma unroll
            for (int p = 0; p < K; ++p) u[p] = p < ku ? U[p * NV + tid] : 0.f;
            for (int q = 0; q < ku; ++q) {
              float w = W[q * NV + tid];
#pragma unroll
              for (int p = 0; p < K; ++p)
                if (p < ku) w = fmaf(-0.25f * (z.Bm[p * K + q] + z.Bm[q * K + p]), u[p], w);
              W[q * NV + tid] = w;
            }
          }
          __syncthreads();
          for (int q = 0; q < ku; ++q) {
            float uc[NC], wc[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              uc[c] = U[q * NV + lane + 32 * c];
              wc[c] = W[q * NV + lane + 32 * c];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float ur = U[q * NV + g.r0 + i], wr = W[q * NV + g.r0 + i];
#pragma unroll
              for (int c = 0; c < NC; ++c)
                g.A[i][c] = fmaf(-wr, uc[c], fmaf(-ur, wc[c], g.A[i][c]));
            }
          }
          const float f2 = stage(c0);
          fl += fl_deflate(n, ku);
          PHASE(3, 5);
          if (eig_power_cert<CL>(g, M, tmem, bar, phase, f2, n, fx, s.red, a.err)) {
            k = kk;
            lanczos_ok = true;
          }
          PHASE(3, 8);
        }
      }
    }
  }
  if (lanczos_ok && g.rank == 0) {
    // keep the Ritz vectors for the next call's warm start
    const int kw = min(ku, kBigWarm);
    float* wdst = ws.warm + (size_t)b * kBigWarm * n;
    for (int e = tid; e < n * kw; e += NT) {
      const int q = e / n, r = e - q * n;
      wdst[e] = U[q * NV + r];
    }
    if (tid == 0) ws.kwarm[b] = kw;
    // V_f (row-major, ld n) for the rebuild
    float* Y = ws.Y + (size_t)b * ws.ystride;
    for (int e = tid; e < n * k; e += NT) {
      const int i = e / k, q = e - i * k;
      const float sig = sqrtf(z.Bm[q * K + q]);
      Y[(size_t)i * n + q] = U[q * NV + i] * sqrtf(fmaxf(1.f - a.tau / sig, 0.f));
    }
  }
  if (tid == 0 && g.rank == 0) {
    if (a.cnt) atomicAdd(a.cnt + 5, (unsigned long long)fl);
    // k < 0: not settled here; tridiag_kernel takes the block
    ws.k[b] = k;
    if (k < 0) {
      if (ws.kwarm) ws.kwarm[b] = 0;
    } else {
      if (a.rank_out) a.rank_out[b] = k;
      if (a.cnt) {
        if (skipped) atomicAdd(a.cnt, 1ull);
        if (k == 0) atomicAdd(a.cnt + 1, 1ull);
        if (lanczos_ok) atomicAdd(a.cnt + 2, 1ull);
      }
      if (a.nuc_acc && k > 0) {
        double t = 0.0;
        for (int q = 0; q < k; ++q) t += (double)fmaxf(sqrtf(z.Bm[q * K + q]) - a.tau, 0.f);
        atomicAdd(a.nuc_acc, t);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  g.barrier();  // no CTA leaves while the other may write its shared memory
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols)
                 : "memory");
}

}  // namespace

cudaError_t configure_eig() {
  if (cudaError_t e = cudaFuncSetAttribute(eig_cluster_kernel<1>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           eig_smem_bytes(1)))
    return e;
  return cudaFuncSetAttribute(eig_cluster_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              eig_smem_bytes(2));
}

cudaError_t launch_eig(const ScaleLaunch& s, const BigWorkspace& ws, int nblocks, cudaStream_t st) {
  const int n = s.m < s.n ? s.m : s.n;
  const int CL = n <= kERows ? 1 : 2;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL * nblocks);
  cfg.blockDim = dim3(kENT);
  cfg.dynamicSmemBytes = eig_smem_bytes(CL);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (CL == 1) return cudaLaunchKernelEx(&cfg, eig_cluster_kernel<1>, s, (const float*)ws.G, ws);
  return cudaLaunchKernelEx(&cfg, eig_cluster_kernel<2>, s, (const float*)ws.G, ws);
}

}  // namespace msllr

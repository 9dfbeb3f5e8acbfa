// Block SVTs of the narrowest blocks (min(m, n) <= 8, max(m, n) <= 16),
// several to a warp: W lanes per block (4 or 8), lane c holds the whole column
// c of C (R rows) in registers -- eq:bsvt under the Sec. 9 shift.  The steps
// and tests are those of warp_block.cuh (bounds, Cholesky certificate,
// one-sided Jacobi without rotations that cannot matter, rebuild); only the
// sums run inside a lane.  One block per warp left half to seven eighths of
// the lanes without a column; adjacent blocks of a warp also read adjacent
// row segments.  A block's result does not depend on its neighbours in the
// warp: sweeps that run on for another block find nothing to rotate in a
// settled one.
#pragma once

#include "warp_block.cuh"

namespace msllr {
namespace {

template <int W>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Block b (of this lane's group; any valid index where !on) by W lanes; `vs`:
// the warp's 32 x W shared scratch; a2 as in warp_block_svt.
template <int W, int R, bool ST, class SRC>
__device__ __forceinline__ void pack_block_svt(const ScaleLaunch& a, int b, bool on, float* vs,
                                               const SRC& a2) {
  const int lane = threadIdx.x & 31, c = lane & (W - 1), base = lane & ~(W - 1);
  const BlockGeom g = block_geom_t<ST>(a, b);
  const int mm = g.mm(), nn = g.nn();
  const bool tr = g.transposed();
  const bool col = on && c < nn;

  float x[R];
  float fro = 0.f;
  {
    float y[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const bool in = col && i < mm;
      const int rr = in ? i : 0, cc = in ? c : 0;
      const size_t off = tr ? g.offset(cc, rr) : g.offset(rr, cc);
      x[i] = in ? __ldg(a.A1 + off) : 0.f;
      y[i] = in ? (tr ? a2(off, cc, rr) : a2(off, rr, cc)) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      x[i] += y[i];
      fro = fmaf(x[i], x[i], fro);
    }
  }
  fro = group_sum<W>(fro);
  const float thr = a.tau * a.tau;
  bool skipped = !on || (a.skip_bound && fro <= thr);
  float fl = 0.f;  // flops of the steps run
  if (a.skip_bound && __any_sync(kFull, !skipped)) {
    // G = C^T C: lane c forms row c
    float gr[W];
#pragma unroll
    for (int j = 0; j < W; ++j) gr[j] = 0.f;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < W; ++j) gr[j] = fmaf(x[i], __shfl_sync(kFull, x[i], base | j), gr[j]);
    float rs = 0.f;
#pragma unroll
    for (int j = 0; j < W; ++j) rs += fabsf(gr[j]);
    // Gershgorin: lambda_max(G) <= max_c sum_j |G_cj| (Sec. 8)
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) rs = fmaxf(rs, __shfl_xor_sync(kFull, rs, o));
    const float gbound = fminf(fro, rs);
    if (!skipped) fl += (float)(2 * mm * nn * nn + 2 * nn * nn);
    const bool test = !skipped && !(gbound <= thr);
    if (gbound <= thr) skipped = true;
    if (__any_sync(kFull, test)) {
      // certified lambda_max(G) < tau^2 by the Cholesky factorisation of
      // c0 I - G (see warp_block.cuh); lane c holds row c
      const int n8 = (nn + 7) & ~7;
      const float c0 = thr - (float)(n8 * n8) * FLT_EPSILON * (thr + gbound);
      bool pd = c0 > 0.f;
#pragma unroll
      for (int j = 0; j < W; ++j) gr[j] = (j == c ? c0 : 0.f) - gr[j];
#pragma unroll
      for (int kk = 0; kk < W; ++kk) {
        if (kk < nn) {
          const float d = __shfl_sync(kFull, gr[kk], base | kk);
          pd = pd && d > 0.f;
          const float l = gr[kk] * rsqrtf(d > 0.f ? d : 1.f);  // L(c, kk) for c > kk
#pragma unroll
          for (int j = kk + 1; j < W; ++j)
            if (j < nn) gr[j] = fmaf(-l, __shfl_sync(kFull, l, base | j), gr[j]);
        }
      }
      if (test) {
        fl += (float)(nn * nn * nn) / 3.f;
        skipped = pd;
      }
    }
  }

  float z[R];
#pragma unroll
  for (int i = 0; i < R; ++i) z[i] = 0.f;
  int k = 0;
  int sweeps = 0;
  if (__any_sync(kFull, !skipped)) {
    // one-sided Jacobi: y = C V, V = I at the start (see warp_block.cuh)
    float y[R], v[W];
#pragma unroll
    for (int i = 0; i < R; ++i) y[i] = x[i];
#pragma unroll
    for (int i = 0; i < W; ++i) v[i] = i == c ? 1.f : 0.f;
    const float inv_fro = 1.f / fro;
    const int np = (nn + 1) & ~1;
    bool live = !skipped;
    for (int s = 0; s < kMaxSweeps && __any_sync(kFull, live); ++s) {
      if (live) ++sweeps;
      float al = 0.f;
#pragma unroll
      for (int i = 0; i < R; ++i) al = fmaf(y[i], y[i], al);
      const float small = group_sum<W>(al <= thr ? al : 0.f);
      float large = al <= thr ? FLT_MAX : al;
#pragma unroll
      for (int o = W / 2; o > 0; o >>= 1) large = fminf(large, __shfl_xor_sync(kFull, large, o));
      const float skip =
          (a.skip_bound && small <= 0.9999f * thr && small <= kSkipRatio * large) ? thr : -1.f;
      bool rotated = false;
#pragma unroll 1
      for (int rd = 0; rd < np - 1; ++rd) {
        int o = 2 * rd - c;
        if (o < 0) o += np - 1;
        else if (o >= np - 1) o -= np - 1;
        if (c == rd) o = np - 1;
        if (c == np - 1) o = rd;
        if (c >= np) o = c;
        const int src = base | o;
        const float be = __shfl_sync(kFull, al, src);
        float yo[R];
        float g0 = 0.f, g1 = 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          yo[i] = __shfl_sync(kFull, y[i], src);
          if (i & 1) g1 = fmaf(y[i], yo[i], g1);
          else g0 = fmaf(y[i], yo[i], g0);
        }
        const float ga = g0 + g1;
        const bool lo = c < o;
        const float a_lo = lo ? al : be, a_hi = lo ? be : al;
        const float gn = ga * inv_fro;
        float cr = 1.f, sr = 0.f, t = 0.f;
        if (live && o != c && fmaxf(a_lo, a_hi) > skip && fminf(a_lo, a_hi) > kTinyCol * fro &&
            gn * gn > (kRotTol * kRotTol) * ((a_lo * inv_fro) * (a_hi * inv_fro))) {
          const float dn = (a_hi - a_lo) * inv_fro;
          const float q2 = fmaf(dn, dn, 4.f * gn * gn);
          float rq = rsqrtf(q2);
          rq = rq * fmaf(-0.5f * q2 * rq, rq, 1.5f);
          const float hh = fmaf(0.5f * fabsf(dn), rq, 0.5f);
          float rh = rsqrtf(hh);
          rh = rh * fmaf(-0.5f * hh * rh, rh, 1.5f);
          cr = hh * rh;
          sr = copysignf(1.f, dn) * gn * rq * rh;
          t = sr * rh;  // tan phi = s / c
          rotated = true;
        }
        const float so = lo ? -sr : sr;  // weight of the partner column
        al = lo ? fmaf(-t, ga, al) : fmaf(t, ga, al);
#pragma unroll
        for (int i = 0; i < R; ++i) y[i] = fmaf(so, yo[i], cr * y[i]);
#pragma unroll
        for (int i = 0; i < W; ++i) {
          const float vo = __shfl_sync(kFull, v[i], src);
          v[i] = fmaf(so, vo, cr * v[i]);
        }
      }
      // settled once a whole sweep of the group's columns rotated nothing
      const unsigned rot = __ballot_sync(kFull, rotated);
      live = live && ((rot >> base) & ((1u << W) - 1u)) != 0u;
    }
    float al = 0.f;
#pragma unroll
    for (int i = 0; i < R; ++i) al = fmaf(y[i], y[i], al);
    const float sig = sqrtf(al);
    const float f = (!skipped && col && sig > a.tau) ? 1.f - a.tau / sig : 0.f;
    const unsigned act = __ballot_sync(kFull, f > 0.f);
    k = __popc((act >> base) & ((1u << W) - 1u));
    if (act) {
      if (a.nuc_acc) {
        double t = f > 0.f ? (double)(sig - a.tau) : 0.0;
        t = warp_sum_d(t);
        if (lane == 0) atomicAdd(a.nuc_acc, t);
      }
      // Z' = sum over kept j of f_j (C V)_j V_j^T; lane c needs V(c, j)
      float* vg = vs + base * W;
#pragma unroll
      for (int i = 0; i < W; ++i) vg[i * W + c] = v[i];
      __syncwarp();
#pragma unroll 1
      for (int j = 0; j < W; ++j) {
        const float fj = __shfl_sync(kFull, f, base | j);
        if (!__any_sync(kFull, fj > 0.f)) continue;
        const float w = fj * vg[c * W + j];
#pragma unroll
        for (int i = 0; i < R; ++i) z[i] = fmaf(__shfl_sync(kFull, y[i], base | j), w, z[i]);
      }
      __syncwarp();
    }
  }
  // scatter Z' and W' = 2 Z' - A through Shift_{-s}
#pragma unroll
  for (int i = 0; i < R; ++i) {
    if (col && i < mm) {
      const size_t off = tr ? g.offset(c, i) : g.offset(i, c);
      a.Zout[off] = z[i];
      if (a.Wout) a.Wout[off] = 2.f * z[i] - x[i];
    }
  }
  if (a.rank_out && on && c == 0) a.rank_out[b] = k;
  if (a.cnt) {
    // one atomic per warp and counter
    const bool lead = on && c == 0;
    const unsigned ms = __ballot_sync(kFull, lead && skipped);
    const unsigned mz = __ballot_sync(kFull, lead && k == 0);
    const unsigned mj = __ballot_sync(kFull, lead && !skipped);
    const int npr = (nn + 1) & ~1;
    const double fj =
        (double)sweeps * (npr - 1) * (npr / 2) * (12.0 * mm + 96.0) + 2.0 * mm * nn * k;
    const double fs = warp_sum_d(lead ? fj + fl : 0.0);
    if (lane == 0) {
      if (ms) atomicAdd(a.cnt, (unsigned long long)__popc(ms));
      if (mz) atomicAdd(a.cnt + 1, (unsigned long long)__popc(mz));
      if (mj) atomicAdd(a.cnt + 3, (unsigned long long)__popc(mj));
      if (fs > 0.0) atomicAdd(a.cnt + 5, (unsigned long long)fs);
    }
  }
}

}  // namespace

// lanes per block where the packed path takes m x n blocks (0: it does not),
// and rows per lane
__host__ __device__ constexpr int pack_lanes(int m, int n) {
  return (m < n ? m : n) > 8 || (m < n ? n : m) > 16 ? 0
         : (m < n ? m : n) <= 4 && (m < n ? n : m) <= 8 ? 4
                                                        : 8;
}
__host__ __device__ constexpr int pack_rows(int m, int n) {
  return pack_lanes(m, n) == 4 ? ((m < n ? n : m) <= 4 ? 4 : 8) : ((m < n ? n : m) <= 8 ? 8 : 16);
}

}  // namespace msllr

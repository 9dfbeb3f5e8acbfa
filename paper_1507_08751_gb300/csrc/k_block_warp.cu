// Block SVT of narrow blocks (min(m, n) <= 16, max(m, n) <= 32): one warp
// per block (warp_block.cuh), or several blocks per warp up to 8 x 16
// (pack_block.cuh), one warp per CTA -- eq:bsvt under the Sec. 9 shift.
#include "pack_block.cuh"

namespace msllr {

cudaError_t set_phase_buffer_warp(unsigned long long* p) {
  return cudaMemcpyToSymbol(g_phase_acc, &p, sizeof(p));
}

namespace {

// RPL: rows of C per lane (mm <= 2 RPL); NP: columns in the rotation order
// when fixed at compile time (16 for blocks 15 or 16 wide), 0 to take it
// from the block
template <int RPL, bool ST, int NP>
__global__ void __launch_bounds__(kWT, RPL <= 8 ? 32 : 16)
blocksvt_warp_kernel(ScaleLaunch a, int nblocks) {
  __shared__ float vsh[kWarps][16][17];  // V of each warp, for the rebuild
  const int wid = threadIdx.x >> 5;
  const int b = blockIdx.x * kWarps + wid;
  if (b >= nblocks) return;  // the whole warp leaves together
  warp_block_svt<RPL, ST, NP>(a, b, vsh[wid], A2Global{a.A2});
}

// W lanes and R rows per lane for a block, 32 / W blocks per warp
template <int W, int R, bool ST>
__global__ void __launch_bounds__(kWT, R <= 8 ? 32 : 16)
blocksvt_pack_kernel(ScaleLaunch a, int nblocks) {
  __shared__ float vs[32 * W];
  const int b = blockIdx.x * (32 / W) + (threadIdx.x & 31) / W;
  const bool on = b < nblocks;
  pack_block_svt<W, R, ST>(a, on ? b : nblocks - 1, on, vs, A2Global{a.A2});
}

template <int W, int R>
void launch_pack(const ScaleLaunch& s, int nblocks, cudaStream_t st) {
  const int per = 32 / W, grid = (nblocks + per - 1) / per;
  if (s.fw || s.rows) blocksvt_pack_kernel<W, R, true><<<grid, kWT, 0, st>>>(s, nblocks);
  else blocksvt_pack_kernel<W, R, false><<<grid, kWT, 0, st>>>(s, nblocks);
}

}  // namespace

bool warp_path(int m, int n) {
  const int nn = m < n ? m : n, mm = m < n ? n : m;
  return nn >= 1 && nn <= 16 && mm <= 32;
}

cudaError_t launch_warp(const ScaleLaunch& s, cudaStream_t st, Prof* prof) {
  const int mm = s.m >= s.n ? s.m : s.n;
  const int nblocks = (s.M / s.m) * (s.N / s.n);
  const int grid = (nblocks + kWarps - 1) / kWarps;
  if (prof)
    if (cudaError_t e = prof->before(st, KK_FUSED)) return e;
  const int nn = s.m < s.n ? s.m : s.n;
  const bool gen = s.fw || s.rows, w16 = nn >= 15;
  if (const int w = pack_lanes(s.m, s.n)) {
    const int r = pack_rows(s.m, s.n);
    if (w == 4) {
      if (r == 4) launch_pack<4, 4>(s, nblocks, st);
      else launch_pack<4, 8>(s, nblocks, st);
    } else {
      if (r == 8) launch_pack<8, 8>(s, nblocks, st);
      else launch_pack<8, 16>(s, nblocks, st);
    }
  } else if (mm <= 16) {
    if (w16) {
      if (gen) blocksvt_warp_kernel<8, true, 16><<<grid, kWT, 0, st>>>(s, nblocks);
      else blocksvt_warp_kernel<8, false, 16><<<grid, kWT, 0, st>>>(s, nblocks);
    } else {
      if (gen) blocksvt_warp_kernel<8, true, 0><<<grid, kWT, 0, st>>>(s, nblocks);
      else blocksvt_warp_kernel<8, false, 0><<<grid, kWT, 0, st>>>(s, nblocks);
    }
  } else {
    if (w16) {
      if (gen) blocksvt_warp_kernel<16, true, 16><<<grid, kWT, 0, st>>>(s, nblocks);
      else blocksvt_warp_kernel<16, false, 16><<<grid, kWT, 0, st>>>(s, nblocks);
    } else {
      if (gen) blocksvt_warp_kernel<16, true, 0><<<grid, kWT, 0, st>>>(s, nblocks);
      else blocksvt_warp_kernel<16, false, 0><<<grid, kWT, 0, st>>>(s, nblocks);
    }
  }
  if (prof)
    if (cudaError_t e = prof->after(st)) return e;
  return cudaGetLastError();
}

}  // namespace msllr

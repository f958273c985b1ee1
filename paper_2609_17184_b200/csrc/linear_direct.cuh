// Stand-alone linear map for a few token rows in ONE launch: y[m][n] = sum_k x[m][k] W[n][k], W row-major bf16 read once and
// in place, x fp32 split into its three exact bf16 planes in registers by the warp that multiplies them.  Bound by the
// weight stream and, for small matrices, by the launch itself: the three-launch form it replaces (planes of x, a tile-major
// copy of W, the cluster GEMM) moved W three times and took 14 us on the device for 2048 x 2048.
//
// A warp owns one 16-row tile of W and one of `cs` contiguous k-ranges; the warps of a CTA cover 8 / cs tiles.  Sums are those
// of gemm_bf16_kernel bit for bit - the same k-ranges, three accumulator chains per range folded hi + (mid + lo), ranges added in
// order - so calls of more rows, which run that kernel, give a row the same bits.
#pragma once
#include "gemm.cuh"

namespace ls {

struct LinearDirectParams {
  const __nv_bfloat16* W;  // [N][K]
  const float* x;          // [M][K]
  float* y;                // [M][N]
  int M, N, K, cs;
};

// the three planes of eight values as B-fragment pieces
__device__ __forceinline__ void split_piece(const float4& a, const float4& b, uint4 (&pl)[3]) {
  const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  unsigned short s[3][8];
#pragma unroll
  for (int i = 0; i < 8; ++i) split3(v[i], s[0][i], s[1][i], s[2][i]);
#pragma unroll
  for (int p = 0; p < 3; ++p)
    pl[p] = make_uint4(s[p][0] | ((unsigned)s[p][1] << 16), s[p][2] | ((unsigned)s[p][3] << 16), s[p][4] | ((unsigned)s[p][5] << 16),
                       s[p][6] | ((unsigned)s[p][7] << 16));
}

// T tiles per warp (they share the split of x).  Two k-blocks are fetched together, so that both 64-byte halves of a row's
// 128-byte line are requested at once.
template <int NG, int T>
__global__ void __launch_bounds__(256, NG * T == 1 ? 2 : 1) linear_direct_kernel(const __grid_constant__ LinearDirectParams p) {
  constexpr int DEPTH = 4;  // k-blocks in flight per warp and tile
  __shared__ float s_red[8][T][8 * NG][16];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int tpc = 8 / p.cs, n_tiles = p.N / 16;
  const int tile0 = (blockIdx.x * tpc + warp / p.cs) * T;
  int lo, hi;
  gemm_krange((p.K + 31) / 32, p.cs, warp % p.cs, lo, hi);
  const __nv_bfloat16* w_lo[T];
#pragma unroll
  for (int q = 0; q < T; ++q) w_lo[q] = p.W + (size_t)(min(tile0 + q, n_tiles - 1) * 16 + g) * p.K + t * 8;  // (tiles beyond the matrix repeat the last one)
  const size_t w_hi = (size_t)8 * p.K;
  const float* xr[NG];
#pragma unroll
  for (int n = 0; n < NG; ++n) xr[n] = p.x + (size_t)min(n * 8 + g, p.M - 1) * p.K + t * 8;  // (columns beyond M repeat the last row and are not stored)

  uint4 wl[DEPTH][T], wh[DEPTH][T];
  float4 xa[DEPTH][NG], xb[DEPTH][NG];
  auto fetch = [&](int u, int kb) {
    const bool live = kb < hi && kb * 32 + t * 8 < p.K;
#pragma unroll
    for (int q = 0; q < T; ++q) {
      wl[u][q] = wh[u][q] = make_uint4(0, 0, 0, 0);
      if (live) {
        wl[u][q] = __ldcs(reinterpret_cast<const uint4*>(w_lo[q] + kb * 32));
        wh[u][q] = __ldcs(reinterpret_cast<const uint4*>(w_lo[q] + w_hi + kb * 32));
      }
    }
#pragma unroll
    for (int n = 0; n < NG; ++n) {
      xa[u][n] = xb[u][n] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (live) {
        xa[u][n] = __ldg(reinterpret_cast<const float4*>(xr[n] + kb * 32));
        xb[u][n] = __ldg(reinterpret_cast<const float4*>(xr[n] + kb * 32) + 1);
      }
    }
  };
  float acc[T][3][NG][4];
#pragma unroll
  for (int q = 0; q < T; ++q)
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
      for (int n = 0; n < NG; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[q][s][n][i] = 0.f;
#pragma unroll
  for (int u = 0; u < DEPTH; ++u) fetch(u, lo + u);
  for (int kb = lo; kb < hi; kb += DEPTH) {
#pragma unroll
    for (int u0 = 0; u0 < DEPTH; u0 += 2) {
#pragma unroll
      for (int u = u0; u < u0 + 2; ++u) {
        if (kb + u < hi) {
#pragma unroll
          for (int n = 0; n < NG; ++n) {
            uint4 b[3];
            split_piece(xa[u][n], xb[u][n], b);
#pragma unroll
            for (int q = 0; q < T; ++q)
#pragma unroll
              for (int s = 0; s < 3; ++s) {
                mma_bf16(acc[q][s][n], wl[u][q].x, wh[u][q].x, wl[u][q].y, wh[u][q].y, b[s].x, b[s].y);
                mma_bf16(acc[q][s][n], wl[u][q].z, wh[u][q].z, wl[u][q].w, wh[u][q].w, b[s].z, b[s].w);
              }
          }
        }
      }
      fetch(u0, kb + u0 + DEPTH);
      fetch(u0 + 1, kb + u0 + 1 + DEPTH);
    }
  }
#pragma unroll
  for (int q = 0; q < T; ++q)
#pragma unroll
    for (int n = 0; n < NG; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) s_red[warp][q][n * 8 + 2 * t + (i & 1)][g + 8 * (i >> 1)] = acc[q][0][n][i] + (acc[q][1][n][i] + acc[q][2][n][i]);
  __syncthreads();
  for (int idx = tid; idx < tpc * T * p.M * 16; idx += 256) {
    const int row = idx & 15, rest = idx >> 4, c = rest % p.M, tl = rest / p.M, w = (tl / T) * p.cs;
    const int n = (blockIdx.x * tpc * T + tl) * 16 + row;
    float v = s_red[w][tl % T][c][row];
    for (int r = 1; r < p.cs; ++r) v += s_red[w + r][tl % T][c][row];  // k-ranges in order
    if (n < p.N) p.y[(size_t)c * p.N + n] = v;
  }
}

}  // namespace ls

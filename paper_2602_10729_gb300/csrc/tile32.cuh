// 32 x 32 tiles of fp32 matrices in shared memory: products by groups of 64 threads,
// and the Cholesky factor of a diagonal tile with its inverse by two warps.
#pragma once

#include "common.cuh"

namespace boute {

constexpr int kFcTile = 32 * 32;

// Word of element (r, q) of a tile: 16-byte groups permuted by the row's quad, so
// that a product's operand reads (rows 4 apart) and result accesses are free of conflicts.
__device__ __forceinline__ int fc_off(int r, int q) {
  return r * 32 + ((((q >> 2) ^ (r >> 2)) & 7) << 2) + (q & 3);
}

// acc[u][v] = sum_q X(4 ty + u, q) Y(4 tx + v, q) by 64 threads (t = 8 ty + tx), each
// an fmaf chain over q = 0 .. 31 in order.
__device__ __forceinline__ void fc_product(const float *X, const float *Y, int t,
                                           float (&acc)[4][4]) {
  const int tx = t & 7, ty = t >> 3;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
  const float4 *X4 = (const float4 *)X + 4 * ty * 8, *Y4 = (const float4 *)Y + 4 * tx * 8;
#pragma unroll 2
  for (int g = 0; g < 8; ++g) {
    float4 x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = X4[u * 8 + (g ^ ty)];
#pragma unroll
    for (int v = 0; v < 4; ++v) y[v] = Y4[v * 8 + (g ^ tx)];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        acc[u][v] = fmaf(x[u].x, y[v].x, acc[u][v]);
        acc[u][v] = fmaf(x[u].y, y[v].y, acc[u][v]);
        acc[u][v] = fmaf(x[u].z, y[v].z, acc[u][v]);
        acc[u][v] = fmaf(x[u].w, y[v].w, acc[u][v]);
      }
  }
}

// The diagonal tile by warps 0 and 1: tile = L L^T factored by warp 0 (lane = row) and
// W_pp = L^-1 formed by warp 1 (lane = column of W_pp), eight columns of L behind. W_pp
// goes to wpp (row, column) and, transposed, to wtpp and into the tile. dg: the tile's
// diagonal of K. Each warp holds a window of its row (column) that moves four columns
// per iteration, so that register indices are static and the code stays small (unrolled
// over the 32 columns it ran three times longer, waiting for instructions); column c
// of L reaches the row updates as broadcast 16-byte loads, and only the entry that the
// next pivot waits for as a shuffle.
struct FcDiag {
  float colL[34 * 32];  // columns of L_pp (rows from the diagonal on); the windows' reads
                        // run up to 28 words past a column
  float invs[32];       // 1 / L_cc
};
__device__ __forceinline__ void fc_diagonal(float *tile, const float *dg, FcDiag &sh, float *wpp,
                                            float *wtpp, int *fbad) {
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  if (threadIdx.x < 32) {
    float a[36];  // columns c0 .. c0 + 31 of the lane's row (those beyond 31: never used)
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const float4 v = ((const float4 *)tile)[lane * 8 + ((g ^ (lane >> 2)) & 7)];
      a[4 * g] = v.x;
      a[4 * g + 1] = v.y;
      a[4 * g + 2] = v.z;
      a[4 * g + 3] = v.w;
    }
    a[32] = a[33] = a[34] = a[35] = 0.f;
    bool ok = true;
    auto recip_root = [](float piv) {  // 1 / L_cc: one Newton step
      const float inv = rsqrtf(piv);
      return inv * fmaf(-0.5f * piv * inv, inv, 1.5f);
    };
    float piv = __shfl_sync(FULL, a[0], 0), inv = recip_root(piv);
#pragma unroll 1
    for (int c0 = 0; c0 < 32; c0 += 4) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j;
        const float l = lane == c ? piv * inv : a[j] * inv;  // (rows above c: never used)
        float *col = sh.colL + c * 32;
        col[lane] = l;
        if (lane == 0) sh.invs[c] = inv;
        // the next pivot: lane c + 1's entry, which needs that lane's l alone; its
        // reciprocal root is formed while the row's update waits for its operands
        const float next = __shfl_sync(FULL, fmaf(-l, l, a[j + 1]), (c + 1) & 31);
        a[j + 1] = fmaf(-l, __shfl_sync(FULL, l, (c + 1) & 31), a[j + 1]);
        __syncwarp();
        float4 v[8];
#pragma unroll
        for (int g = (j + 2) / 4; g < 8; ++g) v[g] = *(const float4 *)(col + c0 + 4 * g);
        if (!(piv > 16.f * 1.1920929e-7f * dg[c])) ok = false;
        piv = next;
        inv = recip_root(piv);  // (unused after c = 31)
#pragma unroll
        for (int g = (j + 2) / 4; g < 8; ++g) {  // the window's columns j + 2 ..
          if (4 * g > j + 1) a[4 * g] = fmaf(-l, v[g].x, a[4 * g]);
          if (4 * g + 1 > j + 1) a[4 * g + 1] = fmaf(-l, v[g].y, a[4 * g + 1]);
          if (4 * g + 2 > j + 1) a[4 * g + 2] = fmaf(-l, v[g].z, a[4 * g + 2]);
          if (4 * g + 3 > j + 1) a[4 * g + 3] = fmaf(-l, v[g].w, a[4 * g + 3]);
        }
      }
      if (c0 & 4) named_barrier_arrive(9 + (c0 >> 3), 64);  // eight columns for warp 1
#pragma unroll
      for (int k = 0; k < 32; ++k) a[k] = a[k + 4];
    }
    if (!ok && lane == 0) *fbad = 1;
  } else {
    float r[36];  // rows c0 .. c0 + 31 of column `lane`: the remainders
#pragma unroll
    for (int c = 0; c < 36; ++c) r[c] = (c == lane) ? 1.f : 0.f;
#pragma unroll 1
    for (int c0 = 0; c0 < 32; c0 += 4) {
      if (!(c0 & 4)) named_barrier_sync(9 + (c0 >> 3), 64);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j;
        const float *col = sh.colL + c * 32;
        r[j] *= sh.invs[c];  // W_c,lane
#pragma unroll
        for (int g = (j + 1) / 4; g < 8; ++g) {  // r_i -= L_ic W_c,lane, rows below c
          const float4 v = *(const float4 *)(col + c0 + 4 * g);
          if (4 * g > j) r[4 * g] = fmaf(-v.x, r[j], r[4 * g]);
          if (4 * g + 1 > j) r[4 * g + 1] = fmaf(-v.y, r[j], r[4 * g + 1]);
          if (4 * g + 2 > j) r[4 * g + 2] = fmaf(-v.z, r[j], r[4 * g + 2]);
          if (4 * g + 3 > j) r[4 * g + 3] = fmaf(-v.w, r[j], r[4 * g + 3]);
        }
        wpp[fc_off(c, lane)] = r[j];
      }
      const float4 v = make_float4(r[0], r[1], r[2], r[3]);
      const int o = lane * 8 + (((c0 >> 2) ^ (lane >> 2)) & 7);
      ((float4 *)wtpp)[o] = v;
      ((float4 *)tile)[o] = v;
#pragma unroll
      for (int k = 0; k < 32; ++k) r[k] = r[k + 4];
    }
  }
  __syncwarp();
}

}  // namespace boute

// Noisy acquisition (Sec. 5.2, constrained qNEHVI with q = 1): the
// expectation runs over joint posterior draws of the objectives at the n
// observed points and at the candidate, so the front a candidate improves on
// is itself drawn, sample by sample.
//
// With K = K_nn + sigma^2 I = L L^T, W = L^-1 and the in-sample posterior
// covariance Sigma = K_nn - K_nn K^-1 K_nn = sigma^2 (I - sigma^2 K^-1), a
// joint draw s is the Cholesky factor of the joint covariance (jitter on the
// in-sample block) applied to the normals (z_s, eps_s):
//   f_s(X) = mu_n + F z_s,  F = chol(Sigma + jitter s2 I),  mu_n = y - sigma^2 alpha
//   f_s(x) = mean(x) + l^T z_s + sqrt(cvar) eps_s,  l = F^-1 Sigma_nx
// with Sigma_nx = sigma^2 K^-1 k*. Both per-candidate terms are contractions
// of k*: l^T z_s = k*^T G_s with G = H Z, H = sigma^2 K^-1 F^-T, and
// cvar = k(x,x) - |W k*|^2 - |H^T k*|^2. H^T and G^T therefore become dense
// output blocks of the posterior's tensor-core contraction beside W.
//
//   insample_factor_kernel one CTA per problem-objective after the fit: K^-1, F and H
//                          (fp32 tiles in shared memory, n <= 128); then
//   insample_draws_kernel, insample_pack_kernel: the draws, G, and its operand images
//   insample_front_kernel  one warp per (problem, draw): the Pareto front of
//                          the feasible in-sample draws as vertical strips
//   nehvi2_kernel          one thread per candidate: the draws' hypervolume
//                          improvements over their own fronts, averaged
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "tile32.cuh"

namespace boute {

namespace {

constexpr int kInsThreads = 512;

// Row stride of the shared-memory matrices: odd, so that a warp reading one
// column (32 consecutive rows) touches 32 different banks.
__host__ __device__ __forceinline__ int ins_ld(int n) { return n | 1; }

__device__ __forceinline__ void atomic_max_pos(unsigned *a, float v) {
  atomicMax(a, __float_as_uint(v));  // non-negative floats order as their bits
}

__device__ __forceinline__ int scale_exp(float mx) { return mx > 0.f ? 13 - ilogbf(mx) : 0; }

// Workspace of one problem-objective: F (n x n, zero above the diagonal),
// H^T (n x n), mu_n (n), and max |G| (one word, as float bits).
__host__ __device__ __forceinline__ size_t ins_ws_floats(int n) {
  return 2 * (size_t)n * n + (size_t)n + 4;
}

// The operand image of one output row of a dense block: K positions k, k + 1
// of row `row` of block q, scaled, as fp16 hi/lo pairs (zero beyond n).
__device__ __forceinline__ void pack_dense_pair(float w0, float w1, int n, int k, float scl, int q,
                                                int row, const PostPlan &plan, uint16_t *img) {
  const float v0 = k < n ? w0 * scl : 0.f, v1 = k + 1 < n ? w1 * scl : 0.f;
  uint32_t hi, lo;
  split_f16x2(v0, v1, hi, lo);
  const int ncol = plan.ncol[q], cidx = k / BOUTE_ACHUNK;
  uint32_t *blk = (uint32_t *)(img + plan.off[q] + (long long)cidx * 2 * ncol * BOUTE_ACHUNK);
  const int o = sw128_off16(row % BOUTE_BLKCOLS, k % BOUTE_ACHUNK) >> 1;
  const long long base = plan.off[q] + (long long)cidx * 2 * ncol * BOUTE_ACHUNK;
  (void)base;  // (used by the debug build's checks)
  if (BOUTE_INB(base + 2 * ((ncol * BOUTE_ACHUNK >> 1) + o) + 1, plan.image_halves) &&
      BOUTE_INB(k, plan.nchunk * BOUTE_ACHUNK)) {
    blk[o] = hi;
    blk[(ncol * BOUTE_ACHUNK >> 1) + o] = lo;
  }
}

// (1) one CTA per problem-objective: the sequential part. K^-1 = W^T W, the
// jittered in-sample covariance and its Cholesky factor F, H^T = sigma^2
// F^-1 K^-1 by forward substitution; F, H^T and mu_n go to the workspace,
// H^T's operand images and scale exponent to the handle. Everything is 32 x 32 tiles
// in shared memory, products by eight groups of 64 threads: W and H as transposes
// (tile (K, I) of WT holds W_KI^T), the right-hand sides H updated with the factor's
// trailing matrix in one right-looking loop, so that what bounds it is four diagonal
// tiles' chains and about 100 tile products (n = 128: 149 -> 46 us; scalar loops
// over rows and columns, with serial substitutions, before).
__global__ void __launch_bounds__(kInsThreads, 1)
    insample_factor_kernel(const float *Wws, int npad, float *xt, int DP, int nxt,
                           const double *Ys, const double *s2, const double *noise, int n, int m,
                           float *ws, uint16_t *bop, PostPlan plan, int *status) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int bad;
  __shared__ unsigned mxh;
  const int bt = blockIdx.x;
  const int tid = threadIdx.x;
  const int nb = (n + 31) / 32, nt = nb * (nb + 1) / 2;
  // W^T (then F) and the covariance: lower tiles; H^T transposed: nb x nb tiles, column
  // tile c of block row q at (q nb + c); the diagonal tile's inverse, both ways
  float *WT = sm, *A = WT + nt * kFcTile, *HT = A + nt * kFcTile;
  float *vpp = HT + nb * nb * kFcTile, *vtt = vpp + kFcTile, *mu = vtt + kFcTile;
  __shared__ __align__(16) FcDiag dsh;
  __shared__ float zero[32];
  auto tri = [](int I, int J) { return (I * (I + 1) / 2 + J) * kFcTile; };
  const double s2d = s2[bt];
  const double nzd = noise[bt] > 1e-12 * s2d ? noise[bt] : 1e-12 * s2d;  // the fit's floor
  const float sig2 = (float)nzd, jit = (float)(kInsJitter * s2d);
  const int cf = xt_chunk_floats(DP);
  float *x0 = xt + (size_t)bt * nxt * cf;
  float *wsb = ws + (size_t)bt * ins_ws_floats(n);
  pdl_wait();  // the fit's W and alpha
  if (tid == 0) {
    bad = *status == BOUTE_ERR_NOT_PD;
    mxh = 0u;
    wsb[2 * (size_t)n * n + n] = 0.f;  // max |G|, raised by the draws kernel
  }
  // W (lower triangle) and mu_n = y - sigma^2 alpha (alpha = hi + lo)
  const float *W = Wws + (size_t)bt * npad * (npad + 1);
  const int warp = tid >> 5, lane = tid & 31;
  for (int e = warp; e < 4 * nt; e += kInsThreads / 32) {  // eight rows of a tile per warp
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= (e >> 2)) ++I;
    const int J = (e >> 2) - I * (I + 1) / 2, r0 = 8 * (e & 3), k = 32 * J + lane;
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 32 * I + r0 + u;
      v[u] = (i < n && k <= i) ? W[(size_t)i * (npad + 1) + k] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) WT[tri(I, J) + fc_off(lane, r0 + u)] = v[u];
  }
  if (tid < 32) zero[tid] = 0.f;
  const int b = bt / m, t = bt % m;
  for (int i = tid; i < n; i += kInsThreads) {
    const float *ca = x0 + (size_t)(i / BOUTE_KCHUNK) * cf + xt_alpha_offset(DP) + i % BOUTE_KCHUNK;
    const double al = (double)ca[0] + (double)ca[BOUTE_KCHUNK];
    mu[i] = (float)(Ys[((size_t)b * n + i) * m + t] - nzd * al);
    wsb[2 * (size_t)n * n + i] = mu[i];
  }
  __syncthreads();
  if (bad) return;
  const int grp = tid >> 6, gt = tid & 63, tx = gt & 7, ty = gt >> 3;
  constexpr int kGroups = kInsThreads / 64;
  float acc[4][4];
  auto store = [&](float *T) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      ((float4 *)T)[(4 * ty + u) * 8 + (tx ^ ty)] =
          make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
  };
  // K^-1 = W^T W by lower tiles, sum over K >= I of W_KI^T W_KJ; from it sigma^2 K^-1
  // (H's right-hand sides, both triangles) and the covariance Sigma + jitter s2 I =
  // sigma^2 (I - sigma^2 K^-1) + jitter s2 I (the longest sums first)
  for (int e = grp; e < nt; e += kGroups) {
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= e) ++I;
    const int J = e - I * (I + 1) / 2;
    float sum[4][4] = {};
    for (int K = I; K < nb; ++K) {
      fc_product(WT + tri(K, I), WT + tri(K, J), gt, acc);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) sum[u][v] += acc[u][v];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int r = 4 * ty + u, c = 4 * tx + v;
        const float kv = sig2 * sum[u][v];  // sigma^2 K^-1
        HT[(J * nb + I) * kFcTile + fc_off(r, c)] = kv;  // (row tile J, column tile I)^T
        if (I != J) HT[(I * nb + J) * kFcTile + fc_off(c, r)] = kv;
        const bool dia = I == J && r == c;
        const float a = sig2 * ((dia ? 1.f : 0.f) - kv);
        acc[u][v] = dia ? a + jit : a;
      }
    store(A + tri(I, J));
  }
  __shared__ int badp;
  if (tid == 0) badp = 0;
  __syncthreads();
  // Panel p: the diagonal tile's factor and inverse V = F_pp^-1 (any positive pivot is
  // accepted); F_Ip = A_Ip V^T into F's tiles (the space of W^T) and H_p^T = V (its
  // right-hand sides); then A_IJ -= F_Ip F_Jp^T and H_I^T -= F_Ip H_p^T.
  float *F = WT;
  float hmax = 0.f;
  for (int p = 0; p < nb; ++p) {
    if (grp == 0) {
      fc_diagonal(A + tri(p, p), zero, dsh, vpp, vtt, &badp);
    }
    __syncthreads();
    if (badp) {  // (uniform)
      if (tid == 0) set_status(status, BOUTE_ERR_NOT_PD);
      return;
    }
    for (int e = tid; e < kFcTile; e += kInsThreads) {  // F_pp, zero above the diagonal
      const int r = e & 31, c = e >> 5;
      F[tri(p, p) + fc_off(r, c)] = c <= r ? dsh.colL[c * 32 + r] : 0.f;
    }
    const int T = nb - 1 - p;
    for (int e = grp; e < T + nb; e += kGroups) {
      if (e < T) {
        const int I = p + 1 + e;
        fc_product(A + tri(I, p), vpp, gt, acc);
        store(F + tri(I, p));
      } else {
        float *H = HT + (p * nb + e - T) * kFcTile;
        fc_product(H, vpp, gt, acc);
        named_barrier_sync(1 + grp, 64);  // the tile is read
        store(H);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) hmax = fmaxf(hmax, fabsf(acc[u][v]));
      }
    }
    __syncthreads();
    const int na = T * (T + 1) / 2;
    for (int e = grp; e < na + T * nb; e += kGroups) {
      float *D;
      if (e < na) {
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        const int I = p + 1 + i, J = p + 1 + e - i * (i + 1) / 2;
        fc_product(F + tri(I, p), F + tri(J, p), gt, acc);
        D = A + tri(I, J);
      } else {
        const int I = p + 1 + (e - na) / nb, c = (e - na) % nb;
        fc_product(HT + (p * nb + c) * kFcTile, F + tri(I, p), gt, acc);
        D = HT + (I * nb + c) * kFcTile;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float4 *q = (float4 *)D + (4 * ty + u) * 8 + (tx ^ ty);
        float4 v = *q;
        v.x -= acc[u][0];
        v.y -= acc[u][1];
        v.z -= acc[u][2];
        v.w -= acc[u][3];
        *q = v;
      }
    }
    __syncthreads();
  }
  for (int i = warp; i < n; i += kInsThreads / 32)  // F, zero above the diagonal
    for (int k = lane; k < n; k += 32)
      wsb[(size_t)i * n + k] =
          k <= i ? F[tri(i >> 5, k >> 5) + fc_off(i & 31, k & 31)] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hmax = fmaxf(hmax, __shfl_xor_sync(0xffffffffu, hmax, o));
  if (lane == 0) atomic_max_pos(&mxh, hmax);
  __syncthreads();
  auto hval = [&](int r, int c) {  // H^T
    return HT[((r >> 5) * nb + (c >> 5)) * kFcTile + fc_off(c & 31, r & 31)];
  };
  for (int i = warp; i < n; i += kInsThreads / 32)
    for (int k = lane; k < n; k += 32) wsb[(size_t)n * n + (size_t)i * n + k] = hval(i, k);
  pdl_trigger();
  // H^T's operand images (output rows of the H blocks) and scale
  const int eh = scale_exp(__uint_as_float(mxh));
  if (tid == 0) x0[xt_param_offset(DP) + 2 * DP + kParEH] = (float)eh;
  const float sh = exp2i(eh);
  const int kpairs = plan.nchunk * (BOUTE_ACHUNK / 2);
  uint16_t *img = bop + (size_t)bt * plan.image_halves;
  for (int row = warp; row < n; row += kInsThreads / 32)
    for (int e = lane; e < kpairs; e += 32) {
      const int k = 2 * e;
      pack_dense_pair(k < n ? hval(row, k) : 0.f, k + 1 < n ? hval(row, k + 1) : 0.f, n, k, sh,
                      plan.nwblk + row / BOUTE_BLKCOLS, row, plan, img);
    }
}

// (2) the draws, kInsDraws per CTA (grid: draw groups x problem-objectives),
// a warp per draw: Yin[s] = mu_n + F z_s and G^T row s = H^T^T z_s, four
// rows per lane as independent chains; max |G| by atomics.
constexpr int kInsDraws = 4, kDrawThreads = 32 * kInsDraws;

__global__ void __launch_bounds__(kDrawThreads)
    insample_draws_kernel(int n, int S, const float *z, float *Yin, float *gws, float *ws,
                          const int *status) {
  extern __shared__ __align__(16) float sm[];
  const int bt = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ld = ins_ld(n);
  float *F = sm, *Ht = F + (size_t)n * ld, *zs = Ht + (size_t)n * ld, *mu = zs + kInsDraws * kInsMaxN;
  float *wsb = ws + (size_t)bt * ins_ws_floats(n);
  pdl_wait();
  pdl_trigger();
  if (*status == BOUTE_ERR_NOT_PD) return;
  for (int i = warp; i < n; i += kInsDraws) {  // a warp per row, eight loads in flight
    float f[kInsMaxN / 32], h[kInsMaxN / 32];
#pragma unroll
    for (int r = 0; r < kInsMaxN / 32; ++r) {
      const int k = lane + 32 * r;
      f[r] = k < n ? wsb[(size_t)i * n + k] : 0.f;
      h[r] = k < n ? wsb[(size_t)n * n + (size_t)i * n + k] : 0.f;
    }
#pragma unroll
    for (int r = 0; r < kInsMaxN / 32; ++r)
      if (lane + 32 * r < n) {
        F[(size_t)i * ld + lane + 32 * r] = f[r];
        Ht[(size_t)i * ld + lane + 32 * r] = h[r];
      }
  }
  for (int i = threadIdx.x; i < n; i += kDrawThreads) mu[i] = wsb[2 * (size_t)n * n + i];
  const int s = blockIdx.x * kInsDraws + warp;
  const size_t zoff = (size_t)bt * S * n;
  float *zw = zs + warp * kInsMaxN;
  if (s < S)
    for (int j = lane; j < n; j += 32) zw[j] = z[zoff + (size_t)s * n + j];
  __syncthreads();
  if (s >= S) return;
  constexpr int R = kInsMaxN / 32;
  float y[R], g[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    y[r] = lane + 32 * r < n ? mu[lane + 32 * r] : 0.f;
    g[r] = 0.f;
  }
  for (int j = 0; j < n; ++j) {
    const float zj = zw[j];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = lane + 32 * r;
      if (i < n) {
        y[r] = fmaf(F[(size_t)i * ld + j], zj, y[r]);  // zero above the diagonal
        g[r] = fmaf(Ht[(size_t)j * ld + i], zj, g[r]);
      }
    }
  }
  float gm = 0.f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = lane + 32 * r;
    if (i < n && BOUTE_INB(zoff + (long long)s * n + i, (long long)gridDim.y * S * n)) {
      Yin[zoff + (size_t)s * n + i] = y[r];
      gws[zoff + (size_t)s * n + i] = g[r];
      gm = fmaxf(gm, fabsf(g[r]));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  if (lane == 0) atomic_max_pos((unsigned *)(wsb + 2 * (size_t)n * n + n), gm);
}

// (3) G^T's operand images (the G blocks) with the scale of max |G|.
__global__ void __launch_bounds__(256)
    insample_pack_kernel(int n, int S, const float *gws, const float *ws, float *xt, int DP,
                         int nxt, uint16_t *bop, PostPlan plan, const int *status) {
  const int bt = blockIdx.y;
  pdl_wait();
  pdl_trigger();
  if (*status == BOUTE_ERR_NOT_PD) return;
  const float *wsb = ws + (size_t)bt * ins_ws_floats(n);
  const int eg = scale_exp(wsb[2 * (size_t)n * n + n]);
  if (blockIdx.x == 0 && threadIdx.x == 0)
    xt[(size_t)bt * nxt * xt_chunk_floats(DP) + xt_param_offset(DP) + 2 * DP + kParEG] = (float)eg;
  const float sg = exp2i(eg);
  const int kpairs = plan.nchunk * (BOUTE_ACHUNK / 2);
  uint16_t *img = bop + (size_t)bt * plan.image_halves;
  const float *gb = gws + (size_t)bt * S * n;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < S * kpairs; e += gridDim.x * blockDim.x) {
    const int row = e / kpairs, k = 2 * (e % kpairs);
    const float *g = gb + (size_t)row * n;
    pack_dense_pair(k < n ? g[k] : 0.f, k + 1 < n ? g[k + 1] : 0.f, n, k, sg,
                    plan.nwblk + plan.nhblk + row / BOUTE_BLKCOLS, row, plan, img);
  }
}

}  // namespace

size_t insample_smem_bytes(int n) {
  const int nb = (n + 31) / 32;
  return ((size_t)(nb * (nb + 1) + nb * nb + 2) * kFcTile + 32 * nb) * sizeof(float);
}

size_t insample_ws_floats(int n) { return ins_ws_floats(n); }

int launch_insample(Gp *gp, const double *Ys, const double *s2, const double *noise,
                    const float *z, float *Yin, cudaStream_t s) {
  const int n = gp->n, BM = gp->B * gp->m, S = gp->plan.S_in;
  if (S < 1 || n > kInsMaxN) return BOUTE_ERR_UNSUPPORTED;
  const size_t smem = insample_smem_bytes(n);
  prefer_shared(insample_factor_kernel);
  cudaFuncSetAttribute(insample_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem);
  launch_pdl(insample_factor_kernel, dim3(BM), dim3(kInsThreads), smem, s,
             (const float *)gp->Wws, gp->plan.npad, gp->xt, gp->DP, gp->plan.nxt, Ys, s2, noise,
             n, gp->m, gp->iws, gp->bop, gp->plan, gp->status);
  const size_t smem2 = (2 * (size_t)n * ins_ld(n) + kInsDraws * kInsMaxN + kInsMaxN) * sizeof(float);
  prefer_shared(insample_draws_kernel);
  cudaFuncSetAttribute(insample_draws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem2);
  launch_pdl(insample_draws_kernel, dim3((S + kInsDraws - 1) / kInsDraws, BM), dim3(kDrawThreads),
             smem2, s, n, S, z, Yin, gp->gws, gp->iws, (const int *)gp->status);
  const int kpairs = gp->plan.nchunk * (BOUTE_ACHUNK / 2);
  const unsigned gx = (unsigned)std::min(64, (S * kpairs + 255) / 256);
  launch_pdl(insample_pack_kernel, dim3(gx, BM), dim3(256), 0, s, n, S,
             (const float *)gp->gws, (const float *)gp->iws, gp->xt, gp->DP, gp->plan.nxt,
             gp->bop, gp->plan, (const int *)gp->status);
  count_launch(3);
  return last_launch_status();
}

namespace {

constexpr int kFrontPts = kInsMaxN / 32;  // in-sample points per lane
constexpr int kFrontWarps = 4;

// The Pareto front (minimisation) of one draw's feasible in-sample points
// that lie strictly inside the reference box, as the vertical strips of the
// region the front leaves undominated: with the front sorted by f1 (f2 then
// decreasing) q_0 .. q_{P-1},
//   strip 0: (-inf, q_0.f1) x (-inf, r2),  strip i: [q_{i-1}.f1, q_i.f1) x (-inf, q_{i-1}.f2),
//   strip P: [q_{P-1}.f1, r1) x (-inf, q_{P-1}.f2),
// stored as (l1, u1, u2); a point's hypervolume improvement is the sum over
// the strips of (u1 - max(l1, y1))+ (u2 - y2)+. Duplicates keep their lowest
// index, as the front of the observed outcomes does.
__global__ void __launch_bounds__(32 * kFrontWarps)
    insample_front_kernel(const float *Yin, int B, int n, int S, const double *ref,
                          const double *cons, float4 *strips, int *counts) {
  __shared__ float f1s[kFrontWarps][kInsMaxN];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bs = blockIdx.x * kFrontWarps + w;  // (problem, draw)
  pdl_wait();
  pdl_trigger();
  if (bs >= B * S) return;
  const int b = bs / S, s = bs % S;
  const float r1 = (float)ref[(size_t)b * 2], r2 = (float)ref[(size_t)b * 2 + 1];
  const bool hc = cons != nullptr;
  const float c1 = hc ? (float)cons[(size_t)b * 2] : 0.f, c2 = hc ? (float)cons[(size_t)b * 2 + 1] : 0.f;
  const float *y1 = Yin + ((size_t)(b * 2) * S + s) * n, *y2 = Yin + ((size_t)(b * 2 + 1) * S + s) * n;
  float p1[kFrontPts], p2[kFrontPts];
  bool ok[kFrontPts];
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r) {
    const int i = lane + 32 * r;
    ok[r] = i < n;
    p1[r] = ok[r] ? y1[i] : 0.f;
    p2[r] = ok[r] ? y2[i] : 0.f;
    ok[r] = ok[r] && p1[r] < r1 && p2[r] < r2 && (!hc || (p1[r] <= c1 && p2[r] <= c2));
  }
  // dominance: every candidate point against every other (shuffles)
  bool keep[kFrontPts];
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r) keep[r] = ok[r];
#pragma unroll
  for (int r2 = 0; r2 < kFrontPts; ++r2) {
    if (32 * r2 >= n) break;
    for (int src = 0; src < 32; ++src) {
      const float q1 = __shfl_sync(0xffffffffu, p1[r2], src);
      const float q2 = __shfl_sync(0xffffffffu, p2[r2], src);
      const bool qv = __shfl_sync(0xffffffffu, ok[r2] ? 1 : 0, src) != 0;
      const int j = src + 32 * r2;
      if (!qv) continue;
#pragma unroll
      for (int r = 0; r < kFrontPts; ++r) {
        const int i = lane + 32 * r;
        const bool le = q1 <= p1[r] && q2 <= p2[r];
        const bool lt = q1 < p1[r] || q2 < p2[r];
        if (j != i && le && (lt || j < i)) keep[r] = false;  // dominated, or a later duplicate
      }
    }
  }
  // count and rank: on the front f1 values are distinct
  int P = 0;
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r) P += __popc(__ballot_sync(0xffffffffu, keep[r]));
  // compact the front's f1 values into shared memory, then rank by f1
  int base = 0;
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r) {
    const unsigned bal = __ballot_sync(0xffffffffu, keep[r]);
    if (keep[r]) f1s[w][base + __popc(bal & ((1u << lane) - 1u))] = p1[r];
    base += __popc(bal);
  }
  __syncwarp();
  float4 *st = strips + (size_t)bs * (n + 1);
  int rank[kFrontPts];
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r) {
    rank[r] = 0;
    if (keep[r])
      for (int q = 0; q < P; ++q) rank[r] += f1s[w][q] < p1[r] ? 1 : 0;
  }
  __syncwarp();
  // the f1 values in sorted order
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r)
    if (keep[r]) f1s[w][rank[r]] = p1[r];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < kFrontPts; ++r)
    if (keep[r] && BOUTE_INB(rank[r] + 1, n + 1)) {
      const float u1 = rank[r] + 1 < P ? f1s[w][rank[r] + 1] : r1;
      st[rank[r] + 1] = make_float4(p1[r], u1, p2[r], 0.f);
    }
  if (lane == 0) {
    st[0] = make_float4(-INFINITY, P > 0 ? f1s[w][0] : r1, r2, 0.f);
    counts[bs] = P + 1;
  }
}

// One thread per candidate: draw s is y_t = mean_t + shift_t,s + sqrt(cvar_t)
// eps_t,s; with constraints only a feasible draw counts; its improvement is
// summed over draw s's strips. Every thread of a block walks the draws in the
// same order, so a block stages all draws' strips in shared memory once
// (packed, by an exclusive scan of the counts) and reads them as broadcasts;
// when they do not fit it reads them from global memory the same way. VEC:
// the normals load four draws at a time.
constexpr int kAcqThreads = 128;
constexpr int kStripSmem = 3072;  // float4 strips staged per block (48 KB)

template <bool VEC>
__global__ void __launch_bounds__(kAcqThreads)
    nehvi2_kernel(const float *mean, const float *cvar, const float *shift, long long N, int S,
                  const float *eps, long long eps_stride, const float4 *strips, const int *counts,
                  int n, const double *cons, float *acq) {
  extern __shared__ __align__(16) float4 st_s[];
  __shared__ int off_s[kInsMaxS + 1];
  __shared__ int total_s;
  const int b = blockIdx.y;
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_trigger();
  const float4 *stb = strips + (size_t)b * S * (n + 1);
  const int *cnt = counts + (size_t)b * S;
  // exclusive scan of the counts (S <= 1024): loaded by all, scanned by warp 0
  for (int s = threadIdx.x; s < S; s += kAcqThreads) off_s[s + 1] = cnt[s];
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int carry = 0;
    for (int base = 0; base < S; base += 32) {
      int v = base + lane < S ? off_s[base + lane + 1] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      if (base + lane < S) off_s[base + lane + 1] = carry + v;
      carry += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) {
      off_s[0] = 0;
      total_s = carry;
    }
  }
  __syncthreads();
  const bool staged = total_s <= kStripSmem;
  if (staged)  // strip q belongs to the draw s with off[s] <= q < off[s + 1]
    for (int q = threadIdx.x; q < total_s; q += kAcqThreads) {
      int lo = 0, hi = S;  // off[lo] <= q < off[hi]
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off_s[mid] <= q) lo = mid;
        else hi = mid;
      }
      if (BOUTE_INB(q - off_s[lo], n + 1)) st_s[q] = stb[(size_t)lo * (n + 1) + (q - off_s[lo])];
    }
  __syncthreads();
  if (c >= N) return;
  const size_t o0 = ((size_t)b * 2) * N + c, o1 = o0 + N;
  const float m0 = mean[o0], m1 = mean[o1];
  const float sd0 = sqrtf(fmaxf(cvar[o0], 0.f)), sd1 = sqrtf(fmaxf(cvar[o1], 0.f));
  const bool hc = cons != nullptr;
  const float c0 = hc ? (float)cons[(size_t)b * 2] : INFINITY;
  const float c1 = hc ? (float)cons[(size_t)b * 2 + 1] : INFINITY;
  const float *e = eps + ((size_t)b * N + c) * eps_stride + (eps_stride == 0 ? (size_t)b * 2 * S : 0);
  const float *sh0 = shift + ((size_t)b * 2) * S * N + c, *sh1 = sh0 + (size_t)S * N;
  // the candidate's normals and its last shift lie inside their arrays
  if (!BOUTE_INB((eps_stride ? ((long long)b * N + c) * eps_stride : (long long)b * 2 * S) + 2 * S - 1,
                 eps_stride ? (long long)gridDim.y * N * eps_stride : (long long)gridDim.y * 2 * S) ||
      !BOUTE_INB((((long long)b * 2 + 1) * S + S - 1) * N + c, (long long)gridDim.y * 2 * S * N))
    return;
  float acc = 0.f;
  auto draw = [&](int s, float e0, float e1, float h0, float h1) {
    const float ya = fmaf(sd0, e0, m0 + h0);
    const float yb = fmaf(sd1, e1, m1 + h1);
    if (!(ya <= c0 && yb <= c1)) return;  // infeasible (or no improvement possible)
    const int k = BOUTE_INB(off_s[s + 1] - off_s[s] - 1, n + 1) ? off_s[s + 1] - off_s[s] : 0;
    const float4 *st = staged ? st_s + off_s[s] : stb + (size_t)s * (n + 1);
    float h = 0.f;
    for (int j = 0; j < k; ++j) {
      const float4 q = st[j];
      const float wdt = fmaxf(q.y - fmaxf(q.x, ya), 0.f), hgt = fmaxf(q.z - yb, 0.f);
      h = fmaf(wdt, hgt, h);
    }
    acc += h;
  };
  // eight draws' shifts and normals are loaded before any is evaluated, so
  // that their latencies overlap
  constexpr int D = 8;
  int s = 0;
  if (VEC) {
    for (; s + D <= S; s += D) {
      float h0[D], h1[D];
#pragma unroll
      for (int u = 0; u < D; ++u) {
        h0[u] = sh0[(size_t)(s + u) * N];
        h1[u] = sh1[(size_t)(s + u) * N];
      }
      float ea[D], eb[D];
#pragma unroll
      for (int u = 0; u < D; u += 4) {
        const float4 a4 = *(const float4 *)(e + s + u), b4 = *(const float4 *)(e + S + s + u);
        ea[u] = a4.x; ea[u + 1] = a4.y; ea[u + 2] = a4.z; ea[u + 3] = a4.w;
        eb[u] = b4.x; eb[u + 1] = b4.y; eb[u + 2] = b4.z; eb[u + 3] = b4.w;
      }
#pragma unroll
      for (int u = 0; u < D; ++u) draw(s + u, ea[u], eb[u], h0[u], h1[u]);
    }
  }
  for (; s < S; ++s) draw(s, e[s], e[S + s], sh0[(size_t)s * N], sh1[(size_t)s * N]);
  if (BOUTE_INB((long long)b * N + c, (long long)gridDim.y * N)) acq[(size_t)b * N + c] = acc / (float)S;
}

}  // namespace

BOUTE_BOUNDS_READER(insample)

int launch_insample_fronts(const float *Yin, int B, int n, int S, const double *ref,
                           const double *cons, float *strips, int *counts, cudaStream_t s) {
  if (n > kInsMaxN) return BOUTE_ERR_UNSUPPORTED;
  const int units = B * S;
  launch_pdl(insample_front_kernel, dim3((units + kFrontWarps - 1) / kFrontWarps),
             dim3(32 * kFrontWarps), 0, s, Yin, B, n, S, ref, cons, (float4 *)strips, counts);
  count_launch();
  return last_launch_status();
}

int launch_nehvi2(const float *mean, const float *cvar, const float *shift, int B, long long N,
                  int S, const float *eps, long long eps_stride, const float *strips,
                  const int *counts, int n, const double *cons, float *acq, cudaStream_t s) {
  const unsigned gx = (unsigned)((N + kAcqThreads - 1) / kAcqThreads);
  const size_t smem = (size_t)kStripSmem * sizeof(float4);
  const bool vec = S % 4 == 0 && eps_stride % 4 == 0 && ((uintptr_t)eps & 15) == 0;
  auto go = [&](auto kern) {
    prefer_shared(kern);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(kern, dim3(gx, B), dim3(kAcqThreads), smem, s, mean, cvar, shift, N, S, eps,
               eps_stride, (const float4 *)strips, counts, n, cons, acq);
  };
  if (vec) go(nehvi2_kernel<true>);
  else go(nehvi2_kernel<false>);
  count_launch();
  return last_launch_status();
}

}  // namespace boute

// GP fit on the device (Sec. 5.2, one exact GP per objective; Sec. 6,
// Matern-5/2 ARD kernel with outputscale on standardised outcomes):
// standardisation, kernel matrix, Cholesky factor, triangular inverse, alpha,
// and the prepacked tensor-core operands of the posterior contraction. The
// kernel matrix is formed in fp64 and kept as an fp32 pair; the factor and its
// inverse are fp32, and alpha is refined against the fp64-accurate matrix
// with double-float residuals (the paper runs its GP kernels in double
// precision, Appendix C; fp64 throughput is low on this part).
#include <math.h>

#include <algorithm>

#include <type_traits>

#include "internal.h"
#include "tile32.cuh"

namespace boute {

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double *red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < nw; ++w) t += red[w];
  return t;
}

// ---- Standardize (one block per (problem, objective)) --------------------
// (codes: outcome transforms, objective_code)
__global__ void standardize_kernel(const double *Y, int n, int m, int codes, double *Ys) {
  __shared__ double red[32];
  const int b = blockIdx.x / m, t = blockIdx.x % m;
  const int code = objective_code(codes, t);
  const double *y = Y + (size_t)b * n * m + t;
  double *ys = Ys + (size_t)b * n * m + t;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += outcome_transform(y[(size_t)i * m], code);
  const double mean = block_sum(s, red) / n;
  double ss = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double z = outcome_transform(y[(size_t)i * m], code) - mean;
    ss += z * z;
  }
  ss = block_sum(ss, red);
  double sd = n > 1 ? sqrt(ss / (n - 1)) : 1.0;
  if (!(sd >= 1e-8)) sd = 1.0;
  const double isd = 1.0 / sd;  // one division; fp64 divides are slow on this part
  __syncthreads();  // every thread has read its inputs before (aliased) outputs land
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    ys[(size_t)i * m] = (outcome_transform(y[(size_t)i * m], code) - mean) * isd;
}

// ---- fit set-up, one launch: K = s2 M52(X, X) + noise I and the side input --
// Blocks [0, nkt) of problem-objective bt compute K in fp64, one half (16 x 8)
// of a 16 x 16 tile on or below the diagonal per block of 128 threads, each
// value written to both (i, j) and (j, i), stored as an fp32 pair (hi = K
// rounded, lo = K - hi): the factorisation works on hi, the refinement of
// alpha on hi + lo. (The set-up is bound by fp64 throughput: the lower
// triangle alone, spread over as many SMs as possible.) The remaining blocks
// write the posterior's side input: scaled training inputs x / l as fp32
// hi/lo pairs (dimension-major per 32-point chunk), and in every chunk the
// objective's 1/l (hi, lo) and outputscale. Block 0 of the first problem
// clears the fit status.
// Composite kernel (kp != null: [s2_c, s2_x, beta, s_0 .. s_{d-1}] of this
// problem-objective, s_k = 0 for the routing features [0, dtau)), Sec. 5.2
// "Additive kernels" and S5 as Sec. 6 assembles them:
//   k = s2 k52(r_t) + s2_c w_i w_j k32(r_c) + s2_x k52(r_t) k32(r_c),
// r_t over the routing features, r_c over the deployment features,
// w = exp(beta sum_k s_k x_k). Its side input holds, in place of the
// coordinates' lo parts, the training points' weights w_j and beta s_k, and
// s2_c, s2_x, dtau after the outputscale.
constexpr int kSetupThreads = 128;
__host__ __device__ inline int kmat_units(int n) {
  const int tn = (n + 15) / 16;
  return tn * (tn + 1);  // tiles on or below the diagonal, two halves each
}
// COMP: the composite kernel (kp its parameters); the Matern-5/2
// instantiation carries none of its code.
template <bool COMP>
__device__ void kmat_tile(const double *X, int n, int d, int b, const double *l, double s2,
                          double noise, int unit, float *Kh, float *Kl, double *il,
                          const double *kp, int dtau) {
  for (int t = threadIdx.x; t < d; t += blockDim.x) il[t] = 1.0 / l[t];
  __syncthreads();
  const int tile = unit >> 1, half = unit & 1;
  int ti = (int)((sqrtf(8.f * tile + 1.f) - 1.f) * 0.5f);  // tile = ti (ti + 1) / 2 + tj
  while (ti * (ti + 1) / 2 > tile) --ti;
  while ((ti + 1) * (ti + 2) / 2 <= tile) ++ti;
  const int tj = tile - ti * (ti + 1) / 2;
  const int i = ti * 16 + threadIdx.x / 8, j = tj * 16 + half * 8 + threadIdx.x % 8;
  if (i >= n || j >= n) return;
  const double *xi = X + ((size_t)b * n + i) * d, *xj = X + ((size_t)b * n + j) * d;
  double r2 = 0.0, r2c = 0.0;
  const int dt = COMP ? dtau : d;
  for (int t = 0; t < dt; ++t) {
    const double z = (xi[t] - xj[t]) * il[t];
    r2 = fma(z, z, r2);
  }
  if (COMP) {
    for (int t = dt; t < d; ++t) {
      const double z = (xi[t] - xj[t]) * il[t];
      r2c = fma(z, z, r2c);
    }
  }
  const double r = sqrt(r2), sr = sqrt(5.0) * r;
  double k;
  if (!COMP) {
    k = s2 * (1.0 + sr + 5.0 * r2 / 3.0) * exp(-sr);
  } else {
    const double k52 = (1.0 + sr + 5.0 * r2 / 3.0) * exp(-sr);
    const double sc = sqrt(3.0) * sqrt(r2c), k32 = (1.0 + sc) * exp(-sc);
    double ei = 0.0, ej = 0.0;
    for (int t = dtau; t < d; ++t) {
      ei = fma(kp[3 + t], xi[t], ei);
      ej = fma(kp[3 + t], xj[t], ej);
    }
    k = s2 * k52 + kp[0] * exp(kp[2] * (ei + ej)) * k32 + kp[1] * k52 * k32;
  }
  if (i == j) k += noise;
  const float kh = (float)k, kl = (float)(k - (double)kh);
  Kh[(size_t)i * n + j] = kh;
  Kl[(size_t)i * n + j] = kl;
  if (i != j) {  // (the same value: the squared differences are symmetric)
    Kh[(size_t)j * n + i] = kh;
    Kl[(size_t)j * n + i] = kl;
  }
}

template <bool COMP>
__device__ void prep_part(const double *X, int n, int d, int b, int DP, int npad,
                          const double *l, double s2, double noise, float *x, int blk, int nblk,
                          const double *kp, int dtau) {
  const int cf = xt_chunk_floats(DP);
  const int total = npad * DP;
  for (int e = blk * blockDim.x + threadIdx.x; e < total; e += nblk * blockDim.x) {
    const int j = e / DP, t = e % DP;
    const double cs = (COMP && t >= dtau) ? kCoordScale32 : kCoordScale52;
    double v = (j < n && t < d) ? X[((size_t)b * n + j) * d + t] / l[t] * cs : 0.0;
    float hi = (float)v, lo = (float)(v - (double)hi);
    const int c = j / BOUTE_KCHUNK, jj = j % BOUTE_KCHUNK;
    float *q = x + (size_t)c * cf;  // dimension-major: [DP][32] hi, [DP][32] lo
    q[t * BOUTE_KCHUNK + jj] = hi;
    if (!COMP) q[BOUTE_KCHUNK * DP + t * BOUTE_KCHUNK + jj] = lo;
  }
  if (COMP) {  // composite kernel: w_j (row 0 of the lo block), beta s_k (row 1)
    for (int e = blk * blockDim.x + threadIdx.x; e < npad; e += nblk * blockDim.x) {
      double ej = 0.0;
      if (e < n)
        for (int t = dtau; t < d; ++t) ej = fma(kp[3 + t], X[((size_t)b * n + e) * d + t], ej);
      x[(size_t)(e / BOUTE_KCHUNK) * cf + BOUTE_KCHUNK * DP + e % BOUTE_KCHUNK] =
          e < n ? (float)exp(kp[2] * ej) : 0.f;
    }
    for (int e = blk * blockDim.x + threadIdx.x; e < (npad / BOUTE_KCHUNK) * DP;
         e += nblk * blockDim.x) {
      const int c = e / DP, k = e % DP;
      x[(size_t)c * cf + BOUTE_KCHUNK * DP + BOUTE_KCHUNK + k] =
          (k >= dtau && k < d) ? (float)(kp[2] * kp[3 + k]) : 0.f;
    }
  }
  const int po = xt_param_offset(DP), nch = npad / BOUTE_KCHUNK, np = 2 * DP + 8;
  for (int e = blk * blockDim.x + threadIdx.x; e < nch * np; e += nblk * blockDim.x) {
    const int c = e / np, k = e % np;
    float v = 0.f;
    // the coordinates' scale over l (hi, lo)
    if (k < DP) v = k < d ? (float)(((COMP && k >= dtau) ? kCoordScale32 : kCoordScale52) / l[k]) : 0.f;
    else if (k < 2 * DP) {
      const int t = k - DP;
      if (t < d) {
        const double iv = ((COMP && t >= dtau) ? kCoordScale32 : kCoordScale52) / l[t];
        v = (float)(iv - (double)(float)iv);
      }
    } else if (k == 2 * DP + kParS2) v = (float)s2;
    else if (COMP && k == 2 * DP + kParS2c) v = (float)kp[0];
    else if (COMP && k == 2 * DP + kParS2x) v = (float)kp[1];
    else if (COMP && k == 2 * DP + kParDtau) v = (float)dtau;
    else if (k == 2 * DP + kParEW)  // the prior variance bounds K's diagonal from above
      v = (float)w_scale_exp(noise, COMP ? s2 + kp[0] + kp[1] : s2);
    x[(size_t)c * cf + po + k] = v;
  }
}

template <bool COMP>
__global__ void __launch_bounds__(kSetupThreads) fit_setup_kernel(
    const double *X, int n, int d, int m, int DP, int npad, const double *ls, const double *s2,
    const double *noise, float *Kh_all, float *Kl_all, float *xt, float *s2f, int nkt, int nprep,
    int early_trigger, int *status, const double *kpar, int dtau) {
  __shared__ double il[BOUTE_MAX_D];
  const int bt = blockIdx.y, b = bt / m;
  if (early_trigger) pdl_trigger();  // the whole grid is resident: the fit may launch now
  const double *l = ls + (size_t)bt * d;
  const double *kp = COMP ? kpar + (size_t)bt * (3 + d) : nullptr;
  if (blockIdx.x == 0 && bt == 0 && threadIdx.x == 0) *status = BOUTE_OK;
  if ((int)blockIdx.x < nkt) {
    kmat_tile<COMP>(X, n, d, b, l, s2[bt], noise[bt], blockIdx.x, Kh_all + (size_t)bt * n * n,
                    Kl_all + (size_t)bt * n * n, il, kp, dtau);
  } else {
    float *x = xt + (size_t)bt * (npad / BOUTE_KCHUNK) * xt_chunk_floats(DP);
    prep_part<COMP>(X, n, d, b, DP, npad, l, s2[bt], noise[bt], x, blockIdx.x - nkt, nprep, kp,
                    dtau);
    // the prior variance's constant part (composite: s2 + s2_x; the
    // posterior adds s2_c w(x)^2)
    if (blockIdx.x == nkt && threadIdx.x == 0) s2f[bt] = (float)(COMP ? s2[bt] + kp[1] : s2[bt]);
  }
}

// The fp16 hi/lo operand images of W = L^-1 scaled by 2^e_W (see PostPlan):
// the pair of elements (g, k), (g, k + 1) of W (row g = output column, k
// even), zero above the diagonal and beyond n. Returns false if a scaled
// element reaches the fp16 range (W beyond four times its bound 1/sigma_n:
// the fp32 factor is numerically singular).
__device__ __forceinline__ bool pack_values(float w0, float w1, int g, int k, const PostPlan &plan,
                                            float scale, uint16_t *img) {
  const int n = plan.n;
  const float v0 = (k < n && g < n && k <= g) ? w0 * scale : 0.f;
  const float v1 = (k + 1 < n && g < n && k + 1 <= g) ? w1 * scale : 0.f;
  uint32_t hi, lo;
  split_f16x2(v0, v1, hi, lo);
  const int q = g / BOUTE_BLKCOLS, c = k / BOUTE_ACHUNK, ncol = plan.ncol[q];
  uint32_t *blk = (uint32_t *)(img + plan.off[q] + (long long)c * 2 * ncol * BOUTE_ACHUNK);
  const int o = sw128_off16(g % BOUTE_BLKCOLS, k % BOUTE_ACHUNK) >> 1;
  const long long base = plan.off[q] + (long long)c * 2 * ncol * BOUTE_ACHUNK;
  (void)base;  // (used by the debug build's checks)
  if (BOUTE_INB(base + 2 * ((ncol * BOUTE_ACHUNK >> 1) + o) + 1, plan.image_halves) &&
      BOUTE_INB(q, plan.nwblk)) {
    blk[o] = hi;
    blk[(ncol * BOUTE_ACHUNK >> 1) + o] = lo;
  }
  return fabsf(v0) < 32768.f && fabsf(v1) < 32768.f;
}
// Error-free product and sum on fp32 pairs (Dekker / Knuth).
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
  p = a * b;
  e = fmaf(a, b, -p);
}
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// The standardisation of one outcome column (stride m) by one warp: with
// standardize != 0 the column's mean and 1 / (sample standard deviation) (1
// when that is below 1e-8 or n = 1), as standardize_kernel computes them,
// else 0 and 1; lane 0 stores them.
__device__ __forceinline__ void standardize_stats(const double *y, int n, int m, int standardize,
                                                  int lane, double &mu, double &isd) {
  if (!standardize) {
    if (lane == 0) {
      mu = 0.0;
      isd = 1.0;
    }
    return;
  }
  double sum = 0.0;
  for (int i = lane; i < n; i += 32) sum += y[(size_t)i * m];
  const double mean = warp_sum(sum) / n;
  double ss = 0.0;
  for (int i = lane; i < n; i += 32) {
    const double z = y[(size_t)i * m] - mean;
    ss += z * z;
  }
  ss = warp_sum(ss);
  double sd = n > 1 ? sqrt(ss / (n - 1)) : 1.0;
  if (!(sd >= 1e-8)) sd = 1.0;
  if (lane == 0) {
    mu = mean;
    isd = 1.0 / sd;
  }
}

// The largest preference weight w_j of problem-objective bt (composite
// kernel), by one warp, into its parameter slot.
__device__ __forceinline__ void composite_wmax(float *xt, int bt, const PostPlan &plan, int DP,
                                               int n, int lane) {
  const int cf = xt_chunk_floats(DP);
  float *x0 = xt + (size_t)bt * plan.nxt * cf;
  const float *xw = x0 + BOUTE_KCHUNK * DP;
  float wm = 0.f;
  for (int j = lane; j < n; j += 32) wm = fmaxf(wm, xw[(size_t)(j / BOUTE_KCHUNK) * cf + j % BOUTE_KCHUNK]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
  if (lane == 0) x0[xt_param_offset(DP) + 2 * DP + kParWmax] = wm;
}

// ---- factorisation on a thread-block cluster ---------------------------------------
// The Cholesky factor of K (its fp32 rounding), W = L^-1 and alpha. fp32 arithmetic on
// the FP32 pipes: the fp32 factor is as accurate as the posterior needs, while alpha,
// which carries the condition number, gets two steps of iterative refinement against
// the fp64-accurate K = hi + lo with double-float residuals. A pivot at or below 16 *
// eps32 times its original diagonal entry counts as not positive.
// One cluster of C = Pr x Pc CTAs per problem-objective runs the whole fit after
// the set-up in one launch: K's lower triangle as 32 x 32 tiles, tile (I, J) owned
// by the CTA (I mod Pr, J mod Pc) and kept in its shared memory (n > 1024: below),
// updated in place:
//   before panel J it holds A_IJ (the trailing matrix), afterwards the transpose of
//   R_IJ = -sum_{J <= K <= p} L_IK W_KJ, and W_IJ^T = (W_II R_IJ)^T from panel I on.
// Panel p: two warps of the owner factor the diagonal tile and invert it (fc_diagonal)
// and send W_pp to the CTAs of its block row and column; cluster barrier; these form
// L_Ip = A_Ip W_pp^T (I > p) and W_pJ = W_pp R_pJ (J < p) and send each to the CTAs
// whose tiles need it; cluster barrier; every CTA updates its tiles, A_IJ -= L_Ip L_Jp^T
// (J > p) and R_IJ -= L_Ip W_pJ (J <= p), the owner of the next diagonal tile that one
// first and factoring it beside the rest, and the owners of block row p write W and its
// operand images. Then alpha and its two refinement steps from the tiles. Tiles and
// vectors travel by stores to the other CTAs' shared memory, ordered by the barriers.
// Sums run in an order that does not depend on C. What bounds it is the chain of a
// panel (two barriers, two tile products, the diagonal tile: about 15 thousand clocks at
// n = 512), for n = 1024 as much the updates' shared-memory reads.
// Fit with its set-up, against three launches a panel, nine for alpha and one block
// per problem-objective in large batches: n = 203, m = 3 174 -> 98 us; n = 512, m = 2
// 385 -> 230 us; n = 777, B = 3, m = 2 1193 -> 754 us; n = 1024, m = 3 1226 -> 943 us;
// n = 256, B = 16, m = 2 560 -> 250 us. Against one block per problem-objective with K
// and W as matrices in shared memory (n <= 160, m = 2): n = 32 32 -> 28 us, n = 128
// 69 -> 50 us, n = 160 100 -> 65 us.
constexpr int kFcThreads = 512, kFcGroups = kFcThreads / 64;
constexpr int kFcMaxCluster = 16;

__host__ __device__ inline int fc_rows(int C) { return C >= 8 ? 4 : C >= 2 ? 2 : 1; }
// tiles of the lower triangle owned by CTA (a, b) of Pr x Pc
__host__ __device__ inline int fc_slots(int nb, int a, int b, int Pr, int Pc) {
  int t = 0;
  for (int I = a; I < nb; I += Pr) t += I >= b ? (I - b) / Pc + 1 : 0;
  return t;
}
// the largest number of tiles of any CTA, and the operand tiles of a panel
__host__ __device__ inline int fc_max_slots(int nb, int C) {
  const int Pr = fc_rows(C), Pc = C / Pr;
  int t = 0;
  for (int a = 0; a < Pr; ++a)
    for (int b = 0; b < Pc; ++b) {
      const int q = fc_slots(nb, a, b, Pr, Pc);
      t = q > t ? q : t;
    }
  return t;
}
__host__ __device__ inline int fc_ops(int nb, int C) {
  const int Pr = fc_rows(C), Pc = C / Pr;
  return (nb + Pr - 1) / Pr + (nb + Pc - 1) / Pc;
}
// Shared memory of CTA `rank` of the cluster at this CTA's address p, and stores there.
__device__ __forceinline__ uint32_t fc_remote(const float *p, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void fc_store4(uint32_t a, const float4 &v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void fc_store1(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// Word offset of tile (I, J) among the lower triangle's, row by row, and the coordinates
// of the e-th.
__device__ __forceinline__ size_t tri_tile(int I, int J) {
  return (size_t)(I * (I + 1) / 2 + J) * kFcTile;
}
__device__ __forceinline__ void tri_coords(int e, int &I, int &J) {
  I = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
  while (I * (I + 1) / 2 > e) --I;
  while ((I + 1) * (I + 2) / 2 <= e) ++I;
  J = e - I * (I + 1) / 2;
}

// Rows r0 .. r0 + 7 of W_IJ, from the final tile T = W_IJ^T, by one warp: W itself and its
// operand images (false if an element does not fit them).
__device__ __forceinline__ bool fc_output(const float *T, int I, int J, int r0, int lane, int NP,
                                          const PostPlan &plan, float wscale, float *W,
                                          uint16_t *img) {
  const int n = plan.n, gmax = BOUTE_BLKCOLS * (plan.nwblk - 1) + plan.ncol[plan.nwblk - 1];
  bool fits = true;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = 32 * I + r0 + u, k = 32 * J + lane;
    if (i < n && k <= i) W[(size_t)i * (NP + 1) + k] = T[fc_off(lane, r0 + u)];
  }
  const int kk = 2 * (lane & 15);
#pragma unroll 1
  for (int u = 0; u < 8; u += 2) {
    const int r = r0 + u + (lane >> 4), g = 32 * I + r;
    if (g >= gmax) continue;
    fits &= pack_values(T[fc_off(kk, r)], T[fc_off(kk + 1, r)], g, 32 * J + kk, plan, wscale, img);
    if (I == J)  // zeros right of the diagonal tile, as far as the block's chunks reach
#pragma unroll 1
      for (int k = 32 * (J + 1) + kk; k < BOUTE_ACHUNK * plan.kc[g / BOUTE_BLKCOLS]; k += 32)
        pack_values(0.f, 0.f, g, k, plan, wscale, img);
  }
  return fits;
}

// TS: the tiles in shared memory; otherwise factored tiles in the workspace, alpha alone.
template <bool TS>
__global__ void __launch_bounds__(kFcThreads, 1) fitc_kernel(
    const float *Kh_all, const float *Kl_all, const double *Ys, int standardize, int n, int m,
    int NP, int C, int max_slots, float *Aws, float *Wws, float *xt, int DP, PostPlan plan,
    uint16_t *bop, int comp, int *status, int *fbad_all) {
  extern __shared__ __align__(16) float sm[];
  __shared__ __align__(16) FcDiag dsh;
  __shared__ double ymu, yisd;
  __shared__ int row_first[BOUTE_MAX_N / 32 + 1];  // the first slot of each block row of this CTA
  __shared__ int next_item, item[kFcGroups];       // the updates' queue beside a diagonal tile
  const int bt = blockIdx.x / C, rank = blockIdx.x % C, b = bt / m, t = bt % m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kFcThreads / 32;
  const int grp = tid >> 6, gt = tid & 63;
  const int nb = NP / 32, Pr = fc_rows(C), Pc = C / Pr, ra = rank % Pr, rb = rank / Pr;
  const int sr = 31 - __clz(Pr), sc = 31 - __clz(Pc);  // (powers of two)
  const int nR = (nb + Pr - 1) / Pr, nC = (nb + Pc - 1) / Pc;
  // operand tiles of a panel (rows: L_Ip; columns: L_Jp or W_pJ^T), W_pp, W_pp^T of
  // two panels, K's diagonal at this CTA's block rows, the slots' block coordinates
  float *rop = sm, *cop = rop + (size_t)nR * kFcTile, *wpp = cop + (size_t)nC * kFcTile;
  float *wt = wpp + kFcTile, *dg = wt + 2 * kFcTile;
  unsigned short *slotI = (unsigned short *)(dg + 32 * nR), *slotJ = slotI + max_slots;
  float *tiles = TS ? dg + 32 * nR + ((max_slots + 3) & ~3) : Aws + (size_t)bt * NP * (NP + 1);
  int *fbad = fbad_all + bt;
  auto sync = [&]() {
    __syncwarp();
    if (C > 1)
      asm volatile(
          "barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
              : "memory");
    else
      __syncthreads();
  };
  // this CTA's block rows I = ra + Pr i, each with the columns J = rb + Pc j <= I
  const int lrows = ra < nb ? ((nb - 1 - ra) >> sr) + 1 : 0;
  auto row_count = [&](int I) { return I >= rb ? ((I - rb) >> sc) + 1 : 0; };
  int nslots = 0;
  if constexpr (TS) {
    for (int i = tid; i <= lrows; i += kFcThreads) {
      int q = 0;
      for (int e = 0; e < i; ++e) q += row_count(ra + (e << sr));
      row_first[i] = q;
    }
    __syncthreads();
    nslots = row_first[lrows];
    for (int i = warp; i < lrows; i += nw)
      for (int j = lane; j < row_count(ra + (i << sr)); j += 32) {
        slotI[row_first[i] + j] = (unsigned short)(ra + (i << sr));
        slotJ[row_first[i] + j] = (unsigned short)(rb + (j << sc));
      }
  }
  const double *y = Ys + (size_t)b * n * m + t;
  if (warp == nw - 1) standardize_stats(y, n, m, standardize, lane, ymu, yisd);
  // everything below reads what the set-up kernel wrote
  pdl_wait();
  const float *Kh = Kh_all + (size_t)bt * n * n, *Kl = Kl_all + (size_t)bt * n * n;
  const int cf = xt_chunk_floats(DP);
  float *x0 = xt + (size_t)bt * plan.nxt * cf;
  bool fits = true;
  auto at = [&](const float *q, int r) { return fc_remote(q, r); };
  if constexpr (TS) {
    if (rank == 0 && tid == 0) __stcg(fbad, 0);
    for (int e = tid; e < 32 * lrows; e += kFcThreads) {
      const int i = 32 * (ra + ((e >> 5) << sr)) + (e & 31);
      dg[e] = i < n ? Kh[(size_t)i * n + i] : 1.f;
    }
    __syncthreads();
    for (int e = warp; e < 4 * nslots; e += nw) {  // eight rows of a tile per warp
      const int s = e >> 2, r0 = 8 * (e & 3), i0 = 32 * slotI[s] + r0, k = 32 * slotJ[s] + lane;
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u;
        v[u] = (i < n && k < n) ? Kh[(size_t)i * n + k] : (i == k ? 1.f : 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) tiles[(size_t)s * kFcTile + fc_off(r0 + u, lane)] = v[u];
    }
    __syncthreads();
    // W_pp and W_pp^T, from this CTA's wpp and wt, to the CTAs of block row and column p
    auto send_diagonal = [&](int p) {
      const int a = p & (Pr - 1), c = p & (Pc - 1), par = p & 1;
      float4 v[4], w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = ((const float4 *)wpp)[gt + 64 * u];
        w[u] = ((const float4 *)(wt + par * kFcTile))[gt + 64 * u];
      }
      for (int q = 0; q < Pr + Pc; ++q) {
        const int r = q < Pr ? q + Pr * c : a + Pr * (q - Pr);
        if (r == rank) continue;
        const uint32_t dst = at(wpp, r) + 16 * gt, dwt = at(wt + par * kFcTile, r) + 16 * gt;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          fc_store4(dst + 1024 * u, v[u]);
          if (q < Pr) fc_store4(dwt + 1024 * u, w[u]);
        }
      }
    };
    sync();  // every CTA of the cluster runs: its shared memory may be written
    if (rank == 0 && grp == 0) {
      fc_diagonal(tiles, dg, dsh, wpp, wt, fbad);
      named_barrier_sync(1, 64);
      send_diagonal(0);
    }
    float acc[4][4];
    const int tx = gt & 7, ty = gt >> 3;
    // block row p of W (final after panel p's products): W itself and its operand images
    const float wscale = exp2i((int)x0[xt_param_offset(DP) + 2 * DP + kParEW]);
    uint16_t *img = bop + (size_t)bt * plan.image_halves;
    float *W = Wws + (size_t)bt * NP * (NP + 1);
    auto output_row = [&](int p) {
      const int f = row_first[(p - ra) >> sr], cnt = 4 * row_count(p);
#pragma unroll 1
      for (int e = warp; e < cnt; e += nw) {  // eight rows of a tile per warp
        const int s = f + (e >> 2);
        fits &= fc_output(tiles + (size_t)s * kFcTile, p, slotJ[s], 8 * (e & 3), lane, NP, plan,
                          wscale, W, img);
      }
      __syncwarp();
    };
    for (int p = 0; p < nb; ++p) {
      sync();  // W_pp has arrived; the previous panel's operands are consumed
      // L_Ip = A_Ip W_pp^T and W_pJ^T = R_pJ^T W_pp^T
      const int i1 = p < ra ? 0 : ((p - ra) >> sr) + 1;  // first block row of this CTA below p
      const int f1 = row_first[i1], a = p & (Pr - 1), c = p & (Pc - 1);
      const int nl = rb == c ? lrows - i1 : 0;
      const int nwt = ra == a ? row_count(p) - (rb == c ? 1 : 0) : 0;
      if (tid == 0) next_item = f1;
      for (int e = grp; e < nl + nwt; e += kFcGroups) {
        int s, X;
        if (e < nl) {
          X = ra + ((i1 + e) << sr);
          s = row_first[i1 + e] + ((p - rb) >> sc);
        } else {
          s = row_first[(p - ra) >> sr] + (e - nl);
          X = rb + ((e - nl) << sc);
        }
        float *T = tiles + (size_t)s * kFcTile;
        fc_product(T, wpp, gt, acc);
        // to the column operands of CTAs (., X mod Pc) and, L_Ip, the row operands of
        // CTAs (X mod Pr, .)
        const int o = ((4 * ty) * 8 + (tx ^ ty)) * 16;
        if (p < nb - 1)
          for (int q = 0; q < (e < nl ? Pr + Pc : Pr); ++q) {
            const uint32_t dst =
                o + (q < Pr ? at(cop + (size_t)(X >> sc) * kFcTile, q + Pr * (X & (Pc - 1)))
                            : at(rop + (size_t)(X >> sr) * kFcTile,
                                 (X & (Pr - 1)) + Pr * (q - Pr)));
#pragma unroll
            for (int u = 0; u < 4; ++u)
              fc_store4(dst + 128 * u, make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]));
          }
        if (e >= nl) {
          named_barrier_sync(1 + grp, 64);  // the tile is read
#pragma unroll
          for (int u = 0; u < 4; ++u)
            ((float4 *)T)[(4 * ty + u) * 8 + (tx ^ ty)] =
                make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
        }
      }
      if (p == nb - 1) break;
      sync();  // L_Ip and W_pJ have arrived
      // update: the slots from block row i1 on; the next diagonal tile first, by group 0
      auto update = [&](int s) {
        const int I = slotI[s], J = slotJ[s];
        const float *L = rop + (size_t)(I >> sr) * kFcTile;
        const float *Q = J == p ? wt + (p & 1) * kFcTile : cop + (size_t)(J >> sc) * kFcTile;
        float *T = tiles + (size_t)s * kFcTile;
        fc_product(J > p ? L : Q, J > p ? Q : L, gt, acc);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float4 *q = (float4 *)T + (4 * ty + u) * 8 + (tx ^ ty);
          float4 v = J == p ? make_float4(0.f, 0.f, 0.f, 0.f) : *q;
          v.x -= acc[u][0];
          v.y -= acc[u][1];
          v.z -= acc[u][2];
          v.w -= acc[u][3];
          *q = v;
        }
      };
      const bool own = ((p + 1) & (Pr - 1)) == ra && ((p + 1) & (Pc - 1)) == rb;
      if (own) {
        // Beside the diagonal tile's two warps only the groups of the other two
        // schedulers work (odd groups); the rest join them afterwards.
        const int sd = row_first[i1] + ((p + 1) >> sc);  // the diagonal tile's slot
        if (grp == 0) {
          update(sd);
          named_barrier_sync(1, 64);
          fc_diagonal(tiles + (size_t)sd * kFcTile, dg + 32 * i1, dsh, wpp,
                      wt + ((p + 1) & 1) * kFcTile, fbad);
          named_barrier_sync(1, 64);
          send_diagonal(p + 1);
        }
        if (!(grp & 1)) named_barrier_sync(13, 32 * nw / 2);
        for (;;) {
          if (gt == 0) item[grp] = atomicAdd(&next_item, 1);
          __syncwarp();
          named_barrier_sync(1 + grp, 64);
          const int s = item[grp];
          if (s >= nslots) break;
          if (s != sd) update(s);
          named_barrier_sync(1 + grp, 64);  // (item is read)
        }
      } else {
        for (int s = f1 + grp; s < nslots; s += kFcGroups) update(s);
      }
      if (ra == a) output_row(p);
    }
    pdl_trigger();
    __syncthreads();
    if (ra == ((nb - 1) & (Pr - 1))) output_row(nb - 1);
  } else {  // (factored by the fitg_* kernels)
    pdl_trigger();
    sync();  // every CTA of the cluster runs: its shared memory may be written
  }
  // ---- alpha0 = W^T (W y), refined twice against K = hi + lo ----------------------
  // (vectors in the operands' space: x, alpha, y hi, y lo, the partial sums of the CTA's
  // block rows and of every column, four classes of tiles each)
  float *x = sm, *al = x + NP, *yv = al + NP, *ylo = yv + NP, *pt = ylo + NP, *pw = pt + 4 * NP;
  {
    const double mu = ymu, isd = yisd;
    for (int i = tid; i < NP; i += kFcThreads) {  // standardised y as an fp32 pair
      const double ys = i < n ? (y[(size_t)i * m] - mu) * isd : 0.0;
      yv[i] = x[i] = (float)ys;
      ylo[i] = (float)(ys - (double)yv[i]);
    }
  }
  __syncthreads();
  // out(k, (W^T (W x))_k) for every k, in every CTA. W x: a warp per block row and class
  // J mod 4, lane = row; W^T: a warp per block column and class I mod 4, lane = column;
  // tiles in ascending order, then the classes.
  const int kr = 4 / Pr, kcl = 4 / Pc;  // classes of block rows and columns in this CTA
  const int lcols = rb < nb ? ((nb - 1 - rb) >> sc) + 1 : 0;
  // tile (row i, column j) of this CTA's; in the workspace the triangle's tiles in order
  auto tile_at = [&](int i, int j) {
    if (TS) return tiles + (size_t)(row_first[i] + j) * kFcTile;
    return tiles + tri_tile(ra + (i << sr), rb + (j << sc));
  };
  auto solve = [&](auto out) {
#pragma unroll 1
    for (int e = warp; e < lrows * kcl; e += nw) {
      const int i = e / kcl, q = rb + Pc * (e % kcl), I = ra + (i << sr);
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
      for (int J = q; J <= I; J += 4) {
        const float *T = tile_at(i, J >> sc), *xj = x + 32 * J;
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          s0 = fmaf(T[fc_off(k, lane)], xj[k], s0);
          s1 = fmaf(T[fc_off(k + 1, lane)], xj[k + 1], s1);
          s2 = fmaf(T[fc_off(k + 2, lane)], xj[k + 2], s2);
          s3 = fmaf(T[fc_off(k + 3, lane)], xj[k + 3], s3);
        }
      }
      const float v = (s0 + s1) + (s2 + s3);
      for (int r = 0; r < Pc; ++r) fc_store1(at(pw + q * 32 * nR + 32 * i + lane, ra + Pr * r), v);
    }
    sync();
    for (int e = tid; e < 32 * lrows; e += kFcThreads) {  // (class 0's words take the sum)
      const int w = 32 * nR;
      pw[e] = (pw[e] + pw[e + w]) + (pw[e + 2 * w] + pw[e + 3 * w]);
    }
    __syncthreads();
#pragma unroll 1
    for (int e = warp; e < lcols * kr; e += nw) {
      const int j = e / kr, q = ra + Pr * (e % kr), J = rb + (j << sc);
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
      for (int I = q; I < nb; I += 4) {
        if (I < J) continue;
        const int i = (I - ra) >> sr;
        const float4 *T4 = (const float4 *)tile_at(i, j) + lane * 8;
        const float4 *v4 = (const float4 *)(pw + 32 * i);
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const float4 w = T4[(g ^ (lane >> 2)) & 7], v = v4[g];
          s0 = fmaf(w.x, v.x, s0);
          s1 = fmaf(w.y, v.y, s1);
          s2 = fmaf(w.z, v.z, s2);
          s3 = fmaf(w.w, v.w, s3);
        }
      }
      const float v = (s0 + s1) + (s2 + s3);
      for (int r = 0; r < C; ++r) fc_store1(at(pt + q * NP + 32 * J + lane, r), v);
    }
    sync();
    for (int k = tid; k < NP; k += kFcThreads)
      out(k, (pt[k] + pt[k + NP]) + (pt[k + 2 * NP] + pt[k + 3 * NP]));
    __syncthreads();
  };
  solve([&](int k, float v) { al[k] = v; });
#pragma unroll 1
  for (int step = 0; step < 2; ++step) {
    // r = y - K alpha in double-float, a half warp per row, eight loads of each of K
    // hi and K lo per lane in flight; to every CTA's x
    const int hl = lane & 15;
#pragma unroll 1
    for (int i = rank * (kFcThreads / 16) + (tid >> 4); i < NP; i += C * (kFcThreads / 16)) {
      float sh = 0.f, sl = 0.f;
      if (i < n) {
#pragma unroll 1
        for (int k0 = 0; k0 < n; k0 += 128) {
          float h8[8], l8[8], a8[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int k = k0 + hl + 16 * u;
            const bool in = k < n;
            a8[u] = in ? al[k] : 0.f;
            h8[u] = in ? Kh[(size_t)i * n + k] : 0.f;
            l8[u] = in ? Kl[(size_t)i * n + k] : 0.f;
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            float pr, e, s_, e2;
            two_prod(h8[u], a8[u], pr, e);
            two_sum(sh, pr, s_, e2);
            sh = s_;
            sl += e2 + fmaf(l8[u], a8[u], e);
          }
        }
      }
      const unsigned half = 0xffffu << (lane & 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {  // within the half warp
        const float oh = __shfl_xor_sync(half, sh, o);
        const float ol = __shfl_xor_sync(half, sl, o);
        float s_, e;
        two_sum(sh, oh, s_, e);
        sh = s_;
        sl += ol + e;
      }
      // (the lanes' sl may differ in the last bit: every CTA gets the first lane's)
      const float r = __shfl_sync(half, i < n ? (yv[i] - sh) + (ylo[i] - sl) : 0.f, 0, 16);
      if (hl < C) fc_store1(at(x + i, hl), r);
    }
    sync();
    // the second correction is kept exactly: alpha = hi + lo, hi = fl(alpha + delta)
    solve([&](int k, float v) {
      float s_, e;
      two_sum(al[k], v, s_, e);
      al[k] = s_;
      if (step == 1) x[k] = e;  // (before that other CTAs may be sending the next residual)
    });
  }
  // (cluster barriers lie between the last pivot and here)
  const bool bad = __ldcg(fbad) != 0;
  if (bad || !fits) set_status(status, BOUTE_ERR_NOT_PD);
  if (bad) return;
  float *xa = x0 + xt_alpha_offset(DP);
  for (int k = rank * kFcThreads + tid; k < BOUTE_KCHUNK * plan.nxt; k += C * kFcThreads) {
    float *q = xa + (size_t)(k / BOUTE_KCHUNK) * cf + k % BOUTE_KCHUNK;
    q[0] = k < n ? al[k] : 0.f;
    q[BOUTE_KCHUNK] = k < n ? x[k] : 0.f;
  }
  if (comp && rank == 0 && warp == nw - 1) composite_wmax(xt, bt, plan, DP, n, lane);
}

// ---- factorisation over the whole GPU -------------------------------------------------
// More tiles than a cluster's shared memory holds (n > 1024): the same tiles, sums and
// orders as above, the tiles in the workspace (the triangle's row by row, then L_Ip of the
// present panel, then W_pp), 64 threads a tile product, two launches a panel over as many
// blocks as there are products. What bounds it is the products' operands from L2 (16 KB
// each), for small n the launches (about 6 us a panel). Fit with its set-up, against one
// cluster per problem-objective, whose 16 SMs do all the products: n = 1025, m = 1 776 ->
// 451 us; n = 1025, B = 8, m = 2 3178 -> 2311 us; n = 1536, m = 2 1854 -> 964 us; n = 2048,
// m = 1 3211 -> 1079 us, m = 3 3800 -> 2231 us.

// K's tiles; block 0 factors the first diagonal tile and clears fbad.
__global__ void __launch_bounds__(64)
    fitg_load_kernel(const float *Kh_all, int n, int NP, float *Aws, int *fbad_all) {
  __shared__ __align__(16) float ts[kFcTile];
  __shared__ __align__(16) FcDiag dsh;
  __shared__ float dg[32];
  pdl_wait();
  pdl_trigger();
  const int bt = blockIdx.y, tid = threadIdx.x, lane = tid & 31, nb = NP / 32;
  const float *Kh = Kh_all + (size_t)bt * n * n;
  float *tiles = Aws + (size_t)bt * NP * (NP + 1), *T = tiles + (size_t)blockIdx.x * kFcTile;
  float *dst = blockIdx.x == 0 ? ts : T;
  int I, J;
  tri_coords(blockIdx.x, I, J);
#pragma unroll 8
  for (int r = tid >> 5; r < 32; r += 2) {
    const int i = 32 * I + r, k = 32 * J + lane;
    dst[fc_off(r, lane)] = (i < n && k < n) ? Kh[(size_t)i * n + k] : (i == k ? 1.f : 0.f);
  }
  if (blockIdx.x) return;
  if (tid < 32) dg[tid] = tid < n ? Kh[(size_t)tid * n + tid] : 1.f;
  if (tid == 0) fbad_all[bt] = 0;
  __syncthreads();
  fc_diagonal(ts, dg, dsh, tiles + tri_tile(nb + 1, 0) - kFcTile, T, fbad_all + bt);
}

__device__ __forceinline__ void fitg_copy(float *dst, const float *src, int tid) {
#pragma unroll
  for (int u = 0; u < 4; ++u) ((float4 *)dst)[tid + 64 * u] = ((const float4 *)src)[tid + 64 * u];
}

// Panel p: W_pJ^T (J < p) in place, L_Ip (I > p) beside the tiles.
__global__ void __launch_bounds__(64) fitg_panel_kernel(int NP, float *Aws, int p) {
  __shared__ __align__(16) float ts[kFcTile], ws[kFcTile];
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, nb = NP / 32;
  float *tiles = Aws + (size_t)blockIdx.y * NP * (NP + 1), *L = tiles + tri_tile(nb, 0);
  const int X = (int)blockIdx.x < p ? blockIdx.x : blockIdx.x + 1;
  float *T = tiles + (X > p ? tri_tile(X, p) : tri_tile(p, X));
  fitg_copy(ts, T, tid);
  fitg_copy(ws, L + (size_t)nb * kFcTile, tid);
  __syncthreads();
  float acc[4][4];
  fc_product(ts, ws, tid, acc);
  if (X > p) T = L + (size_t)X * kFcTile;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    ((float4 *)T)[(4 * ty + u) * 8 + (tx ^ ty)] =
        make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
}

// The tiles of the block rows below panel p; block 0 the next diagonal tile, which it factors.
__global__ void __launch_bounds__(64)
    fitg_update_kernel(const float *Kh_all, int n, int NP, float *Aws, int p, int *fbad_all) {
  __shared__ __align__(16) float ls[kFcTile], qs[kFcTile];
  __shared__ __align__(16) FcDiag dsh;
  __shared__ float dg[32];
  pdl_wait();
  pdl_trigger();
  const int bt = blockIdx.y, tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, nb = NP / 32;
  float *tiles = Aws + (size_t)bt * NP * (NP + 1), *L = tiles + tri_tile(nb, 0);
  int I = p + 1, J = p + 1;
  if (blockIdx.x) {  // (the diagonal tile is number p + 1 of its row)
    const int e = (int)blockIdx.x - 1;
    tri_coords((p + 1) * (p + 2) / 2 + e + (e > p ? 1 : 0), I, J);
  }
  float *T = tiles + tri_tile(I, J);
  float4 old[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    old[u] = J == p ? make_float4(0.f, 0.f, 0.f, 0.f)
                    : ((const float4 *)T)[(4 * ty + u) * 8 + (tx ^ ty)];
  fitg_copy(ls, L + (size_t)I * kFcTile, tid);
  fitg_copy(qs, J > p ? L + (size_t)J * kFcTile : tiles + tri_tile(p, J), tid);
  __syncthreads();
  float acc[4][4];
  fc_product(J > p ? ls : qs, J > p ? qs : ls, tid, acc);
  if (blockIdx.x == 0) __syncthreads();  // (ls is read)
  float *D = blockIdx.x == 0 ? ls : T;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    ((float4 *)D)[(4 * ty + u) * 8 + (tx ^ ty)] =
        make_float4(old[u].x - acc[u][0], old[u].y - acc[u][1], old[u].z - acc[u][2],
                    old[u].w - acc[u][3]);
  if (blockIdx.x) return;
  const float *Kh = Kh_all + (size_t)bt * n * n;
  const int i = 32 * I + tid;
  if (tid < 32) dg[tid] = i < n ? Kh[(size_t)i * n + i] : 1.f;
  __syncthreads();
  fc_diagonal(ls, dg, dsh, L + (size_t)nb * kFcTile, T, fbad_all + bt);
}

// W and its operand images, a tile per block.
__global__ void __launch_bounds__(64)
    fitg_output_kernel(int NP, const float *Aws, float *Wws, const float *xt, int DP, PostPlan plan,
                       uint16_t *bop, int *status, const int *fbad_all) {
  pdl_wait();
  pdl_trigger();
  const int bt = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (fbad_all[bt]) return;  // (fitc_kernel reports it)
  const float *x0 = xt + (size_t)bt * plan.nxt * xt_chunk_floats(DP);
  const float *T = Aws + (size_t)bt * NP * (NP + 1) + (size_t)blockIdx.x * kFcTile;
  const float wscale = exp2i((int)x0[xt_param_offset(DP) + 2 * DP + kParEW]);
  int I, J;
  tri_coords(blockIdx.x, I, J);
  bool fits = true;
  for (int r0 = 8 * warp; r0 < 32; r0 += 16)
    fits &= fc_output(T, I, J, r0, lane, NP, plan, wscale, Wws + (size_t)bt * NP * (NP + 1),
                      bop + (size_t)bt * plan.image_halves);
  if (!fits) set_status(status, BOUTE_ERR_NOT_PD);
}

}  // namespace

// Outcome transforms alone (codes != 0), elementwise: Yt = t(Y), count
// values of m objectives.
__global__ void transform_kernel(const double *Y, long long count, int m, int codes, double *Yt) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x)
    Yt[e] = outcome_transform(Y[e], objective_code(codes, (int)(e % m)));
}

int launch_outcome_transform(const double *Y, long long count, int m, int codes, double *Yt,
                             cudaStream_t s) {
  const int blocks = (int)std::min<long long>((count + 255) / 256, 1024);
  transform_kernel<<<std::max(blocks, 1), 256, 0, s>>>(Y, count, m, codes, Yt);
  count_launch();
  return last_launch_status();
}

int launch_standardize(const double *Y, int B, int n, int m, int codes, double *Ys,
                       cudaStream_t s) {
  standardize_kernel<<<B * m, 256, 0, s>>>(Y, n, m, codes, Ys);
  count_launch();
  return last_launch_status();
}

// Dynamic shared memory of fitc_kernel with clusters of C: operands and tiles, or alpha's
// vectors alone.
static size_t fitc_smem(int npad, int C, bool tiles) {
  const int nb = npad / 32, ms = fc_max_slots(nb, C), nR = (nb + fc_rows(C) - 1) / fc_rows(C);
  if (!tiles) return ((size_t)8 * npad + 4 * 32 * nR) * sizeof(float);
  return ((size_t)(fc_ops(nb, C) + 3 + ms) * kFcTile + 32 * nR + ((ms + 3) & ~3)) * sizeof(float);
}
constexpr size_t kFcMaxSmem = 227 * 1024 - 5 * 1024;  // (its static part: 4.9 KB)

// Clusters of the largest size of which the device holds one per problem-objective at
// once (a cluster lies within a GPC, so of 152 SMs clusters of 16 reach 112, of 8 120 and
// of 4 144: the held clusters are asked for, not the SMs divided. n = 512, 16
// problem-objectives: 535 us on clusters of 4, 655 in two waves of 8; n = 256: 154
// against 215; n = 128, 38 of them: 93 on clusters of 2, 122 in two waves of 4), no more
// CTAs than block rows (n = 32 on one CTA 28 us, on two 30; n = 128 on four 50, on
// eight 53; n = 203 on four 101, on eight 98), and enough that operands and tiles fit
// shared memory (n = 256 on single CTAs, n = 1024 on 16; above that the whole GPU factors
// the tiles and the clusters solve for alpha alone).
static int launch_fitc(Gp *gp, const double *Ys, int standardize, cudaStream_t s) {
  const int n = gp->n, m = gp->m, npad = gp->plan.npad, nb = npad / 32;
  const long long BM = (long long)gp->B * m, sms = num_sms();
  int least = 1;
  while (least < kFcMaxCluster && fitc_smem(npad, least, true) > kFcMaxSmem) least *= 2;
  bool tiles = fitc_smem(npad, least, true) <= kFcMaxSmem;
  if (!tiles) least = 1;
  int C = least;
  while (C < kFcMaxCluster && C < nb && 2 * C * BM <= sms) C *= 2;
  // launches unless the device cannot hold `want` clusters of C
  auto go = [&](auto kern, long long want) {
    prefer_shared(kern);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFcMaxSmem);
    if (C > 8) cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(BM * C));
    cfg.blockDim = dim3(kFcThreads);
    cfg.dynamicSmemBytes = fitc_smem(npad, C, tiles);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int held = 0;
    if (C > 1 &&
        (cudaOccupancyMaxActiveClusters(&held, kern, &cfg) != cudaSuccess || held < want)) {
      cudaGetLastError();
      return false;
    }
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, kern, (const float *)gp->Kh, (const float *)gp->Kl, Ys, standardize, n,
                       m, npad, C, fc_max_slots(nb, C), gp->Aws, gp->Wws, gp->xt, gp->DP, gp->plan,
                       gp->bop, gp->kern, gp->status, gp->fbad);
    return true;
  };
  auto factor = [&]() {  // (every lower tile a product for each panel above it)
    const unsigned nt = nb * (nb + 1) / 2, y = (unsigned)BM;
    launch_pdl(fitg_load_kernel, dim3(nt, y), dim3(64), 0, s, (const float *)gp->Kh, n, npad,
               gp->Aws, gp->fbad);
    for (int p = 0; p < nb; ++p) {
      if (nb > 1) launch_pdl(fitg_panel_kernel, dim3(nb - 1, y), dim3(64), 0, s, npad, gp->Aws, p);
      if (p + 1 < nb)
        launch_pdl(fitg_update_kernel, dim3(nt - (p + 1) * (p + 2) / 2, y), dim3(64), 0, s,
                   (const float *)gp->Kh, n, npad, gp->Aws, p, gp->fbad);
    }
    launch_pdl(fitg_output_kernel, dim3(nt, y), dim3(64), 0, s, npad, (const float *)gp->Aws,
               gp->Wws, (const float *)gp->xt, gp->DP, gp->plan, gp->bop, gp->status,
               (const int *)gp->fbad);
    count_launch(2 * nb + 1);
  };
  if (tiles) {
    while (C > least && !go(fitc_kernel<true>, BM)) C /= 2;
    // (a partitioned device may not place clusters of `least`)
    if (C > least || go(fitc_kernel<true>, 1)) {
      count_launch(2);
      return last_launch_status();
    }
    tiles = false;
    C = 1;
  }
  factor();
  while (C > 1 && !go(fitc_kernel<false>, BM)) C /= 2;
  if (C == 1) go(fitc_kernel<false>, 1);
  count_launch(2);
  return last_launch_status();
}

// Ys: standardised outcomes, or raw outcomes when standardize != 0.
static int launch_fit_impl(Gp *gp, const double *X, const double *Ys, int standardize,
                           const double *ls, const double *s2, const double *noise,
                           cudaStream_t s, cudaEvent_t setup_done = nullptr) {
  const int n = gp->n, d = gp->d, m = gp->m, BM = gp->B * gp->m;
  const int xpad = BOUTE_KCHUNK * gp->plan.nxt;
  const int nkt = kmat_units(n);
  const int sms = num_sms();
  // side-input blocks: as many as leave one block per SM (K blocks first), 2 .. 16
  const int nprep = std::max(2, std::min(16, sms / BM - nkt));
  // The set-up lets the fit launch from its first instruction on where its whole grid is
  // resident at once with room to spare (8 blocks an SM, on all but one SM per
  // problem-objective). The fit's CTAs, a whole SM each, come only when every set-up block
  // has started, so they never hold what a later block needs, however many they are; with
  // several waves of set-up blocks they would only wait on SMs that the last wave could use.
  const long long setup_blocks = (long long)(nkt + nprep) * BM;
  const int setup_early = setup_blocks <= 8LL * (sms - BM) ? 1 : 0;
  auto setup = [&](auto kern) {
    prefer_shared(kern);
    kern<<<dim3(nkt + nprep, BM), kSetupThreads, 0, s>>>(X, n, d, m, gp->DP, xpad, ls, s2, noise,
                                                         gp->Kh, gp->Kl, gp->xt, gp->s2f, nkt,
                                                         nprep, setup_early, gp->status,
                                                         gp->kpar, gp->dtau);
  };
  if (gp->kern) setup(fit_setup_kernel<true>);
  else setup(fit_setup_kernel<false>);
  if (setup_done && cudaEventRecord(setup_done, s) != cudaSuccess) return last_launch_status();
  return launch_fitc(gp, Ys, standardize, s);
}

int launch_fit(Gp *gp, const double *X, const double *Ys, const double *ls, const double *s2,
               const double *noise, cudaStream_t s) {
  return launch_fit_impl(gp, X, Ys, 0, ls, s2, noise, s);
}

int launch_fit_raw(Gp *gp, const double *X, const double *Y, const double *ls, const double *s2,
                   const double *noise, cudaStream_t s, cudaEvent_t setup_done) {
  return launch_fit_impl(gp, X, Y, 1, ls, s2, noise, s, setup_done);
}

BOUTE_BOUNDS_READER(fit)

}  // namespace boute

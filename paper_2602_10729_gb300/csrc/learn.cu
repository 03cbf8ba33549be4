// Hyperparameter learning by maximising the GP's log marginal likelihood
// (Sec. 6: the ARD lengthscales and outputscale are learned jointly by
// maximising the marginal likelihood; all kernels in double precision).
//
// One thread-block cluster per (problem, objective, restart) runs the whole
// optimisation: per Adam step it builds K = s2 M52(X, X) + noise I in fp64,
// factors it, inverts the factor and forms K^-1, alpha = K^-1 y, the log
// likelihood (at the end) and its gradient with respect to
// theta = (log l_1 .. log l_d, log s2, log noise),
//   d log p / d theta_q = 1/2 sum_ij (alpha_i alpha_j - K^-1_ij) dK_ij / dtheta_q,
// then takes a bias-corrected Adam ascent step and clamps theta to its bounds.
//
// What bounds it: fp64 issue. Measured here: one fp64 warp instruction every 19
// clocks per SM whatever its active lanes, 110 clocks from a single warp, so
// the work has to fill whole warps on as many SMs as possible, and what is
// serial (a pivot's reciprocal, 350 clocks, per column) has to run beside the
// rest. The matrices are therefore cut into 16 x 16 tiles (one entry per thread
// of 256), spread over the cluster's CTAs, in a workspace in global memory that
// stays in L2 (tile products take 2400 clocks of fp64 issue, their operands 6 KB).
// The factorisation is right-looking over tile columns p, and the rows of
// W = L^-1 and K^-1 = W^T W grow in the same loop:
//   panel phase   L_ip = A_ip W_pp^T (i > p), W_pJ = W_pp B_pJ (J < p)
//   update phase  A_ij -= L_ip L_jp^T, B_iJ -= L_ip W_pJ, K^-1_ij += W_pi^T W_pj:
//                 nb (nb + 1) / 2 tile products for every p, beside which one
//                 CTA updates, factors and inverts the next diagonal tile
// with a cluster barrier (400 clocks) after each phase. n = 128, d = 12, six
// restarts of 20 steps: 3.3 ms on clusters of 16 (one CTA per restart with the
// matrix in shared memory and a barrier per column took 26.3 ms).
#include <math.h>

#include <algorithm>

#include "internal.h"

namespace boute {

namespace {

constexpr int kT = 16;                // tile edge
constexpr int kTE = kT * kT;          // entries of a tile, one per worker thread
constexpr int kLearnWork = kTE;       // worker threads
constexpr int kLearnThreads = kTE + 32;  // and one warp for the pivots' reciprocals
constexpr int kTS = kT + 1;           // row stride of a tile in shared memory
constexpr int kMaxCluster = 16;
constexpr size_t kLearnWsBytes = size_t(1) << 30;  // of workspaces (see launch_learn)
constexpr double kSqrt5d = 2.23606797749978969641;
constexpr double kSqrt3d = 1.73205080756887729353;
constexpr double kLog2Pi = 1.83787706640934548356;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Tile t of the lower triangle of tiles (row by row) -> (i, j).
__device__ __forceinline__ void tri_index(int t, int &i, int &j) {
  int r = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (r * (r + 1) / 2 > t) --r;
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  i = r;
  j = t - r * (r + 1) / 2;
}
__host__ __device__ __forceinline__ size_t tile_off(int i, int j) {
  return ((size_t)i * (i + 1) / 2 + j) * kTE;
}

__device__ __forceinline__ double clamp_d(double v, double lo, double hi) {
  return v < lo ? lo : (v > hi ? hi : v);
}

// theta_q clamped to its bound: q < d log l, d log s2, d + 1 log noise, then
// (composite kernel) d + 2 log s2_c, d + 3 log s2_x, d + 4 beta
__device__ __forceinline__ double clamp_param(int q, int d, double v) {
  if (q < d) return clamp_d(v, BOUTE_LOG_LS_MIN, BOUTE_LOG_LS_MAX);
  if (q == d) return clamp_d(v, BOUTE_LOG_S2_MIN, BOUTE_LOG_S2_MAX);
  if (q == d + 1) return clamp_d(v, BOUTE_LOG_NOISE_MIN, BOUTE_LOG_NOISE_MAX);
  if (q < d + 4) return clamp_d(v, BOUTE_LOG_SC_MIN, BOUTE_LOG_SC_MAX);
  return clamp_d(v, BOUTE_BETA_MIN, BOUTE_BETA_MAX);
}

// Doubles of one cluster's workspace: the lower triangles of tiles of K (then
// L, then K^-1), of B (then W = L^-1) and of two per-pair values kept for the
// gradient (sqrt5 r and exp(-sqrt5 r); composite kernel: exp(-sqrt5 r_t) and
// exp(-sqrt3 r_c)), alpha, the pivots, the CTAs' gradient sums, and a flag word.
__host__ __device__ inline int learn_tiles(int n) { return (n + kT - 1) / kT; }
__host__ __device__ inline size_t learn_ws_doubles(int n) {
  const size_t nb = learn_tiles(n);
  return 4 * (nb * (nb + 1) / 2) * kTE + 2 * nb * kT + (size_t)kMaxCluster * (BOUTE_MAX_D + 5) + 2;
}

constexpr int kMaxP = BOUTE_MAX_D + 5;  // parameters of the composite kernel

// COMP: the composite kernel (routing features [0, dtau), preference entries
// pref: B x m x (d - dtau)), theta extended by (log s2_c, log s2_x, beta):
//   K = s2 k52(r_t) + s2_c w_i w_j k32(r_c) + s2_x k52 k32 + noise I,
//   dK/dlog l_q = (5/3)(1 + sqrt5 r_t) e^(-sqrt5 r_t) z_q^2 (s2 + s2_x k32)  (routing)
//               = 3 e^(-sqrt3 r_c) z_q^2 (s2_c w_i w_j + s2_x k52)        (deployment)
//   dK/dlog s2_c = s2_c w_i w_j k32, dK/dlog s2_x = s2_x k52 k32,
//   dK/dbeta = s2_c w_i w_j k32 (<s, c_i> + <s, c_j>).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ int cluster_rank() {
  int r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

using DTile = double[kT][kTS];

// sum over the P rows of part (one double per worker thread each) into out
__device__ __forceinline__ void reduce_rows(const double *part, int P, double *out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = warp; q < P; q += kLearnThreads / 32) {
    double v = 0.0;
#pragma unroll
    for (int e = 0; e < kLearnWork / 32; ++e) v += part[(size_t)q * kLearnWork + 32 * e + lane];
    v = warp_sum_d(v);
    if (lane == 0) __stcg(out + q, v);
  }
}

template <bool COMP>
__global__ void __launch_bounds__(kLearnThreads, 1) learn_kernel(
    const double *X, const double *Ys, int n, int d, int m, int R, int blk0, int C,
    const double *theta0, int iters, double lr, double *theta_out, double *mll_out,
    double *grad_out, double *ws, int dtau, const double *pref) {
  extern __shared__ __align__(16) double part[];  // P x kLearnWork gradient terms
  __shared__ double th[kMaxP], m1[kMaxP], m2[kMaxP], gr[kMaxP];
  __shared__ double il[kMaxP];  // 1 / l_q, then the scales
  __shared__ DTile ta, tb;  // operand tiles of a product; the diagonal tile's columns
  __shared__ double xi[kT][BOUTE_MAX_D + 1], xj[kT][BOUTE_MAX_D + 1];
  __shared__ double pci[kT], pcj[kT], wvi[kT], wvj[kT], ai[kT], aj[kT];
  __shared__ double inv_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = C > 1 ? cluster_rank() : 0;
  const int slot = blockIdx.x / C, blk = blk0 + slot, bt = blk / R, b = bt / m, t = bt % m;
  const int P = d + (COMP ? 5 : 2), dc = d - dtau, nb = learn_tiles(n), nt = nb * (nb + 1) / 2;
  const bool work = tid < kLearnWork;
  const int r = tid / kT & (kT - 1), c = tid % kT;  // this thread's entry of a tile
  double *KT = ws + (size_t)slot * learn_ws_doubles(n), *WT = KT + (size_t)nt * kTE;
  double *E1 = WT + (size_t)nt * kTE, *E2 = E1 + (size_t)nt * kTE, *av = E2 + (size_t)nt * kTE;
  double *piv = av + (size_t)nb * kT, *gpart = piv + (size_t)nb * kT;
  volatile int *bad = (volatile int *)(gpart + (size_t)kMaxCluster * (BOUTE_MAX_D + 5));
  const double *Xb = X + (size_t)b * n * d, *pb = COMP ? pref + (size_t)bt * dc : nullptr;
  auto sync = [&]() {
    if (C > 1) cluster_sync();
    else __syncthreads();
  };
  // the rows of tiles i and j of X, zero past n (and <s, c>, w of the composite kernel)
  auto load_x = [&](int i, int j) {
    __syncthreads();  // the previous tile's are read
    for (int e = tid; e < 2 * kT * d; e += kLearnThreads) {
      const int h = e >= kT * d, f = h ? e - kT * d : e, row = f / d, q = f - row * d;
      const int g = (h ? j : i) * kT + row;
      (h ? xj : xi)[row][q] = g < n ? Xb[(size_t)g * d + q] : 0.0;
    }
    __syncthreads();
    if (COMP) {
      if (tid < 2 * kT) {
        const int row = tid & (kT - 1);
        const double *x = tid < kT ? xi[row] : xj[row];
        double e = 0.0;
        for (int k = 0; k < dc; ++k) e = fma(pb[k], x[dtau + k], e);
        (tid < kT ? pci : pcj)[row] = e;
        (tid < kT ? wvi : wvj)[row] = exp(th[d + 4] * e);
      }
      __syncthreads();
    }
  };
  // operand tiles into ta and tb
  auto load_ab = [&](const double *A, const double *B) {
    double va = 0.0, vb = 0.0;
    if (work) {
      va = __ldcg(A + tid);
      vb = __ldcg(B + tid);
    }
    __syncthreads();  // the previous product has read its operands
    if (work) {
      ta[r][c] = va;
      tb[r][c] = vb;
    }
    __syncthreads();
  };
  if (tid < P) {
    th[tid] = clamp_param(tid, d, theta0[(size_t)blk * P + tid]);
    m1[tid] = 0.0;
    m2[tid] = 0.0;
  }
  if (rank == 0 && tid == 0) *bad = 0;
  double b1t = 1.0, b2t = 1.0;
  bool failed = false;
  __syncthreads();

  for (int it = 0; it <= iters; ++it) {
    const bool last = it == iters;
    // ---- K and the per-pair values, tile by tile (identity past n)
    if (tid < P) il[tid] = exp(tid < d ? -th[tid] : th[tid]);
    __syncthreads();
    const double s2 = il[d], nz = il[d + 1];
    const double s2c = COMP ? il[d + 2] : 0.0, s2x = COMP ? il[d + 3] : 0.0;
    for (int e = rank; e < nt; e += C) {
      int i, j;
      tri_index(e, i, j);
      load_x(i, j);
      if (!work) continue;
      const int gi = i * kT + r, gj = j * kT + c;
      double rt2 = 0.0, rc2 = 0.0, v1, v2, k;
      for (int q = 0; q < d; ++q) {
        const double z = (xi[r][q] - xj[c][q]) * il[q];
        if (!COMP || q < dtau) rt2 = fma(z, z, rt2);
        else rc2 = fma(z, z, rc2);
      }
      if (COMP) {
        const double st = kSqrt5d * sqrt(rt2), sc = kSqrt3d * sqrt(rc2);
        v1 = exp(-st);
        v2 = exp(-sc);
        const double k52 = (1.0 + st + 5.0 * rt2 / 3.0) * v1, k32 = (1.0 + sc) * v2;
        k = s2 * k52 + s2c * wvi[r] * wvj[c] * k32 + s2x * k52 * k32;
      } else {
        v1 = kSqrt5d * sqrt(rt2);
        v2 = exp(-v1);
        k = s2 * (1.0 + v1 + 5.0 * rt2 / 3.0) * v2;
      }
      if (gi == gj) k += nz;
      if (gi >= n || gj >= n) k = gi == gj ? 1.0 : 0.0;
      const size_t o = tile_off(i, j) + tid;
      __stcg(KT + o, k);
      __stcg(E1 + o, v1);
      __stcg(E2 + o, v2);
    }
    sync();
    // ---- Cholesky, W = L^-1 and K^-1. diag(p): tile p's Schur complement (its
    // entry in x) factored as L~ D L~^T and inverted in place: at step k the
    // entries right of column k still hold A, those up to k hold the rows of
    // L~^-1, and both take the same update x_rc -= (a_rk y_c) / a_kk, with y =
    // column k of A (c > k) or row k of L~^-1 (c <= k), so that a thread has
    // one product ready before the reciprocal and one fma after it.
    auto diag = [&](int p, double x) {
      double *col = &ta[0][0], *row = &tb[0][0];  // column k of A; row k of L~^-1
      for (int k = 0; k < kT; ++k) {
        if (work) {  // (rows and columns past k; row k of L~^-1)
          if (c == k && r >= k) col[r] = x;
          if (r == k) row[c] = c < k ? x : 1.0;
        }
        __syncthreads();
        const double akk = col[k];
        double y = 0.0;
        const bool act = work && 2 * warp + 1 > k;  // (a warp holds two rows)
        if (act) y = col[r] * (c > k ? col[c] : row[c]);
        if (!work) {
          const double iv = 1.0 / akk;
          if (lane == 0) {
            inv_s = iv;
            __stcg(piv + p * kT + k, akk);
            if (!(akk > 0.0)) *bad = 1;
          }
        }
        __syncthreads();
        if (act && r > k) x = fma(-y, inv_s, c == k ? 0.0 : x);
      }
      // W_pp = D^-1/2 L~^-1 (unit diagonal), zero above
      if (work) {
        if (c == r) x = 1.0;
        const double dr = __ldcg(piv + p * kT + r);  // (written by this CTA before the barriers)
        __stcg(WT + tile_off(p, p) + tid, c <= r ? x * rsqrt(dr) : 0.0);
      }
      __syncthreads();
    };
    if (rank == 0) diag(0, work ? __ldcg(KT + tile_off(0, 0) + tid) : 0.0);
    sync();
    failed = *bad != 0;
    for (int p = 0; p < nb && !failed; ++p) {
      // panel phase: tile p of nb is W_pp, done by diag
      for (int e = rank; e < nb; e += C) {
        if (e == p) continue;
        double s = 0.0;
        if (e > p) {  // L_ep = A_ep W_pp^T
          load_ab(KT + tile_off(e, p), WT + tile_off(p, p));
          if (work) {
#pragma unroll
            for (int k = 0; k < kT; ++k) s = fma(ta[r][k], tb[c][k], s);
            __stcg(KT + tile_off(e, p) + tid, s);
          }
        } else {  // W_pe = W_pp B_pe
          load_ab(WT + tile_off(p, p), WT + tile_off(p, e));
          if (work) {
#pragma unroll
            for (int k = 0; k < kT; ++k) s = fma(ta[r][k], tb[k][c], s);
            __stcg(WT + tile_off(p, e) + tid, s);
          }
        }
      }
      sync();
      // update phase. The CTA of the next diagonal tile does only that (all of
      // it with one CTA); tile (i, j) of the triangle is, by its row and column,
      // a trailing tile (j > p), a tile of B (j <= p < i) or one of K^-1 (i <= p)
      const int own = C > 1 && p + 1 < nb ? (p + 1) % C : -1;
      if (p + 1 < nb && rank == (p + 1) % C) {
        const double *L = KT + tile_off(p + 1, p);
        load_ab(L, L);
        double x = 0.0;
        if (work) {
          double s = 0.0;
#pragma unroll
          for (int k = 0; k < kT; ++k) s = fma(ta[r][k], tb[c][k], s);
          x = __ldcg(KT + tile_off(p + 1, p + 1) + tid) - s;
        }
        __syncthreads();
        diag(p + 1, x);
      }
      if (rank != own) {
        const int nw = own >= 0 ? C - 1 : C, me = own >= 0 && rank > own ? rank - 1 : rank;
        for (int e = me; e < nt; e += nw) {
          int i, j;
          tri_index(e, i, j);
          if (i == p + 1 && j == p + 1) continue;
          double *out = (j > p || i <= p ? KT : WT) + tile_off(i, j);
          const bool fresh = j <= p && (i <= p ? i == p : j == p);  // its first term
          const double old = work && !fresh ? __ldcg(out + tid) : 0.0;
          double s = 0.0;
          if (j > p) {
            load_ab(KT + tile_off(i, p), KT + tile_off(j, p));
            if (work) {
#pragma unroll
              for (int k = 0; k < kT; ++k) s = fma(ta[r][k], tb[c][k], s);
              s = old - s;
            }
          } else if (i > p) {
            load_ab(KT + tile_off(i, p), WT + tile_off(p, j));
            if (work) {
#pragma unroll
              for (int k = 0; k < kT; ++k) s = fma(ta[r][k], tb[k][c], s);
              s = old - s;
            }
          } else {
            load_ab(WT + tile_off(p, i), WT + tile_off(p, j));
            if (work) {
#pragma unroll
              for (int k = 0; k < kT; ++k) s = fma(ta[k][r], tb[k][c], s);
              s = old + s;
            }
          }
          if (work) __stcg(out + tid, s);
        }
      }
      sync();
      failed = *bad != 0;
    }
    if (failed) break;  // (the same in every CTA) keeps theta
    // ---- alpha = K^-1 y: a warp per row
    for (int i = rank * (kLearnThreads / 32) + warp; i < n; i += C * (kLearnThreads / 32)) {
      double s = 0.0;
      for (int j = lane; j < n; j += 32) {
        const int hi = max(i, j), lo = min(i, j);
        s = fma(__ldcg(KT + tile_off(hi / kT, lo / kT) + (hi % kT) * kT + lo % kT),
                Ys[((size_t)b * n + j) * m + t], s);
      }
      s = warp_sum_d(s);
      if (lane == 0) __stcg(av + i, s);
    }
    sync();
    if (last) {
      // log likelihood; log det K = sum_j log D_j
      if (rank == 0 && warp == 0) {
        double s = 0.0, l = 0.0;
        for (int i = lane; i < n; i += 32) {
          s = fma(Ys[((size_t)b * n + i) * m + t], __ldcg(av + i), s);
          l += log(__ldcg(piv + i));
        }
        s = warp_sum_d(s);
        l = warp_sum_d(l);
        if (lane == 0) mll_out[blk] = -0.5 * s - 0.5 * l - 0.5 * (double)n * kLog2Pi;
      }
      if (!grad_out) break;
    }
    // ---- gradient: pairs i >= j (an off-diagonal pair stands for two
    // entries); per pair f = s2 (5/3) (1 + sqrt5 r) e^(-sqrt5 r) multiplies
    // (dx_q / l_q)^2 in the lengthscale terms, whose 1 / l_q^2 is left to the end
    double g[BOUTE_MAX_D], gs2 = 0.0, gnz = 0.0, gsc = 0.0, gsx = 0.0, gbe = 0.0;
#pragma unroll
    for (int q = 0; q < BOUTE_MAX_D; ++q) g[q] = 0.0;
    for (int e = rank; e < nt; e += C) {
      int i, j;
      tri_index(e, i, j);
      load_x(i, j);
      if (tid < 2 * kT) {
        const int row = (tid < kT ? i : j) * kT + (tid & (kT - 1));
        (tid < kT ? ai : aj)[tid & (kT - 1)] = row < n ? __ldcg(av + row) : 0.0;
      }
      __syncthreads();
      const int gi = i * kT + r, gj = j * kT + c;
      if (!work || gi >= n || gj > gi) continue;
      const size_t o = tile_off(i, j) + tid;
      const double Q = (gi == gj ? 0.5 : 1.0) * (ai[r] * aj[c] - __ldcg(KT + o));
      const double v1 = __ldcg(E1 + o), v2 = __ldcg(E2 + o);
      double ft, fc = 0.0;
      if (COMP) {
        double rt2 = 0.0, rc2 = 0.0;
        for (int q = 0; q < d; ++q) {
          const double z = (xi[r][q] - xj[c][q]) * il[q];
          if (q < dtau) rt2 = fma(z, z, rt2);
          else rc2 = fma(z, z, rc2);
        }
        const double st = kSqrt5d * sqrt(rt2), sc = kSqrt3d * sqrt(rc2);
        const double k52 = (1.0 + st + 5.0 * rt2 / 3.0) * v1, k32 = (1.0 + sc) * v2;
        const double ww = wvi[r] * wvj[c];
        ft = Q * (5.0 / 3.0) * (1.0 + st) * v1 * (s2 + s2x * k32);
        fc = Q * 3.0 * v2 * (s2c * ww + s2x * k52);
        gs2 = fma(Q, s2 * k52, gs2);
        const double tc = Q * s2c * ww * k32;
        gsc += tc;
        gsx = fma(Q, s2x * k52 * k32, gsx);
        gbe = fma(tc, pci[r] + pcj[c], gbe);
      } else {
        const double qe = Q * s2 * v2;
        ft = qe * (5.0 / 3.0) * (1.0 + v1);
        gs2 = fma(qe, 1.0 + v1 + v1 * v1 / 3.0, gs2);  // (5/3 r^2 = (sqrt5 r)^2 / 3)
      }
      if (gi == gj) gnz = fma(Q, nz, gnz);
#pragma unroll
      for (int q = 0; q < BOUTE_MAX_D; ++q) {
        if (q < d) {
          const double dx = xi[r][q] - xj[c][q];
          g[q] = fma(COMP && q >= dtau ? fc : ft, dx * dx, g[q]);
        }
      }
    }
    if (work) {
#pragma unroll
      for (int q = 0; q < BOUTE_MAX_D; ++q)
        if (q < d) part[(size_t)q * kLearnWork + tid] = g[q];
      part[(size_t)d * kLearnWork + tid] = gs2;
      part[(size_t)(d + 1) * kLearnWork + tid] = gnz;
      if (COMP) {
        part[(size_t)(d + 2) * kLearnWork + tid] = gsc;
        part[(size_t)(d + 3) * kLearnWork + tid] = gsx;
        part[(size_t)(d + 4) * kLearnWork + tid] = gbe;
      }
    }
    __syncthreads();
    reduce_rows(part, P, gpart + (size_t)rank * P);
    sync();
    // ---- the CTAs' sums, then the Adam step, alike in every CTA
    if (work) {
      for (int q = tid / kMaxCluster; q < P; q += kLearnWork / kMaxCluster) {
        double v = tid % kMaxCluster < C ? __ldcg(gpart + (size_t)(tid % kMaxCluster) * P + q) : 0.0;
        const unsigned half = 0xffffu << (lane & 16);
#pragma unroll
        for (int o = kMaxCluster / 2; o > 0; o >>= 1) v += __shfl_xor_sync(half, v, o);
        if (tid % kMaxCluster == 0) gr[q] = q < d ? v * (il[q] * il[q]) : v;
      }
    }
    __syncthreads();
    if (last) {
      if (rank == 0 && tid < P) grad_out[(size_t)blk * P + tid] = gr[tid];
      break;
    }
    b1t *= BOUTE_ADAM_B1;
    b2t *= BOUTE_ADAM_B2;
    if (tid < P) {  // Adam ascent step, bias-corrected moments, then the bounds
      const double v = gr[tid];
      m1[tid] = BOUTE_ADAM_B1 * m1[tid] + (1.0 - BOUTE_ADAM_B1) * v;
      m2[tid] = BOUTE_ADAM_B2 * m2[tid] + (1.0 - BOUTE_ADAM_B2) * v * v;
      const double mh = m1[tid] / (1.0 - b1t), vh = m2[tid] / (1.0 - b2t);
      th[tid] = clamp_param(tid, d, th[tid] + lr * mh / (sqrt(vh) + BOUTE_ADAM_EPS));
    }
    __syncthreads();
  }
  if (rank == 0) {
    if (tid < P) theta_out[(size_t)blk * P + tid] = th[tid];
    if (failed) {  // not positive definite
      if (tid == 0) mll_out[blk] = nan("");
      if (grad_out && tid < P) grad_out[(size_t)blk * P + tid] = nan("");
    }
  }
}

}  // namespace

// dtau, pref: the composite kernel (pref null: the Matern-5/2 kernel)
int launch_learn(const double *X, const double *Ys, int B, int n, int d, int m,
                 const double *theta0, int R, int iters, double lr, double *theta, double *mll,
                 double *grad, int dtau, const double *pref, cudaStream_t s) {
  const int blocks = B * m * R;
  // the largest cluster of which the device holds one per restart at once, an SM to each
  // CTA (clusters lie within a GPC, so fewer fit than SMs / C: 7 of 16 CTAs; 8 restarts
  // at n = 128 took 3.39 ms for 10 Adam steps on clusters of 16, 2.23 on clusters of 8), and
  // no more CTAs than the power of two that covers the triangle's tiles (n = 20, 3 tiles,
  // 20 steps: 1.06 ms on four CTAs, 1.36 on two; n = 48, 6 tiles: 1.37 on eight, 1.71 on four)
  const int nb = learn_tiles(n), nt = nb * (nb + 1) / 2;
  const long long sms = num_sms();
  int C = kMaxCluster;
  while (C > 1 && (C * (long long)blocks > sms || C / 2 >= nt)) C /= 2;
  const size_t smem = (size_t)(d + 5) * kLearnWork * sizeof(double);
  double *ws = nullptr;
  int st = BOUTE_OK;
  auto go = [&](auto kern) {
    prefer_shared(kern);
    constexpr size_t kAlone = 120 * 1024;  // more than half an SM's shared memory
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAlone);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(kLearnThreads);
    cfg.dynamicSmemBytes = kAlone;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (C > 8)
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (;; C /= 2) {
      attr[0].val.clusterDim.x = C;
      cfg.gridDim = dim3((unsigned)(blocks * C));
      int held = 0;
      if (C == 1 || (cudaOccupancyMaxActiveClusters(&held, kern, &cfg) == cudaSuccess &&
                     held >= blocks))
        break;
      cudaGetLastError();
    }
    cfg.dynamicSmemBytes = smem;
    // Workspaces for what runs at once (a CTA's registers take an SM), or for as many rounds
    // of that as kLearnWsBytes hold; further restarts follow in launches of their own that
    // use the same ones, so that the memory does not grow with the restarts. (One launch
    // whose clusters loop over their restarts cost 1 to 2 % at every size.)
    const size_t per = learn_ws_doubles(n) * sizeof(double);
    const long long rounds = std::max<long long>(1, (long long)(kLearnWsBytes / per) / sms);
    const int wave = C > 1 ? blocks : (int)std::min<long long>(blocks, rounds * sms);
    if (cudaMallocAsync((void **)&ws, per * wave, s) != cudaSuccess) {
      cudaGetLastError();
      st = BOUTE_ERR_OOM;
      return;
    }
    for (int blk0 = 0; blk0 < blocks; blk0 += wave) {
      cfg.gridDim = dim3((unsigned)(std::min(wave, blocks - blk0) * C));
      cudaLaunchKernelEx(&cfg, kern, X, Ys, n, d, m, R, blk0, C, theta0, iters, lr, theta, mll,
                         grad, ws, dtau, pref);
      count_launch();
    }
  };
  if (pref) go(learn_kernel<true>);
  else go(learn_kernel<false>);
  if (st) return st;
  st = last_launch_status();
  cudaFreeAsync(ws, s);
  return st;
}

}  // namespace boute

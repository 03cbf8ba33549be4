// Optimising the acquisition over the decision space (Sec. 5.2 step (ii),
// "optimize it over the decision space"): projected Adam ascent on the
// sample-average Monte-Carlo hypervolume improvement of two objectives, from
// given starting points (for instance the best candidates of a pool).
//
// With fixed base normals eps_s the acquisition A(x) = (1/S) sum_s HVI(mu(x) +
// sd(x) eps_s) is a deterministic, piecewise smooth function of x. Its
// gradient runs through the GP posterior of each objective (Matern-5/2):
//   k*_j = s2 (1 + sqrt5 r + 5/3 r^2) e^(-sqrt5 r),
//   dk*_j/dx_k = -5/3 s2 (1 + sqrt5 r) e^(-sqrt5 r) (x_k - X_jk) / l_k^2,
//   mu = k*^T alpha,  var = s2 - |W k*|^2,  dvar/dx = -2 (W^T W k*)^T dk*/dx,
// and the strip sum HVI(y) = sum_k (b_k - max(a_k, y1))+ (u_k - y2)+, whose
// derivatives are -(u_k - y2)+ for the strip containing y1 and
// -sum_k (b_k - max(a_k, y1))+ [y2 < u_k].
//
// One CTA per (problem, starting point) runs all its steps; each step is a chain
// of short phases, so what bounds it is latency. Half of its (16, with many starts of few
// observations 8 or 4) warps take each
// objective: the threads build k* and its gradient factors over the training
// points (the fit's side input: scaled coordinates hi + lo, alpha as a pair);
// a warp takes a row of the fit's W into registers, forms q_i = W_i k* and adds
// q_i W_i to its share of W^T (W k*) in the same pass (n <= 512; two passes
// beyond), W staying in L1 over the steps while it fits; the gradient is a warp
// per coordinate, the S draws are scored four threads to a draw against the
// observed front's strips (in shared memory), and one warp closes the step.
// n = 200, d = 16, S = 128, 10 steps from 32 points: 0.13 ms (4 warps taking the
// objectives in turn, W^T q a thread per column: 0.98 ms).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace boute {

namespace {

constexpr float kLn2f = 0.6931471805599453f;
constexpr float kLn2Sq3f = 0.16015100463940046f;  // (ln 2)^2 / 3
// 1 / (the side input's coordinate scale)^2
constexpr float kInvScale2 = (float)(1.0 / (kCoordScale52 * kCoordScale52));

struct OptArgs {
  const float *Wws, *xt;
  int npad, nxt, DP, n, d, m;
  const float *lower, *upper;  // the observed front's strips (box decomposition)
  const int *K;
  int box_cap;
  const float *eps;  // 2 x S, shared by every point
  int S;
  const float *X0, *xlo, *xhi;
  int P, steps;
  float lr;
  float *X, *acq, *grad;
};

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// acc[u] += q w[u] and back: a row's entries j0 + lane + 32 u up to column i
template <int kRowRegs>
__device__ __forceinline__ void load_row(const float *wr, int i, int j0, int lane,
                                         float (&w)[kRowRegs]) {
#pragma unroll
  for (int u = 0; u < kRowRegs; ++u) {
    const int j = j0 + lane + 32 * u;
    w[u] = j <= i ? wr[j] : 0.f;
  }
}

// kRowRegs: columns of a row of W per lane (n <= 32 kRowRegs, or panels of as many).
template <int kOptThreads, int kRowRegs>
__global__ void __launch_bounds__(kOptThreads) acqopt_kernel(const __grid_constant__ OptArgs a) {
  constexpr int kOptWarps = kOptThreads / 32, kPanel = 32 * kRowRegs;
  constexpr int kObjWarps = kOptWarps / 2, kObjThreads = kOptThreads / 2;  // per objective
  extern __shared__ __align__(16) float sm[];
  __shared__ float xs[BOUTE_MAX_D], xsc[2][BOUTE_MAX_D];  // x, x / l (scaled)
  __shared__ float dmu_s[2][BOUTE_MAX_D], dvar_s[2][BOUTE_MAX_D];
  __shared__ float rmu[kOptWarps], rq[kOptWarps], red[kOptWarps][5];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = warp / kObjWarps, ow = warp % kObjWarps, ot = tid % kObjThreads;  // objective
  const int b = blockIdx.y, p = blockIdx.x;
  const int n = a.n, d = a.d, DP = a.DP, cf = xt_chunk_floats(DP), ldw = a.npad + 1;
  const int pan = min(n, kPanel);
  float *kv = sm + t * n, *cv = sm + (2 + t) * n, *wv = sm + (4 + t) * n;  // k*, c_j, W^T W k*
  float *part = sm + 6 * n + (size_t)t * kObjWarps * pan;  // the warps' shares of a panel of it
  float *strips = sm + 6 * n + 2 * (size_t)kObjWarps * pan;  // (a, b, u) per strip, K <= n + 1
  float *qv = strips + 3 * (n + 1) + t * n;  // W k* (n > kPanel)
  pdl_wait();
  const int K = BOUTE_INB(a.K[b], a.box_cap + 1) ? a.K[b] : 0;
  const float *lo = a.lower + (size_t)b * a.box_cap * 2, *up = a.upper + (size_t)b * a.box_cap * 2;
  const bool staged = K <= n + 1;
  if (staged)
    for (int k = tid; k < K; k += kOptThreads) {
      strips[3 * k] = lo[2 * k];
      strips[3 * k + 1] = up[2 * k];
      strips[3 * k + 2] = up[2 * k + 1];
    }
  const int bt = b * a.m + t;
  const float *x0 = a.xt + (size_t)bt * a.nxt * cf;
  const float *par = x0 + xt_param_offset(DP);  // 1/l hi [DP], 1/l lo [DP], scalars
  const float s2 = par[2 * DP + kParS2];
  const float *W = a.Wws + (size_t)bt * a.npad * ldw;
  // (warp 0, lane = coordinate: the point and Adam's moments)
  float x = 0.f, m1 = 0.f, m2 = 0.f, g = 0.f, val = 0.f;
  if (warp == 0 && lane < d) x = xs[lane] = a.X0[((size_t)b * a.P + p) * d + lane];
  for (int it = 0; it <= a.steps; ++it) {
    __syncthreads();  // x
    if (ow == 0 && lane < d) xsc[t][lane] = fmaf(xs[lane], par[lane], xs[lane] * par[DP + lane]);
    __syncthreads();
    // ---- k* and its gradient factors. r2 = r'^2, the side input's scaled
    // distance: sqrt5 r = ln2 r', exp(-sqrt5 r) = 2^(-r')
    float amu = 0.f;
    for (int j = ot; j < n; j += kObjThreads) {
      const float *ch = x0 + (size_t)(j / BOUTE_KCHUNK) * cf;
      const int jj = j % BOUTE_KCHUNK;
      float r2 = 0.f;
#pragma unroll 8
      for (int k = 0; k < d; ++k) {
        const float dk = (xsc[t][k] - ch[k * BOUTE_KCHUNK + jj]) - ch[(DP + k) * BOUTE_KCHUNK + jj];
        r2 = fmaf(dk, dk, r2);
      }
      const float rs = sqrtf(r2), ex = exp2f(-rs);
      const float k = s2 * fmaf(kLn2Sq3f, r2, fmaf(kLn2f, rs, 1.f)) * ex;
      kv[j] = k;
      cv[j] = -5.f / 3.f * s2 * fmaf(kLn2f, rs, 1.f) * ex;
      const float *al = ch + xt_alpha_offset(DP) + jj;
      amu = fmaf(k, al[0] + al[BOUTE_KCHUNK], amu);
    }
    amu = warp_sum_f(amu);
    if (lane == 0) rmu[warp] = amu;
    __syncthreads();
    // ---- q = W k* and W^T q
    float aq = 0.f;
    if (n <= kPanel) {
      float acc[kRowRegs];
#pragma unroll
      for (int u = 0; u < kRowRegs; ++u) acc[u] = 0.f;
      float kr[kRowRegs];
#pragma unroll
      for (int u = 0; u < kRowRegs; ++u) kr[u] = lane + 32 * u < n ? kv[lane + 32 * u] : 0.f;
      for (int i = ow; i < n; i += 2 * kObjWarps) {  // two rows in flight
        const int i1 = i + kObjWarps;
        float w0[kRowRegs], w1[kRowRegs], q0 = 0.f, q1 = 0.f;
        load_row(W + (size_t)i * ldw, i, 0, lane, w0);
        load_row(W + (size_t)min(i1, n - 1) * ldw, i1 < n ? i1 : -1, 0, lane, w1);
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) {
          q0 = fmaf(w0[u], kr[u], q0);
          q1 = fmaf(w1[u], kr[u], q1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          q0 += __shfl_xor_sync(0xffffffffu, q0, o);
          q1 += __shfl_xor_sync(0xffffffffu, q1, o);
        }
        aq = fmaf(q0, q0, fmaf(q1, q1, aq));
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) acc[u] = fmaf(q0, w0[u], fmaf(q1, w1[u], acc[u]));
      }
#pragma unroll
      for (int u = 0; u < kRowRegs; ++u)
        if (lane + 32 * u < n) part[(size_t)ow * pan + lane + 32 * u] = acc[u];
      if (lane == 0) rq[warp] = aq;
      __syncthreads();
      for (int j = ot; j < n; j += kObjThreads) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < kObjWarps; ++w) v += part[(size_t)w * pan + j];
        wv[j] = v;
      }
    } else {
      for (int i = ow; i < n; i += kObjWarps) {
        const float *wr = W + (size_t)i * ldw;
        float q = 0.f;
        for (int j = lane; j <= i; j += 32) q = fmaf(wr[j], kv[j], q);
        q = warp_sum_f(q);
        aq = fmaf(q, q, aq);
        if (lane == 0) qv[i] = q;
      }
      if (lane == 0) rq[warp] = aq;
      for (int j0 = 0; j0 < n; j0 += kPanel) {  // panels of columns
        __syncthreads();  // q; the previous panel's shares are read
        float acc[kRowRegs];
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) acc[u] = 0.f;
        for (int i = j0 + ow; i < n; i += kObjWarps) {
          float w[kRowRegs];
          load_row(W + (size_t)i * ldw, i, j0, lane, w);
          const float q = qv[i];
#pragma unroll
          for (int u = 0; u < kRowRegs; ++u) acc[u] = fmaf(q, w[u], acc[u]);
        }
#pragma unroll
        for (int u = 0; u < kRowRegs; ++u) part[(size_t)ow * pan + lane + 32 * u] = acc[u];
        __syncthreads();
        for (int j = ot; j < kPanel && j0 + j < n; j += kObjThreads) {
          float v = 0.f;
#pragma unroll
          for (int w = 0; w < kObjWarps; ++w) v += part[(size_t)w * pan + j];
          wv[j0 + j] = v;
        }
      }
    }
    __syncthreads();
    float mu[2], sd[2];  // (every thread)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float sm_ = 0.f, sq = 0.f;
#pragma unroll
      for (int w = 0; w < kObjWarps; ++w) {
        sm_ += rmu[q * kObjWarps + w];
        sq += rq[q * kObjWarps + w];
      }
      const float sq2 = a.xt[(size_t)(b * a.m + q) * a.nxt * cf + xt_param_offset(DP) + 2 * DP + kParS2];
      mu[q] = sm_;
      sd[q] = sqrtf(fmaxf(sq2 - sq, 0.f));
    }
    // ---- d mu / dx_k = sum_j alpha_j c_j df_jk, -1/2 d var / dx_k = sum_j w_j c_j
    // df_jk, df_jk = (x_k - X_jk) / l_k^2 (the side input's scale twice)
    for (int k = ow; k < d; k += kObjWarps) {
      float gm = 0.f, gv = 0.f;
#pragma unroll 4
      for (int j = lane; j < n; j += 32) {
        const float *ch = x0 + (size_t)(j / BOUTE_KCHUNK) * cf;
        const float dk =
            (xsc[t][k] - ch[k * BOUTE_KCHUNK + lane]) - ch[(DP + k) * BOUTE_KCHUNK + lane];
        const float *al = ch + xt_alpha_offset(DP) + lane;
        const float cd = cv[j] * dk;
        gm = fmaf(al[0] + al[BOUTE_KCHUNK], cd, gm);
        gv = fmaf(wv[j], cd, gv);
      }
      gm = warp_sum_f(gm);
      gv = warp_sum_f(gv);
      if (lane == 0) {
        const float f = (par[k] + par[DP + k]) * kInvScale2;
        dmu_s[t][k] = gm * f;
        dvar_s[t][k] = gv * f;
      }
    }
    // ---- the draws against the front's strips: A, dA/dmu_t, dA/dsd_t
    float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    for (int e = tid; e < 4 * a.S; e += kOptThreads) {
      const int s = e >> 2;
      const float e0 = a.eps[s], e1 = a.eps[a.S + s];
      const float y1 = fmaf(sd[0], e0, mu[0]), y2 = fmaf(sd[1], e1, mu[1]);
      float h = 0.f, g1 = 0.f, g2 = 0.f;
      for (int k = e & 3; k < K; k += 4) {
        const float ak = staged ? strips[3 * k] : lo[2 * k];
        const float bk = staged ? strips[3 * k + 1] : up[2 * k];
        const float uk = staged ? strips[3 * k + 2] : up[2 * k + 1];
        const float wdt = fmaxf(bk - fmaxf(ak, y1), 0.f), hgt = fmaxf(uk - y2, 0.f);
        h = fmaf(wdt, hgt, h);
        if (ak < y1 && y1 < bk) g1 -= hgt;
        if (y2 < uk) g2 -= wdt;
      }
      acc[0] += h;
      acc[1] += g1;
      acc[2] += g1 * e0;
      acc[3] += g2;
      acc[4] += g2 * e1;
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      acc[q] = warp_sum_f(acc[q]);
      if (lane == 0) red[warp][q] = acc[q];
    }
    __syncthreads();
    if (warp == 0) {  // ---- value, gradient and the projected Adam step
      float cf5[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        float v = lane < kOptWarps ? red[lane][q] : 0.f;
#pragma unroll
        for (int o = kOptWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        cf5[q] = __shfl_sync(0xffffffffu, v, 0) / (float)a.S;
      }
      val = cf5[0];
      if (lane < d) {
        // d sd = d var / (2 sd)
        const float ds0 = sd[0] > 0.f ? -dvar_s[0][lane] / sd[0] : 0.f;
        const float ds1 = sd[1] > 0.f ? -dvar_s[1][lane] / sd[1] : 0.f;
        g = cf5[1] * dmu_s[0][lane] + cf5[2] * ds0 + cf5[3] * dmu_s[1][lane] + cf5[4] * ds1;
        if (it < a.steps) {  // (the last pass only evaluates)
          const float c1 = 1.f - powf(0.9f, (float)(it + 1)), c2 = 1.f - powf(0.999f, (float)(it + 1));
          m1 = fmaf(0.9f, m1, 0.1f * g);
          m2 = fmaf(0.999f, m2, 0.001f * g * g);
          const float stp = a.lr * (m1 / c1) / (sqrtf(m2 / c2) + 1e-8f);
          x = xs[lane] = fminf(fmaxf(x + stp, a.xlo[lane]), a.xhi[lane]);
        }
      }
    }
  }
  if (warp == 0) {
    if (lane < d) {
      a.X[((size_t)b * a.P + p) * d + lane] = x;
      if (a.grad) a.grad[((size_t)b * a.P + p) * d + lane] = g;
    }
    if (lane == 0) a.acq[(size_t)b * a.P + p] = val;
  }
}

}  // namespace

int launch_acq_optimize(const Gp *gp, const float *lower, const float *upper, const int *K,
                        int box_cap, const float *eps, int S, const float *X0, int P,
                        const float *xlo, const float *xhi, int steps, float lr, float *X,
                        float *acq, float *grad, cudaStream_t s) {
  if (gp->m != 2 || gp->kern || gp->d > BOUTE_MAX_D) return BOUTE_ERR_UNSUPPORTED;
  OptArgs a;
  a.Wws = gp->Wws;
  a.xt = gp->xt;
  a.npad = gp->plan.npad;
  a.nxt = gp->plan.nxt;
  a.DP = gp->DP;
  a.n = gp->n;
  a.d = gp->d;
  a.m = gp->m;
  a.lower = lower;
  a.upper = upper;
  a.K = K;
  a.box_cap = box_cap;
  a.eps = eps;
  a.S = S;
  a.X0 = X0;
  a.xlo = xlo;
  a.xhi = xhi;
  a.P = P;
  a.steps = steps;
  a.lr = lr;
  a.X = X;
  a.acq = acq;
  a.grad = grad;
  const size_t n = gp->n;
  // (the limit on n and d that the call has always had)
  if ((4 * n + n * gp->d) * sizeof(float) > 200 * 1024) return BOUTE_ERR_UNSUPPORTED;
  auto go = [&](auto threads, auto regs) {
    constexpr int T = decltype(threads)::value, R = decltype(regs)::value;
    const size_t panel = 32 * R;
    const size_t smem = (6 * n + (size_t)(T / 32) * std::min(n, panel) + 3 * (n + 1) +
                         (n > panel ? 2 * n : 0)) * sizeof(float);
    // (no shared-memory preference: what it leaves of the SM's memory caches W)
    cudaFuncSetAttribute(acqopt_kernel<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    launch_pdl(acqopt_kernel<T, R>, dim3(P, gp->B), dim3(T), smem, s, a);
  };
  // With at most 128 columns a row of W takes four registers of a lane, and starts beyond one
  // per SM share SMs in smaller blocks: n = 32, d = 6, S = 64, 5 steps: 256 starts 27 us
  // with 256 threads (42 with 512), 1024 starts 49 with 128 (74 with 256, 137 with 512, 171
  // with 16 registers); n = 100, S = 128, 3 steps, 4096 starts: 274 (749 with 512 and 16).
  // More columns keep 16 registers and the block of 512: n = 700, 1024 starts, 2 steps 2.0
  // ms against 2.2 with 128.
  using std::integral_constant;
  const long long blocks = (long long)P * gp->B, sms = num_sms();
  if (n > 128) go(integral_constant<int, 512>{}, integral_constant<int, 16>{});
  else if (blocks <= sms) go(integral_constant<int, 512>{}, integral_constant<int, 4>{});
  else if (blocks <= 2 * sms) go(integral_constant<int, 256>{}, integral_constant<int, 4>{});
  else go(integral_constant<int, 128>{}, integral_constant<int, 4>{});
  count_launch();
  return last_launch_status();
}

}  // namespace boute

// Pareto front of the observed (standardised) outcomes and the disjoint box
// decomposition of the region that improves on it. One block per problem;
// fronts are small (tens of points), the work is O(n^2) compares.
#include <math.h>

#include "internal.h"

namespace boute {

namespace {

// Order-preserving integer image of a double (-0 taken as +0): x < y exactly
// when key(x) < key(y), for finite values. Comparing keys keeps the O(n^2)
// dominance tests and the boxes' sweep on the integer pipes: an fp64 comparison
// takes a warp about 100 clocks here.
__device__ __forceinline__ long long dkey(double x) {
  long long b = __double_as_longlong(x);
  if (b == (long long)0x8000000000000000ull) b = 0;
  return b >= 0 ? b : (long long)(b ^ 0x7FFFFFFFFFFFFFFFll);
}

// The m keys of point i, taken from component-major arrays of n.
struct Keys {
  long long v[BOUTE_MAX_M];
  __device__ __forceinline__ Keys(const long long *yk, int n, int m, int i) {
#pragma unroll
    for (int t = 0; t < BOUTE_MAX_M; ++t) v[t] = t < m ? yk[(size_t)t * n + i] : 0;
  }
};

// Point j removes point i (minimisation): <= everywhere and < somewhere, or
// equal with the smaller index.
__device__ __forceinline__ bool removes(const Keys &yj, int j, const Keys &yi, int i) {
  bool le = true, lt = false;
#pragma unroll
  for (int t = 0; t < BOUTE_MAX_M; ++t) {
    le = le && yj.v[t] <= yi.v[t];
    lt = lt || yj.v[t] < yi.v[t];
  }
  return le && (lt || j < i);
}

// (Y_j, j) < (Y_i, i) lexicographically
__device__ __forceinline__ bool lex_less(const Keys &yj, int j, const Keys &yi, int i) {
  bool less = j < i;
#pragma unroll
  for (int t = BOUTE_MAX_M - 1; t >= 0; --t)
    less = yj.v[t] < yi.v[t] || (yj.v[t] == yi.v[t] && less);
  return less;
}

// A warp per point, its lanes over the others: a point is dropped as soon as one
// of them removes it (most are within the first 32), and the kept points' ranks are
// counts over the kept points alone. n = 512, m = 2, with the standardisation: 344
// -> 25 us; n = 203, m = 3, with the boxes: 117 -> 40 us (before, all n^2 ordered
// pairs went through the threads twice, each with a 64-bit division).
// smem: n*m keys, n kept indices. Writes mask, front rows, P.
__device__ void pareto_block(const double *Yb, int n, int m, const double *rb,
                             unsigned char *mask, double *front, int *P, void *smem) {
  long long *yk = (long long *)smem;
  int *kept = (int *)(yk + (size_t)n * m);
  __shared__ int count;
  __shared__ long long rk[BOUTE_MAX_M];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int t = 0; t < m; ++t)
    for (int i = threadIdx.x; i < n; i += blockDim.x) yk[(size_t)t * n + i] = dkey(Yb[(size_t)i * m + t]);
  if (threadIdx.x < m) rk[threadIdx.x] = dkey(rb[threadIdx.x]);
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  for (int i = warp; i < n; i += nw) {
    const Keys yi(yk, n, m, i);
    bool drop = false;
#pragma unroll
    for (int t = 0; t < BOUTE_MAX_M; ++t)
      if (t < m && !(yi.v[t] < rk[t])) drop = true;
    for (int j0 = 0; j0 < n && !drop; j0 += 32) {
      const int j = min(j0 + lane, n - 1);
      drop = __any_sync(0xffffffffu, j != i && removes(Keys(yk, n, m, j), j, yi, i));
    }
    if (lane == 0) {
      mask[i] = (unsigned char)!drop;
      if (!drop) kept[atomicAdd(&count, 1)] = i;
    }
  }
  __syncthreads();
  const int K = count;
  for (int q = warp; q < K; q += nw) {
    const int i = kept[q];
    const Keys yi(yk, n, m, i);
    int rank = 0;
    for (int e = lane; e < K; e += 32) {
      const int j = kept[e];
      rank += j != i && lex_less(Keys(yk, n, m, j), j, yi, i);
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane < m) front[(size_t)rank * m + lane] = Yb[(size_t)i * m + lane];
  }
  if (threadIdx.x == 0) *P = K;
  __syncthreads();
}

__global__ void pareto_kernel(const double *Ys, int n, int m, const double *ref,
                              unsigned char *mask, double *front, int *P) {
  extern __shared__ long long smem_keys[];
  const int b = blockIdx.x;
  pareto_block(Ys + (size_t)b * n * m, n, m, ref + (size_t)b * m, mask + (size_t)b * n,
               front + (size_t)b * n * m, P + b, smem_keys);
}

// ---- boxes ---------------------------------------------------------------------
// m = 2: strip i = [a_i, b_i) x (-inf, u_i) of the staircase (P+1 strips).
// m = 3: sweep the front by increasing f3; between consecutive levels the
// cross-section of the improving region is the 2-D staircase region of the
// points below the level. Each strip lives from the level where it appears to
// the level where an inserted point changes it, and becomes one box
// [a, b) x (-inf, u) x [z_birth, z_death); every insertion creates at most two
// strips, so there are at most 2P+1 boxes.
// One problem: F = its front (P rows), r = its reference point, lo/hi = its
// box arrays (capacity 2n+2), *Kout = box count. smem (m = 3): 13 (n+2)
// doubles. The sweep is one thread's chain of comparisons, made on keys.
__device__ void boxes_block(const double *F, int Pb, int n, int m, const double *r, float *lo,
                            float *hi, int *Kout, void *smem) {
  double *ws = (double *)smem;
  const int cap = 2 * n + 2;
  (void)cap;  // (the debug build checks the box count against it)
  if (m == 2) {
    for (int i = threadIdx.x; i <= Pb; i += blockDim.x) {
      if (!BOUTE_INB(i, cap)) break;
      lo[2 * i] = i == 0 ? -INFINITY : (float)F[2 * (i - 1)];
      lo[2 * i + 1] = -INFINITY;
      hi[2 * i] = i == Pb ? (float)r[0] : (float)F[2 * i];
      hi[2 * i + 1] = i == 0 ? (float)r[1] : (float)F[2 * (i - 1) + 1];
    }
    if (threadIdx.x == 0) *Kout = Pb + 1;
    return;
  }
  // m == 3 --------------------------------------------------------------------
  const int L = n + 2;
  double *sx = ws, *sy = sx + L;                          // staircase (f1 asc, f2 desc)
  double *ca = sy + L, *cb = ca + L, *cu = cb + L, *cz = cu + L;  // live strips
  double *na = cz + L, *nb = na + L, *nu = nb + L, *nz = nu + L;  // next strips
  double *fx = nz + L, *fy = fx + L, *fz = fy + L;  // the front by increasing f3
  for (int i = threadIdx.x; i < Pb; i += blockDim.x) {  // order by (f3, index)
    int rank = 0;
    const long long zi = dkey(F[(size_t)i * 3 + 2]);
#pragma unroll 4
    for (int j = 0; j < Pb; ++j) {
      const long long zj = dkey(F[(size_t)j * 3 + 2]);
      rank += zj < zi || (zj == zi && j < i);
    }
    fx[rank] = F[(size_t)i * 3];
    fy[rank] = F[(size_t)i * 3 + 1];
    fz[rank] = F[(size_t)i * 3 + 2];
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  auto lt = [](double x, double y) { return dkey(x) < dkey(y); };
  auto le = [](double x, double y) { return dkey(x) <= dkey(y); };
  auto eq = [](double x, double y) { return dkey(x) == dkey(y); };
  const double r0 = r[0], r1 = r[1], r2 = r[2];
  int ns = 0, nc = 1, K = 0;
  ca[0] = -INFINITY; cb[0] = r0; cu[0] = r1; cz[0] = -INFINITY;
  auto emit = [&](double a, double bb, double u, double z0, double z1) {
    // (a decomposition with more than cap boxes is reported by the debug build)
    if (lt(z0, z1) && lt(a, bb) && BOUTE_INB(K, cap)) {
      lo[K * 3 + 0] = (float)a; lo[K * 3 + 1] = -INFINITY; lo[K * 3 + 2] = (float)z0;
      hi[K * 3 + 0] = (float)bb; hi[K * 3 + 1] = (float)u; hi[K * 3 + 2] = (float)z1;
      ++K;
    }
  };
  for (int q = 0; q < Pb; ++q) {
    const double qx = fx[q], qy = fy[q], qz = fz[q];
    bool covered = false;
    for (int s = 0; s < ns && !covered; ++s)
      if (le(sx[s], qx) && le(sy[s], qy)) covered = true;
    if (covered) continue;
    // new staircase: drop points q weakly dominates in 2-D, insert q in f1 order
    int w = 0, ins = -1;
    for (int s = 0; s < ns; ++s) {
      if (le(qx, sx[s]) && le(qy, sy[s])) continue;
      if (ins < 0 && lt(qx, sx[s])) { ins = w; na[w] = qx; nb[w] = qy; ++w; }
      na[w] = sx[s]; nb[w] = sy[s]; ++w;
    }
    if (ins < 0) { na[w] = qx; nb[w] = qy; ++w; }
    for (int s = 0; s < w; ++s) { sx[s] = na[s]; sy[s] = nb[s]; }
    ns = w;
    // strips of the new staircase; a strip identical to a live one keeps its birth
    int nn = 0, j = 0;
    for (int s = 0; s <= ns; ++s) {
      const double a = s == 0 ? -INFINITY : sx[s - 1];
      const double bb = s == ns ? r0 : sx[s];
      const double u = s == 0 ? r1 : sy[s - 1];
      while (j < nc && lt(ca[j], a)) { emit(ca[j], cb[j], cu[j], cz[j], qz); ++j; }
      double z = qz;
      if (j < nc && eq(ca[j], a) && eq(cb[j], bb) && eq(cu[j], u)) { z = cz[j]; ++j; }
      na[nn] = a; nb[nn] = bb; nu[nn] = u; nz[nn] = z; ++nn;
    }
    while (j < nc) { emit(ca[j], cb[j], cu[j], cz[j], qz); ++j; }
    for (int s = 0; s < nn; ++s) { ca[s] = na[s]; cb[s] = nb[s]; cu[s] = nu[s]; cz[s] = nz[s]; }
    nc = nn;
  }
  for (int j = 0; j < nc; ++j) emit(ca[j], cb[j], cu[j], cz[j], r2);
  *Kout = K;
}

__global__ void boxes_kernel(const double *front, const int *P, int n, int m, const double *ref,
                             float *lower, float *upper, int *Kout) {
  extern __shared__ double ws_boxes[];
  const int b = blockIdx.x, cap = 2 * n + 2;
  boxes_block(front + (size_t)b * n * m, P[b], n, m, ref + (size_t)b * m,
              lower + (size_t)b * cap * m, upper + (size_t)b * cap * m, Kout + b, ws_boxes);
}

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The engine's front stage, one block per problem: standardise the m outcome
// columns, take the Pareto front, decompose the improving region into boxes.
// It depends on the raw outcomes only, so it runs beside the GP fit.
__global__ void front_fused_kernel(const double *Y, int n, int m, const double *ref, double *Ys,
                                   unsigned char *mask, double *front, int *P, float *lower,
                                   float *upper, int *Kout, int want_boxes) {
  extern __shared__ long long smem_front[];
  __shared__ double part[4][BOUTE_MAX_M], means[BOUTE_MAX_M], isds[BOUTE_MAX_M];
  const int b = blockIdx.x, cap = 2 * n + 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double *Yb = Y + (size_t)b * n * m;
  double *Ysb = Ys + (size_t)b * n * m;
  // Four warps per outcome for the sums, one of them for the quotients and the root:
  // few warps issue fp64 (every thread doing them all took 15 of 26 us at n = 32).
  const int t = warp >> 2, q = warp & 3;
  if (t < m) {
    double s = 0.0;
    for (int i = 32 * q + lane; i < n; i += 128) s += Yb[(size_t)i * m + t];
    s = warp_sum_f64(s);
    if (lane == 0) part[q][t] = s;
  }
  __syncthreads();
  if (t < m && q == 0) {
    const double mean = ((part[0][t] + part[1][t]) + (part[2][t] + part[3][t])) / n;
    if (lane == 0) means[t] = mean;
  }
  __syncthreads();
  if (t < m) {
    const double mean = means[t];
    double ss = 0.0;
    for (int i = 32 * q + lane; i < n; i += 128) {
      const double z = Yb[(size_t)i * m + t] - mean;
      ss += z * z;
    }
    ss = warp_sum_f64(ss);
    if (lane == 0) part[q][t] = ss;
  }
  __syncthreads();
  if (t < m && q == 0) {
    const double ss = (part[0][t] + part[1][t]) + (part[2][t] + part[3][t]);
    double sd = n > 1 ? sqrt(ss / (n - 1)) : 1.0;
    if (!(sd >= 1e-8)) sd = 1.0;
    if (lane == 0) isds[t] = 1.0 / sd;
  }
  __syncthreads();
  for (int c = 0; c < m; ++c) {
    const double mean = means[c], isd = isds[c];
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      Ysb[(size_t)i * m + c] = (Yb[(size_t)i * m + c] - mean) * isd;
  }
  __syncthreads();
  __shared__ int Pb;
  pareto_block(Ysb, n, m, ref + (size_t)b * m, mask + (size_t)b * n, front + (size_t)b * n * m,
               &Pb, smem_front);
  if (threadIdx.x == 0) P[b] = Pb;
  if (want_boxes)
    boxes_block(front + (size_t)b * n * m, Pb, n, m, ref + (size_t)b * m,
                lower + (size_t)b * cap * m, upper + (size_t)b * cap * m, Kout + b, smem_front);
}

}  // namespace

int launch_pareto(const double *Ys, int B, int n, int m, const double *ref, unsigned char *mask,
                  double *front, int *P, cudaStream_t s) {
  const size_t smem = (size_t)n * m * sizeof(long long) + (size_t)n * sizeof(int) + 16;
  cudaFuncSetAttribute(pareto_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  pareto_kernel<<<B, 512, smem, s>>>(Ys, n, m, ref, mask, front, P);
  count_launch();
  return last_launch_status();
}

int launch_boxes(const double *front, const int *P, int B, int n, int m, const double *ref,
                 float *lower, float *upper, int *K, cudaStream_t s) {
  size_t smem = 0;
  if (m == 3) smem = (size_t)13 * (n + 2) * sizeof(double);
  else if (m != 2) return BOUTE_ERR_UNSUPPORTED;
  cudaFuncSetAttribute(boxes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  boxes_kernel<<<B, 256, smem, s>>>(front, P, n, m, ref, lower, upper, K);
  count_launch();
  return last_launch_status();
}

size_t front_smem_bytes(int n, int m) {
  const size_t pk = (size_t)n * m * sizeof(long long) + (size_t)n * sizeof(int) + 16;
  const size_t bx = m == 3 ? (size_t)13 * (n + 2) * sizeof(double) : 0;
  return pk > bx ? pk : bx;
}

int launch_front_fused(const double *Y, int B, int n, int m, const double *ref, double *Ys,
                       unsigned char *mask, double *front, int *P, float *lower, float *upper,
                       int *K, int want_boxes, cudaStream_t s) {
  const size_t smem = front_smem_bytes(n, m);
  prefer_shared(front_fused_kernel);
  // (static arrays count against the same 48 KB default: always set)
  cudaFuncSetAttribute(front_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem);
  front_fused_kernel<<<B, 512, smem, s>>>(Y, n, m, ref, Ys, mask, front, P, lower, upper, K,
                                          want_boxes);
  count_launch();
  return last_launch_status();
}

BOUTE_BOUNDS_READER(front)

}  // namespace boute

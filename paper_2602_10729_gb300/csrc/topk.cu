// Deterministic top-k per problem. Values become 64-bit keys (order-preserving
// float bits in the high word, the complement of the index in the low word), so
// one unsigned comparison orders by value descending, then index ascending, and
// no two keys are equal.
//
// A block selects rather than sorts: it holds its segment's keys in registers
// and builds the k-th largest key bit by bit, counting the keys at or above
// each trial with the barrier's own count (__syncthreads_count, one barrier
// per bit). The k-th largest of the threads' maxima comes first: k keys at
// least reach it, and few others do, so that the rest of the search runs on the
// survivors, one or two per thread. When more survive than that, the search runs on
// all of the segment's keys, two bits a barrier (k near the thread count, sorted inputs),
// or, when they tie there (scores that are mostly zero), ends at that value: of values,
// the ties wanted are the first by position, found by one scan.
// Level 1 keeps k keys of each 8192 values; a further level does the same to
// 8192 keys; as soon as 16384 entries (values or keys) are left, one block per
// problem selects the k best and ranks them by counting. What bounds it is the
// chain of barriers (about 70 a level), not the reads.
// Four problems of 1 Mi values, k = 100: 25 us (bitonic sorts of 2048-key
// segments, four launches: 232 us); mostly zero 30. One problem of 4096 values, k = 8:
// 3.5 us, mostly zero 7.2 (a warp's running top 32: 12.5 and 10.4); of 65536, k = 32: 10
// and 13 (14.5 and 10.6).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "warp_select.cuh"

namespace boute {

namespace {

constexpr int kR = 16;                   // entries per thread
constexpr int kSegThreads = 512;         // a level's blocks: segments of 8192 entries
constexpr int kFinThreads = 1024;        // the last level: up to 16384 entries
constexpr int kSeg = kSegThreads * kR;
constexpr int kFin = kFinThreads * kR;
constexpr int kMaxK = 1024;

// Sums over the block's NT threads of three counts of at most kR each, packed ten bits
// apart, for every thread; turn: alternate between two halves of red (2 NT / 32 words), so
// that one barrier a call is enough.
template <int NT>
__device__ __forceinline__ void block_counts(unsigned c, int turn, unsigned *red, int (&sum)[3]) {
  static_assert(32 * kR < 1024, "a warp's counts fit ten bits");
  const int lane = threadIdx.x & 31;
  c = __reduce_add_sync(0xffffffffu, c);
  unsigned *half = red + (turn & 1) * (NT / 32);
  if (lane == 0) half[threadIdx.x >> 5] = c;
  __syncthreads();
  const unsigned w = lane < NT / 32 ? half[lane] : 0u;
#pragma unroll
  for (int u = 0; u < 3; ++u)
    sum[u] = (int)__reduce_add_sync(0xffffffffu, (w >> (10 * u)) & 1023u);
}

// The largest t with at least k keys >= t (count(t): how many are), built from
// the top bit of the low `bits`, above which it has those of `ones`; exact: set when
// exactly k keys reach it.
template <class Count>
__device__ __forceinline__ unsigned kth_word(int k, unsigned ones, int bits, bool &exact,
                                             Count count) {
  unsigned t = ones;
  exact = false;
  for (unsigned bit = 1u << (bits - 1); bit && !exact; bit >>= 1) {
    const int c = count(t | bit);
    if (c >= k) t |= bit;
    exact = c == k;
  }
  return t;
}

// The same for counts over all of the threads' keys (count_of(t): this thread's at or above
// t), two bits a round.
template <int NT, class CountOf>
__device__ __forceinline__ unsigned kth_word_all(int k, unsigned ones, int bits, unsigned *red,
                                                 bool &exact, CountOf count_of) {
  unsigned t = ones;
  exact = false;
  for (int b = (bits + 1) & ~1, turn = 0; b > 0 && !exact; ++turn) {
    b -= 2;
    unsigned c = 0u;
#pragma unroll
    for (unsigned u = 1; u <= 3; ++u) c += count_of(t | (u << b)) << (10 * (u - 1));
    int sum[3];
    block_counts<NT>(c, turn, red, sum);
    const int u = sum[2] >= k ? 3 : sum[1] >= k ? 2 : sum[0] >= k ? 1 : 0;
    t |= (unsigned)u << b;
    exact = u > 0 && (u == 3 ? sum[2] : u == 2 ? sum[1] : sum[0]) == k;
  }
  __syncthreads();  // (red may be used again from its first half)
  return t;
}

// The k largest keys of the block's segment (hi[r], lo(r): the words of this
// thread's keys, hi = 0 for none; the lo words' bits above lo_bits are all ones), in any
// order, into out (shared or global); fewer when the segment holds fewer. POS: keys of
// equal value descend with their position (r, thread). Returns how many.
template <int NT, bool POS, class Lo>
__device__ __forceinline__ int block_select(const unsigned (&hi)[kR], Lo lo, int lo_bits, int k,
                                            unsigned long long *buf, unsigned *red,
                                            unsigned long long *out) {
  __shared__ int nsurv, nout;
  const unsigned ones = lo_bits < 32 ? ~0u << lo_bits : 0u;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) nsurv = nout = 0;
  unsigned m = 0u;
#pragma unroll
  for (int r = 0; r < kR; ++r) m = max(m, hi[r]);
  bool exact = true;
  unsigned t0 = 0u;
  if (k <= NT)
    t0 = kth_word(k, 0u, 32, exact, [&](unsigned t) { return __syncthreads_count(m >= t); });
  else __syncthreads();
  t0 = max(t0, 1u);  // (absent keys never survive)
  const bool value = !exact;  // t0 has all its bits: it may be the k-th value
  // survivors into buf, while they fit
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const unsigned bal = __ballot_sync(0xffffffffu, hi[r] >= t0);
    if (bal == 0u) continue;
    int pos = 0;
    if (lane == 0) pos = atomicAdd(&nsurv, __popc(bal));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & ((1u << lane) - 1u));
    if (hi[r] >= t0 && pos < 2 * NT) buf[pos] = ((unsigned long long)hi[r] << 32) | lo(r);
  }
  __syncthreads();
  const int ns = nsurv;
  unsigned long long thr = 0ull;
  auto take = [&](bool in, unsigned long long key) {  // (k keys at most: thr selects exactly)
    if (in) out[atomicAdd(&nout, 1)] = key;
  };
  if (ns <= 2 * NT) {
    const unsigned long long a = tid < ns ? buf[tid] : 0ull;
    const unsigned long long b = tid + NT < ns ? buf[tid + NT] : 0ull;
    if (ns > k) {
      const unsigned ah = (unsigned)(a >> 32), bh = (unsigned)(b >> 32);
      const bool two = ns > NT;
      auto count_above = [&](unsigned t) {
        const int c = __syncthreads_count(ah > t);
        return two ? c + __syncthreads_count(bh > t) : c;
      };
      unsigned th = t0;  // (the k-th value unless k keys lie above it)
      int above = value ? count_above(t0) : k;
      exact = false;
      if (above >= k) {
        th = kth_word(k, 0u, 32, exact, [&](unsigned t) {
          const int c = __syncthreads_count(ah >= t);
          return two ? c + __syncthreads_count(bh >= t) : c;
        });
        if (!exact) above = count_above(th);
      }
      thr = (unsigned long long)th << 32;
      if (!exact) {  // ties at the k-th value: the smallest indices of them
        thr |= kth_word(k - above, ones, lo_bits, exact, [&](unsigned t) {
          const int c = __syncthreads_count(ah == th && (unsigned)a >= t);
          return two ? c + __syncthreads_count(bh == th && (unsigned)b >= t) : c;
        });
      }
    }
    take(a != 0ull && a >= thr, a);
    take(b != 0ull && b >= thr, b);
  } else {
    // More survivors than that: k near the thread count, or ties at t0 (scores that are
    // mostly zero), where t0 itself is the k-th value unless k keys lie above it.
    auto at_least = [&](unsigned t) {
      unsigned c = 0u;
#pragma unroll
      for (int r = 0; r < kR; ++r) c += hi[r] >= t;
      return c;
    };
    int sum[3];
    auto count_above = [&](unsigned t) {
      block_counts<NT>(t == 0xffffffffu ? 0u : at_least(t + 1u), 0, red, sum);
      __syncthreads();
      return sum[0];
    };
    unsigned th = t0;
    int above = value ? count_above(t0) : k;
    exact = false;
    if (above >= k) {
      th = kth_word_all<NT>(k, 0u, 32, red, exact, at_least);
      if (!exact) above = count_above(th);
    }
    thr = (unsigned long long)th << 32;
    if constexpr (POS) {
      // ties by position (r, thread): their counts per r and warp, scanned by one warp
      const int warp = tid >> 5, need = exact ? NT * kR : k - above;
      unsigned *cnt = (unsigned *)buf;  // (the survivors in it are not used)
      unsigned tie[kR];
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        tie[r] = __ballot_sync(0xffffffffu, hi[r] == th);
        if (lane == 0) cnt[r * (NT / 32) + warp] = __popc(tie[r]);
      }
      __syncthreads();
      if (warp == 0) {
        constexpr int E = kR * NT / 32 / 32;  // entries of a lane
        unsigned c[E], run = 0u;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          c[e] = run;
          run += cnt[lane * E + e];
        }
        unsigned sc = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned u = __shfl_up_sync(0xffffffffu, sc, o);
          if (lane >= o) sc += u;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) cnt[lane * E + e] = c[e] + sc - run;
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const int rank = cnt[r * (NT / 32) + warp] + __popc(tie[r] & ((1u << lane) - 1u));
        take(hi[r] > th || (hi[r] == th && rank < need), ((unsigned long long)hi[r] << 32) | lo(r));
      }
    } else {
      if (!exact)
        thr |= kth_word_all<NT>(k - above, ones, lo_bits, red, exact,
                                [&](unsigned t) {
                                  unsigned c = 0u;
#pragma unroll
                                  for (int r = 0; r < kR; ++r) c += hi[r] == th && lo(r) >= t;
                                  return c;
                                });
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const unsigned long long key = ((unsigned long long)hi[r] << 32) | lo(r);
        take(hi[r] != 0u && key >= thr, key);
      }
    }
  }
  __syncthreads();
  return nout;
}

// Segment blockIdx.x (NT * kR entries) of problem blockIdx.y's `len` entries:
// values (VALUES) or keys. FINAL: the only segment; the k best in order to idx
// and val (acq: the scores that the indices refer to). Otherwise its k best,
// padded with zero keys, to keys_out.
template <int NT, bool VALUES, bool FINAL>
__global__ void __launch_bounds__(NT) topk_kernel(const float *vals,
                                                  const unsigned long long *keys_in,
                                                  long long len, int k,
                                                  unsigned long long *keys_out, const float *acq,
                                                  long long N, long long *idx, float *val) {
  __shared__ unsigned long long buf[2 * NT];
  __shared__ unsigned red[2 * NT / 32];
  __shared__ unsigned long long sel[FINAL ? (NT < kMaxK ? NT : kMaxK) : 1];
  pdl_wait();
  if (!FINAL) pdl_trigger();
  const int b = blockIdx.y, tid = threadIdx.x;
  const long long base = (long long)blockIdx.x * (NT * kR);
  unsigned hi[kR], lw[VALUES ? 1 : kR];
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const long long g = base + r * NT + tid;
    unsigned long long key = 0ull;  // below every real key
    if (g < len)
      key = VALUES ? make_key(__ldcs(vals + (size_t)b * len + g), (unsigned)g)
                   : __ldcg(keys_in + (size_t)b * len + g);
    hi[r] = (unsigned)(key >> 32);
    if (!VALUES) lw[r] = (unsigned)key;
  }
  const int lo_bits = N > 1 ? 64 - __clzll(N - 1) : 1;  // (of 0xffffffff - index, index < N)
  auto lo = [&](int r) {
    if (VALUES) return 0xFFFFFFFFu - (unsigned)(base + r * NT + tid);
    return lw[VALUES ? 0 : r];
  };
  if constexpr (!FINAL) {
    unsigned long long *out = keys_out + ((size_t)b * gridDim.x + blockIdx.x) * k;
    const int got = block_select<NT, VALUES>(hi, lo, lo_bits, k, buf, red, out);
    for (int i = got + tid; i < k; i += NT) out[i] = 0ull;
  } else {
    block_select<NT, VALUES>(hi, lo, lo_bits, k, buf, red, sel);
    // rank of each selected key, `per` threads (a power of two) to a key
    int per = 1;
    while (per < 32 && 2 * per * k <= NT) per *= 2;
    const int q = tid / per, p = tid & (per - 1);
    int rank = 0;
    const unsigned long long key = q < k ? sel[q] : 0ull;
    if (q < k)
      for (int j = p; j < k; j += per) rank += sel[j] > key;
    for (int o = per >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (q < k && p == 0) {
      const unsigned j = key_index(key);
      if (BOUTE_INB(rank, k) && BOUTE_INB(j, N)) {
        idx[(size_t)b * k + rank] = (long long)j;
        val[(size_t)b * k + rank] = acq[(size_t)b * N + j];
      }
    }
  }
}

}  // namespace

// Scratch for the levels after the first: two ping-pong key arrays, at most
// ceil(N / 8192) * k keys per problem and level (the bound counts segments of
// 2048 and k as at least 32, which boute_select_topk_noalloc's limit states).
size_t topk_scratch_bytes(int B, long long N, int k) {
  const long long g1 = (N + 2047) / 2048;
  if (g1 <= 1) return 16;
  return 2 * (size_t)B * g1 * std::max(k, 32) * sizeof(unsigned long long) + 16;
}

// The last level's block for len entries: the fewest threads that hold them and twice k (with
// fewer the k-th of their maxima leaves most entries to the second search: N = 8192, k = 512
// 20 us with 512, 17 with 1024), whose barriers are cheaper and of whose blocks more run at
// once (N = 1024, k = 32, 1000 problems: 8 us with 128 threads, 35 with 1024; N = 4096,
// k = 8, one problem: 3.9 with 256, 5.5).
template <class Go>
static void final_threads(long long len, int k, Go go) {
  if (len <= 128 * kR && k <= 64) go(std::integral_constant<int, 128>{});
  else if (len <= 256 * kR && k <= 128) go(std::integral_constant<int, 256>{});
  else if (len <= 512 * kR && k <= 256) go(std::integral_constant<int, 512>{});
  else go(std::integral_constant<int, kFinThreads>{});
}

int launch_topk(const float *acq, int B, long long N, int k, long long *idx, float *val,
                void *scratch, cudaStream_t s) {
  if (k > kMaxK) return BOUTE_ERR_UNSUPPORTED;
  const unsigned long long *no_keys = nullptr;
  const float *no_vals = nullptr;
  unsigned long long *no_out = nullptr;
  long long *ni = nullptr;
  float *nv = nullptr;
  if (N <= kFin) {
    final_threads(N, k, [&](auto nt) {
      constexpr int NT = decltype(nt)::value;
      launch_pdl(topk_kernel<NT, true, true>, dim3(1, B), dim3(NT), 0, s, acq, no_keys, N, k,
                 no_out, acq, N, idx, val);
    });
    count_launch(1);
    return last_launch_status();
  }
  int launches = 2;
  long long nseg = (N + kSeg - 1) / kSeg, len = nseg * k;
  unsigned long long *ping = (unsigned long long *)scratch, *pong = ping + (size_t)B * len;
  launch_pdl(topk_kernel<kSegThreads, true, false>, dim3((unsigned)nseg, B), dim3(kSegThreads), 0,
             s, acq, no_keys, N, k, ping, acq, N, ni, nv);
  for (; len > kFin; ++launches) {
    nseg = (len + kSeg - 1) / kSeg;
    launch_pdl(topk_kernel<kSegThreads, false, false>, dim3((unsigned)nseg, B), dim3(kSegThreads),
               0, s, no_vals, (const unsigned long long *)ping, len, k, pong, acq, N, ni, nv);
    std::swap(ping, pong);
    len = nseg * k;
  }
  final_threads(len, k, [&](auto nt) {
    constexpr int NT = decltype(nt)::value;
    launch_pdl(topk_kernel<NT, false, true>, dim3(1, B), dim3(NT), 0, s, no_vals,
               (const unsigned long long *)ping, len, k, no_out, acq, N, idx, val);
  });
  count_launch(launches);
  return last_launch_status();
}

BOUTE_BOUNDS_READER(topk)

}  // namespace boute

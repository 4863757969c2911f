// Top-k of one head's scores by histograms of their keys, for one thread block.
// Shared by the stand-alone selection kernel and by the smoothing kernel, which selects straight from the
// smoothed scores it still holds on chip.
#pragma once

#include "common.cuh"

namespace akv {

// Order-preserving map float -> uint32 (larger float, larger key); -0 and +0 share a key.
__device__ __forceinline__ uint32_t score_key(float f) {
  uint32_t u = __float_as_uint(f);
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kSelBins = 2048;
constexpr int kSelCand = 1024;  // keys of the threshold's bin kept in a list
constexpr int kSelSub = 512;    // bins of the histogram over that list
constexpr int kSelRank = 64;    // keys ranked by comparison with one another

struct SelectSmem {
  int hist[kSelBins];
  uint2 cand[kSelCand];  // (key, token)
  int sub[kSelSub];
  uint2 last[kSelRank];
  int wsum[32];
  uint32_t lo;
  int want, cnt, n_cand, n_last;
};

// Loops of a block of T threads over [0, n): get(i) for U elements before the first use(i, value). Without a branch between
// them the loads of the U elements are in flight together.
template <int T, int U, class Get, class Use>
__device__ __forceinline__ void batched_loop(int n, Get get, Use use) {
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += U * T) {
    decltype(get(0)) v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) v[q] = get(min(i + q * T, n - 1));
#pragma unroll
    for (int q = 0; q < U; ++q)
      if (i + q * T < n) use(i + q * T, v[q]);
  }
}

// Exclusive prefix of v over a block of T threads; *total gets the sum.
template <int T>
__device__ __forceinline__ int block_excl_scan_int(int v, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  const int ws = lane < T / 32 ? wsum[lane] : 0;
  int winc = ws;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, winc, o);
    if (lane >= o) winc += t;
  }
  *total = __shfl_sync(0xffffffffu, winc, 31);
  return __shfl_sync(0xffffffffu, winc - ws, warp) + inc - v;
}

// words of shared memory a selection over M entries needs for its bit masks and their prefix sums
__host__ __device__ inline int select_words(int M, bool pair) { return (pair ? 2 : 1) * ((M + 31) / 32); }

// Writes to `out` the k prefix tokens (of P) with the largest keys, ties to the lower index, in ascending token order,
// then the W window tokens P .. P+W-1. The keys come as M entries: PAIR: ld(m) = keys of tokens 2m and 2m + 1 (a token
// >= P is ignored); else ld(m).x = key of token m. kmin and kmax are the smallest and the largest key. Every thread of
// the block calls this with the same arguments. words: select_words(M, PAIR) uint32 of shared memory, which may lie
// over sm->hist; pre: ceil(M / 32) ints of shared memory.
//
// The block reads the keys twice, whatever the distribution is like (once more for each refinement of the histogram):
//   1. a histogram of 2048 bins over [kmin, kmax] (equal steps of the key, that is of the float's bits: about 70 bins
//      an octave for scores spread over thirty octaves; a histogram of the key's top 11 bits has four, so that a few
//      counters took most of the atomic adds, and three passes over every key were needed in any case). A bin that
//      holds the k-th key and more than kSelCand others is histogrammed again;
//   2. one bit per key above that bin, ballots written as words, and a list of the bin's own keys; a histogram over the
//      list and a comparison of the few keys of its threshold bin, (key, lower index), give the bits of the list's keys;
//   3. prefix sums over the words; every kept token's place follows from its word's sum and the bits below its own.
template <int T, bool PAIR, typename Ld>
__device__ __forceinline__ void select_entries(Ld ld, int M, int P, int W, int k, uint32_t kmin, uint32_t kmax,
                                               int32_t* __restrict__ out, SelectSmem* sm, uint32_t* words, int* pre,
                                               int* __restrict__ status) {
  constexpr int A = PAIR ? 2 : 1;
  constexpr int kOwn = kSelBins / T;  // bins per thread
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const int ng = (M + 31) / 32;  // groups of 32 entries: one word (two with PAIR: even and odd tokens) each
  if (k > 0 && k < P) {
    uint32_t lo = kmin;
    const uint32_t range = kmax - kmin;
    int shift = range == 0u ? 0 : max(0, 21 - __clz(range));  // (kmax - kmin) >> shift < 2048
    int want = k, cnt = 0;
    uint32_t bins = kSelBins;  // of which this many belong to the range
#pragma unroll 1
    for (;;) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kOwn; ++i) sm->hist[threadIdx.x + T * i] = 0;
      if (threadIdx.x < kSelSub) sm->sub[threadIdx.x] = 0;
      if (threadIdx.x == 0) sm->n_cand = sm->n_last = 0;
      __syncthreads();
      batched_loop<T, 4>(M, ld, [&](int m, float2 e) {
        const uint32_t a = __float_as_uint(e.x), b = __float_as_uint(e.y);
        const uint32_t da = (a - lo) >> shift, db = (b - lo) >> shift;
        if (a >= lo && da < bins) atomicAdd(&sm->hist[da], 1);
        if (PAIR && b >= lo && db < bins && 2 * m + 1 < P) atomicAdd(&sm->hist[db], 1);
      });
      __syncthreads();
      // thread t owns bins 2047 - kOwn t - i (descending)
      const int top = kSelBins - 1 - kOwn * static_cast<int>(threadIdx.x);
      int c[kOwn], sum = 0;
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        c[i] = sm->hist[top - i];
        sum += c[i];
      }
      int tot;
      int above = block_excl_scan_int<T>(sum, sm->wsum, &tot);
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        if (above < want && want <= above + c[i]) {
          sm->lo = lo + (static_cast<uint32_t>(top - i) << shift);
          sm->want = want - above;
          sm->cnt = c[i];
        }
        above += c[i];
      }
      __syncthreads();
      lo = sm->lo;
      want = sm->want;
      cnt = sm->cnt;
      if (cnt <= kSelCand || shift == 0) break;
      bins = 1u << min(shift, 11);
      shift = max(0, shift - 11);
    }
    // keys in [lo, lo + 2^shift) compete for the last `want` places, keys above it are kept
    const bool ties = shift == 0 && cnt > kSelRank;  // many keys equal to lo: the lowest indices, by prefix sums
#pragma unroll 1
    for (int turn = ties ? 0 : 1; turn < 2; ++turn) {
      // turn 0 (ties): how many of them each group has, as prefix sums in `pre`
      constexpr int U = 2;
#pragma unroll 1
      for (int g0 = warp; g0 < ng; g0 += U * (T / 32)) {
        float2 e[U];
#pragma unroll
        for (int q = 0; q < U; ++q) e[q] = ld(min(32 * (g0 + q * (T / 32)) + lane, M - 1));
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int g = g0 + q * (T / 32), m = 32 * g + lane;
          const uint32_t a = __float_as_uint(e[q].x), b = __float_as_uint(e[q].y);
          const bool va = m < M && a >= lo, vb = PAIR && m < M && 2 * m + 1 < P && b >= lo;
          bool ga = va && ((a - lo) >> shift) > 0, gb = vb && ((b - lo) >> shift) > 0;
          const bool ca = va && !ga, cb = vb && !gb;
          if (ties) {
            const uint32_t ea = __ballot_sync(0xffffffffu, ca), eb = PAIR ? __ballot_sync(0xffffffffu, cb) : 0u;
            if (turn == 0) {
              if (lane == 0 && g < ng) pre[g] = __popc(ea) + __popc(eb);
            } else {
              const int rank = (g < ng ? pre[g] : 0) + __popc(ea & lt) + __popc(eb & lt);
              ga = ga || (ca && rank < want);
              gb = gb || (cb && rank + (ca ? 1 : 0) < want);
            }
          } else {
            if (ca) sm->cand[atomicAdd(&sm->n_cand, 1)] = make_uint2(a, A * m);
            if (cb) sm->cand[atomicAdd(&sm->n_cand, 1)] = make_uint2(b, A * m + 1);
          }
          if (turn == 1) {
            const uint32_t wa = __ballot_sync(0xffffffffu, ga), wb = PAIR ? __ballot_sync(0xffffffffu, gb) : 0u;
            if (lane == 0 && g < ng) {
              words[A * g] = wa;
              if (PAIR) words[A * g + 1] = wb;
            }
          }
        }
      }
      __syncthreads();
      if (turn == 0) {
        const int per = (ng + T - 1) / T, g0 = min(ng, static_cast<int>(threadIdx.x) * per), g1 = min(ng, g0 + per);
        int sum = 0, tot;
        for (int g = g0; g < g1; ++g) sum += pre[g];
        int run = block_excl_scan_int<T>(sum, sm->wsum, &tot);
        for (int g = g0; g < g1; ++g) {
          const int v = pre[g];
          pre[g] = run;
          run += v;
        }
        __syncthreads();
      }
    }
    if (!ties) {
      auto keep = [&](uint32_t tok) {
        const int m = static_cast<int>(tok) / A;
        atomicOr(&words[A * (m >> 5) + (PAIR ? (tok & 1) : 0)], 1u << (m & 31));
      };
      // the list's threshold bin: all of it when the list is short
      int sub_shift = 32, bin = 0;
      if (cnt > kSelRank) {
        sub_shift = max(0, shift - 9);
        for (int i = threadIdx.x; i < cnt; i += T) atomicAdd(&sm->sub[(sm->cand[i].x - lo) >> sub_shift], 1);
        __syncthreads();
        const int mine = threadIdx.x < kSelSub ? sm->sub[kSelSub - 1 - threadIdx.x] : 0;
        int tot;
        const int above = block_excl_scan_int<T>(mine, sm->wsum, &tot);
        if (above < want && want <= above + mine) {
          sm->lo = kSelSub - 1 - threadIdx.x;
          sm->want = want - above;
          sm->cnt = mine;
        }
        __syncthreads();
        bin = static_cast<int>(sm->lo);
        want = sm->want;
      }
      const bool few = (cnt > kSelRank ? sm->cnt : cnt) <= kSelRank;  // else (close keys): ranked within the list itself
      for (int i = threadIdx.x; i < cnt; i += T) {
        const uint2 me = sm->cand[i];
        const int q = sub_shift > 31 ? 0 : static_cast<int>((me.x - lo) >> sub_shift);
        if (q > bin) keep(me.y);
        if (q == bin && few) sm->last[atomicAdd(&sm->n_last, 1)] = me;
        if (q == bin && !few) {
          int rank = 0;
          for (int j = 0; j < cnt; ++j) {
            const uint2 o = sm->cand[j];
            const int oq = static_cast<int>((o.x - lo) >> sub_shift);
            rank += oq == bin && (o.x > me.x || (o.x == me.x && o.y < me.y));
          }
          if (rank < want) keep(me.y);
        }
      }
      __syncthreads();
      if (few) {
        const int n_last = sm->n_last;
        if (static_cast<int>(threadIdx.x) < n_last) {
          const uint2 me = sm->last[threadIdx.x];
          int rank = 0;
#pragma unroll 4
          for (int j = 0; j < n_last; ++j) {
            const uint2 o = sm->last[j];
            rank += o.x > me.x || (o.x == me.x && o.y < me.y);
          }
          if (rank < want) keep(me.y);
        }
        __syncthreads();
      }
    }
    // places: prefix sums over the groups
    const int per = (ng + T - 1) / T, g0 = min(ng, static_cast<int>(threadIdx.x) * per), g1 = min(ng, g0 + per);
    int sum = 0, tot;
    for (int g = g0; g < g1; ++g) sum += __popc(words[A * g]) + (PAIR ? __popc(words[A * g + 1]) : 0);
    int run = block_excl_scan_int<T>(sum, sm->wsum, &tot);
    for (int g = g0; g < g1; ++g) {
      pre[g] = run;
      run += __popc(words[A * g]) + (PAIR ? __popc(words[A * g + 1]) : 0);
    }
    if (tot != k && threadIdx.x == 0) atomicExch(status, AUDIOKV_EDEVICE);  // unordered (NaN) keys
    __syncthreads();
#pragma unroll 2
    for (int g = warp; g < ng; g += T / 32) {
      const uint32_t wa = words[A * g], wb = PAIR ? words[A * g + 1] : 0u;
      int pos = pre[g] + __popc(wa & lt) + __popc(wb & lt);
      const int tok = A * (32 * g + lane);
      if ((wa >> lane) & 1u) {
        if (pos < k) out[pos] = tok;
        ++pos;
      }
      if (PAIR && ((wb >> lane) & 1u) && pos < k) out[pos] = tok + 1;
    }
  } else if (k > 0) {
    for (int j = threadIdx.x; j < k; j += T) out[j] = j;
  }
  for (int i = threadIdx.x; i < W; i += T) out[k + i] = P + i;
  __syncthreads();
}

}  // namespace akv

// Offline head score: for every decode step and head, the top-K tokens of the attention row, how many of them
// fall inside the audio span of the word generated at that step, and the mean of that ratio over the steps.
//
// What bounds it: the rows, read once (64 steps x 784 heads x 8192 tokens are 1.6 GB, 0.25 ms of HBM). So a row belongs to
// one warp, which streams it through registers and keeps the maxima of 32 groups of its values per lane; the k-th largest
// of the lanes' maxima bounds the k-th largest value from below; the few groups that reach the bound are read once more
// (from L2) and their values listed; the listed values inside the span are ranked against the list. No barrier joins
// two warps, so that twenty rows an SM are in different phases and the loads never stop: 289 us, 87 % of the measured
// copy bandwidth. Rows a list cannot serve (top_k above 32, many values equal to the bound, NaN) are left to the
// whole block, a histogram of the keys at a time.
#include "common.cuh"
#include "select.cuh"

namespace akv {
namespace {

constexpr int kHitWarps = 4;                 // warps per block
constexpr int kHitThreads = 32 * kHitWarps;
constexpr int kHitBlocksPerSm = 5;
constexpr int kHitGroups = 32;               // groups of a lane's 16-byte pieces (two pieces each at 8192 values a row)
constexpr int kHitCand = 512;                // listed values of a row
constexpr int kHitListK = 32;                // top_k up to which a warp lists: one maximum a lane bounds the k-th value
constexpr int kHitTurn = 32;                 // rows a warp goes through before the block takes what was left over
constexpr int kHitBins = 2048;
constexpr int kHitRank = 256;                // keys of the threshold's bin that are ranked by comparison

struct HitList {
  float val[kHitCand];
  int idx[kHitCand];
  uint16_t entry[kHitGroups * 32];           // groups that reach the bound: group * 32 + lane
};
struct HitBlock {
  int hist[kHitBins];
  uint32_t key[kHitRank];
  int idx[kHitRank];
  uint32_t red[2][kHitWarps];
  int scan[kHitWarps];
  uint32_t lo;
  int want, cnt, n, hits, gt_in, eq_before, eq_in;
};
union HitSmem {
  HitList warp[kHitWarps];
  HitBlock block;
};

// The larger value, NaN if either is NaN.
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// use(x, j) for every value x at place j of the row, by the whole block, as 16-byte pieces with the singles around them.
template <class Use>
__device__ __forceinline__ void for_row(const float* __restrict__ row, int L, Use use) {
  const int j0 = min(L, static_cast<int>((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) >> 2);
  const int nvec = (L - j0) >> 2, tail = j0 + 4 * nvec;
  const float4* rv = reinterpret_cast<const float4*>(row + j0);
  if (nvec)
    batched_loop<kHitThreads, 8>(nvec, [&](int m) { return __ldg(rv + m); }, [&](int m, float4 v) {
      use(v.x, j0 + 4 * m);
      use(v.y, j0 + 4 * m + 1);
      use(v.z, j0 + 4 * m + 2);
      use(v.w, j0 + 4 * m + 3);
    });
  const int t = threadIdx.x, j = t < 3 ? t : tail + t - 3;
  if (t < 3 ? t < j0 : t < 6 && j < L) use(__ldg(row + j), j);
}

// Exact count for one row of any kind, by the whole block: a histogram of 2048 equal steps between the smallest and the largest
// key (equal steps of the float's bits), again inside the bin of the k-th key while that holds too many, then a comparison
// of its keys; of the keys equal to the k-th the lowest indices count. Keys order a NaN by its bits: above every
// number, or below with the sign bit set. Eight rows of 8192 take 18 us, 1792 of them 50, whatever top_k is.
__device__ __noinline__ int hits_by_block(const float* __restrict__ row, int L, int k, int lo_tok, int hi_tok, HitBlock& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kOwn = kHitBins / kHitThreads;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  for_row(row, L, [&](float x, int) {
    const uint32_t key = score_key(x);
    kmin = min(kmin, key);
    kmax = max(kmax, key);
  });
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  __syncthreads();  // the row before is done with the shared state
  if (lane == 0) {
    sm.red[0][warp] = kmin;
    sm.red[1][warp] = kmax;
  }
  if (threadIdx.x == 0) sm.n = sm.hits = sm.gt_in = sm.eq_before = sm.eq_in = 0;
  __syncthreads();
  for (int w = 0; w < kHitWarps; ++w) {
    kmin = min(kmin, sm.red[0][w]);
    kmax = max(kmax, sm.red[1][w]);
  }
  // keys in [lo, lo + bins << shift) are looked at; `want` of the k largest lie among the bin's keys
  uint32_t lo = kmin, bins = kHitBins;
  int shift = max(0, 21 - __clz((kmax - kmin) | 1u)), want = k, cnt = L;  // (kmax - kmin) >> shift < 2048
#pragma unroll 1
  while (kmax > kmin) {
#pragma unroll
    for (int i = 0; i < kOwn; ++i) sm.hist[threadIdx.x + kHitThreads * i] = 0;
    __syncthreads();
    for_row(row, L, [&](float x, int) {
      const uint32_t key = score_key(x), d = (key - lo) >> shift;
      if (key >= lo && d < bins) atomicAdd(&sm.hist[d], 1);
    });
    __syncthreads();
    const int top = kHitBins - 1 - kOwn * static_cast<int>(threadIdx.x);  // this thread's bins, descending
    int sum = 0;
#pragma unroll
    for (int i = 0; i < kOwn; ++i) sum += sm.hist[top - i];
    int total;
    int above = block_excl_scan_int<kHitThreads>(sum, sm.scan, &total);
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
      const int c = sm.hist[top - i];
      if (above < want && want <= above + c) {
        sm.lo = lo + (static_cast<uint32_t>(top - i) << shift);
        sm.want = want - above;
        sm.cnt = c;
      }
      above += c;
    }
    __syncthreads();
    lo = sm.lo;
    want = sm.want;
    cnt = sm.cnt;
    if (cnt <= kHitRank || shift == 0) break;
    bins = 1u << min(shift, 11);
    shift = max(0, shift - 11);
    __syncthreads();
  }
  const bool ties = cnt > kHitRank;  // then shift is 0: that many keys equal to lo
  int gt_in = 0, eq_before = 0, eq_in = 0;
  for_row(row, L, [&](float x, int j) {
    const uint32_t key = score_key(x);
    if (key < lo) return;
    const bool in = j >= lo_tok && j <= hi_tok, gt = ((key - lo) >> shift) > 0;
    gt_in += gt && in;
    if (gt) return;
    if (ties) {
      eq_before += j < lo_tok;
      eq_in += in;
    } else {
      const int at = atomicAdd(&sm.n, 1);
      sm.key[at] = key;
      sm.idx[at] = j;
    }
  });
  gt_in = __reduce_add_sync(0xffffffffu, gt_in);
  eq_before = __reduce_add_sync(0xffffffffu, eq_before);
  eq_in = __reduce_add_sync(0xffffffffu, eq_in);
  if (lane == 0) {
    atomicAdd(&sm.gt_in, gt_in);
    atomicAdd(&sm.eq_before, eq_before);
    atomicAdd(&sm.eq_in, eq_in);
  }
  __syncthreads();
  if (!ties) {
    const int n = sm.n;
    for (int i = threadIdx.x; i < n; i += kHitThreads) {
      const uint32_t key = sm.key[i];
      const int j = sm.idx[i];
      if (j < lo_tok || j > hi_tok) continue;
      int rank = 0;
#pragma unroll 4
      for (int o = 0; o < n; ++o) rank += sm.key[o] > key || (sm.key[o] == key && sm.idx[o] < j);
      if (rank < want) atomicAdd(&sm.hits, 1);
    }
    __syncthreads();
  }
  return sm.gt_in + (ties ? min(sm.eq_in, max(0, want - sm.eq_before)) : sm.hits);
}

__global__ void __launch_bounds__(kHitThreads, kHitBlocksPerSm)
hit_count_kernel(const float* __restrict__ attn, int n_steps, int n_heads, int64_t row_stride,
                 const int32_t* __restrict__ row_len, const int32_t* __restrict__ span, int top_k,
                 int32_t* __restrict__ counts) {
  __shared__ HitSmem sm_all;
  __shared__ int left[kHitWarps * kHitTurn], n_left;  // rows for the block
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const int n_pairs = n_steps * n_heads;
  // Rows are dealt out over the blocks first, so that few rows have a block each.
#pragma unroll 1
  for (int64_t turn = 0; turn < n_pairs; turn += static_cast<int64_t>(gridDim.x) * kHitWarps * kHitTurn) {
    if (threadIdx.x == 0) n_left = 0;
    __syncthreads();
#pragma unroll 1
    for (int i = warp; i < kHitWarps * kHitTurn; i += kHitWarps) {
      const int64_t pair = turn + static_cast<int64_t>(i) * gridDim.x + blockIdx.x;
      if (pair >= n_pairs) break;
      HitList& sm = sm_all.warp[warp];
      const int t = static_cast<int>(pair) / n_heads, a = static_cast<int>(pair) - t * n_heads;
      const int L = __ldg(row_len + t);
      const float* row = attn + pair * row_stride;
      const int lo = max(__ldg(span + 2 * t), 0), hi = min(__ldg(span + 2 * t + 1), L - 1);
      const int k = min(top_k, L);
      if (lo > hi) continue;  // nothing to count
      if (k >= L) {           // every token is kept
        if (lane == 0) atomicAdd(counts + a, hi - lo + 1);
        continue;
      }
      int n = 0;  // listed values
      if (k <= kHitListK) {
        // the row as up to three single values, 16-byte pieces, up to three single values; piece lane + 32 i is this lane's
        const int j0 = min(L, static_cast<int>((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) >> 2);
        const int nvec = (L - j0) >> 2, tail = j0 + 4 * nvec;
        const float4* rv = reinterpret_cast<const float4*>(row + j0);
        const int gs = (nvec + 32 * kHitGroups - 1) / (32 * kHitGroups);  // pieces of a group: i = g gs .. (g + 1) gs - 1
        float gm[kHitGroups];
#pragma unroll
        for (int g0 = 0; g0 < kHitGroups; g0 += 8) {
#pragma unroll
          for (int g = 0; g < 8; ++g) gm[g0 + g] = -INFINITY;
#pragma unroll 1
          for (int i = 0; i < gs; ++i) {
            float4 v[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const int m = lane + 32 * ((g0 + g) * gs + i);
              v[g] = m < nvec ? __ldg(rv + m) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            }
#pragma unroll
            for (int g = 0; g < 8; ++g) gm[g0 + g] = max_nan(max_nan(gm[g0 + g], max_nan(v[g].x, v[g].y)), max_nan(v[g].z, v[g].w));
          }
        }
        // Lower bound of the k-th largest value: the k-th largest of the 32 lanes' maxima. Of 8192 values and k = 24 about 45 lie
        // at or above it.
        float me = -INFINITY;
#pragma unroll
        for (int g = 0; g < kHitGroups; ++g) me = max_nan(me, gm[g]);
        const bool nan = isnan(me);
        int rank = 0;  // ties to the lower lane
        for (int o = 0; o < 32; ++o) {
          const float other = __shfl_sync(0xffffffffu, me, o);
          rank += other > me || (other == me && o < lane);
        }
        const uint32_t at_k = __ballot_sync(0xffffffffu, rank == k - 1);
        const float bound = at_k ? __shfl_sync(0xffffffffu, me, __ffs(at_k) - 1) : -INFINITY;  // none: NaN
        int n_ent = 0;
#pragma unroll
        for (int g = 0; g < kHitGroups; ++g) {
          const bool in = lane + 32 * (g * gs) < nvec && gm[g] >= bound;  // a short row leaves most groups empty
          const uint32_t b = __ballot_sync(0xffffffffu, in);
          if (in) sm.entry[n_ent + __popc(b & lt)] = static_cast<uint16_t>(g * 32 + lane);
          n_ent += __popc(b);
        }
        __syncwarp();
        auto take = [&](bool have, float x, int j) {  // by the whole warp
          const bool in = have && x >= bound;
          const uint32_t b = __ballot_sync(0xffffffffu, in);
          const int at = n + __popc(b & lt);
          if (in && at < kHitCand) {
            sm.val[at] = x;
            sm.idx[at] = j;
          }
          n += __popc(b);
        };
#pragma unroll 1
        for (int e = 0; e < n_ent && n <= kHitCand; e += 32) {
          const int id = e + lane < n_ent ? sm.entry[e + lane] : 0;
#pragma unroll 2
          for (int i = 0; i < gs; ++i) {
            const int m = (id & 31) + 32 * ((id >> 5) * gs + i);
            const bool have = e + lane < n_ent && m < nvec;
            const float4 x = have ? __ldg(rv + m) : make_float4(0.f, 0.f, 0.f, 0.f);
            const int j = j0 + 4 * m;
            if (!__any_sync(0xffffffffu, have && fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)) >= bound)) continue;
            take(have, x.x, j);
            take(have, x.y, j + 1);
            take(have, x.z, j + 2);
            take(have, x.w, j + 3);
          }
        }
        const int single = lane < 3 ? lane : tail + lane - 3;  // the values before and after the pieces
        const bool have = lane < 3 ? lane < j0 : (lane < 6 && single < L);
        const float xs = have ? __ldg(row + single) : 0.f;
        take(have, xs, single);
        if (__any_sync(0xffffffffu, nan || isnan(xs))) n = 0;  // a NaN compares with nothing
        __syncwarp();
      }
      int c = 0;
      if (n >= k && n <= kHitCand) {
        for (int i = lane; i < n; i += 32) {
          const float x = sm.val[i];
          const int j = sm.idx[i];
          if (j < lo || j > hi) continue;
          int rank = 0;
#pragma unroll 4
          for (int o = 0; o < n; ++o) {
            const float y = sm.val[o];
            rank += y > x || (y == x && sm.idx[o] < j);
          }
          c += rank < k;
        }
        c = __reduce_add_sync(0xffffffffu, c);
        __syncwarp();  // the list is free again
      } else if (lane == 0) {
        left[atomicAdd(&n_left, 1)] = static_cast<int>(pair);
      }
      if (lane == 0 && c) atomicAdd(counts + a, c);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < n_left; ++i) {
      const int pair = left[i], t = pair / n_heads, a = pair - t * n_heads;
      const int L = __ldg(row_len + t);
      const int c = hits_by_block(attn + pair * row_stride, L, min(top_k, L), max(__ldg(span + 2 * t), 0),
                                  min(__ldg(span + 2 * t + 1), L - 1), sm_all.block);
      if (threadIdx.x == 0 && c) atomicAdd(counts + a, c);
    }
    __syncthreads();
  }
  chain_release();  // the ratios are launched under the last rows
}

__global__ void hit_ratio_kernel(const int32_t* __restrict__ counts, int n_heads, int n_steps, int top_k,
                                 float* __restrict__ s_hit) {
  chain_wait();
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < n_heads)
    s_hit[a] = static_cast<float>(static_cast<double>(counts[a]) / (static_cast<double>(top_k) * n_steps));
}

}  // namespace

cudaError_t launch_hit_score(const float* attn, int n_steps, int n_heads, int64_t row_stride, const int32_t* row_len,
                             const int32_t* span, int top_k, int32_t* counts, float* s_hit, Launch ln) {
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(int32_t) * n_heads, ln.stream);
  if (e != cudaSuccess) return e;
  const int64_t n_pairs = static_cast<int64_t>(n_steps) * n_heads;
  const int max_grid = device_sm_count() * kHitBlocksPerSm;
  const int grid = static_cast<int>(n_pairs < max_grid ? n_pairs : max_grid);
  hit_count_kernel<<<grid, kHitThreads, 0, ln.stream>>>(attn, n_steps, n_heads, row_stride, row_len, span, top_k, counts);
  ln.done("hit_count");
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = launch_chained(hit_ratio_kernel, dim3((n_heads + 255) / 256), dim3(256), 0, ln.stream, counts, n_heads, n_steps, top_k, s_hit);
  ln.done("hit_ratio");
  return e;
}

}  // namespace akv

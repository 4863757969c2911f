// Offline head score: for every decode step and head, the top-K tokens of the attention row, how many of them
// fall inside the audio span of the word generated at that step, and the mean of that ratio over the steps.
//
// What bounds it: the rows, read once (64 steps x 784 heads x 8192 tokens are 1.6 GB, 0.25 ms of HBM). So a row belongs to
// one warp, which streams it through registers and keeps the maxima of 32 groups of its values per lane; the k-th largest
// of the lanes' maxima bounds the k-th largest value from below; the few groups that reach the bound are read once more
// (from L2) and their values listed; the listed values inside the span are ranked against the list. No barrier joins
// two warps, so that twenty rows an SM are in different phases and the loads never stop.
// On that workload 295 us, 85 % of the measured copy bandwidth; before: 3.69 ms with a radix select over every row by a block of 1024 threads (five reads of it through
// L2, some twenty barriers); 0.48 ms with this selection by a block of 256 (5.7 us a row and block whether four blocks an SM
// ran on plain loads or three with the next row's copies under way: the chain of a row's phases was the bound).
#include "common.cuh"
#include "select.cuh"

namespace akv {
namespace {

constexpr int kHitWarps = 4;                 // warps per block
constexpr int kHitThreads = 32 * kHitWarps;
constexpr int kHitBlocksPerSm = 5;
constexpr int kHitGroups = 32;               // groups of a lane's 16-byte pieces (two pieces each at 8192 values a row)
constexpr int kHitCand = 512;                // listed values of a row
constexpr int kHitListK = 64;                // top_k up to which the bound is sharp enough for the list

struct HitSmem {
  float val[kHitCand];
  int idx[kHitCand];
  uint16_t entry[kHitGroups * 32];           // groups that reach the bound: group * 32 + lane
};

// The larger value, NaN if either is NaN.
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Exact count for a row the list cannot serve (many equal values, NaN, a large K): the k-th largest key by a search over its
// bits, two bits a pass over the row (L2), then the span's tokens against it; of the keys equal to it the lowest
// indices count. Keys order a NaN by its bits: above every number, or below with the sign bit set. One warp.
__device__ __noinline__ int hits_by_search(const float* __restrict__ row, int L, int k, int lo, int hi) {
  const int lane = threadIdx.x & 31;
  uint32_t key = 0u;  // the largest key x with at least k keys >= x
  for (int shift = 30; shift >= 0; shift -= 2) {
    const uint32_t p1 = key + (1u << shift), p2 = key + (2u << shift), p3 = key + (3u << shift);
    int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll 8
    for (int j = lane; j < L; j += 32) {
      const uint32_t x = score_key(__ldg(row + j));
      c1 += x >= p1;
      c2 += x >= p2;
      c3 += x >= p3;
    }
    c1 = __reduce_add_sync(0xffffffffu, c1);
    c2 = __reduce_add_sync(0xffffffffu, c2);
    c3 = __reduce_add_sync(0xffffffffu, c3);
    key = c3 >= k ? p3 : c2 >= k ? p2 : c1 >= k ? p1 : key;
  }
  int above = 0, eq_before = 0, eq_in = 0, gt_in = 0;
#pragma unroll 4
  for (int j = lane; j < L; j += 32) {
    const uint32_t x = score_key(__ldg(row + j));
    above += x > key;
    if (x == key) {
      eq_before += j < lo;
      eq_in += j >= lo && j <= hi;
    }
    gt_in += x > key && j >= lo && j <= hi;
  }
  above = __reduce_add_sync(0xffffffffu, above);
  eq_before = __reduce_add_sync(0xffffffffu, eq_before);
  eq_in = __reduce_add_sync(0xffffffffu, eq_in);
  gt_in = __reduce_add_sync(0xffffffffu, gt_in);
  return gt_in + min(eq_in, max(0, k - above - eq_before));
}

__global__ void __launch_bounds__(kHitThreads, kHitBlocksPerSm)
hit_count_kernel(const float* __restrict__ attn, int n_steps, int n_heads, int64_t row_stride,
                 const int32_t* __restrict__ row_len, const int32_t* __restrict__ span, int top_k,
                 int32_t* __restrict__ counts) {
  __shared__ HitSmem sm_all[kHitWarps];
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  HitSmem& sm = sm_all[threadIdx.x >> 5];
  const int n_pairs = n_steps * n_heads;
  for (int64_t pair = static_cast<int64_t>(blockIdx.x) * kHitWarps + (threadIdx.x >> 5); pair < n_pairs;
       pair += static_cast<int64_t>(gridDim.x) * kHitWarps) {
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
      // Lower bound of the k-th largest value: the k-th largest of the 32 lanes' maxima (of 64, one for the even and one for
      // the odd groups of a lane, when k > 32). Of 8192 values and k = 24 about 45 lie at or above it.
      float me = -INFINITY, mo = -INFINITY;
#pragma unroll
      for (int g = 0; g < kHitGroups; g += 2) {
        me = max_nan(me, gm[g]);
        mo = max_nan(mo, gm[g + 1]);
      }
      const bool nan = isnan(me) || isnan(mo);
      const bool two = k > 32;
      if (!two) me = fmaxf(me, mo);
      int re = 0, ro = 0;  // ranks, ties to the lower lane, the even half first
      for (int o = 0; o < 32; ++o) {
        const float oe = __shfl_sync(0xffffffffu, me, o), oo = __shfl_sync(0xffffffffu, mo, o);
        re += (oe > me || (oe == me && o < lane)) + (two && oo > me);
        ro += (oe >= mo) + (oo > mo || (oo == mo && o < lane));
      }
      const uint32_t be = __ballot_sync(0xffffffffu, re == k - 1), bo = __ballot_sync(0xffffffffu, two && ro == k - 1);
      float bound = -INFINITY;
      if (be) bound = __shfl_sync(0xffffffffu, me, __ffs(be) - 1);
      else if (bo) bound = __shfl_sync(0xffffffffu, mo, __ffs(bo) - 1);
      int n_ent = 0;
#pragma unroll
      for (int g = 0; g < kHitGroups; ++g) {
        const bool in = gm[g] >= bound;
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
      if (__any_sync(0xffffffffu, nan || isnan(xs))) n = 0;  // a NaN compares with nothing: its row is left to the search
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
    } else {
      c = hits_by_search(row, L, k, lo, hi);
    }
    if (lane == 0 && c) atomicAdd(counts + a, c);
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
  const int64_t n_blocks = (static_cast<int64_t>(n_steps) * n_heads + kHitWarps - 1) / kHitWarps;
  const int max_grid = device_sm_count() * kHitBlocksPerSm;
  const int grid = static_cast<int>(n_blocks < max_grid ? n_blocks : max_grid);
  hit_count_kernel<<<grid, kHitThreads, 0, ln.stream>>>(attn, n_steps, n_heads, row_stride, row_len, span, top_k, counts);
  ln.done("hit_count");
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = launch_chained(hit_ratio_kernel, dim3((n_heads + 255) / 256), dim3(256), 0, ln.stream, counts, n_heads, n_steps, top_k, s_hit);
  ln.done("hit_ratio");
  return e;
}

}  // namespace akv

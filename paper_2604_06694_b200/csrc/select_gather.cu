// Per-head top-k (see select.cuh), ordered compaction of the kept indices, and the
// vectorised gather of the kept K and V rows into the compacted cache.
#include <algorithm>

#include "common.cuh"
#include "select.cuh"

namespace akv {
namespace {

constexpr int kSelThreads = 1024;

// One block per head: the head's keys staged once in shared memory when they fit, then select_entries.
__global__ void __launch_bounds__(kSelThreads, 1)
select_kernel(Shape sh, const ReqDesc* __restrict__ reqs, const float* __restrict__ smoothed,
              const int32_t* __restrict__ budgets, const int32_t* __restrict__ cu_kept,
              int32_t* __restrict__ kept_idx, int smem_keys, int* __restrict__ status) {
  chain_wait();
  extern __shared__ uint32_t skeys[];  // smem_keys keys, then the masks and prefix sums of the longest head
  __shared__ SelectSmem ssm;
  __shared__ uint32_t s_min, s_max;

  for (int u = blockIdx.x; u < sh.total_heads; u += gridDim.x) {
    const int r = u / sh.heads_per_req;
    const ReqDesc rq = reqs[r];
    const int P = rq.P, W = sh.window;
    const float* s = smoothed + rq.score_offset + static_cast<int64_t>(u - rq.head_base) * P;
    int k = budgets[u] - W;
    if (k < 0 || k > P) {
      if (threadIdx.x == 0) atomicExch(status, AUDIOKV_EDEVICE);
      k = k < 0 ? 0 : P;
    }
    const bool staged = P <= smem_keys;
    if (threadIdx.x == 0) {
      s_min = 0xffffffffu;
      s_max = 0u;
    }
    __syncthreads();
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
    for (int j = threadIdx.x; j < P; j += kSelThreads) {
      const uint32_t key = score_key(s[j]);
      if (staged) skeys[j] = key;
      lo = min(lo, key);
      hi = max(hi, key);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&s_min, lo);
      atomicMax(&s_max, hi);
    }
    __syncthreads();
    uint32_t* words = skeys + smem_keys;
    int* pre = reinterpret_cast<int*>(words) + select_words(P, false);
    int32_t* out = kept_idx + cu_kept[u];
    if (staged)
      select_entries<kSelThreads, false>([&](int j) { return make_float2(__uint_as_float(skeys[j]), 0.f); }, P, P, W, k,
                                         s_min, s_max, out, &ssm, words, pre, status);
    else
      select_entries<kSelThreads, false>([&](int j) { return make_float2(__uint_as_float(score_key(s[j])), 0.f); }, P, P,
                                         W, k, s_min, s_max, out, &ssm, words, pre, status);
  }
  chain_release();  // at the end: see the gather
}

// Copies the kept rows. A warp takes eight output rows at a time: lanes 0-7 look up the head of one row each
// (bisection in cu_kept) and its source row; then all lanes copy 16-byte chunks, K chunks first, V chunks after,
// eight independent loads in flight per lane before the stores. log2_chunks: log2 of the chunks per row.
// Rows are read and written once: both sides carry the streaming hint, so that the hundreds of megabytes that pass
// through leave the small, reused state of the pass (tables, scores, statistics, the kernels' code) in L2. Measured
// on the 28-layer L = 8192 pass: the smoothing kernel of the next pass took 35 us instead of 43.
constexpr int kGatherRows = 8;

__global__ void __launch_bounds__(256, 3)  // three blocks per SM: at most 80 registers per thread
gather_kernel(Shape sh, const ReqDesc* __restrict__ reqs, const int32_t* __restrict__ cu_kept,
              const int32_t* __restrict__ kept_idx, const uint4* __restrict__ k, const uint4* __restrict__ v,
              uint4* __restrict__ k_out, uint4* __restrict__ v_out, int log2_chunks, int elems_per_chunk,
              int head_begin, int head_end) {
  // The smoothing kernel lets this one in at its end. (Let in at its start, the blocks here only sat on the SMs that finished their
  // heads first, and a ragged batch ran 7 % slower.)
  chain_wait();
  chain_release();  // the next pass's first scoring sweep may be set up while this kernel drains
  const int64_t first_row = cu_kept[head_begin];  // the rows of heads [head_begin, head_end)
  const int64_t total_rows = cu_kept[head_end];
  const int64_t n_batches = (total_rows - first_row + kGatherRows - 1) / kGatherRows;
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t n_warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  const int chunks = 1 << log2_chunks;
  for (int64_t bt = warp0; bt < n_batches; bt += n_warps) {
    const int64_t row0 = first_row + bt * kGatherRows;
    int64_t my_src = 0;  // lane i < 8: first 16-byte chunk of the source row of output row row0 + i
    if (lane < kGatherRows && row0 + lane < total_rows) {
      const int64_t row = row0 + lane;
      int lo = head_begin, hi = head_end;  // largest u with cu_kept[u] <= row
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(cu_kept + mid) <= row) lo = mid; else hi = mid;
      }
      const int u = lo;
      const ReqDesc rq = reqs[u / sh.heads_per_req];
      const int lh = u - rq.head_base;
      const int l = lh / sh.n_kv_heads, h = lh - l * sh.n_kv_heads;
      const int tok = __ldg(kept_idx + row);
      my_src = (l * sh.kv_stride_layer + h * sh.kv_stride_head + kv_token_offset(sh, rq, u / sh.heads_per_req, tok)) /
               elems_per_chunk;
    }
    const int n_rows = static_cast<int>(min(static_cast<int64_t>(kGatherRows), total_rows - row0));
    int64_t so[kGatherRows];  // every lane gets the eight source rows (all lanes take part in the shuffles)
#pragma unroll
    for (int i = 0; i < kGatherRows; ++i) so[i] = __shfl_sync(0xffffffffu, my_src, i);
    for (int c0 = lane; c0 < 2 * chunks; c0 += 32) {
      const bool is_v = c0 >= chunks;
      const int c = c0 & (chunks - 1);
      const uint4* src = is_v ? v : k;
      uint4* dst = (is_v ? v_out : k_out) + (row0 << log2_chunks) + c;
      uint4 val[kGatherRows];
#pragma unroll
      for (int i = 0; i < kGatherRows; ++i)
        if (i < n_rows) val[i] = __ldcs(src + so[i] + c);
#pragma unroll
      for (int i = 0; i < kGatherRows; ++i)
        if (i < n_rows) __stcs(dst + (static_cast<int64_t>(i) << log2_chunks), val[i]);
    }
  }
}

// The gather beside the smoothing: head by head, in the order in which their selections end. It is let in when the blocks of the
// smoothing kernel have all started, takes the SMs that come free, and follows the list of finished heads (HeadQueue). Where
// some heads need transforms and others do not, the rows of the others move while the transforms run.
// A block is one warp that prepares and eight that copy. The first takes tickets, each a few units of rows (more of them while
// much is left, one at a time at the end, so that the blocks end together), finds the finished heads that they belong to,
// looks up the source rows and deals them out, eight at a time, through a small ring per copying warp: the chain ticket, head,
// indices (three trips to L2) stays out of the way of the rows, which move as in gather_kernel.
// What the smoothing kernel writes while this one runs is read past L1 (indices of two heads can share a line).
constexpr int kCopyWarps = 8;
constexpr int kStreamThreads = (kCopyWarps + 1) * 32;
constexpr int kRing = 2 * kCopyWarps;  // batches of rows prepared ahead
constexpr int kUnitChunks = 512;       // rows of a unit times 16-byte chunks of a row of K
constexpr int kTicketUnits = 4;        // units of a ticket at most
constexpr long long kHeadWaitCycles = 8000000000LL;  // about four seconds without another head finished

struct RowBatch {
  int64_t src;  // 16-byte chunk of the head's row 0 in K and V
  int64_t dst;  // first output row
  int n;        // rows; 0: no more work
  int row[kGatherRows];
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ bool phase_done(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded, like every wait here: false (and a status) after twice the limit of a wait for a head.
__device__ __forceinline__ bool phase_wait(uint32_t bar, uint32_t parity, int* status) {
  if (phase_done(bar, parity)) return true;
  const long long t0 = clock64();
  while (!phase_done(bar, parity))
    if (clock64() - t0 > 2 * kHeadWaitCycles) {
      atomicExch(status, AUDIOKV_ETIMEOUT);
      return false;
    }
  return true;
}
__device__ __forceinline__ void phase_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The head that a unit of rows belongs to: the last one listed at or before it. The warp looks at 32 places of the list at a
// time, from the place of the head it had before.
struct HeadAt {
  int place = 0, u = -1, kept = 0;
  int64_t row = 0;              // first output row
  unsigned begin = 0, end = 0;  // units [begin, end)
};
enum class Found { kHead, kGap, kNoMore, kTimeout };  // a gap: a unit of no head (budgets and prefix sums that disagree)
__device__ Found find_head(HeadAt& h, unsigned unit, const HeadQueue& hq, int n_heads, const int32_t* cu_kept, int lane, int* status) {
  const long long t0 = clock64();
  for (;;) {
    unsigned long long e = 0;
    if (h.place + lane < n_heads)
      asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(e) : "l"(hq.done + h.place + lane) : "memory");
    __syncwarp();  // orders every lane's reads behind the acquires
    const unsigned before = __ballot_sync(0xffffffffu, e != 0 && static_cast<unsigned>(e) <= unit);
    const unsigned listed = __ballot_sync(0xffffffffu, e != 0);
    if (before) {
      const int i = 31 - __clz(before);
      const unsigned long long ei = __shfl_sync(0xffffffffu, e, i);
      h.place += i;
      if (i == 31) continue;  // the next ones may be at or before it as well
      h.u = static_cast<int>(ei >> 32) - 1;
      h.row = __ldcg(cu_kept + h.u);
      h.kept = __ldcg(cu_kept + h.u + 1) - static_cast<int>(h.row);
      h.begin = static_cast<unsigned>(ei);
      h.end = h.begin + (h.kept + hq.unit_rows - 1) / hq.unit_rows;
      if (unit < h.end) return Found::kHead;
      if (h.place == n_heads - 1) return Found::kNoMore;
      if ((listed >> (i + 1)) & 1u) return Found::kGap;
    }
    if (clock64() - t0 > kHeadWaitCycles) {
      if (lane == 0) atomicExch(status, AUDIOKV_ETIMEOUT);
      return Found::kTimeout;
    }
    __nanosleep(200);
  }
}

__global__ void __launch_bounds__(kStreamThreads, 3)  // three blocks per SM: at most 72 registers per thread
gather_stream_kernel(Shape sh, const ReqDesc* __restrict__ reqs, const int32_t* cu_kept, const int32_t* kept_idx,
                     const uint4* __restrict__ k, const uint4* __restrict__ v, uint4* __restrict__ k_out,
                     uint4* __restrict__ v_out, int log2_chunks, int elems_per_chunk, int n_heads, int about_units, HeadQueue hq,
                     int* status) {
  __shared__ RowBatch ring[kRing];
  __shared__ alignas(8) uint64_t full[kRing], empty[kRing];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < kRing) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full[threadIdx.x])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&empty[threadIdx.x])) : "memory");
  }
  __syncthreads();
  if (warp == kCopyWarps) {
    int at = 0;  // next place of the ring, in batches since the start modulo 2 kRing
    bool ok = true;
    HeadAt h;
    int64_t src = 0;
    int ticket = 0, n_next = 1, r = 0;
    if (lane == 0) ticket = atomicAdd(hq.ticket(), n_next);
    while (ok) {
      const int t = __shfl_sync(0xffffffffu, ticket, 0), n = n_next;
      n_next = min(kTicketUnits, max(1, (about_units - t) / (2 * static_cast<int>(gridDim.x))));
      if (lane == 0) ticket = atomicAdd(hq.ticket(), n_next);  // comes back under this ticket's rows
      for (int unit = t; unit < t + n && ok; ++unit) {
        if (h.u < 0 || static_cast<unsigned>(unit) >= h.end) {
          const Found found = find_head(h, unit, hq, n_heads, cu_kept, lane, status);
          if (found == Found::kGap) continue;
          ok = found == Found::kHead;
          if (!ok) break;
          r = h.u / sh.heads_per_req;
          const int lh = h.u - reqs[r].head_base, l = lh / sh.n_kv_heads, kh = lh - l * sh.n_kv_heads;
          src = (l * sh.kv_stride_layer + kh * sh.kv_stride_head + (sh.page_size ? 0 : reqs[r].kv_offset)) / elems_per_chunk;
        }
        const int first = (unit - static_cast<int>(h.begin)) * hq.unit_rows, end = min(h.kept, first + hq.unit_rows);
        for (int row0 = first; row0 < end && ok; row0 += 32) {
          const int row = row0 + lane < end ? kv_token_row(sh, r, __ldcg(kept_idx + h.row + row0 + lane)) : 0;
          const int n_batches = (min(32, end - row0) + kGatherRows - 1) / kGatherRows;
          int place = at + lane;  // lanes 0 .. n_batches - 1: the places of the batches
          place -= place >= 2 * kRing ? 2 * kRing : 0;
          const int ring_at = place < kRing ? place : place - kRing;
          bool mine = true;
          if (lane < n_batches) {
            mine = phase_wait(smem_addr(&empty[ring_at]), place < kRing ? 1 : 0, status);
            ring[ring_at].src = src;
            ring[ring_at].dst = h.row + row0 + lane * kGatherRows;
            ring[ring_at].n = min(kGatherRows, end - row0 - lane * kGatherRows);
          }
          ok = __all_sync(0xffffffffu, mine);
          const int to = __shfl_sync(0xffffffffu, ring_at, lane / kGatherRows);
          if (lane / kGatherRows < n_batches) ring[to].row[lane % kGatherRows] = row;
          __syncwarp();
          if (lane < n_batches) phase_arrive(smem_addr(&full[ring_at]));
          at += n_batches;
          at -= at >= 2 * kRing ? 2 * kRing : 0;
        }
      }
    }
    // The last block to find no more rows leaves the queue as the next pass wants it.
    int last = 0;
    if (lane == 0) last = atomicAdd(hq.blocks(), 1) == static_cast<int>(gridDim.x) - 1;
    if (__shfl_sync(0xffffffffu, last, 0)) {
      for (int i = lane; i < n_heads; i += 32) hq.done[i] = 0;
      if (lane == 0) {
        *hq.listed = 0;
        *hq.ticket() = *hq.blocks() = 0;
      }
    }
    // the end, to every copying warp
    int place = at + lane;
    place -= place >= 2 * kRing ? 2 * kRing : 0;
    const int ring_at = place < kRing ? place : place - kRing;
    if (lane < kCopyWarps && phase_wait(smem_addr(&empty[ring_at]), place < kRing ? 1 : 0, status)) {
      ring[ring_at].n = 0;
      phase_arrive(smem_addr(&full[ring_at]));
    }
  } else {
    const int chunks = 1 << log2_chunks;
    const int64_t row_stride = sh.kv_stride_tok / elems_per_chunk;  // in 16-byte chunks
    uint32_t parity = 0;
    for (int at = warp;;) {
      if (!phase_wait(smem_addr(&full[at]), parity, status)) break;
      const RowBatch& rb = ring[at];
      const int n = rb.n;
      if (n == 0) break;
      for (int c0 = lane; c0 < 2 * chunks; c0 += 32) {
        const bool is_v = c0 >= chunks;
        const int c = c0 & (chunks - 1);
        const uint4* src = (is_v ? v : k) + rb.src + c;
        uint4* dst = (is_v ? v_out : k_out) + (rb.dst << log2_chunks) + c;
        uint4 val[kGatherRows];
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i)
          if (i < n) val[i] = __ldcs(src + rb.row[i] * row_stride);
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i)
          if (i < n) __stcs(dst + (static_cast<int64_t>(i) << log2_chunks), val[i]);
      }
      __syncwarp();
      if (lane == 0) phase_arrive(smem_addr(&empty[at]));
      at += kCopyWarps;
      if (at >= kRing) {
        at -= kRing;
        parity ^= 1;
      }
    }
  }
  chain_wait();  // every head is through, so the kernel before is as good as over
  chain_release();
}

}  // namespace

cudaError_t launch_select(const Shape& sh, const ReqDesc* d_reqs, const float* smoothed, const int32_t* budgets,
                          const int32_t* cu_kept, int32_t* kept_idx, int max_P, int* status, Launch ln) {
  const int smem_keys = max_P <= 40 * 1024 ? max_P : 40 * 1024;
  const size_t smem = (static_cast<size_t>(smem_keys) + 2 * select_words(max_P, false)) * sizeof(uint32_t);
  cudaError_t e = cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int max_grid = device_sm_count() * 4;
  const int grid = sh.total_heads < max_grid ? sh.total_heads : max_grid;
  e = launch_chained(select_kernel, dim3(grid), dim3(kSelThreads), smem, ln.stream, sh, d_reqs, smoothed, budgets, cu_kept, kept_idx,
                     smem_keys, status);
  ln.done("select");
  return e;
}

cudaError_t launch_gather(const Shape& sh, const ReqDesc* d_reqs, const int32_t* cu_kept, const int32_t* kept_idx,
                          const void* k, const void* v, void* k_out, void* v_out, int head_begin, int head_end,
                          Launch ln) {
  const int esize = sh.dtype == AUDIOKV_F32 ? 4 : 2;
  const int elems_per_chunk = 16 / esize;
  const int chunks_per_row = sh.head_dim / elems_per_chunk;  // 8 .. 64: head_dim is 64, 128 or 256
  int log2_chunks = 0;
  while ((1 << log2_chunks) < chunks_per_row) ++log2_chunks;
  cudaError_t e = launch_chained(gather_kernel, dim3(device_sm_count() * 8), dim3(256), 0, ln.stream, sh, d_reqs, cu_kept, kept_idx,
                                 (const uint4*)k, (const uint4*)v, (uint4*)k_out, (uint4*)v_out, log2_chunks, elems_per_chunk,
                                 head_begin, head_end);
  ln.done("gather");
  return e;
}

int gather_unit_rows(const Shape& sh) { return kUnitChunks * (16 / (sh.dtype == AUDIOKV_F32 ? 4 : 2)) / sh.head_dim; }

cudaError_t launch_gather_stream(const Shape& sh, const ReqDesc* d_reqs, const int32_t* cu_kept, const int32_t* kept_idx,
                                 const void* k, const void* v, void* k_out, void* v_out, int n_heads, int64_t kept_rows,
                                 HeadQueue hq, int* status, Launch ln) {
  const int elems_per_chunk = 16 / (sh.dtype == AUDIOKV_F32 ? 4 : 2);
  const int chunks_per_row = sh.head_dim / elems_per_chunk;
  int log2_chunks = 0;
  while ((1 << log2_chunks) < chunks_per_row) ++log2_chunks;
  const int about_units = static_cast<int>(std::min<int64_t>(kept_rows / hq.unit_rows + n_heads / 2, 1 << 30));
  // An SM that a smoothing block has just left is set up for that block's shared memory, and what is left as L1 bounds the
  // loads in flight: without this, 48 layers of L 16384 took 846 us a pass, with it 796.
  cudaError_t e = cudaFuncSetAttribute(gather_stream_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxL1);
  if (e != cudaSuccess) return e;
  e = launch_chained(gather_stream_kernel, dim3(device_sm_count() * 3), dim3(kStreamThreads), 0, ln.stream, sh, d_reqs,
                     cu_kept, kept_idx, (const uint4*)k, (const uint4*)v, (uint4*)k_out, (uint4*)v_out, log2_chunks,
                     elems_per_chunk, n_heads, about_units, hq, status);
  ln.done("gather");
  return e;
}

}  // namespace akv

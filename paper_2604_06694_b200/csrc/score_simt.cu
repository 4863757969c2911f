// Importance scores on the fp32 FMA pipe, for any element type.
//
// This is the path for fp32 inputs (which must not be rounded to TF32) and the fallback for shapes the tensor-core kernels
// do not take. A column sum mixes rows with different normalisers, which are known only when every key has been seen.
//
// What bounds it: the FMAs of Q K^T, 26.3 GFLOP for 28 layers of the 7B shape at 4096 keys, 0.35 ms of the fp32 pipe if
// they are done once. So where there is room they are done once: the product kernel writes exp2(z - m) of its tile, m the
// row's maximum over the tile's keys, and (m, sum) per row; a merge gives every row c = -(max + log2 sum) over all keys;
// the sum kernel adds exp2(m + c) exp2(z - m) over the rows of every key, a stream at memory speed. Heads go through in
// chunks of up to 256 MB of exponentials, or what room the caller has. A head too long for it, and the entry point with
// fixed scratch, run the product twice: statistics, merge, column sums.
// The product is a register-tiled matrix product, 8 keys x 4, 7 or 8 query rows a thread. The tile's keys lie transposed in shared
// memory for as long as the tile lasts, two neighbouring keys make a packed pair of accumulators, and the query rows
// come in panels of 32 dimensions by asynchronous copies, the next one under the arithmetic of this one, across row tiles.
// 128 registers, 16 warps an SM: 180 to 191 us for 28 heads at 4096 keys (the FMA pipe 61 % busy by its counter, its throttle the
// first stall). What was tried on the way on that launch: scalar FMAs in this layout 217 us, in rows of either side 240 us, held up by
// dispatch stalls of three-operand reads; pairs of even and odd dimensions 218 us, and 201 us with half the address
// arithmetic: twice the accumulators leave two warps a scheduler, which do not cover their latencies.
// Logits are kept in base 2 (scale * log2 e folded into one multiply).
#include <algorithm>

#include "common.cuh"

namespace akv {
namespace {

constexpr int kThreads = 256;  // of the merge and the sum kernel
constexpr int kPanel = 32;     // dimensions per stage of query rows
constexpr int kStages = 2;
// Keys per tile: 64 KB of shared memory (32 KB at head_dim 64) with two blocks an SM.
__host__ __device__ constexpr int tile_keys(int head_dim) { return head_dim == 256 ? 64 : 128; }

struct HeadCoord {
  int r, l, h;
};
__device__ __forceinline__ HeadCoord head_coord(const Shape& sh, int u) {
  HeadCoord c;
  c.r = u / sh.heads_per_req;
  int lh = u - c.r * sh.heads_per_req;
  c.l = lh / sh.n_kv_heads;
  c.h = lh - c.l * sh.n_kv_heads;
  return c;
}

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair_of(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// Four elements as fp32, from shared or global memory.
__device__ __forceinline__ float4 four(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 four(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                     __uint_as_float(raw.y & 0xffff0000u));
}
// 16 bytes to shared memory without passing through registers.
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// 2^x; arguments are at most 0, and what lies below 2^-126 of a row's maximum counts as nothing
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

enum { kStore = 0, kStats = 1, kColsum = 2 };

// A panel row in shared memory: 32 elements and 16 bytes of padding, which puts neighbouring rows' 16-byte pieces on
// different banks.
constexpr int panel_row_bytes(int esize) { return kPanel * esize + 16; }
constexpr int tile_smem_bytes(int d, int rpt, int esize, int rows) {
  return tile_keys(d) * d * 4 + kStages * 16 * rpt * panel_row_bytes(esize) + (rows + 16 * rpt) * static_cast<int>(sizeof(void*));
}

// MODE kStore: one tile of keys per slab; its exponentials and row statistics. kStats: row statistics of a slab. kColsum: column
// sums of a slab's prefix keys, the rows' c given (see merge_kernel). Heads u0, u0 + 1, ...; statistics of head u at u - u0.
template <typename T, int D, int RPT, int MODE>
__global__ void __launch_bounds__(2 * tile_keys(D), 2)
score_tile_kernel(Shape sh, const ReqDesc* __restrict__ reqs, const T* __restrict__ q, const T* __restrict__ k,
                  float* __restrict__ scores, float2* __restrict__ stats, float* __restrict__ exps, int n_slab, int slab_keys,
                  int u0, int beside) {
  constexpr int kKeys = tile_keys(D), kThr = 2 * kKeys, kTx = kKeys / 8, kRows = 16 * RPT;
  constexpr int kRowBytes = panel_row_bytes(static_cast<int>(sizeof(T))), kStage = kRows * kRowBytes;
  constexpr int kPieces = kPanel * static_cast<int>(sizeof(T)) / 16;  // 16-byte pieces of a panel row
  constexpr int kPanels = D / kPanel;
  extern __shared__ __align__(16) unsigned char smem[];
  float* kt_s = reinterpret_cast<float*>(smem);               // [D][kKeys]: the tile's keys, transposed
  unsigned char* q_s = smem + kKeys * D * 4;                  // kStages panels of query rows
  const T** rows = reinterpret_cast<const T**>(q_s + kStages * kStage);  // the head's query rows, whole row tiles

  // The budget kernel launched just before (see launch_score_umma's `beside`) lets this one in when everything earlier on the
  // stream is complete, and computes nothing that is read here: the two run side by side, and every block waits for it at its
  // end, which the kernels behind then need not do (6 us of a pass over 2 heads of 1024 keys, 59 in all).
  chain_release();
  if (!beside) chain_wait();  // the request table may be the work of the kernel before
  const int uc = blockIdx.x / n_slab, slab = blockIdx.x - uc * n_slab, u = u0 + uc;
  const HeadCoord hc = head_coord(sh, u);
  const ReqDesc rq = reqs[hc.r];
  const int R = sh.window * sh.group, G = sh.group;
  const int ty = threadIdx.x / kTx, tx = threadIdx.x % kTx;  // rows ty + 16 a; keys 4 tx .. + 3 of either half of the tile
  const int j0 = slab * slab_keys;
  const int j1 = min(MODE == kColsum ? rq.P : rq.L, j0 + slab_keys);  // column sums: prefix keys only
  float2* my_stats = stats + (static_cast<int64_t>(uc) * n_slab + slab) * R;
  const T* kbase = k + hc.l * sh.kv_stride_layer + hc.h * sh.kv_stride_head;  // the token term: kv_token_offset
  const T* qbase = q + rq.q_offset + hc.l * sh.q_stride_layer + static_cast<int64_t>(hc.h) * G * sh.q_stride_head;
  if (j0 >= j1) {  // no keys of this request here
    if (MODE != kColsum)
      for (int r = threadIdx.x; r < R; r += kThr) my_stats[r] = make_float2(-INFINITY, 0.f);
    if (beside) chain_wait();
    return;
  }
  const int n_rt = (R + kRows - 1) / kRows;  // row tiles; rows past the end repeat the last one, their logits are dropped
  for (int i = threadIdx.x; i < n_rt * kRows; i += kThr) {
    const int rr = min(i, R - 1), w = rr / G;
    rows[i] = qbase + w * sh.q_stride_tok + (rr - w * G) * sh.q_stride_head;
  }

  const uint32_t q_smem = static_cast<uint32_t>(__cvta_generic_to_shared(q_s));
  // Panel g of the query rows (row tile g / kPanels, dimensions 32 (g % kPanels) ..) into stage g % 2.
  auto load_q = [&](int g) {
    const int rt = g / kPanels, p = g - rt * kPanels;
    const int my_row = threadIdx.x / kPieces, from = p * (kPanel * static_cast<int>(sizeof(T))) + threadIdx.x % kPieces * 16;
    const uint32_t to = q_smem + (g & 1) * kStage + my_row * kRowBytes + threadIdx.x % kPieces * 16;
    constexpr int kStep = kThr / kPieces;  // rows per turn
#pragma unroll
    for (int i = 0; i < (kRows + kStep - 1) / kStep; ++i)
      if (kRows % kStep == 0 || my_row + i * kStep < kRows)
        copy16(to + i * kStep * kRowBytes, reinterpret_cast<const unsigned char*>(rows[rt * kRows + my_row + i * kStep]) + from);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // Keys kt .. of the tile into shared memory, transposed: a lane holds a key, so that the stores run along the banks.
  // Keys past the end repeat the last one: their logits are masked or dropped.
  auto load_k = [&](int kt) {
    const int key = threadIdx.x % kKeys, c0 = threadIdx.x / kKeys;  // pieces of four dimensions: c0, c0 + 2, ...
    const T* src = kbase + kv_token_offset(sh, rq, hc.r, min(kt + key, j1 - 1));
#pragma unroll 1
    for (int c = c0; c < D / 4; c += 16) {
      float4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = four(src + 4 * (c + 2 * i));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float* dst = kt_s + 4 * (c + 2 * i) * kKeys + key;
        dst[0] = v[i].x;
        dst[kKeys] = v[i].y;
        dst[2 * kKeys] = v[i].z;
        dst[3 * kKeys] = v[i].w;
      }
    }
  };
  // acc[a][b] = <Q row ty + 16 a of row tile rt, key b of this thread>; the first panel of the row tile is on its way, and the
  // first of row tile `next` (if not negative) is when this returns.
  f32x2 sum[RPT][4];
  float acc[8];
  auto product = [&](int rt, int next) {
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) sum[a][b] = 0ull;
#pragma unroll 1
    for (int p = 0; p < kPanels; ++p) {
      const int g = rt * kPanels + p;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();  // panel g (and the keys) are in place; everybody is done with panel g - 1
      if (p + 1 < kPanels) load_q(g + 1);
      else if (next >= 0) load_q(next * kPanels);  // the stages alternate: kPanels is even
      const unsigned char* qr = q_s + (g & 1) * kStage + ty * kRowBytes;
      const float* kr = kt_s + p * kPanel * kKeys + 4 * tx;
#pragma unroll 1
      for (int t = 0; t < kPanel; t += 4) {
        float4 qv[RPT];
#pragma unroll
        for (int a = 0; a < RPT; ++a) qv[a] = four(reinterpret_cast<const T*>(qr + 16 * a * kRowBytes) + t);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const ulonglong2 k0 = *reinterpret_cast<const ulonglong2*>(kr + (t + i) * kKeys);
          const ulonglong2 k1 = *reinterpret_cast<const ulonglong2*>(kr + (t + i) * kKeys + kKeys / 2);
#pragma unroll
          for (int a = 0; a < RPT; ++a) {
            const float s = i == 0 ? qv[a].x : i == 1 ? qv[a].y : i == 2 ? qv[a].z : qv[a].w;
            const f32x2 s2 = pair_of(s, s);
            sum[a][0] = fma2(s2, k0.x, sum[a][0]);
            sum[a][1] = fma2(s2, k0.y, sum[a][1]);
            sum[a][2] = fma2(s2, k1.x, sum[a][2]);
            sum[a][3] = fma2(s2, k1.y, sum[a][3]);
          }
        }
      }
    }
  };
  auto row_logits = [&](int a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) unpack(sum[a][b], acc[2 * b], acc[2 * b + 1]);
  };
  auto key_of = [&](int b) { return (b >> 2) * (kKeys / 2) + 4 * tx + (b & 3); };
  __syncthreads();  // the row pointers are in place
  load_q(0);
  if constexpr (MODE == kColsum) {
    const float2* hs = stats + static_cast<int64_t>(uc) * n_slab * R;  // c of row r: .y of the head's first slab
    for (int kt = j0; kt < j1; kt += kKeys) {
      load_k(kt);
      float col[8];
#pragma unroll
      for (int b = 0; b < 8; ++b) col[b] = 0.f;
      for (int rt = 0; rt < n_rt; ++rt) {
        product(rt, rt + 1 < n_rt ? rt + 1 : kt + kKeys < j1 ? 0 : -1);
#pragma unroll
        for (int a = 0; a < RPT; ++a) {
          const int rr = rt * kRows + ty + 16 * a;
          const float c = rr < R ? hs[rr].y : -INFINITY;
          row_logits(a);
#pragma unroll
          for (int b = 0; b < 8; ++b) col[b] += ex2(fmaf(acc[b], sh.scale_log2e, c));
        }
      }
      __syncthreads();  // the keys make room for the sums of the 16 thread rows
      float* red = kt_s;
#pragma unroll
      for (int b = 0; b < 8; ++b) red[ty * kKeys + key_of(b)] = col[b];
      __syncthreads();
      if (threadIdx.x < kKeys && kt + static_cast<int>(threadIdx.x) < j1) {
        float s = 0.f;
#pragma unroll
        for (int y = 0; y < 16; ++y) s += red[y * kKeys + threadIdx.x];
        scores[rq.score_offset + (static_cast<int64_t>(hc.l) * sh.n_kv_heads + hc.h) * rq.P + kt + threadIdx.x] = s;
      }
      __syncthreads();  // and the sums for the next keys
    }
  } else {
    if (MODE == kStore) load_k(j0);
    for (int rt = 0; rt < n_rt; ++rt) {
      float m[RPT], Z[RPT];
#pragma unroll
      for (int a = 0; a < RPT; ++a) {
        m[a] = -INFINITY;
        Z[a] = 0.f;
      }
      for (int kt = j0; kt < j1; kt += kKeys) {
        if (MODE == kStats) {
          __syncthreads();  // everybody is done with the keys before
          load_k(kt);
        }
        product(rt, kt + kKeys < j1 ? rt : rt + 1 < n_rt ? rt + 1 : -1);
        const bool masked = kt + kKeys > min(j1, rq.P + 1);  // the tile reaches past the keys or into the window: causal mask
#pragma unroll
        for (int a = 0; a < RPT; ++a) {
          const int rr = rt * kRows + ty + 16 * a;
          row_logits(a);
          if (masked) {
            const int last = min(j1 - 1, rq.P + rr / G) - kt;  // last visible key of this row
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[b] = key_of(b) <= last ? acc[b] : -INFINITY;
          }
          float top = acc[0];
#pragma unroll
          for (int b = 1; b < 8; ++b) top = fmaxf(top, acc[b]);
          if (MODE == kStore) {  // one reference for the row's keys of the tile
#pragma unroll
            for (int o = 1; o < kTx; o <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
          }
          const float ref = fmaxf(m[a], top * sh.scale_log2e);
          const float safe = ref == -INFINITY ? 0.f : ref;  // nothing visible yet: the exponentials are zeros
          float s = 0.f;
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            acc[b] = ex2(fmaf(acc[b], sh.scale_log2e, -safe));
            s += acc[b];
          }
          Z[a] = MODE == kStore ? s : Z[a] * ex2(m[a] - safe) + s;  // kStore: one tile
          m[a] = ref;
          if (MODE == kStore && rr < R) {
            float* e = exps + ((static_cast<int64_t>(uc) * n_slab + slab) * R + rr) * kKeys + 4 * tx;
            *reinterpret_cast<float4*>(e) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            *reinterpret_cast<float4*>(e + kKeys / 2) = make_float4(acc[4], acc[5], acc[6], acc[7]);
          }
        }
      }
#pragma unroll
      for (int a = 0; a < RPT; ++a) {
#pragma unroll
        for (int o = 1; o < kTx; o <<= 1) {
          const float zo = __shfl_xor_sync(0xffffffffu, Z[a], o);
          if (MODE == kStore) {
            Z[a] += zo;
          } else {
            const float mo = __shfl_xor_sync(0xffffffffu, m[a], o);
            const float mn = fmaxf(m[a], mo), safe = mn == -INFINITY ? 0.f : mn;
            Z[a] = Z[a] * ex2(m[a] - safe) + zo * ex2(mo - safe);
            m[a] = mn;
          }
        }
        const int rr = rt * kRows + ty + 16 * a;
        if (tx == 0 && rr < R) my_stats[rr] = make_float2(m[a], Z[a]);
      }
    }
  }
  if (beside) chain_wait();
}

// c = -(max + log2 sum) of every row over its head's slabs, into .y of the row's entry of the first slab (whose sum is no
// longer needed; its maximum stays). One block per 32 rows of a head: eight warps share the slabs.
__global__ void __launch_bounds__(kThreads) merge_kernel(float2* __restrict__ stats, int n_slab, int R) {
  __shared__ float2 part[8][32];
  chain_release();
  chain_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = blockIdx.y * 32 + lane;
  float2* hs = stats + static_cast<int64_t>(blockIdx.x) * n_slab * R;
  float M = -INFINITY, Z = 0.f;
  auto add = [&](float2 st) {
    if (!(st.y > 0.f)) return;
    const float mn = fmaxf(M, st.x);
    Z = Z * exp2f(M - mn) + st.y * exp2f(st.x - mn);
    M = mn;
  };
  if (r < R) {
#pragma unroll 4
    for (int s = warp; s < n_slab; s += 8) add(hs[static_cast<int64_t>(s) * R + r]);
  }
  part[warp][lane] = make_float2(M, Z);
  __syncthreads();
  if (warp == 0 && r < R) {
    for (int w = 1; w < 8; ++w) add(part[w][lane]);
    hs[r].y = -(M + log2f(Z));
  }
}

// Column sums from the stored exponentials: one block per tile; KEYS / 4 lanes read one row at a time.
template <int KEYS>
__global__ void __launch_bounds__(kThreads)
colsum_kernel(Shape sh, const ReqDesc* __restrict__ reqs, float* __restrict__ scores, const float2* __restrict__ stats,
              const float* __restrict__ exps, int n_slab, int u0) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* f = reinterpret_cast<float*>(smem);                   // [R] factor of every row
  constexpr int kLanes = KEYS / 4, kTurn = kThreads / kLanes;  // rows at a time
  __shared__ float4 red[kTurn][kLanes];
  chain_release();
  chain_wait();
  const int uc = blockIdx.x / n_slab, slab = blockIdx.x - uc * n_slab, u = u0 + uc;
  const HeadCoord hc = head_coord(sh, u);
  const ReqDesc rq = reqs[hc.r];
  const int R = sh.window * sh.group, j0 = slab * KEYS;
  const int lane = threadIdx.x % kLanes, first = threadIdx.x / kLanes;
  if (j0 >= rq.P) return;
  const float2* hs = stats + static_cast<int64_t>(uc) * n_slab * R;
  const float4* e = reinterpret_cast<const float4*>(exps + (static_cast<int64_t>(uc) * n_slab + slab) * R * KEYS) + lane;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 v[8];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldcs(e + static_cast<int64_t>(min(r0 + i * kTurn, R - 1)) * kLanes);
  };
  fetch(first);  // the first rows run beside the factors' loads
  for (int r = threadIdx.x; r < R; r += kThreads) f[r] = exp2f(hs[static_cast<int64_t>(slab) * R + r].x + hs[r].y);
  __syncthreads();
  for (int r0 = first; r0 < R;) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float w = r0 + i * kTurn < R ? f[r0 + i * kTurn] : 0.f;
      s.x = fmaf(v[i].x, w, s.x);
      s.y = fmaf(v[i].y, w, s.y);
      s.z = fmaf(v[i].z, w, s.z);
      s.w = fmaf(v[i].w, w, s.w);
    }
    r0 += 8 * kTurn;
    if (r0 < R) fetch(r0);
  }
  red[first][lane] = s;
  __syncthreads();
  if (threadIdx.x < KEYS && j0 + static_cast<int>(threadIdx.x) < rq.P) {
    const float* col = reinterpret_cast<const float*>(red) + threadIdx.x;
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kTurn; ++w) t += col[w * KEYS];
    scores[rq.score_offset + (static_cast<int64_t>(hc.l) * sh.n_kv_heads + hc.h) * rq.P + j0 + threadIdx.x] = t;
  }
}

template <typename T, int D, int RPT, int MODE>
cudaError_t launch_tile(const Shape& sh, const ReqDesc* d_reqs, const void* q, const void* k, float* scores, float2* stats,
                        float* exps, int n_slab, int slab_keys, int u0, int heads, Launch ln, bool beside) {
  auto kern = score_tile_kernel<T, D, RPT, MODE>;
  const int smem = tile_smem_bytes(D, RPT, static_cast<int>(sizeof(T)), sh.window * sh.group);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = launch_chained(kern, dim3(static_cast<unsigned>(n_slab) * heads), dim3(2 * tile_keys(D)), smem, ln.stream, sh, d_reqs,
                     static_cast<const T*>(q), static_cast<const T*>(k), scores, stats, exps, n_slab, slab_keys, u0, beside ? 1 : 0);
  ln.done(MODE == kStore ? "score_simt_exps" : MODE == kStats ? "score_simt_stats" : "score_simt_colsum");
  return e;
}

// Heads of a chunk, at most `most`: as few waves of blocks over all chunks as possible, two blocks an SM, a chunk's three
// launches counted as a third of a wave. (112 heads of 32 tiles in room for 36: 28 heads a chunk are 3.03 waves, so four chunks
// of four, 0.77 ms; 36 heads are 3.9, three chunks of four and one of one.)
int heads_per_chunk(int most, int total, int tiles) {
  const int64_t slots = 2LL * device_sm_count();
  int best = most;
  double cost = 1e30;
  for (int h = most; h >= 1 && (h > most / 2 || h > most - 64); --h) {
    const int full = total / h, rest = total - full * h;
    const double c = full * (static_cast<double>((static_cast<int64_t>(h) * tiles + slots - 1) / slots) + 0.33) +
                     (rest ? static_cast<double>((static_cast<int64_t>(rest) * tiles + slots - 1) / slots) + 0.33 : 0.0);
    if (c < cost) {
      cost = c;
      best = h;
    }
  }
  return best;
}

// Exponentials of one head, in floats, and their row statistics, in float2.
int64_t head_exps(int max_L, int rows, int head_dim) {
  const int keys = tile_keys(head_dim);
  return static_cast<int64_t>((max_L + keys - 1) / keys) * keys * rows;
}
// Of a chunk. Every chunk ends in a wave of blocks that is not full, a merge and a stream, so fewer are better, even though the
// exponentials no longer stay in L2: 112 heads of 4096 keys, 224 rows (411 MB): 878 us a pass at 96 MB, 853 at 128 (four chunks), 805
// at 256 (two), 788 in one, which would make a context 1.5 ms longer to create.
constexpr int64_t kMaxExps = (256LL << 20) / sizeof(float);
constexpr int64_t kMaxHeadExps = (128LL << 20) / sizeof(float);  // a head with more has its product done twice

// room: where the exponentials of a chunk of heads and then their statistics may go.
template <typename T, int D, int RPT>
cudaError_t launch_typed(const Shape& sh, const ReqDesc* d_reqs, const void* q, const void* k, float* scores, float2* stats,
                         int n_slab, int slab_keys, void* room, size_t room_bytes, int max_L, Launch ln, bool beside) {
  constexpr int kKeys = tile_keys(D);
  const int R = sh.window * sh.group, n_tile = (max_L + kKeys - 1) / kKeys;
  const int64_t per_head = head_exps(max_L, R, D);
  const int64_t fit = per_head > kMaxHeadExps ? 0 : std::min<int64_t>(room_bytes / (per_head / kKeys * (kKeys * sizeof(float) + sizeof(float2))), kMaxExps / per_head);
  const bool store = fit >= 1;
  const int slabs = store ? n_tile : n_slab;
  const int most = static_cast<int>(std::min<int64_t>(store ? fit : 0x7fffffffLL / slabs, sh.total_heads));
  const int chunk = store ? heads_per_chunk(most, sh.total_heads, slabs) : most;
  float* exps = static_cast<float*>(room);
  if (store) stats = reinterpret_cast<float2*>(exps + chunk * per_head);
  cudaError_t e = cudaSuccess;
  for (int u0 = 0; u0 < sh.total_heads && e == cudaSuccess; u0 += chunk) {
    const int heads = sh.total_heads - u0 < chunk ? sh.total_heads - u0 : chunk;
    if (store) e = launch_tile<T, D, RPT, kStore>(sh, d_reqs, q, k, scores, stats, exps, slabs, kKeys, u0, heads, ln, beside && u0 == 0);
    else e = launch_tile<T, D, RPT, kStats>(sh, d_reqs, q, k, scores, stats, exps, slabs, slab_keys, u0, heads, ln, beside && u0 == 0);
    if (e != cudaSuccess) return e;
    e = launch_chained(merge_kernel, dim3(heads, (R + 31) / 32), dim3(kThreads), 0, ln.stream, stats, slabs, R);
    ln.done("score_simt_merge");
    if (e != cudaSuccess) return e;
    if (store) {
      // The blocks follow the product's on the SM and would keep its shared memory: 40 % of it holds eight of them, the rest is L1 for
      // their loads in flight (23 us for 36 heads of 4096 keys with what the product leaves, 18 so).
      e = cudaFuncSetAttribute(colsum_kernel<kKeys>, cudaFuncAttributePreferredSharedMemoryCarveout, 40);
      if (e != cudaSuccess) return e;
      e = launch_chained(colsum_kernel<kKeys>, dim3(static_cast<unsigned>(slabs) * heads), dim3(kThreads), sizeof(float) * R, ln.stream, sh,
                         d_reqs, scores, stats, exps, slabs, u0);
      ln.done("score_simt_colsum");
    } else {
      e = launch_tile<T, D, RPT, kColsum>(sh, d_reqs, q, k, scores, stats, exps, slabs, slab_keys, u0, heads, ln, false);
    }
  }
  return e;
}

// Rows per thread: the tile height that leaves the fewest padding rows, the larger one on a tie.
template <typename T, int D>
cudaError_t launch_rows(const Shape& sh, const ReqDesc* d_reqs, const void* q, const void* k, float* scores, float2* stats,
                        int n_slab, int slab_keys, void* room, size_t room_bytes, int max_L, Launch ln, bool beside) {
  const int R = sh.window * sh.group;
  auto padded = [R](int rows) { return (R + rows - 1) / rows * rows; };
  if (R <= 64) return launch_typed<T, D, 4>(sh, d_reqs, q, k, scores, stats, n_slab, slab_keys, room, room_bytes, max_L, ln, beside);
  if (padded(112) < padded(128)) return launch_typed<T, D, 7>(sh, d_reqs, q, k, scores, stats, n_slab, slab_keys, room, room_bytes, max_L, ln, beside);
  return launch_typed<T, D, 8>(sh, d_reqs, q, k, scores, stats, n_slab, slab_keys, room, room_bytes, max_L, ln, beside);
}

}  // namespace

size_t score_simt_room(int total_heads, int max_L, int rows, int head_dim) {
  const int keys = tile_keys(head_dim);
  const int64_t exps = std::min(head_exps(max_L, rows, head_dim) * total_heads, kMaxExps);
  return static_cast<size_t>(exps / keys) * (keys * sizeof(float) + sizeof(float2));
}

cudaError_t launch_score_simt(const Shape& sh, const ReqDesc* d_reqs, const void* q, const void* k, float* scores,
                              float2* stats_ws, int n_slab, int slab_keys, void* room, size_t room_bytes, int max_L, Launch ln, bool beside) {
#define AKV_CASE(T, D) return launch_rows<T, D>(sh, d_reqs, q, k, scores, stats_ws, n_slab, slab_keys, room, room_bytes, max_L, ln, beside)
  if (sh.dtype == AUDIOKV_F32) {
    if (sh.head_dim == 64) AKV_CASE(float, 64);
    if (sh.head_dim == 128) AKV_CASE(float, 128);
    if (sh.head_dim == 256) AKV_CASE(float, 256);
  } else {
    if (sh.head_dim == 64) AKV_CASE(__nv_bfloat16, 64);
    if (sh.head_dim == 128) AKV_CASE(__nv_bfloat16, 128);
    if (sh.head_dim == 256) AKV_CASE(__nv_bfloat16, 256);
  }
#undef AKV_CASE
  return cudaErrorInvalidValue;
}

}  // namespace akv

// ---------------------------------------------------------------------------------------
// Scoring without any allocation.
//
// Some hosts of this library may not allocate device memory at the moment they need the
// scores: code that runs inside a memory-pool or arena whose owner forbids cudaMalloc once
// serving has started, plug-ins that are handed a stream and buffers but no allocator, and
// callers that must not risk the implicit device synchronisation an allocation can cause.
// For them the scratch of the two-sweep scoring (the per-slab row statistics) and the small
// request table live in one fixed array that is part of the library image: every GPU that
// loads the library holds kNoAllocBytes of it until the process exits.
#include <mutex>

namespace akv {
namespace {

constexpr size_t kNoAllocBytes = 8u << 20;     // 8 MiB per GPU, fixed
constexpr size_t kNoAllocTableBytes = 4096;    // request table at the front, statistics after it
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kNoAllocMaxDevices] = {};  // device address of the array, per device ordinal

// The request table reaches the scratch as a kernel argument (2.5 KB, copied at launch): no host
// buffer has to outlive the call.
constexpr int kNoAllocMaxReq = 64;
struct NoAllocTable {
  ReqDesc r[kNoAllocMaxReq];
};
__global__ void noalloc_table_kernel(const NoAllocTable t, int n, ReqDesc* dst) {
  if (threadIdx.x < n) dst[threadIdx.x] = t.r[threadIdx.x];
}

// The array's name is only a host-side handle; kernels need the address the runtime reports
// for the current device.
cudaError_t noalloc_scratch(int device, void** out) {
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[device] = p;
  }
  *out = g_noalloc_ptr[device];
  return cudaSuccess;
}

}  // namespace
}  // namespace akv

extern "C" int audiokv_score_noalloc(int device, const audiokv_params* p, const void* q_win, const void* k,
                                     float* scores, audiokv_stream stream) {
  using namespace akv;
  if (!p || !p->seq_len || !q_win || !k || !scores) return AUDIOKV_EINVAL;
  if (device < 0 || device >= kNoAllocMaxDevices) return AUDIOKV_EINVAL;
  if (p->dtype != AUDIOKV_F32 && p->dtype != AUDIOKV_BF16) return AUDIOKV_EINVAL;
  if (p->n_layers < 1 || p->n_kv_heads < 1 || p->n_q_heads < 1 || p->n_q_heads % p->n_kv_heads) return AUDIOKV_EINVAL;
  if (p->n_req < 1 || p->n_req > kNoAllocMaxReq || p->window < 1) return AUDIOKV_EINVAL;
  if (p->head_dim != 64 && p->head_dim != 128 && p->head_dim != 256) return AUDIOKV_EUNSUPPORTED;
  if (p->page_size != 0) return AUDIOKV_EUNSUPPORTED;  // contiguous K only
  const int G = p->n_q_heads / p->n_kv_heads;
  const int64_t R = static_cast<int64_t>(p->window) * G;
  if (R > 1024) return AUDIOKV_EUNSUPPORTED;
  if (static_cast<int64_t>(p->n_layers) * p->n_kv_heads > 2048) return AUDIOKV_EUNSUPPORTED;  // as audiokv_score
  const int per16 = p->dtype == AUDIOKV_F32 ? 4 : 8;
  const int64_t strides[] = {p->q_stride_req, p->q_stride_layer, p->q_stride_tok, p->q_stride_head,
                             p->kv_stride_layer, p->kv_stride_tok, p->kv_stride_head};
  for (int64_t s : strides) {
    if (s < 0) return AUDIOKV_EINVAL;
    if (s % per16) return AUDIOKV_EALIGN;
  }
  if ((reinterpret_cast<uintptr_t>(q_win) | reinterpret_cast<uintptr_t>(k)) & 15u) return AUDIOKV_EALIGN;
  static_assert(sizeof(ReqDesc) * kNoAllocMaxReq <= kNoAllocTableBytes, "request table must fit its slot");

  Shape sh{};
  sh.dtype = p->dtype;
  sh.n_layers = p->n_layers;
  sh.n_q_heads = p->n_q_heads;
  sh.n_kv_heads = p->n_kv_heads;
  sh.head_dim = p->head_dim;
  sh.n_req = p->n_req;
  sh.window = p->window;
  sh.group = G;
  sh.heads_per_req = p->n_layers * p->n_kv_heads;
  sh.total_heads = sh.heads_per_req * p->n_req;
  sh.q_stride_layer = p->q_stride_layer;
  sh.q_stride_tok = p->q_stride_tok;
  sh.q_stride_head = p->q_stride_head;
  sh.kv_stride_layer = p->kv_stride_layer;
  sh.kv_stride_tok = p->kv_stride_tok;
  sh.kv_stride_head = p->kv_stride_head;
  sh.softmax_scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(static_cast<float>(p->head_dim));
  sh.scale_log2e = static_cast<float>(static_cast<double>(sh.softmax_scale) * 1.4426950408889634);

  NoAllocTable table{};
  ReqDesc* reqs = table.r;
  int max_L = 0;
  int64_t score_off = 0;
  for (int r = 0; r < p->n_req; ++r) {
    const int L = p->seq_len[r];
    if (L <= p->window || L > AUDIOKV_MAX_SEQ_LEN) return AUDIOKV_EINVAL;
    const int64_t off = p->kv_req_offset ? p->kv_req_offset[r] : 0;
    if (off < 0) return AUDIOKV_EINVAL;
    if (off % per16) return AUDIOKV_EALIGN;
    const int64_t q_off = p->q_req_offset ? p->q_req_offset[r] : r * p->q_stride_req;
    if (q_off < 0) return AUDIOKV_EINVAL;
    if (q_off % per16) return AUDIOKV_EALIGN;
    reqs[r] = ReqDesc{L, L - p->window, r * sh.heads_per_req, 0, off, q_off, score_off};
    score_off += static_cast<int64_t>(sh.heads_per_req) * (L - p->window);
    max_L = L > max_L ? L : max_L;
  }
  constexpr int kSlabKeys = 512;
  const int n_slab = (max_L + kSlabKeys - 1) / kSlabKeys;
  const size_t need = sizeof(float2) * static_cast<size_t>(sh.total_heads) * n_slab * static_cast<size_t>(R);
  if (need > kNoAllocBytes - kNoAllocTableBytes) return AUDIOKV_EWORKSPACE;  // beyond the fixed scratch

  if (cudaSetDevice(device) != cudaSuccess) return AUDIOKV_ECUDA;
  void* base = nullptr;
  if (noalloc_scratch(device, &base) != cudaSuccess) return AUDIOKV_ECUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  noalloc_table_kernel<<<1, kNoAllocMaxReq, 0, s>>>(table, p->n_req, static_cast<ReqDesc*>(base));
  if (cudaGetLastError() != cudaSuccess) return AUDIOKV_ECUDA;
  int64_t launches = 0;
  Launch ln{s, &launches, nullptr};
  // Sweep 1 writes every statistics entry that sweep 2 reads, so nothing has to start at zero.
  cudaError_t e = launch_score_simt(sh, static_cast<const ReqDesc*>(base), q_win, k, scores,
                                    reinterpret_cast<float2*>(static_cast<unsigned char*>(base) + kNoAllocTableBytes),
                                    n_slab, kSlabKeys, nullptr, 0, max_L, ln);
  return e == cudaSuccess ? AUDIOKV_OK : AUDIOKV_ECUDA;
}

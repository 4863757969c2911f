// C boundary of the AudioKV eviction pass: argument checks, the per-shape plan (request
// table, FFT plans and tables, workspace layout) and the launch sequence of each entry point.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <unordered_map>
#include <vector>

#include "common.cuh"

using namespace akv;

namespace {

constexpr size_t kAlign = 256;
constexpr int kSlabKeys = 256;          // keys per slab of the softmax statistics (two K tiles of the tensor-core kernel)
constexpr int kMaxRows = 1024;          // W * G
constexpr int kMaxHeadsPerReq = 2048;
constexpr int kHostChunks = 8;          // the host-buffer call evicts one request in at most this many runs of layers

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Byte offsets inside the workspace; status .. ctas, up to blob_end, are uploaded as one piece with a plan. What only
// audiokv_evict_host needs lies behind the rest, so that the rest stays where a captured graph has it.
struct Layout {
  size_t status, reqs, plans, order, units, ctas, ready, blob_end, tables, stats, fft_scratch, scores, kstar, aux, end;
  size_t host_units, host_ctas, host_stats, host_end;
};

// Runs of the tensor-core scoring: both sweeps of every schedule.
struct ScoreTables {
  std::vector<ScoreUnit> units;
  std::vector<int32_t> ctas;             // per-CTA run offsets of every (schedule, sweep)
  std::vector<ScoreSchedule> schedules;
  int parts = 1;                         // statistics slots per head
};

struct Plan {
  bool valid = false;
  bool host_call = false;       // has the schedules of audiokv_evict_host, in host_score
  audiokv_params p{};
  std::vector<int32_t> seq_len;
  std::vector<int64_t> kv_off, q_off;
  Shape sh{};
  std::vector<ReqDesc> reqs;
  std::vector<FftPlan> fft;
  ScoreTables score;            // one schedule per run of requests
  ScoreTables host_score;       // one per chunk of layers of a single request
  std::vector<int32_t> sss_order;  // heads in the order the smoothing blocks take them (see build_plan)
  int64_t table_len = 0;        // float2 elements
  int64_t scores_len = 0;
  int max_L = 0, max_P = 0;
  int n_slab = 0;
  size_t score_room = 0;        // bytes of workspace behind everything else that the FMA scoring puts to use
  int sss_grid = 0;
  size_t sss_smem = 0;
  int64_t scratch_per_block = 0;  // float2 elements
  Layout lay{};
};

// Host arrays of the per-head problem that audiokv_reevict derives from its arguments.
struct ReevictArrays {
  std::vector<int32_t> len;
  std::vector<int64_t> kv_off, q_off, budget;
};

}  // namespace

struct audiokv_ctx {
  int device = 0;
  char* ws = nullptr;
  size_t ws_bytes = 0;
  Plan plan;
  bool plan_uploaded = false;
  bool host_uploaded = false;             // plan.host_score too
  uint64_t plan_id = 0;      // counts plan rebuilds
  ScoreMapCache score_maps;
  cudaEvent_t plan_ready = nullptr;
  cudaStream_t plan_stream = nullptr;     // where the plan went up
  bool plan_settled = false;              // the upload was seen complete
  std::vector<char> blob;                 // the plan as it goes up
  cudaStream_t side = nullptr;            // audiokv_evict_host copies in here
  cudaEvent_t fork = nullptr;
  // audiokv_evict_host: copies in on `side`, kernels on the caller's stream, copies out on `out`, chunk by chunk
  static constexpr int kMaxChunks = kHostChunks;
  cudaStream_t out = nullptr;
  cudaEvent_t chunk_in[kMaxChunks] = {}, chunk_done[kMaxChunks] = {}, copies_out = nullptr;
  int64_t launches = 0;
  int score_path = 0;  // route of the last scoring: 0 none yet, 1 tensor cores, 2 fp32 FMA
  Profiler prof;
  std::string cuda_error;
  ReevictArrays re;  // audiokv_reevict: the per-head problem it hands to the eviction pass
};

namespace {

int esize(int dtype) { return dtype == AUDIOKV_F32 ? 4 : 2; }

int check_params(const audiokv_params* p) {
  if (!p || !p->seq_len) return AUDIOKV_EINVAL;
  if (p->dtype != AUDIOKV_F32 && p->dtype != AUDIOKV_BF16) return AUDIOKV_EINVAL;
  if (p->n_layers < 1 || p->n_kv_heads < 1 || p->n_q_heads < 1 || p->n_q_heads % p->n_kv_heads) return AUDIOKV_EINVAL;
  if (p->n_req < 1 || p->n_req > AUDIOKV_MAX_REQ || p->window < 1) return AUDIOKV_EINVAL;
  if (!(p->rho > 0.f && p->rho <= 1.f) || !(p->alpha >= 0.f && p->alpha <= 1.f)) return AUDIOKV_EINVAL;
  if (p->transition_bins < 0 || p->base_per_head < 0) return AUDIOKV_EINVAL;
  if (p->smooth_mode < AUDIOKV_SMOOTH_SSS || p->smooth_mode > AUDIOKV_SMOOTH_MAX_POOL) return AUDIOKV_EINVAL;
  if (p->smooth_mode == AUDIOKV_SMOOTH_FIXED_FRACTION && !(p->smooth_kappa >= 0.f && p->smooth_kappa <= 1.f))
    return AUDIOKV_EINVAL;
  if (p->smooth_mode >= AUDIOKV_SMOOTH_AVG_POOL && (p->pool_kernel < 1 || p->pool_kernel > 1023 || p->pool_kernel % 2 == 0))
    return AUDIOKV_EINVAL;
  for (int r = 0; r < p->n_req; ++r) {
    if (p->seq_len[r] <= p->window || p->seq_len[r] > AUDIOKV_MAX_SEQ_LEN) return AUDIOKV_EINVAL;
    if (p->kv_req_offset && p->kv_req_offset[r] < 0) return AUDIOKV_EINVAL;
    if (p->q_req_offset && p->q_req_offset[r] < 0) return AUDIOKV_EINVAL;
  }
  if (p->head_dim != 64 && p->head_dim != 128 && p->head_dim != 256) return AUDIOKV_EUNSUPPORTED;
  const int64_t rows = static_cast<int64_t>(p->window) * (p->n_q_heads / p->n_kv_heads);
  if (rows > kMaxRows) return AUDIOKV_EUNSUPPORTED;
  if (static_cast<int64_t>(p->n_layers) * p->n_kv_heads > kMaxHeadsPerReq) return AUDIOKV_EUNSUPPORTED;
  const int per16 = 16 / esize(p->dtype);
  const int64_t strides[] = {p->q_stride_req, p->q_stride_layer, p->q_stride_tok, p->q_stride_head,
                             p->kv_stride_layer, p->kv_stride_tok, p->kv_stride_head};
  for (int64_t s : strides) {
    if (s < 0) return AUDIOKV_EINVAL;
    if (s % per16) return AUDIOKV_EALIGN;
  }
  if (p->page_size != 0) {
    if (p->page_size != 16 && p->page_size != 32 && p->page_size != 64 && p->page_size != 128) return AUDIOKV_EUNSUPPORTED;
    if (p->n_pages < 1 || !p->page_table || p->kv_stride_tok < 1) return AUDIOKV_EINVAL;
    if (static_cast<int64_t>(p->n_pages) * p->page_size > 0x7fffffffLL) return AUDIOKV_EUNSUPPORTED;
    for (int r = 0; r < p->n_req; ++r)
      if ((p->seq_len[r] + p->page_size - 1) / p->page_size > p->page_table_stride) return AUDIOKV_EINVAL;
  }
  for (int r = 0; r < p->n_req; ++r) {
    if (p->kv_req_offset && p->kv_req_offset[r] % per16) return AUDIOKV_EALIGN;
    if (p->q_req_offset && p->q_req_offset[r] % per16) return AUDIOKV_EALIGN;
  }
  return AUDIOKV_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool same_plan(const Plan& pl, const audiokv_params* p) {
  if (!pl.valid) return false;
  const audiokv_params& a = pl.p;
  if (a.dtype != p->dtype || a.n_layers != p->n_layers || a.n_q_heads != p->n_q_heads ||
      a.n_kv_heads != p->n_kv_heads || a.head_dim != p->head_dim || a.n_req != p->n_req || a.window != p->window ||
      a.q_stride_layer != p->q_stride_layer ||
      a.q_stride_tok != p->q_stride_tok || a.q_stride_head != p->q_stride_head ||
      a.kv_stride_layer != p->kv_stride_layer || a.kv_stride_tok != p->kv_stride_tok ||
      a.kv_stride_head != p->kv_stride_head || a.softmax_scale != p->softmax_scale || a.rho != p->rho ||
      a.alpha != p->alpha || a.transition_bins != p->transition_bins || a.base_per_head != p->base_per_head ||
      a.smooth_mode != p->smooth_mode || a.smooth_kappa != p->smooth_kappa || a.pool_kernel != p->pool_kernel ||
      a.page_size != p->page_size || a.n_pages != p->n_pages || a.page_table_stride != p->page_table_stride)
    return false;
  for (int r = 0; r < p->n_req; ++r) {
    if (pl.seq_len[r] != p->seq_len[r]) return false;
    if (pl.kv_off[r] != (p->kv_req_offset ? p->kv_req_offset[r] : 0)) return false;
    if (pl.q_off[r] != (p->q_req_offset ? p->q_req_offset[r] : r * p->q_stride_req)) return false;
  }
  return true;
}

// What a smoothing block can have in dynamic shared memory, in float2: 227 KB less what it uses beside it.
int sss_room() { return (232448 - sss_static_smem()) / static_cast<int>(sizeof(float2)); }

// Radix sequence for a complex length N: primes 11..127 first (descending), then 7, 5, 3, 4s, 2.
// Returns false when N has a prime factor above 127.
bool factor_len(int N, FftSeq* sq) {
  sq->N = N;
  sq->n_pass = 0;
  int rest = N, twos = 0;
  while (rest % 2 == 0) {
    rest /= 2;
    ++twos;
  }
  std::vector<int> odd;
  for (int q = 3; q <= kMaxPrime && rest > 1; q += 2)
    while (rest % q == 0) {
      odd.push_back(q);
      rest /= q;
    }
  if (rest != 1) return false;
  std::vector<int> seq;
  for (auto it = odd.rbegin(); it != odd.rend(); ++it) seq.push_back(*it);
  for (int i = 0; i < twos / 2; ++i) seq.push_back(4);
  if (twos % 2) seq.push_back(2);
  if (seq.size() > static_cast<size_t>(kMaxRadices)) return false;
  for (size_t i = 0; i < seq.size(); ++i) sq->radix[i] = seq[i];
  sq->n_pass = static_cast<int>(seq.size());
  return true;
}

// Rough cost of a transform, in arbitrary units: index arithmetic, shared-memory traffic and butterflies of the small
// radices are much alike per pass; a prime radix is a p x p product.
double seq_cost(const FftSeq& sq) {
  double c = 0.5;
  for (int i = 0; i < sq.n_pass; ++i) c += sq.radix[i] > 13 ? 1.5 + sq.radix[i] / 20.0 : 1.0;
  return c * sq.N;
}

// Places for the matrices of a sequence's prime radices.
void seq_tables(FftSeq* sq, int64_t* table_len) {
  sq->base = *table_len = (*table_len + 1) & ~int64_t(1);  // matrices and filters are read as float4
  int off = 0;
  for (int i = 0; i < sq->n_pass; ++i) {
    sq->mat[i] = off;
    if (sq->radix[i] > kMaxSmall) off += (sq->radix[i] - 1) / 2 * fft_mat_cols(sq->radix[i]);
  }
  *table_len += off;
}

void build_fft_plan(int n, FftPlan* fp, int64_t* table_len) {
  memset(fp, 0, sizeof(*fp));
  fp->n = n;
  fp->packed = (n % 2 == 0) ? 1 : 0;
  fp->N = fp->packed ? n / 2 : n;
  const int N = fp->N;
  if (!factor_len(N, &fp->seq)) {
    fp->bluestein = 1;
    // An odd real length is transformed at full complex length N = n, but only bins 0 .. (n-1)/2 are wanted (the rest
    // mirror them) and only those go back into the inverse: differences between input and output indices then span
    // N + (N-1)/2 values instead of 2N - 1, and the convolution may be that much shorter.
    fp->half = fp->packed ? 0 : 1;
    const int64_t need = fp->half ? static_cast<int64_t>(N) + (N - 1) / 2 : 2LL * N - 1;
    // convolution length: the smallest 2^a 3^b 5^c 7^d (a >= 2) that holds `need` points; close to it
    // instead of up to twice that for a power of two, which also keeps more transforms in shared memory
    int M = 0;
    for (int64_t p7 = 4; M == 0 || p7 < M; p7 *= 7)
      for (int64_t p5 = p7; M == 0 || p5 < M; p5 *= 5)
        for (int64_t p3 = p5; M == 0 || p3 < M; p3 *= 3) {
          int64_t p2 = p3;
          while (p2 < need) p2 *= 2;
          if (M == 0 || p2 < M) M = static_cast<int>(p2);
        }
    fp->M = M;
    factor_len(M, &fp->seq);
  }
  const int len = fp->seq.N;
  fp->root_mult = fp->packed && !fp->bluestein ? 2 : 1;  // an even n's post-twiddles are roots of order 2N
  fp->root_count = root_entries(len * fp->root_mult);
  fp->root_count2 = fp->bluestein ? root_entries(2 * N) : 0;
  const int room = sss_room() - 2 * (fp->root_count + fp->root_count2);  // for the work buffer
  fp->in_smem = sss_slots(len) <= room ? 1 : 0;
  if (!fp->in_smem) {
    // leading passes on the global buffer until a block fits on chip; then as many blocks at a time as fit
    const int cap = (room - 4) / 273 * 256;  // sss_slots(cap) <= room
    int blk = len;
    while (fp->g_pass < fp->seq.n_pass && blk > cap) blk /= fp->seq.radix[fp->g_pass++];
    fp->chunk = cap / blk * blk;
  }
  fp->root_at = sss_slots(fp->in_smem ? len : fp->chunk);
  fp->root_offset = *table_len = (*table_len + 1) & ~int64_t(1);
  *table_len += 2 * (fp->root_count + fp->root_count2);
  seq_tables(&fp->seq, table_len);
  if (!fp->bluestein) {
    fp->wide_pos = N > 65536 ? 1 : 0;
    fp->pos_offset = *table_len;
    *table_len += (N / 2 + 1) * (1 + fp->wide_pos) / 2 + 1;
  } else {
    fp->filter_offset = *table_len = (*table_len + 1) & ~int64_t(1);
    *table_len += fp->M;  // even
    if (fp->half) {
      fp->filter2_offset = *table_len;
      *table_len += fp->M;
    }
  }
}

int host_chunks(int n_layers) { return n_layers < kHostChunks ? n_layers : kHostChunks; }
int host_chunk_layer(int n_layers, int c) { return static_cast<int>(static_cast<int64_t>(n_layers) * c / host_chunks(n_layers)); }

// Schedules of the tensor-core scoring. A schedule covers a set of heads; the key tiles of those heads, in the order
// the sweep walks them, are dealt out evenly over the CTAs, CTA c taking tiles [c T / grid, (c + 1) T / grid): a few
// runs of consecutive tiles of one head. Sweep 1 walks the heads in order over all L keys (the runs of a head number
// its statistics slots); sweep 2 walks them backwards over the prefix keys (the heads sweep 1 touched last are the
// ones still in L2).
// chunks: not the schedules of whole requests but those of audiokv_evict_host, which evicts one request in chunks of layers
void build_score_schedules(const Plan& pl, bool chunks, ScoreTables* tab) {
  const Shape& sh = pl.sh;
  *tab = ScoreTables{};
  if (!score_umma_takes(sh)) return;
  // a head whose W * G query rows exceed the kernel's Q tile is scored in chunks of window rows (runs of their own)
  const int w_chunk = score_window_chunk(sh);
  const int n_wchunks = (sh.window + w_chunk - 1) / w_chunk;
  std::vector<int32_t> parts_of(static_cast<size_t>(sh.total_heads) * n_wchunks, 0);
  auto add = [&](bool whole, int r_begin, int r_end, int head_begin, int head_end) {
    ScoreSchedule sc{};
    sc.whole_requests = whole ? 1 : 0;
    sc.r_begin = r_begin;
    sc.r_end = r_end;
    sc.head_begin = head_begin;
    sc.head_end = head_end;
    struct Q {
      int u, r, hr, ch;
    };
    std::vector<Q> qs;  // the (head, window chunk) pairs of this schedule, in sweep-1 order
    for (int r = r_begin; r < r_end; ++r)
      for (int hr = whole ? 0 : head_begin; hr < (whole ? sh.heads_per_req : head_end); ++hr)
        for (int ch = 0; ch < n_wchunks; ++ch) qs.push_back(Q{pl.reqs[r].head_base + hr, r, hr, ch});
    for (int sweep = 1; sweep <= 2; ++sweep) {
      if (sweep == 2) std::reverse(qs.begin(), qs.end());
      int64_t total = 0;
      for (const Q& x : qs) {
        const int range = sweep == 1 ? pl.reqs[x.r].L : pl.reqs[x.r].P;
        total += (range + 127) / 128;
      }
      const int grid = static_cast<int>(total < kScoreCtas ? total : kScoreCtas);
      sc.unit_off[sweep - 1] = static_cast<int32_t>(tab->units.size());
      sc.cta_off[sweep - 1] = static_cast<int32_t>(tab->ctas.size());
      sc.grid[sweep - 1] = grid;
      const size_t first = tab->units.size();
      int64_t tile = 0;  // tiles before the current head in the sweep's sequence
      int c = 0;         // CTA whose range holds the next tile
      tab->ctas.push_back(0);
      for (const Q& x : qs) {
        const ReqDesc& d = pl.reqs[x.r];
        const int range = sweep == 1 ? d.L : d.P;
        const int n_tiles = (range + 127) / 128;
        int t = 0, part = 0;
        while (t < n_tiles) {
          // the CTA that owns tile `tile + t`, and how far its range reaches into this head
          while (c + 1 < grid && (static_cast<int64_t>(c + 1) * total) / grid <= tile + t) {
            ++c;
            tab->ctas.push_back(static_cast<int32_t>(tab->units.size() - first));
          }
          const int64_t c_end = (static_cast<int64_t>(c + 1) * total) / grid;
          const int take = static_cast<int>(std::min<int64_t>(n_tiles - t, c_end - (tile + t)));
          ScoreUnit un{};
          un.u = x.u;
          un.r = x.r;
          un.l = x.hr / sh.n_kv_heads;
          un.h = x.hr % sh.n_kv_heads;
          un.part = part++;
          un.kt0 = t * 128;
          un.n_tiles = take;
          un.P = d.P;
          un.score_base = d.score_offset + static_cast<int64_t>(x.hr) * d.P;
          un.w0 = x.ch * w_chunk;
          un.wn = sh.window - un.w0 < w_chunk ? sh.window - un.w0 : w_chunk;
          un.qid = x.u * n_wchunks + x.ch;
          un.head_parts = 0;  // set below
          tab->units.push_back(un);
          t += take;
        }
        if (sweep == 1) {
          parts_of[static_cast<size_t>(x.u) * n_wchunks + x.ch] = part;
          tab->parts = part > tab->parts ? part : tab->parts;
        }
        tile += n_tiles;
      }
      while (static_cast<int>(tab->ctas.size()) - sc.cta_off[sweep - 1] < grid + 1)
        tab->ctas.push_back(static_cast<int32_t>(tab->units.size() - first));
      for (size_t i = first; i < tab->units.size(); ++i) tab->units[i].head_parts = parts_of[tab->units[i].qid];
    }
    tab->schedules.push_back(sc);
  };
  if (!chunks) {
    const int cap = score_map_chunk(sh.n_req);
    for (int r0 = 0; r0 < sh.n_req; r0 += cap) add(true, r0, r0 + cap < sh.n_req ? r0 + cap : sh.n_req, 0, 0);
  } else if (sh.n_req == 1 && sh.n_layers > 1) {
    const int n_chunks = host_chunks(sh.n_layers);
    for (int c = 0; c < n_chunks; ++c)
      add(false, 0, 1, host_chunk_layer(sh.n_layers, c) * sh.n_kv_heads, host_chunk_layer(sh.n_layers, c + 1) * sh.n_kv_heads);
  }
}

// Softmax statistics of the tensor-core kernels: [head][part][group][row].
size_t stat_entries(const Plan& pl, const ScoreTables& tab) {
  return static_cast<size_t>(pl.sh.total_heads) * tab.parts * score_stat_sets() * pl.sh.window * pl.sh.group;
}

int build_plan(const audiokv_params* p, Plan* pl) {
  int rc = check_params(p);
  if (rc) return rc;
  pl->valid = false;
  pl->p = *p;
  pl->seq_len.assign(p->seq_len, p->seq_len + p->n_req);
  pl->kv_off.assign(p->n_req, 0);
  if (p->kv_req_offset) pl->kv_off.assign(p->kv_req_offset, p->kv_req_offset + p->n_req);
  pl->q_off.resize(p->n_req);
  for (int r = 0; r < p->n_req; ++r) pl->q_off[r] = p->q_req_offset ? p->q_req_offset[r] : r * p->q_stride_req;
  pl->p.seq_len = nullptr;
  pl->p.kv_req_offset = nullptr;
  pl->p.q_req_offset = nullptr;
  pl->p.page_table = nullptr;

  Shape& sh = pl->sh;
  sh.dtype = p->dtype;
  sh.n_layers = p->n_layers;
  sh.n_q_heads = p->n_q_heads;
  sh.n_kv_heads = p->n_kv_heads;
  sh.head_dim = p->head_dim;
  sh.n_req = p->n_req;
  sh.window = p->window;
  sh.group = p->n_q_heads / p->n_kv_heads;
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
  sh.rho = p->rho;
  sh.alpha = p->alpha;
  sh.transition_bins = p->transition_bins;
  sh.base_per_head = p->base_per_head;
  sh.smooth_mode = p->smooth_mode;
  sh.smooth_kappa = p->smooth_kappa;
  sh.pool_kernel = p->pool_kernel;
  sh.page_size = p->page_size;
  sh.page_shift = 0;
  while (p->page_size && (1 << sh.page_shift) < p->page_size) ++sh.page_shift;
  sh.n_pages = p->n_pages;
  sh.page_table_stride = p->page_table_stride;
  sh.page_table = nullptr;  // set per call, with the status word
  sh.page_status = nullptr;

  pl->reqs.assign(p->n_req, ReqDesc{});
  pl->fft.clear();
  pl->table_len = 0;
  pl->scores_len = 0;
  pl->max_L = pl->max_P = 0;
  std::unordered_map<int, int> plan_of;  // prefix length -> index into pl->fft
  for (int r = 0; r < p->n_req; ++r) {
    ReqDesc& d = pl->reqs[r];
    d.L = p->seq_len[r];
    d.P = d.L - p->window;
    d.head_base = r * sh.heads_per_req;
    d.kv_offset = pl->kv_off[r];
    d.q_offset = pl->q_off[r];
    d.score_offset = pl->scores_len;
    pl->scores_len += static_cast<int64_t>(sh.heads_per_req) * d.P;
    pl->max_L = d.L > pl->max_L ? d.L : pl->max_L;
    pl->max_P = d.P > pl->max_P ? d.P : pl->max_P;
    auto it = plan_of.find(d.P);
    if (it == plan_of.end()) {
      FftPlan fp;
      build_fft_plan(d.P, &fp, &pl->table_len);
      fp.id = static_cast<int>(pl->fft.size());
      pl->fft.push_back(fp);
      it = plan_of.emplace(d.P, static_cast<int>(pl->fft.size()) - 1).first;
    }
    d.fft_plan = it->second;
  }
  pl->n_slab = (pl->max_L + kSlabKeys - 1) / kSlabKeys;
  build_score_schedules(*pl, false, &pl->score);
  pl->host_score = ScoreTables{};
  pl->host_call = false;
  // one block per head at a time, as many blocks as the planning SM count (the plan, and with it the workspace size,
  // does not depend on the device)
  pl->sss_grid = sh.total_heads < kScoreCtas ? sh.total_heads : kScoreCtas;
  {
    // The smoothing blocks take the heads from a queue, in this order: by an estimate of their transform's cost, so that the
    // last ones to be taken are cheap.
    auto cost = [&](int r) -> double {
      const FftPlan& fp = pl->fft[pl->reqs[r].fft_plan];
      return seq_cost(fp.seq) * (fp.bluestein ? 2.0 : 1.0) * (fp.in_smem ? 1.0 : 1.5) + 8.0 * fp.n;
    };
    // the heads of a request cost the same: the requests are sorted, and their heads follow in order
    std::vector<std::pair<double, int32_t>> by_cost(p->n_req);
    for (int r = 0; r < p->n_req; ++r) by_cost[r] = {cost(r), r};
    std::stable_sort(by_cost.begin(), by_cost.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    pl->sss_order.resize(sh.total_heads);
    for (int i = 0; i < sh.total_heads; ++i)
      pl->sss_order[i] = pl->reqs[by_cost[i / sh.heads_per_req].second].head_base + i % sh.heads_per_req;
  }
  int smem_c = 64;
  pl->scratch_per_block = 0;
  for (const FftPlan& fp : pl->fft) {
    const int need = fp.root_at + 2 * (fp.root_count + fp.root_count2);
    smem_c = need > smem_c ? need : smem_c;
    if (!fp.in_smem) pl->scratch_per_block = fp.seq.N > pl->scratch_per_block ? fp.seq.N : pl->scratch_per_block;
  }
  pl->sss_smem = static_cast<size_t>(smem_c) * sizeof(float2);

  Layout& L = pl->lay;
  size_t off = 0;
  L.status = off;      off = align_up(off + 64);
  L.reqs = off;        off = align_up(off + sizeof(ReqDesc) * pl->reqs.size());
  L.plans = off;       off = align_up(off + sizeof(FftPlan) * pl->fft.size());
  L.order = off;       off = align_up(off + sizeof(int32_t) * pl->sss_order.size());
  L.units = off;       off = align_up(off + sizeof(ScoreUnit) * pl->score.units.size());
  L.ctas = off;        off = align_up(off + sizeof(int32_t) * pl->score.ctas.size());
  L.ready = off;       off = align_up(off + sizeof(uint64_t) * static_cast<size_t>(sh.total_heads));  // goes up as zeros
  L.blob_end = off;
  L.tables = off;      off = align_up(off + sizeof(float2) * static_cast<size_t>(pl->table_len));
  {
    // softmax statistics: [head][slab][row] for the FMA kernels
    const int rows = sh.window * sh.group;
    const size_t entries = std::max(static_cast<size_t>(sh.total_heads) * pl->n_slab * rows, stat_entries(*pl, pl->score));
    L.stats = off;     off = align_up(off + sizeof(float2) * entries);
    pl->score_room = score_umma_takes(sh) ? 0 : score_simt_room(sh.total_heads, pl->max_L, rows, sh.head_dim);
  }
  L.fft_scratch = off; off = align_up(off + sizeof(float2) * static_cast<size_t>(pl->scratch_per_block) * pl->sss_grid);
  L.scores = off;      off = align_up(off + sizeof(float) * static_cast<size_t>(pl->scores_len));
  L.kstar = off;       off = align_up(off + sizeof(int32_t) * static_cast<size_t>(sh.total_heads));
  L.aux = off;         off = align_up(off + 2 * sizeof(int32_t) * static_cast<size_t>(sh.total_heads));  // audiokv_reevict
  L.end = L.host_end = off;
  pl->valid = true;
  return AUDIOKV_OK;
}

// The schedules by chunks of layers that audiokv_evict_host runs through, and their place in the workspace (a serving loop whose
// every prompt brings a new length builds a plan a call, so the others go without).
void add_host_part(Plan* pl) {
  build_score_schedules(*pl, true, &pl->host_score);
  Layout& L = pl->lay;
  size_t off = L.end;
  if (!pl->host_score.units.empty()) {
    L.host_units = off;  off = align_up(off + sizeof(ScoreUnit) * pl->host_score.units.size());
    L.host_ctas = off;   off = align_up(off + sizeof(int32_t) * pl->host_score.ctas.size());
    L.host_stats = off;  off = align_up(off + sizeof(float2) * stat_entries(*pl, pl->host_score));
  }
  L.host_end = off;
  pl->host_call = true;
}

int cuda_fail(audiokv_ctx* ctx, cudaError_t e) {
  ctx->cuda_error = cudaGetErrorString(e);
  return AUDIOKV_ECUDA;
}

// Makes ctx->plan match p and its tables resident on the device (stream-ordered).
int prepare(audiokv_ctx* ctx, const audiokv_params* p, cudaStream_t stream, bool host_call = false) {
  if (!ctx) return AUDIOKV_EINVAL;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  if (!same_plan(ctx->plan, p)) {
    int rc = build_plan(p, &ctx->plan);
    ctx->plan_id += 1;
    if (rc) return rc;
    ctx->plan_uploaded = ctx->host_uploaded = false;
  }
  Plan& pl = ctx->plan;
  if (host_call && !pl.host_call) add_host_part(&pl);
  if ((host_call ? pl.lay.host_end : pl.lay.end) > ctx->ws_bytes) return AUDIOKV_EWORKSPACE;
  pl.sh.page_table = p->page_size ? p->page_table : nullptr;  // device data of this call, not part of the plan
  pl.sh.page_status = reinterpret_cast<int*>(ctx->ws + pl.lay.status);
  if (!ctx->plan_uploaded) {
    // A graph that held the upload would bring this plan back at every replay, over the one the context then has: the first
    // call with a given shape has to run outside capture (later ones add nothing but the kernels of the pass).
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(stream, &cap)) != cudaSuccess) return cuda_fail(ctx, e);
    if (cap != cudaStreamCaptureStatusNone) {
      ctx->cuda_error = "the plan of these params is not on the device yet: make one call outside stream capture first";
      return AUDIOKV_ECUDA;
    }
    // The request table, FFT plans, order and schedules go up as one piece, and the status word starts clean with it. It travels
    // as arguments of kernels, for which the host does not wait (a prompt of a new length then costs no round trip); a
    // plan too large for some of these, thousands of heads or requests, goes up from pageable memory, for which it does.
    const size_t blob = pl.lay.blob_end;
    const bool inlined = blob <= kPlanParts * kPlanPartBytes;
    ctx->blob.resize(blob);
    char* src = ctx->blob.data();
    memset(src, 0, 64);
    memset(src + pl.lay.ready, 0, blob - pl.lay.ready);
    auto put = [&](size_t at, const void* data, size_t bytes) {
      if (bytes) memcpy(src + at, data, bytes);
    };
    put(pl.lay.reqs, pl.reqs.data(), sizeof(ReqDesc) * pl.reqs.size());
    put(pl.lay.plans, pl.fft.data(), sizeof(FftPlan) * pl.fft.size());
    put(pl.lay.units, pl.score.units.data(), sizeof(ScoreUnit) * pl.score.units.size());
    put(pl.lay.ctas, pl.score.ctas.data(), sizeof(int32_t) * pl.score.ctas.size());
    put(pl.lay.order, pl.sss_order.data(), sizeof(int32_t) * pl.sss_order.size());
    if (!inlined && (e = cudaMemcpyAsync(ctx->ws, src, blob, cudaMemcpyHostToDevice, stream)) != cudaSuccess) return cuda_fail(ctx, e);
    Launch ln{stream, &ctx->launches, &ctx->prof};
    e = launch_fft_tables(static_cast<int>(pl.fft.size()), inlined ? src : nullptr, blob, pl.lay.units, ctx->ws, pl.lay.plans,
                          reinterpret_cast<float2*>(ctx->ws + pl.lay.tables), pl.sss_smem, ln);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if ((e = cudaEventRecord(ctx->plan_ready, stream)) != cudaSuccess) return cuda_fail(ctx, e);
    ctx->plan_stream = stream;
    ctx->plan_settled = false;
    ctx->plan_uploaded = true;
  } else if (!ctx->plan_settled) {
    // Calls on the stream of the upload are ordered behind it. On another stream, or inside a capture (which must not wait for
    // an event from outside), the upload has to be complete: seen so once, no later call asks again.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(stream, &cap)) != cudaSuccess) return cuda_fail(ctx, e);
    if (stream != ctx->plan_stream || cap != cudaStreamCaptureStatusNone) {
      cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // the event is not the capture's: waiting for it is safe
      if ((e = cudaThreadExchangeStreamCaptureMode(&mode)) != cudaSuccess) return cuda_fail(ctx, e);
      e = cudaEventSynchronize(ctx->plan_ready);
      const cudaError_t e2 = cudaThreadExchangeStreamCaptureMode(&mode);
      if (e != cudaSuccess || e2 != cudaSuccess) return cuda_fail(ctx, e != cudaSuccess ? e : e2);
      ctx->plan_settled = true;
    }
  }
  if (host_call && !ctx->host_uploaded) {
    // from pageable memory: this call waits on the host in any case
    const ScoreTables& t = pl.host_score;
    if (!t.units.empty() &&
        ((e = cudaMemcpyAsync(ctx->ws + pl.lay.host_units, t.units.data(), sizeof(ScoreUnit) * t.units.size(),
                              cudaMemcpyHostToDevice, stream)) != cudaSuccess ||
         (e = cudaMemcpyAsync(ctx->ws + pl.lay.host_ctas, t.ctas.data(), sizeof(int32_t) * t.ctas.size(),
                              cudaMemcpyHostToDevice, stream)) != cudaSuccess))
      return cuda_fail(ctx, e);
    ctx->host_uploaded = true;
  }
  return AUDIOKV_OK;
}

// The per-kernel timing of one call, from here (event 0) to its end, when profiling is on.
struct ProfiledCall {
  Profiler& pf;
  ProfiledCall(audiokv_ctx* ctx, cudaStream_t stream) : pf(ctx->prof) {
    if (!pf.on) return;
    pf.n = 0;
    pf.recording = true;
    pf.mark("begin", stream);
  }
  ~ProfiledCall() { pf.recording = false; }
};

const ReqDesc* d_reqs(audiokv_ctx* c) { return reinterpret_cast<const ReqDesc*>(c->ws + c->plan.lay.reqs); }
// The first 64 bytes of the workspace: the status word, from int 4 on the queue of the smoothing kernel, from int 8 on the
// counters of the queue between smoothing and gather.
int* d_status(audiokv_ctx* c) { return reinterpret_cast<int*>(c->ws + c->plan.lay.status); }

// used: bytes at the front of the workspace that the call needs; the FMA scoring may have the rest. head_end >= 0 (one request,
// tensor-core path only): the heads [head_begin, head_end) alone, a chunk of audiokv_evict_host.
int do_score(audiokv_ctx* ctx, const void* q, const void* k, float* scores, cudaStream_t stream, size_t used, int head_begin = 0,
             int head_end = -1, bool beside = false) {
  Plan& pl = ctx->plan;
  Launch ln{stream, &ctx->launches, &ctx->prof};
  float2* stats = reinterpret_cast<float2*>(ctx->ws + pl.lay.stats);
  cudaError_t e = cudaErrorNotSupported;
  if (score_umma_takes(pl.sh)) {
    const bool chunk = head_end >= 0;
    const ScoreTables& t = chunk ? pl.host_score : pl.score;
    e = launch_score_umma(pl.sh, pl.reqs.data(), reinterpret_cast<const ScoreUnit*>(ctx->ws + (chunk ? pl.lay.host_units : pl.lay.units)),
                          reinterpret_cast<const int32_t*>(ctx->ws + (chunk ? pl.lay.host_ctas : pl.lay.ctas)), t.schedules.data(),
                          static_cast<int>(t.schedules.size()), q, k, scores,
                          chunk ? reinterpret_cast<float2*>(ctx->ws + pl.lay.host_stats) : stats, t.parts, d_status(ctx), ln,
                          head_begin, head_end, &ctx->score_maps, ctx->plan_id, beside);
  }
  if (head_end >= 0 && e != cudaSuccess) return cuda_fail(ctx, e);  // no head ranges in the FMA kernel
  ctx->score_path = 1;
  if (e == cudaErrorNotSupported) {
    // fp32 inputs (which must not be rounded to TF32), a GQA group above 256 query heads, or strides the copy
    // engine cannot take; audiokv_last_score_path tells the caller which route ran
    ctx->score_path = 2;
    e = launch_score_simt(pl.sh, d_reqs(ctx), q, k, scores, stats, pl.n_slab, kSlabKeys, ctx->ws + used,
                          std::min(pl.score_room, ctx->ws_bytes - used), pl.max_L, ln, beside && !score_umma_takes(pl.sh));
  }
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

// Smoothing; with budgets, cu_kept and kept_idx it also selects each head's kept tokens (smoothed may then be null).
// head_end < 0: all heads, in the plan's cost-sorted order; else the heads [head_begin, head_end) in index order.
int do_smooth(audiokv_ctx* ctx, const float* scores, float* smoothed, int32_t* kstar, const int32_t* budgets,
              const int32_t* cu_kept, int32_t* kept_idx, cudaStream_t stream, int head_begin = 0, int head_end = -1,
              HeadQueue hq = {}) {
  Plan& pl = ctx->plan;
  Launch ln{stream, &ctx->launches, &ctx->prof};
  const bool all = head_end < 0;
  const int count = all ? static_cast<int>(pl.sss_order.size()) : head_end - head_begin;
  cudaError_t e = launch_sss(pl.sh, d_reqs(ctx), reinterpret_cast<const FftPlan*>(ctx->ws + pl.lay.plans),
                             reinterpret_cast<const float2*>(ctx->ws + pl.lay.tables), scores, smoothed, kstar,
                             reinterpret_cast<float2*>(ctx->ws + pl.lay.fft_scratch), pl.scratch_per_block,
                             all ? pl.sss_grid : (count < pl.sss_grid ? count : pl.sss_grid), pl.sss_smem,
                             all ? reinterpret_cast<const int32_t*>(ctx->ws + pl.lay.order) : nullptr, count,
                             head_begin, budgets, cu_kept, kept_idx, d_status(ctx), d_status(ctx) + 4, hq, ln);
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

int do_gather(audiokv_ctx* ctx, const int32_t* cu_kept, const int32_t* kept_idx, const void* k, const void* v,
              void* k_out, void* v_out, cudaStream_t stream, int head_begin = 0, int head_end = -1) {
  Plan& pl = ctx->plan;
  Launch ln{stream, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_gather(pl.sh, d_reqs(ctx), cu_kept, kept_idx, k, v, k_out, v_out, head_begin,
                                head_end < 0 ? pl.sh.total_heads : head_end, ln);
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

// Smoothing, selection and gather of all heads; kept_rows: about how many rows they keep.
int do_smooth_gather(audiokv_ctx* ctx, const float* scores, float* smoothed, int32_t* kstar, const int32_t* budgets,
                     const int32_t* cu_kept, int32_t* kept_idx, const void* k, const void* v, void* k_out, void* v_out,
                     int64_t kept_rows, cudaStream_t stream) {
  Plan& pl = ctx->plan;
  // The gather beside the smoothing pays as soon as some heads can end well before others: when the blocks take a second turn
  // (48 layers of 2048 tokens, 192 heads: 145.9 -> 133.0 us a pass) or when a transform takes long beside a head that needs none
  // (28 layers, 30 % of heads with transforms: 8192 tokens 269.7 -> 247.8, 32768 908 -> 812). It costs 2 to 3 us more where no
  // head needs one, which its own work has to be long against: with less than 80 MB to read and write (14 layers of 1500 tokens,
  // half kept: 42 MB) 64.6 -> 67.7, above (2500 tokens: 70 MB; 5000: 140 MB) 75.4 -> 74.3 and 107.1 -> 103.7.
  const int64_t moved = kept_rows * pl.sh.head_dim * esize(pl.sh.dtype) * 4;
  const bool follow = pl.sh.total_heads > pl.sss_grid || (pl.max_P >= 1400 && moved >= (80LL << 20));
  int* words = d_status(ctx);
  const HeadQueue hq{reinterpret_cast<unsigned long long*>(words + 8), words + 10,
                     follow ? reinterpret_cast<unsigned long long*>(ctx->ws + pl.lay.ready) : nullptr, gather_unit_rows(pl.sh)};
  int rc = do_smooth(ctx, scores, smoothed, kstar, budgets, cu_kept, kept_idx, stream, 0, -1, hq);
  if (rc || !follow) return rc ? rc : do_gather(ctx, cu_kept, kept_idx, k, v, k_out, v_out, stream);
  Launch ln{stream, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_gather_stream(pl.sh, d_reqs(ctx), cu_kept, kept_idx, k, v, k_out, v_out, pl.sh.total_heads, kept_rows, hq,
                                       d_status(ctx), ln);
  if (e == cudaSuccess) return AUDIOKV_OK;
  ctx->plan_uploaded = false;  // the queue keeps this call's heads: it goes up again, empty
  return cuda_fail(ctx, e);
}

int check_budgets(const Plan& pl, const int64_t* total_budget) {
  if (!total_budget) return AUDIOKV_EINVAL;
  const int64_t N = pl.sh.heads_per_req, f = static_cast<int64_t>(pl.sh.window) + pl.sh.base_per_head;
  for (int r = 0; r < pl.sh.n_req; ++r) {
    if (f > pl.reqs[r].L) return AUDIOKV_EINVAL;
    if (total_budget[r] < N * f || total_budget[r] > N * pl.reqs[r].L) return AUDIOKV_EINVAL;
  }
  return AUDIOKV_OK;
}

int do_allocate(audiokv_ctx* ctx, const float* head_scores, const int64_t* total_budget, int32_t* budgets,
                int32_t* cu_kept, cudaStream_t stream) {
  Plan& pl = ctx->plan;
  int rc = check_budgets(pl, total_budget);
  if (rc) return rc;
  Launch ln{stream, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_allocate(pl.sh, d_reqs(ctx), head_scores, total_budget, budgets, cu_kept, d_status(ctx), ln);
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

int do_select_gather(audiokv_ctx* ctx, const float* smoothed, const int32_t* budgets, const int32_t* cu_kept,
                     const void* k, const void* v, void* k_out, void* v_out, int32_t* kept_idx, cudaStream_t stream) {
  Plan& pl = ctx->plan;
  Launch ln{stream, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_select(pl.sh, d_reqs(ctx), smoothed, budgets, cu_kept, kept_idx, pl.max_P, d_status(ctx), ln);
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  return do_gather(ctx, cu_kept, kept_idx, k, v, k_out, v_out, stream);
}

// Where audiokv_evict_host keeps the device copies of its buffers: byte offsets behind the plan's own part of the workspace.
struct HostStaging {
  size_t q, k, v, head_scores, k_out, v_out, kept_idx, budgets, cu_kept, end;
  int64_t rows;
};
HostStaging host_staging(const Plan& pl, int64_t q_elems, int64_t kv_elems, const int64_t* total_budget) {
  HostStaging h{};
  const size_t es = esize(pl.sh.dtype), TH = static_cast<size_t>(pl.sh.total_heads);
  for (int r = 0; r < pl.sh.n_req; ++r) h.rows += total_budget[r];
  const size_t row_bytes = static_cast<size_t>(h.rows) * pl.sh.head_dim * es;
  size_t off = pl.lay.host_end;
  h.q = off;           off = align_up(off + q_elems * es);
  h.k = off;           off = align_up(off + kv_elems * es);
  h.v = off;           off = align_up(off + kv_elems * es);
  h.head_scores = off; off = align_up(off + sizeof(float) * TH);
  h.k_out = off;       off = align_up(off + row_bytes);
  h.v_out = off;       off = align_up(off + row_bytes);
  h.kept_idx = off;    off = align_up(off + h.rows * sizeof(int32_t));
  h.budgets = off;     off = align_up(off + sizeof(int32_t) * TH);
  h.cu_kept = off;     off = align_up(off + sizeof(int32_t) * (TH + 1));
  h.end = off;
  return h;
}

}  // namespace

extern "C" {

size_t audiokv_params_size(void) { return sizeof(audiokv_params); }

const char* audiokv_strerror(int status) {
  switch (status) {
    case AUDIOKV_OK: return "ok";
    case AUDIOKV_EINVAL: return "invalid argument";
    case AUDIOKV_EALIGN: return "pointer or stride not 16-byte aligned";
    case AUDIOKV_EUNSUPPORTED: return "shape not supported";
    case AUDIOKV_EWORKSPACE: return "workspace too small";
    case AUDIOKV_ECUDA: return "CUDA runtime error";
    case AUDIOKV_ETIMEOUT: return "a kernel gave up a bounded wait";
    case AUDIOKV_EDEVICE: return "a kernel found an index out of range";
    default: return "unknown status";
  }
}

int64_t audiokv_budget_from_ratio(double c, int32_t n_heads_total, int32_t seq_len, int32_t window) {
  if (!(c >= 0.0 && c <= 1.0) || n_heads_total < 1 || seq_len < 1 || window < 0 || window > seq_len) return -1;
  const int64_t hi = static_cast<int64_t>(n_heads_total) * seq_len, lo = static_cast<int64_t>(n_heads_total) * window;
  int64_t b = static_cast<int64_t>(floor(c * static_cast<double>(hi)));
  return b < lo ? lo : (b > hi ? hi : b);
}

int64_t audiokv_scores_len(const audiokv_params* p) {
  int rc = check_params(p);
  if (rc) return rc;
  int64_t n = 0;
  for (int r = 0; r < p->n_req; ++r)
    n += static_cast<int64_t>(p->n_layers) * p->n_kv_heads * (p->seq_len[r] - p->window);
  return n;
}

size_t audiokv_workspace_bytes(const audiokv_params* p) {
  Plan pl;
  if (build_plan(p, &pl)) return 0;
  return pl.lay.end + pl.score_room;
}

size_t audiokv_workspace_bytes_host(const audiokv_params* p, int64_t q_elems, int64_t kv_elems,
                                    const int64_t* total_budget) {
  Plan pl;
  if (build_plan(p, &pl) || !total_budget || q_elems < 0 || kv_elems < 0) return 0;
  add_host_part(&pl);
  return host_staging(pl, q_elems, kv_elems, total_budget).end + pl.score_room;
}

int audiokv_create(audiokv_ctx** out, int device, size_t workspace_bytes) {
  if (!out || workspace_bytes == 0) return AUDIOKV_EINVAL;
  *out = nullptr;
  if (cudaSetDevice(device) != cudaSuccess) return AUDIOKV_ECUDA;
  audiokv_ctx* c = new audiokv_ctx();
  c->device = device;
  if (cudaMalloc(&c->ws, workspace_bytes) != cudaSuccess) {
    delete c;
    return AUDIOKV_ECUDA;
  }
  c->ws_bytes = workspace_bytes;
  if (workspace_bytes < 64 || cudaMemset(c->ws, 0, 64) != cudaSuccess) {  // the status word starts clean
    cudaFree(c->ws);
    delete c;
    return workspace_bytes < 64 ? AUDIOKV_EINVAL : AUDIOKV_ECUDA;
  }
  if (cudaEventCreateWithFlags(&c->plan_ready, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&c->fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) != cudaSuccess) {
    if (c->plan_ready) cudaEventDestroy(c->plan_ready);
    if (c->fork) cudaEventDestroy(c->fork);
    cudaFree(c->ws);
    delete c;
    return AUDIOKV_ECUDA;
  }
  bool ok = cudaStreamCreateWithFlags(&c->out, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&c->copies_out, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; i < audiokv_ctx::kMaxChunks && ok; ++i)
    ok = cudaEventCreateWithFlags(&c->chunk_in[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&c->chunk_done[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    audiokv_destroy(c);
    return AUDIOKV_ECUDA;
  }
  *out = c;
  return AUDIOKV_OK;
}

int audiokv_destroy(audiokv_ctx* ctx) {
  if (!ctx) return AUDIOKV_EINVAL;
  cudaSetDevice(ctx->device);
  cudaEventDestroy(ctx->plan_ready);
  cudaEventDestroy(ctx->fork);
  cudaStreamDestroy(ctx->side);
  if (ctx->out) cudaStreamDestroy(ctx->out);
  if (ctx->copies_out) cudaEventDestroy(ctx->copies_out);
  for (int i = 0; i < audiokv_ctx::kMaxChunks; ++i) {
    if (ctx->chunk_in[i]) cudaEventDestroy(ctx->chunk_in[i]);
    if (ctx->chunk_done[i]) cudaEventDestroy(ctx->chunk_done[i]);
  }
  for (cudaEvent_t e : ctx->prof.ev) cudaEventDestroy(e);
  cudaFree(ctx->ws);
  delete ctx;
  return AUDIOKV_OK;
}

int audiokv_last_device_status(audiokv_ctx* ctx, audiokv_stream stream) {
  if (!ctx) return AUDIOKV_EINVAL;
  int st = 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(&st, ctx->ws, sizeof(int), cudaMemcpyDeviceToHost, s);  // first word of the workspace
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && st != 0) e = cudaMemsetAsync(ctx->ws, 0, sizeof(int), s);  // reported once, then clean again
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  return st;
}

const char* audiokv_last_cuda_error(const audiokv_ctx* ctx) { return ctx ? ctx->cuda_error.c_str() : ""; }

int64_t audiokv_launch_count(const audiokv_ctx* ctx) { return ctx ? ctx->launches : 0; }

const char* audiokv_last_score_path(const audiokv_ctx* ctx) {
  if (!ctx || ctx->score_path == 0) return "none";
  return ctx->score_path == 1 ? "tcgen05" : "fma";
}

int64_t audiokv_set_wait_limit(int64_t cycles) {
  const int64_t before = score_wait_cycles();
  set_score_wait_cycles(cycles);
  return before;
}

int audiokv_profile_enable(audiokv_ctx* ctx, int on) {
  if (!ctx) return AUDIOKV_EINVAL;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return AUDIOKV_ECUDA;
  Profiler& pf = ctx->prof;
  if (on && !pf.reserve(32)) return AUDIOKV_ECUDA;  // enough for a pass of one request; longer ones add theirs
  pf.on = on != 0;
  pf.n = 0;
  return AUDIOKV_OK;
}

int audiokv_profile_count(const audiokv_ctx* ctx) { return ctx && ctx->prof.n > 0 ? ctx->prof.n - 1 : 0; }

const char* audiokv_profile_name(const audiokv_ctx* ctx, int i) {
  if (!ctx || i < 0 || i + 1 >= ctx->prof.n) return "";
  return ctx->prof.name[i + 1];
}

float audiokv_profile_ms(audiokv_ctx* ctx, int i) {
  if (!ctx || i < 0 || i + 1 >= ctx->prof.n) return -1.f;
  float ms = -1.f;
  if (cudaEventSynchronize(ctx->prof.ev[i + 1]) != cudaSuccess) return -1.f;
  if (cudaEventElapsedTime(&ms, ctx->prof.ev[i], ctx->prof.ev[i + 1]) != cudaSuccess) return -1.f;
  return ms;
}

int audiokv_score(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, const void* k, float* scores,
                  audiokv_stream stream) {
  if (!q_win || !k || !scores) return AUDIOKV_EINVAL;
  if (!aligned16(q_win) || !aligned16(k)) return AUDIOKV_EALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  return do_score(ctx, q_win, k, scores, s, ctx->plan.lay.end);
}

int audiokv_smooth(audiokv_ctx* ctx, const audiokv_params* p, const float* scores, float* smoothed,
                   int32_t* kstar_or_null, audiokv_stream stream) {
  if (!scores || !smoothed) return AUDIOKV_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  return do_smooth(ctx, scores, smoothed, kstar_or_null, nullptr, nullptr, nullptr, s);
}

int audiokv_allocate(audiokv_ctx* ctx, const audiokv_params* p, const float* head_scores,
                     const int64_t* total_budget, int32_t* budgets, int32_t* cu_kept, audiokv_stream stream) {
  if (!head_scores || !total_budget || !budgets || !cu_kept) return AUDIOKV_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  return do_allocate(ctx, head_scores, total_budget, budgets, cu_kept, s);
}

int audiokv_select_gather(audiokv_ctx* ctx, const audiokv_params* p, const float* smoothed, const int32_t* budgets,
                          const int32_t* cu_kept, const void* k, const void* v, void* k_out, void* v_out,
                          int32_t* kept_idx, audiokv_stream stream) {
  if (!smoothed || !budgets || !cu_kept || !k || !v || !k_out || !v_out || !kept_idx) return AUDIOKV_EINVAL;
  if (!aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out)) return AUDIOKV_EALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  return do_select_gather(ctx, smoothed, budgets, cu_kept, k, v, k_out, v_out, kept_idx, s);
}

namespace {

// audiokv_evict; used: bytes at the front of the workspace that the caller needs, if more than the plan's.
int evict_pass(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, const void* k, const void* v,
               const float* head_scores, const int64_t* total_budget, void* k_out, void* v_out,
               int32_t* kept_idx, int32_t* budgets, int32_t* cu_kept, audiokv_stream stream, size_t used) {
  if (!q_win || !k || !v || !head_scores || !total_budget || !k_out || !v_out || !kept_idx || !budgets || !cu_kept)
    return AUDIOKV_EINVAL;
  if (!aligned16(q_win) || !aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out))
    return AUDIOKV_EALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  Plan& pl = ctx->plan;
  float* ws_scores = reinterpret_cast<float*>(ctx->ws + pl.lay.scores);
  int32_t* ws_kstar = reinterpret_cast<int32_t*>(ctx->ws + pl.lay.kstar);
  const ProfiledCall timed(ctx, s);
  // The budgets depend on nothing the GPU computes, and only the selection needs them. The allocation kernel waits for
  // everything earlier on the stream and then lets its dependents in; the first scoring sweep, a programmatic dependent, runs beside it and waits for it at its
  // own end, so that the smoothing and selection, two chained kernels later, find the budgets complete. With per-kernel
  // timing on, every kernel waits for the one before it.
  const bool beside = !ctx->prof.on;
  rc = do_allocate(ctx, head_scores, total_budget, budgets, cu_kept, s);
  if (!rc) rc = do_score(ctx, q_win, k, ws_scores, s, std::max(used, pl.lay.end), 0, -1, beside);
  if (rc) return rc;
  // the pooling variants hand their result to the selection through the score buffer itself
  float* ws_smoothed = pl.sh.smooth_mode >= AUDIOKV_SMOOTH_AVG_POOL ? ws_scores : nullptr;
  int64_t rows = 0;
  for (int r = 0; r < pl.sh.n_req; ++r) rows += total_budget[r];
  return do_smooth_gather(ctx, ws_scores, ws_smoothed, ws_kstar, budgets, cu_kept, kept_idx, k, v, k_out, v_out, rows, s);
}

}  // namespace

int audiokv_evict(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, const void* k, const void* v,
                  const float* head_scores, const int64_t* total_budget, void* k_out, void* v_out,
                  int32_t* kept_idx, int32_t* budgets, int32_t* cu_kept, audiokv_stream stream) {
  return evict_pass(ctx, p, q_win, k, v, head_scores, total_budget, k_out, v_out, kept_idx, budgets, cu_kept, stream, 0);
}

int audiokv_evict_kstar(audiokv_ctx* ctx, int32_t* kstar, audiokv_stream stream) {
  if (!ctx || !kstar) return AUDIOKV_EINVAL;
  if (!ctx->plan.valid || !ctx->plan_uploaded) return AUDIOKV_EINVAL;  // no pass has run on this context yet
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  e = cudaMemcpyAsync(kstar, ctx->ws + ctx->plan.lay.kstar, sizeof(int32_t) * ctx->plan.sh.total_heads,
                      cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

int audiokv_evict_budgeted(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, const void* k, const void* v,
                           const int32_t* budgets, void* k_out, void* v_out, int32_t* kept_idx, int32_t* cu_kept,
                           audiokv_stream stream) {
  if (!q_win || !k || !v || !budgets || !k_out || !v_out || !kept_idx || !cu_kept) return AUDIOKV_EINVAL;
  if (!aligned16(q_win) || !aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out))
    return AUDIOKV_EALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  Plan& pl = ctx->plan;
  float* ws_scores = reinterpret_cast<float*>(ctx->ws + pl.lay.scores);
  int32_t* ws_kstar = reinterpret_cast<int32_t*>(ctx->ws + pl.lay.kstar);
  int32_t* ws_budgets = reinterpret_cast<int32_t*>(ctx->ws + pl.lay.aux);  // the checked copy the selection reads
  const ProfiledCall timed(ctx, s);
  Launch ln{s, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_budget_prefix(pl.sh, d_reqs(ctx), budgets, ws_budgets, cu_kept, d_status(ctx), ln);
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  if ((rc = do_score(ctx, q_win, k, ws_scores, s, pl.lay.end, 0, -1, !ctx->prof.on))) return rc;
  float* ws_smoothed = pl.sh.smooth_mode >= AUDIOKV_SMOOTH_AVG_POOL ? ws_scores : nullptr;
  // only the device knows the budgets: a guess
  const int64_t rows = pl.scores_len / 3 + static_cast<int64_t>(pl.sh.total_heads) * pl.sh.window;
  return do_smooth_gather(ctx, ws_scores, ws_smoothed, ws_kstar, ws_budgets, cu_kept, kept_idx, k, v, k_out, v_out, rows, s);
}

namespace {

// The per-head problem of a re-eviction: every head of the compacted cache becomes a request of one layer and one
// KV head, with its own length, its own place in the packed cache and its own slice of the window queries.
int reevict_problem(ReevictArrays* a, const audiokv_params* p, const int32_t* cu_cache, const int32_t* new_budgets,
                    audiokv_params* dp) {
  if (!a || !p || !cu_cache) return AUDIOKV_EINVAL;
  if (p->n_layers < 1 || p->n_kv_heads < 1 || p->n_q_heads < 1 || p->n_q_heads % p->n_kv_heads || p->n_req < 1 ||
      p->head_dim < 1)
    return AUDIOKV_EINVAL;
  const int64_t TH = static_cast<int64_t>(p->n_req) * p->n_layers * p->n_kv_heads;
  if (TH > AUDIOKV_MAX_REQ) return AUDIOKV_EUNSUPPORTED;
  const int G = p->n_q_heads / p->n_kv_heads;
  a->len.resize(TH);
  a->kv_off.resize(TH);
  a->q_off.resize(TH);
  a->budget.resize(TH);
  if (cu_cache[0] != 0) return AUDIOKV_EINVAL;
  int64_t u = 0;
  for (int r = 0; r < p->n_req; ++r) {
    const int64_t q_r = p->q_req_offset ? p->q_req_offset[r] : r * p->q_stride_req;
    for (int l = 0; l < p->n_layers; ++l)
      for (int h = 0; h < p->n_kv_heads; ++h, ++u) {
        const int64_t n = static_cast<int64_t>(cu_cache[u + 1]) - cu_cache[u];
        if (n <= p->window || n > AUDIOKV_MAX_SEQ_LEN) return AUDIOKV_EINVAL;
        a->len[u] = static_cast<int32_t>(n);
        a->kv_off[u] = static_cast<int64_t>(cu_cache[u]) * p->head_dim;
        a->q_off[u] = q_r + l * p->q_stride_layer + static_cast<int64_t>(h) * G * p->q_stride_head;
        if (new_budgets) {
          if (new_budgets[u] < p->window || new_budgets[u] > n) return AUDIOKV_EINVAL;
          a->budget[u] = new_budgets[u];
        }
      }
  }
  *dp = *p;
  dp->n_req = static_cast<int32_t>(TH);
  dp->n_layers = 1;
  dp->n_kv_heads = 1;
  dp->n_q_heads = G;
  dp->seq_len = a->len.data();
  dp->q_stride_req = 0;
  dp->q_stride_layer = 0;
  dp->kv_stride_layer = 0;
  dp->kv_stride_head = 0;
  dp->kv_stride_tok = p->head_dim;
  dp->kv_req_offset = a->kv_off.data();
  dp->q_req_offset = a->q_off.data();
  dp->base_per_head = 0;
  dp->page_size = 0;  // the compacted cache is packed, not paged
  dp->n_pages = 0;
  dp->page_table = nullptr;
  dp->page_table_stride = 0;
  return AUDIOKV_OK;
}

}  // namespace

size_t audiokv_reevict_workspace_bytes(const audiokv_params* p, const int32_t* cu_cache) {
  ReevictArrays tmp;
  audiokv_params dp;
  if (reevict_problem(&tmp, p, cu_cache, nullptr, &dp)) return 0;
  return audiokv_workspace_bytes(&dp);
}

int audiokv_reevict(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, const void* k_cache,
                    const void* v_cache, const int32_t* cu_cache, const int32_t* new_budgets, void* k_out, void* v_out,
                    int32_t* kept_idx, int32_t* cu_kept, audiokv_stream stream) {
  if (!ctx || !new_budgets) return AUDIOKV_EINVAL;
  audiokv_params dp;
  int rc = reevict_problem(&ctx->re, p, cu_cache, new_budgets, &dp);
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if ((rc = prepare(ctx, &dp, s))) return rc;
  // One head per request: the allocation hands each its whole total, whatever the weight. The weights and the
  // per-head budgets it writes live in the workspace.
  const size_t TH = ctx->re.len.size();
  float* weights = reinterpret_cast<float*>(ctx->ws + ctx->plan.lay.aux);
  int32_t* budgets = reinterpret_cast<int32_t*>(weights + TH);
  cudaError_t e = cudaMemsetAsync(weights, 0x3f, sizeof(float) * TH, s);  // 0x3f3f3f3f = 0.747
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  return audiokv_evict(ctx, &dp, q_win, k_cache, v_cache, weights, ctx->re.budget.data(), k_out, v_out, kept_idx,
                       budgets, cu_kept, s);
}

int audiokv_hit_score(audiokv_ctx* ctx, const float* attn, int32_t n_steps, int32_t n_heads, int64_t row_stride,
                      const int32_t* row_len, const int32_t* span, int32_t top_k, int32_t* hit_counts, float* s_hit,
                      audiokv_stream stream) {
  if (!ctx || !attn || !row_len || !span || !hit_counts || !s_hit) return AUDIOKV_EINVAL;
  if (n_steps < 1 || n_heads < 1 || row_stride < 1 || top_k < 1 || top_k > 1024) return AUDIOKV_EINVAL;
  if (static_cast<int64_t>(n_steps) * n_heads > 0x7fffffffLL || ctx->ws_bytes < 64) return AUDIOKV_EINVAL;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return cuda_fail(ctx, e);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  Launch ln{s, &ctx->launches, &ctx->prof};
  e = launch_hit_score(attn, n_steps, n_heads, row_stride, row_len, span, top_k, hit_counts, s_hit, ln);
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

int audiokv_selection_spread(audiokv_ctx* ctx, const audiokv_params* p, const int32_t* kept_idx,
                             const int32_t* cu_kept, int32_t n_bins, int32_t* hist, float* stats,
                             audiokv_stream stream) {
  if (!kept_idx || !cu_kept || !hist || !stats) return AUDIOKV_EINVAL;
  if (n_bins < 1 || n_bins > 4096) return AUDIOKV_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s);
  if (rc) return rc;
  Launch ln{s, &ctx->launches, &ctx->prof};
  cudaError_t e = launch_selection_spread(ctx->plan.sh, d_reqs(ctx), kept_idx, cu_kept, n_bins, hist, stats,
                                          d_status(ctx), ln);
  return e == cudaSuccess ? AUDIOKV_OK : cuda_fail(ctx, e);
}

int audiokv_evict_host(audiokv_ctx* ctx, const audiokv_params* p, const void* q_win, int64_t q_elems, const void* k,
                       const void* v, int64_t kv_elems, const float* head_scores, const int64_t* total_budget,
                       void* k_out, void* v_out, int32_t* kept_idx, int32_t* budgets, int32_t* cu_kept,
                       audiokv_stream stream) {
  if (!q_win || !k || !v || !head_scores || !total_budget || !k_out || !v_out || !kept_idx || !budgets || !cu_kept)
    return AUDIOKV_EINVAL;
  if (p && p->page_size != 0) return AUDIOKV_EUNSUPPORTED;  // a page table is device data: use audiokv_evict
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = prepare(ctx, p, s, true);
  if (rc) return rc;
  Plan& pl = ctx->plan;
  if (q_elems < 0 || kv_elems < 0) return AUDIOKV_EINVAL;
  const HostStaging hs = host_staging(pl, q_elems, kv_elems, total_budget);
  if (hs.rows < 0) return AUDIOKV_EINVAL;
  if (hs.end > ctx->ws_bytes) return AUDIOKV_EWORKSPACE;
  const size_t es = esize(p->dtype);
  const int64_t rows = hs.rows;
  const int TH = pl.sh.total_heads;
  char *dq = ctx->ws + hs.q, *dk = ctx->ws + hs.k, *dv = ctx->ws + hs.v, *dS = ctx->ws + hs.head_scores;
  char *dko = ctx->ws + hs.k_out, *dvo = ctx->ws + hs.v_out, *dki = ctx->ws + hs.kept_idx, *db = ctx->ws + hs.budgets;
  char* dcu = ctx->ws + hs.cu_kept;
  cudaError_t e;
#define AKV_CP_ON(st, dst, src, n, kind) \
  if ((e = cudaMemcpyAsync(dst, src, n, kind, st)) != cudaSuccess) return cuda_fail(ctx, e)
#define AKV_CP(dst, src, n, kind) AKV_CP_ON(s, dst, src, n, kind)
  // One request whose K and V are laid out layer by layer, scored on the tensor cores: the pass runs in chunks of
  // layers, so that the copy of the next chunk's K and V (in), this chunk's kernels, and the copy of the previous
  // chunk's kept rows (out) overlap; in and out use the two directions of the link. Everything else: in, pass, out.
  const int NL = pl.sh.n_layers, Hkv = pl.sh.n_kv_heads;
  const bool layered = pl.sh.n_req == 1 && NL > 1 && score_umma_takes(pl.sh) && !ctx->prof.on &&
                       p->kv_stride_layer > 0 && kv_elems == static_cast<int64_t>(NL) * p->kv_stride_layer &&
                       p->kv_stride_layer >= p->kv_stride_tok * pl.reqs[0].L && p->kv_stride_layer >= p->kv_stride_head * Hkv;
  if (layered) {
    const int n_chunks = host_chunks(NL);
    int32_t* d_budgets = reinterpret_cast<int32_t*>(db);
    int32_t* d_cu = reinterpret_cast<int32_t*>(dcu);
    AKV_CP(dq, q_win, q_elems * es, cudaMemcpyHostToDevice);
    AKV_CP(dS, head_scores, sizeof(float) * TH, cudaMemcpyHostToDevice);
    if ((rc = do_allocate(ctx, reinterpret_cast<float*>(dS), total_budget, d_budgets, d_cu, s))) return rc;
    // the chunk boundaries of the output: the prefix sums come back first (a few hundred bytes)
    AKV_CP(budgets, db, sizeof(int32_t) * TH, cudaMemcpyDeviceToHost);
    AKV_CP(cu_kept, dcu, sizeof(int32_t) * (TH + 1), cudaMemcpyDeviceToHost);
    if ((e = cudaEventRecord(ctx->fork, s)) != cudaSuccess) return cuda_fail(ctx, e);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return cuda_fail(ctx, e);
    // the copy streams start behind everything the caller's stream holds so far (the workspace may be in use)
    if ((e = cudaStreamWaitEvent(ctx->side, ctx->fork, 0)) != cudaSuccess) return cuda_fail(ctx, e);
    if ((e = cudaStreamWaitEvent(ctx->out, ctx->fork, 0)) != cudaSuccess) return cuda_fail(ctx, e);
    float* ws_scores = reinterpret_cast<float*>(ctx->ws + pl.lay.scores);
    int32_t* ws_kstar = reinterpret_cast<int32_t*>(ctx->ws + pl.lay.kstar);
    float* ws_smoothed = pl.sh.smooth_mode >= AUDIOKV_SMOOTH_AVG_POOL ? ws_scores : nullptr;
    const size_t layer_bytes = static_cast<size_t>(p->kv_stride_layer) * es, row_bytes = static_cast<size_t>(p->head_dim) * es;
    // V is only ever read by the gather, and only its kept rows: when the caller's V is pinned memory the device can
    // address, the gather fetches those rows straight from it and the rest of V never crosses the link.
    const void* v_src = dv;
    {
      cudaPointerAttributes at{};
      if (cudaPointerGetAttributes(&at, v) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer &&
          aligned16(at.devicePointer))
        v_src = at.devicePointer;
      else
        cudaGetLastError();  // pageable memory is reported as an error by older drivers: not one of this call's
    }
    for (int c = 0; c < n_chunks; ++c) {
      const int l0 = host_chunk_layer(NL, c), l1 = host_chunk_layer(NL, c + 1);
      const size_t off = l0 * layer_bytes, len = (l1 - l0) * layer_bytes;
      AKV_CP_ON(ctx->side, dk + off, static_cast<const char*>(k) + off, len, cudaMemcpyHostToDevice);
      if (v_src == dv) AKV_CP_ON(ctx->side, dv + off, static_cast<const char*>(v) + off, len, cudaMemcpyHostToDevice);
      if ((e = cudaEventRecord(ctx->chunk_in[c], ctx->side)) != cudaSuccess) return cuda_fail(ctx, e);
      if ((e = cudaStreamWaitEvent(s, ctx->chunk_in[c], 0)) != cudaSuccess) return cuda_fail(ctx, e);
      const int u0 = l0 * Hkv, u1 = l1 * Hkv;
      if ((rc = do_score(ctx, dq, dk, ws_scores, s, hs.end, u0, u1))) return rc;
      if ((rc = do_smooth(ctx, ws_scores, ws_smoothed, ws_kstar, d_budgets, d_cu, reinterpret_cast<int32_t*>(dki), s, u0, u1)))
        return rc;
      if ((rc = do_gather(ctx, d_cu, reinterpret_cast<int32_t*>(dki), dk, v_src, dko, dvo, s, u0, u1))) return rc;
      if ((e = cudaEventRecord(ctx->chunk_done[c], s)) != cudaSuccess) return cuda_fail(ctx, e);
      if ((e = cudaStreamWaitEvent(ctx->out, ctx->chunk_done[c], 0)) != cudaSuccess) return cuda_fail(ctx, e);
      const size_t r0 = static_cast<size_t>(cu_kept[u0]), r1 = static_cast<size_t>(cu_kept[u1]);  // host copy, read above
      AKV_CP_ON(ctx->out, static_cast<char*>(k_out) + r0 * row_bytes, dko + r0 * row_bytes, (r1 - r0) * row_bytes,
                cudaMemcpyDeviceToHost);
      AKV_CP_ON(ctx->out, static_cast<char*>(v_out) + r0 * row_bytes, dvo + r0 * row_bytes, (r1 - r0) * row_bytes,
                cudaMemcpyDeviceToHost);
      AKV_CP_ON(ctx->out, reinterpret_cast<char*>(kept_idx) + r0 * sizeof(int32_t), dki + r0 * sizeof(int32_t),
                (r1 - r0) * sizeof(int32_t), cudaMemcpyDeviceToHost);
    }
    // the caller's stream ends behind the last copy out, then the host waits for it
    if ((e = cudaEventRecord(ctx->copies_out, ctx->out)) != cudaSuccess) return cuda_fail(ctx, e);
    if ((e = cudaStreamWaitEvent(s, ctx->copies_out, 0)) != cudaSuccess) return cuda_fail(ctx, e);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return cuda_fail(ctx, e);
    return AUDIOKV_OK;
  }
  AKV_CP(dq, q_win, q_elems * es, cudaMemcpyHostToDevice);
  AKV_CP(dk, k, kv_elems * es, cudaMemcpyHostToDevice);
  AKV_CP(dv, v, kv_elems * es, cudaMemcpyHostToDevice);
  AKV_CP(dS, head_scores, sizeof(float) * TH, cudaMemcpyHostToDevice);
  rc = evict_pass(ctx, p, dq, dk, dv, reinterpret_cast<float*>(dS), total_budget, dko, dvo, reinterpret_cast<int32_t*>(dki),
                  reinterpret_cast<int32_t*>(db), reinterpret_cast<int32_t*>(dcu), s, hs.end);
  if (rc) return rc;
  AKV_CP(k_out, dko, rows * p->head_dim * es, cudaMemcpyDeviceToHost);
  AKV_CP(v_out, dvo, rows * p->head_dim * es, cudaMemcpyDeviceToHost);
  AKV_CP(kept_idx, dki, rows * sizeof(int32_t), cudaMemcpyDeviceToHost);
  AKV_CP(budgets, db, sizeof(int32_t) * TH, cudaMemcpyDeviceToHost);
  AKV_CP(cu_kept, dcu, sizeof(int32_t) * (TH + 1), cudaMemcpyDeviceToHost);
#undef AKV_CP
#undef AKV_CP_ON
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return cuda_fail(ctx, e);
  return AUDIOKV_OK;
}

}  // extern "C"

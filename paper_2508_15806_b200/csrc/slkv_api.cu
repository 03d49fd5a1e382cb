// extern "C" entry points of libslkv: argument validation, workspace carve-up, launch sequencing.
// No step of the method runs here; every step is a kernel in the other translation units.
#include <atomic>
#include <cstring>
#include <mutex>
#include <vector>

#include "slkv_internal.cuh"

namespace slkv {
namespace {

thread_local int g_last_cuda_error = 0;
thread_local int g_last_launches = 0;
thread_local int g_expire_next_layer_wait = 0;

// ---- per-kernel timing (off by default) -----------------------------------------------------------
struct TimedLaunch { int kid; cudaEvent_t a, b; };
thread_local int g_prof_on = 0;          // 0 off, 1 every kernel, 2 the score kernels only
thread_local std::vector<TimedLaunch>* g_prof = nullptr;      // records of the current thread
thread_local std::vector<cudaEvent_t>* g_prof_free = nullptr;

cudaEvent_t prof_event() {
  if (g_prof_free && !g_prof_free->empty()) {
    cudaEvent_t e = g_prof_free->back();
    g_prof_free->pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

constexpr int kMaxWindow = 256;

int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return SLKV_ERR_CUDA;
}

struct Layout {
  size_t hist_off, tile_off, pooled, sync, total;
  size_t layer0, layer_bytes;                  // per-layer part: layer i's begins at layer0 + i * layer_bytes
  size_t vote, part, gather_src, win_m, win_z; // ... with these in it
};

// Validates p and cu_seqlens_host and fills the host-known fields of `pb`.
int describe(const slkv_params* p, const int32_t* cu_host, Problem* pb) {
  if (!p || !cu_host) return SLKV_ERR_NULL_PTR;
  if (p->dtype != SLKV_F32 && p->dtype != SLKV_BF16) return SLKV_ERR_BAD_DTYPE;
  if (p->pool_mode != SLKV_POOL_MAX && p->pool_mode != SLKV_POOL_AVG) return SLKV_ERR_BAD_DTYPE;
  if (p->softmax_domain != SLKV_HISTORY && p->softmax_domain != SLKV_ALL_CAUSAL) return SLKV_ERR_BAD_DTYPE;
  if (p->lse_units != SLKV_LSE_LN && p->lse_units != SLKV_LSE_LOG2) return SLKV_ERR_BAD_DTYPE;
  if (p->history_only != 0 && p->history_only != 1) return SLKV_ERR_BAD_DTYPE;
  if (p->history_only && p->n_seqs != 1) return SLKV_ERR_BAD_SHAPE;
  if (p->score_path < SLKV_PATH_AUTO || p->score_path > SLKV_PATH_TENSOR) return SLKV_ERR_BAD_DTYPE;
  if (p->n_seqs < 1 || p->n_seqs > (1 << 20)) return SLKV_ERR_BAD_SHAPE;
  if (p->n_kv_heads < 1 || p->n_kv_heads > 65535 || p->n_q_heads < p->n_kv_heads ||
      p->n_q_heads % p->n_kv_heads != 0)
    return SLKV_ERR_BAD_SHAPE;
  if (p->head_dim != 64 && p->head_dim != 128) return SLKV_ERR_BAD_SHAPE;
  if (p->window < 1 || p->window > kMaxWindow) return SLKV_ERR_BAD_SHAPE;
  if (p->pool_kernel < 1 || p->pool_kernel % 2 == 0 || p->pool_kernel > 1025) return SLKV_ERR_BAD_SHAPE;
  const int elem = p->dtype == SLKV_F32 ? 4 : 2;
  const int64_t row = p->head_dim;
  if (p->k_stride_head < row || p->v_stride_head < row || p->q_stride_head < row ||
      p->k_stride_tok < row || p->v_stride_tok < row || p->q_stride_row < row || p->q_stride_seq < row)
    return SLKV_ERR_BAD_SHAPE;
  const int64_t strides[] = {p->k_stride_tok, p->k_stride_head, p->v_stride_tok, p->v_stride_head,
                             p->q_stride_seq, p->q_stride_row, p->q_stride_head};
  for (int64_t s : strides)
    if ((s * elem) % 16 != 0) return SLKV_ERR_BAD_ALIGN;
  if (cu_host[0] != 0) return SLKV_ERR_BAD_SHAPE;
  // History rows only: the kernels are told about a sequence of rows + window tokens whose last `window` rows they
  // never read (the window rows are only ever read as keys by the all-causal window statistics, which such a call
  // does not run); the K tensor map still ends at the rows that exist.
  const int64_t rows_given = cu_host[p->n_seqs];
  if (p->history_only && (cu_host[1] < 0 || (int64_t)cu_host[1] + p->window >= (1ll << 31))) return SLKV_ERR_BAD_SHAPE;
  const int32_t cu_virtual[2] = {0, p->history_only ? cu_host[1] + p->window : 0};
  if (p->history_only) cu_host = cu_virtual;
  int64_t total_hist = 0, tiles = 0;
  int max_hist = 0;
  for (int s = 0; s < p->n_seqs; ++s) {
    int64_t len = (int64_t)cu_host[s + 1] - cu_host[s];
    if (len < 0) return SLKV_ERR_BAD_SHAPE;
    int64_t nh = len > p->window ? len - p->window : 0;
    total_hist += nh;
    tiles += (nh + 127) / 128;
    if (nh > max_hist) max_hist = (int)nh;
  }
  const int64_t T = cu_host[p->n_seqs];
  if ((int64_t)p->n_kv_heads * T >= (1ll << 31)) return SLKV_ERR_BAD_SHAPE;
  std::memset(pb, 0, sizeof(*pb));
  pb->p = *p;
  pb->G = p->n_q_heads / p->n_kv_heads;
  pb->R = pb->G * p->window;
  pb->elem = elem;
  pb->max_hist = max_hist;
  pb->total_tokens = rows_given;
  if (p->history_only) {
    pb->p.softmax_domain = SLKV_HISTORY;
    pb->cu_virtual[0] = cu_virtual[0]; pb->cu_virtual[1] = cu_virtual[1];
  }
  pb->total_hist = total_hist;
  pb->n_tiles128 = tiles * p->n_kv_heads;
  pb->n_seg = p->n_seqs * p->n_kv_heads;
  if (p->n_seqs <= kInlineSeqs) {
    pb->tab.n_inline = p->n_seqs;
    long long hacc = 0;
    int tacc = 0;
    for (int s = 0; s <= p->n_seqs; ++s) {
      pb->tab.cu[s] = cu_host[s];
      pb->tab.hist_off[s] = hacc;
      pb->tab.tile_off[s] = tacc;
      if (s < p->n_seqs) {
        long long nh = (long long)cu_host[s + 1] - cu_host[s] - p->window;
        if (nh < 0) nh = 0;
        hacc += nh;
        tacc += (int)((nh + 127) / 128);
      }
    }
  }
  if (pb->n_seg > 65535 * 16) return SLKV_ERR_BAD_SHAPE;
  if (pb->R > 1024) return SLKV_ERR_BAD_SHAPE;
  return SLKV_OK;
}

// Overlapped calls are launched as lists where the tensor-core score kernel and a list selection take the shape.
bool list_supported(const Problem& pb) {
  return tensor_path_supported(pb.p) && pb.p.score_path != SLKV_PATH_SIMT && pb.tab.n_inline > 0 && pb.max_hist > 0 &&
         (select_list_supported(pb) || select_cluster_supported(pb));
}

// Layers of a list.  A list costs some 23 us beside its layers (pipeline fill and tail, selections and gathers that nothing
// runs beside), and its layers wait for the last of them to be called: it goes out when it holds about 0.4 ms of work, 32768
// products of 128 keys x 128 rows, or eight layers (with two passes over them; with log-sum-exps handed in, one pass, half as long).  Steps
// of 32 layers, both passes, us in a row / by themselves from an idle GPU, with 32, 16, 8 and 4 layers to a list:
//   4001 tokens, 128 rows    132 / 197    154 / 191    202 / 228    329 / 348
//   32768 tokens, 128 rows   734 / 879    756 / 889    804 / 887    946 / 1017
//   131072 tokens, 256 rows  5175 / 5717  5147 / 5690  5130 / 5697  5101 / 5746
// At 32768 tokens 32 layers to a list would be 1-3 % quicker than the 16 of the rule, for twice the workspace.  Lists that go with one
// product (slkv_bound.cu) were not measured at other lengths.
constexpr int64_t kListProducts = 32768;
constexpr int kListMinLayers = 8;      // four: eight ragged sequences of 147k tokens, held, 6504 -> 6696 us
int list_layers(const Problem& pb) {
  const int64_t per_layer = pb.n_tiles128 * ((pb.R + 127) / 128);
  const int64_t n = per_layer > 0 ? (kListProducts + per_layer - 1) / per_layer : kListMaxLayers;
  return n < kListMinLayers ? kListMinLayers : (n > kListMaxLayers ? kListMaxLayers : (int)n);
}

Layout layout_of(const Problem& pb, bool overlapped = false) {
  Layout L;
  size_t o = 0;
  L.hist_off = o; o = align_up(o + (size_t)(pb.p.n_seqs + 1) * sizeof(int64_t));
  L.tile_off = o; o = align_up(o + (size_t)(pb.p.n_seqs + 1) * sizeof(int32_t));
  const size_t votes = (size_t)pb.p.n_kv_heads * (size_t)pb.total_hist * sizeof(float);
  L.pooled = o; o = align_up(o + votes);
  L.sync = o; o = align_up(o + kSyncBytes);
  // Every layer of a list has its own votes, row statistics and source-row list; ordinary calls use the first.
  L.layer0 = o;
  size_t q = 0;
  L.vote = q; q = align_up(q + votes);
  // row statistics: StatView (tensor cores), SimtStats
  const size_t shares = (size_t)tensor_slot_stride(pb);
  const size_t by_tensor = (size_t)pb.n_seg * ((shares * 8 + 12) * (size_t)pb.R + kMaxSplit / 8);
  const size_t by_simt = simt_part_bytes(pb);
  L.part = q; q = align_up(q + (by_tensor > by_simt ? by_tensor : by_simt));
  L.gather_src = q; q = align_up(q + (size_t)pb.p.n_kv_heads * (size_t)pb.total_tokens * sizeof(int32_t));
  // row statistics over the window keys (all-causal softmax domain): [n_seg][R] maxima and sums
  const size_t wins = (size_t)pb.n_seg * pb.R * sizeof(float);
  L.win_m = q; q = align_up(q + wins);
  L.win_z = q; q = align_up(q + wins);
  L.layer_bytes = q;
  L.total = o + q * (size_t)(overlapped && list_supported(pb) ? list_layers(pb) : 1);
  return L;
}

// Picks the score path; SLKV_ERR_* when the requested one cannot take the shape.
int resolve_path(const Problem& pb, int* path) {
  int want = pb.p.score_path;
  const bool tensor_ok = tensor_path_supported(pb.p);
  if (want == SLKV_PATH_AUTO) want = tensor_ok ? SLKV_PATH_TENSOR : SLKV_PATH_SIMT;
  if (want == SLKV_PATH_TENSOR && !tensor_ok) return SLKV_ERR_BAD_DTYPE;
  *path = want;
  return SLKV_OK;
}

// slot: the layer's place in the list (overlapped calls)
void carve(Problem* pb, const Layout& L, void* ws, int slot) {
  unsigned char* b = static_cast<unsigned char*>(ws);
  pb->hist_off = reinterpret_cast<int64_t*>(b + L.hist_off);
  pb->tile_off = reinterpret_cast<int32_t*>(b + L.tile_off);
  pb->tab.tile_ptr = pb->tile_off;
  pb->tab.hist_ptr = reinterpret_cast<const long long*>(pb->hist_off);
  pb->pooled_ws = reinterpret_cast<float*>(b + L.pooled);
  pb->sync = reinterpret_cast<unsigned long long*>(b + L.sync);
  unsigned char* l = b + L.layer0 + (size_t)slot * L.layer_bytes;
  pb->vote = reinterpret_cast<float*>(l + L.vote);
  pb->part = l + L.part;
  pb->gather_src = reinterpret_cast<int32_t*>(l + L.gather_src);
  pb->win_m = reinterpret_cast<float*>(l + L.win_m);
  pb->win_z = reinterpret_cast<float*>(l + L.win_z);
}
int bind_workspace(Problem* pb, void* ws, size_t ws_bytes) {
  if (!ws) return SLKV_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % kAlign != 0) return SLKV_ERR_BAD_ALIGN;
  const Layout L = layout_of(*pb);
  if (ws_bytes < L.total) return SLKV_ERR_WORKSPACE;
  carve(pb, L, ws, 0);
  return SLKV_OK;
}

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// The window keys' row statistics, where the softmax runs over all causally visible keys and the caller has not
// supplied the rows' log-sum-exp (Eq. 3-4 over the prefill attention's own key set).
int enqueue_window_stats(const Problem& pb, int path, cudaStream_t st, int* launches) {
  if (pb.lse_opt || pb.p.softmax_domain != SLKV_ALL_CAUSAL) return SLKV_OK;
  cudaError_t e = launch_window_stats(pb, path == SLKV_PATH_TENSOR && tensor_q_head_inner(pb.p), st, launches);
  if (e != cudaSuccess) return cuda_fail(e);
  return SLKV_OK;
}

// window votes of every history key (device pointers resolved); with the caller's row statistics the vote pass alone
int enqueue_votes(const Problem& pb, int path, const int32_t* cu_host, int32_t* status, cudaStream_t st,
                  int* launches) {
  int rc = enqueue_window_stats(pb, path, st, launches);
  if (rc != SLKV_OK) return rc;
  const int passes = pb.lse_opt ? 2 : 3;
  cudaError_t e = path == SLKV_PATH_TENSOR ? launch_score_tensor(pb, cu_host, status, passes == 3 && bound_shape(pb) ? kScoreWide : passes, nullptr, false, st, launches)
                                           : launch_score_simt(pb, status, passes, st, launches);
  if (e != cudaSuccess) return cuda_fail(e);
  return SLKV_OK;
}

// CTAs per segment where one launch does the whole layer, else 0.  A wait for words in memory that is to run out
// (slkv_debug_expire_next_wait) is one of the other kernels'.
int layer_cluster(const Problem& pb, int path, bool select) {
  if (next_wait_expires()) return 0;
  return path == SLKV_PATH_TENSOR ? layer_tc_cluster(pb, select) : layer_fma_cluster(pb, select);
}
cudaError_t launch_layer(const Problem& pb, int path, int cs, const TailLayer* tail, float* pooled, int32_t* status, cudaStream_t st,
                         int* launches) {
  return path == SLKV_PATH_TENSOR ? launch_layer_tc(pb, cs, tail, pooled, status, st, launches)
                                  : launch_layer_fma(pb, cs, tail, pooled, status, st, launches);
}

// ---- overlapped calls ---------------------------------------------------------------------------------------
// A call queues its layer; a list of layers goes out as three launches on the caller's stream -- scores, selections,
// gathers, each over all layers of the list -- when it is full (list_layers) or at a join.  What a list gives over single calls: the
// statistics of one layer overlap the votes of another, all layers' selections fill the SMs side by side, and the host
// makes three launches instead of 48.
struct ListState {
  bool open = false;             // the shape below is valid
  slkv_params p;
  std::vector<int32_t> cu_host;
  const int32_t* cu_dev = nullptr;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  bool with_lse = false;
  Problem pb;                    // of the shape; the per-layer pointers are set call by call
  Layout layout;
  ScorePlan plan;
  int n = 0, n_max = 0;          // layers queued; those a list goes out at
  ScoreLayer score[kListMaxLayers];
  TailLayer tail[kListMaxLayers];
  bool in_flight = false;        // lists have gone out since this stream's last join
  cudaEvent_t event = nullptr;   // orders another stream behind this one
};
// One state per (device, caller's stream): calls made on different streams (by different host threads, or by one)
// never share a queue, so each stream's calls keep their own order whatever the others do.
constexpr int kMaxDevices = 64;
constexpr int kStatesPerDevice = 8;
struct DeviceStates {
  ListState st[kStatesPerDevice];
  cudaStream_t owner[kStatesPerDevice] = {};
  bool used[kStatesPerDevice] = {};
  unsigned long long last_use[kStatesPerDevice] = {};
  unsigned long long tick = 0;
};
DeviceStates* g_lists[kMaxDevices] = {};
std::mutex g_lists_mu;

// The queued layers of a state go out on its stream (g_lists_mu held).
cudaError_t flush_list(ListState* s, cudaStream_t owner, int* launches) {
  if (s->n == 0) return cudaSuccess;
  const int n = s->n;
  s->n = 0;
  s->in_flight = true;
  cudaError_t e;
  const bool bound = !s->with_lse && bound_list_supported(s->pb, s->tail, n);
  bool pooled = false;
  for (int i = 0; i < n; ++i) pooled = pooled || s->tail[i].pooled_out != nullptr;
  if (bound && !pooled) {
    e = launch_bound_list(s->pb, s->plan.sh, s->score, s->tail, n, owner, launches);
    if (e == cudaSuccess) e = launch_gather(s->pb, s->tail, n, owner, launches);
    if (e != cudaErrorNotSupported) return e;
  }
  e = launch_score_list(s->plan.sh, s->score, n, s->with_lse ? 2 : bound || bound_shape(s->pb) ? kScoreWide : 3, s->pb.sync, owner, launches);
  if (e == cudaSuccess)
    e = select_list_supported(s->pb) ? launch_select_list(s->pb, s->tail, n, owner, launches)
                                     : launch_select_cluster(s->pb, s->tail, n, owner, launches);
  if (e == cudaSuccess) e = launch_gather(s->pb, s->tail, n, owner, launches);
  return e;
}

// Orders `st` behind everything of a state that has gone out.
cudaError_t order_behind(ListState* s, cudaStream_t owner, cudaStream_t st) {
  if (!s->in_flight || owner == st) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  if (!s->event) e = cudaEventCreateWithFlags(&s->event, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(s->event, owner);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(st, s->event, 0);
  return e;
}

cudaError_t device_states(DeviceStates** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!g_lists[dev]) g_lists[dev] = new DeviceStates();
  *out = g_lists[dev];
  return cudaSuccess;
}

// The state of overlapped calls made on `st` on the current device (g_lists_mu held).  All eight in use by other
// streams: the one used longest ago is handed over once its queued layers have gone out on its own stream.
cudaError_t list_state(cudaStream_t st, ListState** out, DeviceStates** states, int* launches) {
  DeviceStates* d = nullptr;
  cudaError_t e = device_states(&d);
  if (e != cudaSuccess) return e;
  *states = d;
  int idx = -1;
  for (int i = 0; i < kStatesPerDevice; ++i)
    if (d->used[i] && d->owner[i] == st) idx = i;
  if (idx < 0) {
    for (int i = 0; i < kStatesPerDevice && idx < 0; ++i)
      if (!d->used[i]) idx = i;
    if (idx < 0) {
      int oldest = 0, oldest_idle = -1;
      for (int i = 0; i < kStatesPerDevice; ++i) {
        if (d->last_use[i] < d->last_use[oldest]) oldest = i;
        if (d->st[i].n == 0 && !d->st[i].in_flight && (oldest_idle < 0 || d->last_use[i] < d->last_use[oldest_idle])) oldest_idle = i;
      }
      idx = oldest_idle >= 0 ? oldest_idle : oldest;
      e = flush_list(&d->st[idx], d->owner[idx], launches);
      // a later join on any stream must still cover these calls: the stream that takes the state over stands for them
      if (e == cudaSuccess) e = order_behind(&d->st[idx], d->owner[idx], st);
      if (e != cudaSuccess) return e;
      d->st[idx].open = false;
    }
    d->used[idx] = true;
    d->owner[idx] = st;
  }
  d->last_use[idx] = ++d->tick;
  *out = &d->st[idx];
  return cudaSuccess;
}

// Calls on other streams whose workspace overlaps [ws, ws + bytes): their queued layers go out and `st` waits for what
// they have in flight, before a call on `st` carves that memory up for itself (g_lists_mu held).
cudaError_t drain_states_sharing(DeviceStates* d, const ListState* mine, const void* ws, size_t bytes, cudaStream_t st,
                                 int* launches) {
  const char* lo = static_cast<const char*>(ws);
  for (int i = 0; i < kStatesPerDevice; ++i) {
    ListState& s = d->st[i];
    if (!d->used[i] || &s == mine || !s.ws || (s.n == 0 && !s.in_flight)) continue;
    const char* olo = static_cast<const char*>(s.ws);
    if (olo + s.ws_bytes <= lo || lo + bytes <= olo) continue;
    cudaError_t e = flush_list(&s, d->owner[i], launches);
    if (e == cudaSuccess) e = order_behind(&s, d->owner[i], st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Sends out what is queued on this device and makes `st` wait for every overlapped call still in flight, whatever
// stream it was made on (no host wait).  Only the calls made on `st` itself are then forgotten: the others stay in
// flight for a join on their own stream, which still has to be ordered behind them.
cudaError_t join_lists(cudaStream_t st, int* launches) {
  std::lock_guard<std::mutex> lock(g_lists_mu);
  DeviceStates* d = nullptr;
  cudaError_t e = device_states(&d);
  if (e != cudaSuccess) return e == cudaErrorInvalidDevice ? cudaSuccess : e;
  for (int i = 0; i < kStatesPerDevice; ++i) {
    if (!d->used[i]) continue;
    ListState& s = d->st[i];
    e = flush_list(&s, d->owner[i], launches);
    if (e == cudaSuccess) e = order_behind(&s, d->owner[i], st);
    if (e != cudaSuccess) return e;
    if (d->owner[i] == st) s.in_flight = false;
  }
  return cudaSuccess;
}

// Workspace of the context-parallel packing: totals per head and counts per slice and head (above, equal), source rows
// of the packed rows.
struct CpWorkspace {
  int32_t *totals, *cnt_gt, *cnt_eq, *gather_src;
  size_t bytes;
  CpWorkspace(void* ws, int32_t n_kv_heads, int32_t own_count, int64_t capacity) {
    const size_t heads = 2 * align_up((size_t)n_kv_heads * sizeof(int32_t));
    const size_t slices = align_up((size_t)cp_slices(own_count) * (size_t)n_kv_heads * sizeof(int32_t));
    char* w = static_cast<char*>(ws);
    totals = reinterpret_cast<int32_t*>(w);
    cnt_gt = reinterpret_cast<int32_t*>(w + heads);
    cnt_eq = reinterpret_cast<int32_t*>(w + heads + slices);
    gather_src = reinterpret_cast<int32_t*>(w + heads + 2 * slices);
    bytes = heads + 2 * slices + align_up((size_t)capacity * sizeof(int32_t));
  }
};

TailLayer tail_of(const Problem& pb, const int32_t* budgets, void* k_out, void* v_out, int64_t capacity, int32_t* offsets,
                  int32_t* kept_idx, float* pooled_opt, int32_t* status) {
  TailLayer t;
  t.vote = pb.vote; t.budgets = budgets; t.offsets = offsets; t.kept_idx = kept_idx; t.gather_src = pb.gather_src;
  t.pooled_out = pooled_opt; t.status = status; t.k = pb.k; t.v = pb.v; t.k_out = k_out; t.v_out = v_out;
  t.kept_copy = t.offsets_copy = nullptr;
  t.capacity = capacity;
  return t;
}

int compress_impl(const slkv_params* p, const void* q_win, const void* k, const void* v, const int32_t* cu_dev,
                  const int32_t* cu_host, const int32_t* budgets, const float* lse_opt, void* k_out, void* v_out,
                  int64_t capacity, int32_t* offsets, int32_t* kept_idx, float* pooled_opt, int32_t* status, void* ws,
                  size_t ws_bytes, cudaStream_t st, bool overlapped = false, int32_t* kept_copy = nullptr,
                  int32_t* offsets_copy = nullptr) {
  g_last_launches = 0;
  if (!q_win || !k || !v || !cu_dev || !budgets || !k_out || !v_out || !offsets || !kept_idx)
    return SLKV_ERR_NULL_PTR;
  int launches = 0;
  if (overlapped && p && cu_host && ws) {
    // the shape of the calls before this one: everything that depends on it alone is there already
    std::lock_guard<std::mutex> lock(g_lists_mu);
    ListState* s = nullptr;
    DeviceStates* d = nullptr;
    cudaError_t e = list_state(st, &s, &d, &launches);
    if (e != cudaSuccess) overlapped = false;                // the ordinary path reports it, behind bad arguments
    const bool with_lse = lse_opt != nullptr;
    const bool same = overlapped && s->open && s->ws == ws && s->ws_bytes == ws_bytes && s->with_lse == with_lse && s->cu_dev == cu_dev &&
                      std::memcmp(&s->p, p, sizeof(*p)) == 0 &&
                      std::memcmp(s->cu_host.data(), cu_host, s->cu_host.size() * sizeof(int32_t)) == 0;
    if (overlapped && !same) {
      Problem pb;
      int rc = describe(p, cu_host, &pb);
      if (rc != SLKV_OK) return rc;
      if (p->history_only) return SLKV_ERR_BAD_SHAPE;        // nothing to append behind the selected rows
      int path = 0;
      rc = resolve_path(pb, &path);
      if (rc != SLKV_OK) return rc;
      overlapped = path == SLKV_PATH_TENSOR && list_supported(pb);
      if (overlapped) {
        if (reinterpret_cast<uintptr_t>(ws) % kAlign != 0) return SLKV_ERR_BAD_ALIGN;
        const Layout L = layout_of(pb, true);
        if (ws_bytes < L.total) return SLKV_ERR_WORKSPACE;
        e = flush_list(s, st, &launches);                    // layers of the shape before
        if (e != cudaSuccess) return cuda_fail(e);
        s->open = false;
        carve(&pb, L, ws, 0);
        pb.cu = cu_dev; pb.tab.cu_ptr = cu_dev;
        pb.q = q_win; pb.k = k; pb.v = v; pb.lse_opt = lse_opt;
        e = plan_score_tensor(pb, cu_host, status, &s->plan);
        if (e != cudaSuccess) return cuda_fail(e);
        s->p = *p; s->cu_host.assign(cu_host, cu_host + p->n_seqs + 1); s->cu_dev = cu_dev;
        s->ws = ws; s->ws_bytes = ws_bytes; s->with_lse = with_lse; s->pb = pb; s->layout = L;
        s->n_max = list_layers(pb);
        s->open = true;
      }
    }
    if (overlapped) {
      if (capacity < 0) return SLKV_ERR_CAPACITY;
      if (!aligned16(q_win) || !aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out))
        return SLKV_ERR_BAD_ALIGN;
      e = drain_states_sharing(d, s, ws, ws_bytes, st, &launches);
      if (e != cudaSuccess) return cuda_fail(e);
      Problem& pb = s->pb;
      carve(&pb, s->layout, ws, s->n);
      pb.q = q_win; pb.k = k; pb.v = v; pb.lse_opt = lse_opt;
      e = plan_score_layer(pb, status, &s->score[s->n]);
      if (e != cudaSuccess) return cuda_fail(e);
      const int rc = enqueue_window_stats(pb, SLKV_PATH_TENSOR, st, &launches);
      if (rc != SLKV_OK) return rc;
      s->tail[s->n] = tail_of(pb, budgets, k_out, v_out, capacity, offsets, kept_idx, pooled_opt, status);
      if (++s->n == s->n_max) {
        e = flush_list(s, st, &launches);
        if (e != cudaSuccess) return cuda_fail(e);
      }
      g_last_launches = launches;
      return SLKV_OK;
    }
  }
  // an ordinary call (or a shape that is not taken as a list): on the caller's stream, after whatever overlapped calls
  // are still in flight
  Problem pb;
  int rc = describe(p, cu_host, &pb);
  if (rc != SLKV_OK) return rc;
  if (p->history_only) return SLKV_ERR_BAD_SHAPE;            // nothing to append behind the selected rows
  if (capacity < 0) return SLKV_ERR_CAPACITY;
  if (!aligned16(q_win) || !aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out))
    return SLKV_ERR_BAD_ALIGN;
  int path = 0;
  rc = resolve_path(pb, &path);
  if (rc != SLKV_OK) return rc;
  rc = bind_workspace(&pb, ws, ws_bytes);
  if (rc != SLKV_OK) return rc;
  cudaError_t e = join_lists(st, &launches);
  if (e != cudaSuccess) return cuda_fail(e);
  pb.cu = cu_dev; pb.q = q_win; pb.k = k; pb.v = v;
  pb.tab.cu_ptr = cu_dev;
  pb.lse_opt = lse_opt;
  TailLayer tail = tail_of(pb, budgets, k_out, v_out, capacity, offsets, kept_idx, pooled_opt, status);
  // One launch for the whole layer where that is quicker.  With pooled_opt the call takes the general path, launch by launch:
  // that is a caller who looks into the steps, and how the two are held against each other on the same inputs.
  if (const int cs = !kept_copy && !offsets_copy && !pooled_opt ? layer_cluster(pb, path, true) : 0) {
    e = launch_layer(pb, path, cs, &tail, nullptr, status, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
    g_last_launches = launches;
    return SLKV_OK;
  }
  const bool one_kernel = select_list_supported(pb) || select_cluster_supported(pb);
  if (!one_kernel || pb.tab.n_inline == 0) {       // tables in global memory and / or the packed offsets
    e = launch_setup(pb, one_kernel ? nullptr : budgets, offsets, capacity, status, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  rc = enqueue_votes(pb, path, cu_host, status, st, &launches);
  if (rc != SLKV_OK) return rc;
  tail.kept_copy = kept_copy;
  tail.offsets_copy = offsets_copy;
  if (one_kernel) {
    // pooling, offsets and selection in one kernel
    e = select_list_supported(pb) ? launch_select_list(pb, &tail, 1, st, &launches)
                                  : launch_select_cluster(pb, &tail, 1, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
  } else {
    float* pooled = pooled_opt ? pooled_opt : pb.pooled_ws;
    e = launch_pool(pb, pooled, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
    e = launch_select(pb, pooled, budgets, offsets, kept_idx, capacity, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  e = launch_gather(pb, &tail, 1, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e);
  g_last_launches = launches;
  return SLKV_OK;
}

}  // namespace

// Launch number times an odd constant: none looks like a small number or an address, which workspaces are full of, and in
// 2^40 - 1 launches none comes twice and none is zero, in the low 40 bits either.
unsigned long long next_launch_tag() {
  static std::atomic<unsigned long long> launches{0};
  unsigned long long n;
  do n = launches.fetch_add(1, std::memory_order_relaxed) + 1; while ((n & ((1ull << 40) - 1)) == 0);
  return n * 0x9E3779B97F4A7C15ull;
}

void expire_next_layer_wait(int on) { g_expire_next_layer_wait = on; }
int take_expire_next_layer_wait(bool sums) {
  const int v = g_expire_next_layer_wait;
  if (v == 1 && !sums) return 0;
  g_expire_next_layer_wait = 0;
  return v;
}

LaunchScope::LaunchScope(int kid, cudaStream_t st, int* launches) : kid_(kid), st_(st), slot_(-1) {
  ++*launches;
  if (!g_prof_on) return;
  const bool score_kid = kid == KID_SCORE_LSE || kid == KID_SCORE_VOTE || kid == KID_SCORE_FUSED || kid == KID_SCORE_LIST || kid == KID_SCORE_BOUND;
  if (g_prof_on == 2 && !score_kid) return;
  if (!g_prof) g_prof = new std::vector<TimedLaunch>();
  TimedLaunch t{kid, prof_event(), prof_event()};
  if (!t.a || !t.b) return;
  cudaEventRecord(t.a, st);
  g_prof->push_back(t);
  slot_ = (int)g_prof->size() - 1;
}
LaunchScope::~LaunchScope() {
  if (slot_ >= 0) cudaEventRecord((*g_prof)[slot_].b, st_);
}

}  // namespace slkv

using namespace slkv;

extern "C" {

const char* slkv_strerror(int status) {
  switch (status) {
    case SLKV_OK: return "SLKV_OK";
    case SLKV_ERR_NULL_PTR: return "SLKV_ERR_NULL_PTR: a required pointer is NULL";
    case SLKV_ERR_BAD_SHAPE: return "SLKV_ERR_BAD_SHAPE: size, count or stride out of range";
    case SLKV_ERR_BAD_DTYPE: return "SLKV_ERR_BAD_DTYPE: unknown or unsupported dtype / mode / path";
    case SLKV_ERR_BAD_ALIGN: return "SLKV_ERR_BAD_ALIGN: pointer or stride not 16-byte aligned";
    case SLKV_ERR_BUDGET_SUM: return "SLKV_ERR_BUDGET_SUM: total smaller than heads * fixed";
    case SLKV_ERR_NEG_INF_SC: return "SLKV_ERR_NEG_INF_SC: INF_sc negative or not finite";
    case SLKV_ERR_CAPACITY: return "SLKV_ERR_CAPACITY: packed output capacity too small";
    case SLKV_ERR_WORKSPACE: return "SLKV_ERR_WORKSPACE: workspace missing or too small";
    case SLKV_ERR_CUDA: return "SLKV_ERR_CUDA: a CUDA runtime call failed";
    case SLKV_ERR_DEVICE_TIMEOUT: return "SLKV_ERR_DEVICE_TIMEOUT: a bounded device-side wait ran out";
    default: return "unknown slkv status";
  }
}

int slkv_profile_enable(int on) {
  g_prof_on = on < 0 ? 0 : (on > 2 ? 1 : on);
  return SLKV_OK;
}

int slkv_profile_collect(float* total_ms, int32_t* launches, int32_t n_kernels) {
  if (!total_ms || !launches) return SLKV_ERR_NULL_PTR;
  for (int i = 0; i < n_kernels; ++i) { total_ms[i] = 0.f; launches[i] = 0; }
  if (!g_prof) return SLKV_OK;
  if (!g_prof_free) g_prof_free = new std::vector<cudaEvent_t>();
  int rc = SLKV_OK;
  for (TimedLaunch& t : *g_prof) {
    float ms = 0.f;
    cudaError_t e = cudaEventSynchronize(t.b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, t.a, t.b);
    if (e != cudaSuccess) rc = cuda_fail(e);
    else if (t.kid < n_kernels) { total_ms[t.kid] += ms; launches[t.kid] += 1; }
    g_prof_free->push_back(t.a);
    g_prof_free->push_back(t.b);
  }
  g_prof->clear();
  return rc;
}

const char* slkv_kernel_name(int kernel_id) {
  static const char* names[KID_COUNT] = {"k_setup", "k_score_lse", "k_score_vote", "k_pool", "k_select",
                                         "k_gather", "k_alloc", "k_score_fused", "k_score_list", "k_window_stats",
                                         "k_merge_lse", "k_behavior", "k_cp", "k_layer", "k_score_bound"};
  return (kernel_id >= 0 && kernel_id < KID_COUNT) ? names[kernel_id] : "";
}

int slkv_kernel_count(void) { return KID_COUNT; }

int slkv_trace_set_buffer(void* dev_buf, size_t bytes) {
  set_tensor_trace(dev_buf, dev_buf ? bytes : 0);
  return SLKV_OK;
}

int slkv_last_cuda_error(void) { return g_last_cuda_error; }
int slkv_last_launch_count(void) { return g_last_launches; }
int slkv_version(void) { return 300; }

int slkv_debug_list_way(int way) {
  set_list_way(way == 1 || way == 2 ? way : 0);
  return SLKV_OK;
}

int slkv_debug_expire_next_wait(int on) {
  const int layer = on == 3 || on == 4 ? on - 2 : 0;
  expire_next_layer_wait(layer);
  expire_next_wait(layer ? 0 : on == 2 ? 2 : on != 0);
  return SLKV_OK;
}

int slkv_behavior_scores(const float* attn, int64_t n_rows, int32_t row_len, int64_t row_stride,
                         const int32_t* needle_idx, int32_t n_needle, int64_t needle_stride, const int32_t* topk_idx,
                         int32_t n_topk, int64_t topk_stride, float* sf_sc, float* lg_sc, float* inf_sc, void* stream) {
  if (!attn || !needle_idx || !topk_idx || !sf_sc || !lg_sc || !inf_sc) return SLKV_ERR_NULL_PTR;
  if (n_rows < 0 || n_rows > (1ll << 34) || row_len < 1 || row_stride < 0 || n_needle < 0 || n_needle > 4096 ||
      n_topk < 0 || n_topk > 4096 || needle_stride < 0 || topk_stride < 0)
    return SLKV_ERR_BAD_SHAPE;
  cudaError_t e = launch_behavior(attn, row_stride, row_len, n_rows, needle_idx, n_needle, needle_stride, topk_idx,
                                  n_topk, topk_stride, sf_sc, lg_sc, inf_sc, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  return SLKV_OK;
}

// ---- context-parallel selection (slkv_cp.cu) -----------------------------------------------------------------
int slkv_cp_merge_lse(const slkv_params* p, const float* lse_parts, int32_t n_parts, float* lse_out, void* stream) {
  if (!p || !lse_parts || !lse_out) return SLKV_ERR_NULL_PTR;
  if (n_parts < 1 || n_parts > 4096 || p->n_seqs != 1 || p->n_q_heads < 1 || p->window < 1 || p->window > kMaxWindow)
    return SLKV_ERR_BAD_SHAPE;
  if (p->lse_units != SLKV_LSE_LN && p->lse_units != SLKV_LSE_LOG2) return SLKV_ERR_BAD_DTYPE;
  int launches = 0;
  const float to_log2 = p->lse_units == SLKV_LSE_LOG2 ? 1.0f : 1.4426950408889634f;
  cudaError_t e = launch_cp_merge_lse(lse_parts, n_parts, (long long)p->n_q_heads * p->window, to_log2, lse_out,
                                      (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

int slkv_cp_select_init(const int32_t* budgets, int32_t n_kv_heads, int32_t window, int64_t seq_len, uint32_t* prefix,
                        int32_t* need, void* stream) {
  if (!budgets || !prefix || !need) return SLKV_ERR_NULL_PTR;
  if (n_kv_heads < 1 || n_kv_heads > 65535 || window < 1 || window > kMaxWindow || seq_len < 0 || seq_len >= (1ll << 31))
    return SLKV_ERR_BAD_SHAPE;
  CpStep a = {};
  a.budgets = budgets; a.n_kv_heads = n_kv_heads; a.window = window; a.seq_len = seq_len;
  a.prefix_out = prefix; a.need_out = need;
  int launches = 0;
  cudaError_t e = launch_cp_step(a, (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

int slkv_cp_histogram(const float* pooled, int32_t n_kv_heads, int64_t row_stride, int32_t own_begin, int32_t own_count,
                      int32_t level, const uint32_t* prefix, int32_t* hist, void* stream) {
  if (!pooled || !prefix || !hist) return SLKV_ERR_NULL_PTR;
  if (n_kv_heads < 1 || n_kv_heads > 65535 || row_stride < 0 || own_begin < 0 || own_count < 0 ||
      (int64_t)own_begin + own_count > row_stride || level < 0 || level > 2)
    return SLKV_ERR_BAD_SHAPE;
  cudaError_t e = cudaMemsetAsync(hist, 0, (size_t)n_kv_heads * kCpBins * sizeof(int32_t), (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  CpStep a = {};
  a.prefix_in = prefix; a.n_kv_heads = n_kv_heads; a.pooled = pooled; a.row_stride = row_stride;
  a.own_begin = own_begin; a.own_count = own_count; a.level_out = level; a.hist = hist;
  int launches = 0;
  e = launch_cp_step(a, (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

int slkv_cp_descend(const int32_t* hist, int32_t n_kv_heads, int32_t level, uint32_t* prefix, int32_t* need,
                    void* stream) {
  if (!hist || !prefix || !need) return SLKV_ERR_NULL_PTR;
  if (n_kv_heads < 1 || n_kv_heads > 65535 || level < 0 || level > 2) return SLKV_ERR_BAD_SHAPE;
  CpStep a = {};
  a.prefix_in = prefix; a.need_in = need; a.prefix_out = prefix; a.need_out = need;
  a.n_kv_heads = n_kv_heads; a.hist_sum = hist; a.level_in = level;
  int launches = 0;
  cudaError_t e = launch_cp_step(a, (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

int slkv_cp_local_ties(const int32_t* hist_local, const uint32_t* prefix, int32_t n_kv_heads, int32_t* ties,
                       void* stream) {
  if (!hist_local || !prefix || !ties) return SLKV_ERR_NULL_PTR;
  if (n_kv_heads < 1 || n_kv_heads > 65535) return SLKV_ERR_BAD_SHAPE;
  int launches = 0;
  cudaError_t e = launch_cp_local_ties(hist_local, prefix, n_kv_heads, ties, (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

size_t slkv_cp_workspace_bytes(int32_t n_kv_heads, int32_t own_count, int64_t out_capacity_rows) {
  if (n_kv_heads < 1 || own_count < 0 || out_capacity_rows < 0) return 0;
  return CpWorkspace(nullptr, n_kv_heads, own_count, out_capacity_rows).bytes;
}

int slkv_cp_step(const int32_t* budgets, int32_t n_kv_heads, int32_t window, int64_t seq_len, int32_t level,
                 int32_t* state, const int32_t* hist_sum, const float* pooled, int64_t row_stride, int32_t own_begin,
                 int32_t own_count, int32_t* hist, int32_t* totals, void* clear, size_t clear_bytes, void* workspace,
                 size_t workspace_bytes, void* stream) {
  if (!state || !pooled || (level == 0 ? !budgets : !hist_sum) || (level < 3 ? !hist : !totals) || (clear_bytes && !clear))
    return SLKV_ERR_NULL_PTR;
  if (n_kv_heads < 1 || n_kv_heads > 65535 || window < 1 || window > kMaxWindow || seq_len < 0 ||
      seq_len >= (1ll << 31) || row_stride < 0 || own_begin < 0 || own_count < 0 ||
      (int64_t)own_begin + own_count > row_stride || level < 0 || level > 3 || clear_bytes % 16 != 0)
    return SLKV_ERR_BAD_SHAPE;
  if (!aligned16(clear)) return SLKV_ERR_BAD_ALIGN;
  CpStep a = {};
  a.n_kv_heads = n_kv_heads; a.window = window; a.seq_len = seq_len;
  a.pooled = pooled; a.row_stride = row_stride; a.own_begin = own_begin; a.own_count = own_count;
  a.clear = clear; a.clear_bytes = (long long)clear_bytes;
  int32_t* mine = state + (size_t)level * 2 * n_kv_heads;          // state[level]: prefix, need
  a.prefix_out = reinterpret_cast<unsigned*>(mine);
  a.need_out = mine + n_kv_heads;
  if (level == 0) {
    a.budgets = budgets;
  } else {
    a.prefix_in = a.prefix_out - 2 * n_kv_heads;
    a.need_in = a.need_out - 2 * n_kv_heads;
    a.hist_sum = hist_sum;
    a.level_in = level - 1;
  }
  if (level < 3) {
    a.hist = hist;
    a.level_out = level;
  } else {
    const CpWorkspace w(workspace, n_kv_heads, own_count, 0);
    if (!workspace || workspace_bytes < w.bytes || reinterpret_cast<uintptr_t>(workspace) % kAlign != 0)
      return SLKV_ERR_WORKSPACE;
    a.cnt_gt = w.cnt_gt; a.cnt_eq = w.cnt_eq; a.tot_gt = totals; a.tot_eq = totals + n_kv_heads;
  }
  int launches = 0;
  cudaError_t e = launch_cp_step(a, (cudaStream_t)stream, &launches);
  return e == cudaSuccess ? SLKV_OK : cuda_fail(e);
}

int slkv_cp_emit_counted(const slkv_params* p, const void* k, const void* v, int64_t rows, const float* pooled,
                         int64_t row_stride, int32_t own_begin, int32_t own_count, int64_t pos0,
                         const uint32_t* threshold, const int32_t* need, const int32_t* ties_all, int32_t n_parts,
                         int32_t part, int32_t window_rows, int64_t window_pos0, const int32_t* totals, void* k_out,
                         void* v_out, int64_t out_capacity_rows, int32_t* offsets, int32_t* kept_idx, int32_t* status,
                         void* workspace, size_t workspace_bytes, void* stream) {
  g_last_launches = 0;
  if (!p || !k || !v || !pooled || !threshold || !need || !ties_all || !k_out || !v_out || !offsets || !kept_idx)
    return SLKV_ERR_NULL_PTR;
  const int32_t cu1[2] = {0, (int32_t)(rows < (1ll << 31) && rows >= 0 ? rows : -1)};
  Problem pb;
  int rc = describe(p, cu1, &pb);                    // validates dtype, head counts, strides
  if (rc != SLKV_OK) return rc;
  if (n_parts < 1 || part < 0 || part >= n_parts || window_rows < 0 || window_rows > p->window || window_rows > rows ||
      own_begin < 0 || own_count < 0 || (int64_t)own_begin + own_count > rows - window_rows ||
      (int64_t)own_begin + own_count > row_stride || pos0 < 0 || pos0 + own_count >= (1ll << 31) || window_pos0 < 0 ||
      window_pos0 + window_rows >= (1ll << 31))
    return SLKV_ERR_BAD_SHAPE;
  if (out_capacity_rows < 0) return SLKV_ERR_CAPACITY;
  if (!aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out)) return SLKV_ERR_BAD_ALIGN;
  const CpWorkspace w(workspace, p->n_kv_heads, own_count, out_capacity_rows);
  if (!workspace || workspace_bytes < w.bytes || reinterpret_cast<uintptr_t>(workspace) % kAlign != 0)
    return SLKV_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  int launches = 0;
  cudaError_t e = cudaSuccess;
  const bool counted = totals != nullptr;
  if (!counted) {                                    // the counts of slkv_cp_step's last level
    CpStep a = {};
    a.prefix_in = threshold; a.n_kv_heads = p->n_kv_heads; a.pooled = pooled; a.row_stride = row_stride;
    a.own_begin = own_begin; a.own_count = own_count;
    a.cnt_gt = w.cnt_gt; a.cnt_eq = w.cnt_eq; a.tot_gt = w.totals; a.tot_eq = w.totals + p->n_kv_heads;
    e = cudaMemsetAsync(w.totals, 0, 2 * (size_t)p->n_kv_heads * sizeof(int32_t), st);
    if (e == cudaSuccess) e = launch_cp_step(a, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
    totals = w.totals;
  }
  CpEmit m = {};
  m.pooled = pooled; m.threshold = threshold; m.need = need; m.ties_all = ties_all;
  m.cnt_gt = w.cnt_gt; m.cnt_eq = w.cnt_eq; m.tot_gt = totals; m.tot_eq = totals + p->n_kv_heads;
  m.offsets = offsets; m.kept_idx = kept_idx; m.gather_src = w.gather_src; m.status = status;
  m.row_stride = row_stride; m.pos0 = pos0; m.window_row0 = rows - window_rows; m.window_pos0 = window_pos0;
  m.capacity = out_capacity_rows;
  m.n_kv_heads = p->n_kv_heads; m.part = part; m.window_rows = window_rows; m.own_begin = own_begin;
  m.own_count = own_count; m.fill_tail = counted;
  e = launch_cp_emit(m, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e);
  pb.total_tokens = rows;
  pb.n_seg = p->n_kv_heads;
  pb.k = k; pb.v = v;
  pb.gather_src = w.gather_src;
  const TailLayer tail = tail_of(pb, nullptr, k_out, v_out, out_capacity_rows, offsets, kept_idx, nullptr, status);
  e = launch_gather(pb, &tail, 1, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e);
  g_last_launches = launches;
  return SLKV_OK;
}

int slkv_cp_emit(const slkv_params* p, const void* k, const void* v, int64_t rows, const float* pooled,
                 int64_t row_stride, int32_t own_begin, int32_t own_count, int64_t pos0, const uint32_t* threshold,
                 const int32_t* need, const int32_t* ties_all, int32_t n_parts, int32_t part, int32_t window_rows,
                 int64_t window_pos0, void* k_out, void* v_out, int64_t out_capacity_rows, int32_t* offsets,
                 int32_t* kept_idx, int32_t* status, void* workspace, size_t workspace_bytes, void* stream) {
  return slkv_cp_emit_counted(p, k, v, rows, pooled, row_stride, own_begin, own_count, pos0, threshold, need, ties_all,
                              n_parts, part, window_rows, window_pos0, nullptr, k_out, v_out, out_capacity_rows, offsets,
                              kept_idx, status, workspace, workspace_bytes, stream);
}

int slkv_alloc_budgets_ex(const float* inf_sc, int32_t n_layers, int32_t n_heads, int32_t fixed, int64_t total,
                          const slkv_alloc_options* opt, int32_t* budgets, int32_t* status, void* stream) {
  if (!inf_sc || !budgets) return SLKV_ERR_NULL_PTR;
  if (n_layers < 1 || n_heads < 1 || n_layers > 1024 || (int64_t)n_layers * n_heads > 16384)
    return SLKV_ERR_BAD_SHAPE;
  const int64_t n = (int64_t)n_layers * n_heads;
  if (fixed < 0 || total < n * fixed) return SLKV_ERR_BUDGET_SUM;
  if (total > 0x7fffffffll) return SLKV_ERR_BAD_SHAPE;
  int within = 0, paper = 0;
  long long cap = -1;
  if (opt) {
    if (opt->head_normaliser != SLKV_NORM_GLOBAL && opt->head_normaliser != SLKV_NORM_WITHIN_LAYER) return SLKV_ERR_BAD_DTYPE;
    if (opt->rounding != SLKV_ROUND_SUM_EXACT && opt->rounding != SLKV_ROUND_PAPER) return SLKV_ERR_BAD_DTYPE;
    if (opt->cap < 0 || opt->cap > 0x7fffffffll) return SLKV_ERR_BAD_SHAPE;
    within = opt->head_normaliser == SLKV_NORM_WITHIN_LAYER;
    paper = opt->rounding == SLKV_ROUND_PAPER;
    if (opt->cap > 0) {
      cap = opt->cap;
      // a cap below the fixed part, or a total that does not fit under the cap (where the total is to be met)
      if (cap < fixed || (!paper && total > n * cap)) return SLKV_ERR_BUDGET_SUM;
    }
  }
  cudaError_t e = launch_alloc(inf_sc, n_layers, n_heads, fixed, total, within, paper, cap, budgets, status,
                               (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  return SLKV_OK;
}

int slkv_alloc_budgets(const float* inf_sc, int32_t n_layers, int32_t n_heads, int32_t fixed, int64_t total,
                       int32_t* budgets, int32_t* status, void* stream) {
  return slkv_alloc_budgets_ex(inf_sc, n_layers, n_heads, fixed, total, nullptr, budgets, status, stream);
}

size_t slkv_workspace_bytes(const slkv_params* p, const int32_t* cu_seqlens_host) {
  Problem pb;
  if (describe(p, cu_seqlens_host, &pb) != SLKV_OK) return 0;
  return layout_of(pb).total;
}

size_t slkv_workspace_bytes_overlapped(const slkv_params* p, const int32_t* cu_seqlens_host) {
  Problem pb;
  if (describe(p, cu_seqlens_host, &pb) != SLKV_OK) return 0;
  return layout_of(pb, true).total;
}

int slkv_compress_overlapped(const slkv_params* p, const void* q_win, const void* k, const void* v,
                             const int32_t* cu_seqlens_dev, const int32_t* cu_seqlens_host, const int32_t* budgets,
                             const float* lse_opt, void* k_out, void* v_out, int64_t out_capacity_rows,
                             int32_t* offsets, int32_t* kept_idx, float* pooled_opt, int32_t* status, void* workspace,
                             size_t workspace_bytes, void* stream) {
  return compress_impl(p, q_win, k, v, cu_seqlens_dev, cu_seqlens_host, budgets, lse_opt, k_out, v_out,
                       out_capacity_rows, offsets, kept_idx, pooled_opt, status, workspace, workspace_bytes,
                       (cudaStream_t)stream, true);
}

int slkv_join(void* stream) {
  int launches = 0;
  cudaError_t e = join_lists((cudaStream_t)stream, &launches);
  g_last_launches = launches;
  if (e != cudaSuccess) return cuda_fail(e);
  return SLKV_OK;
}

int64_t slkv_pooled_elems(const slkv_params* p, const int32_t* cu_seqlens_host) {
  Problem pb;
  if (describe(p, cu_seqlens_host, &pb) != SLKV_OK) return -1;
  return (int64_t)pb.p.n_kv_heads * pb.total_hist;
}

int64_t slkv_packed_rows_upper_bound(const slkv_params* p, const int32_t* cu_seqlens_host) {
  Problem pb;
  if (describe(p, cu_seqlens_host, &pb) != SLKV_OK) return -1;
  return (int64_t)pb.p.n_kv_heads * pb.total_tokens;
}

namespace {
// slkv_score and slkv_row_lse: the votes pooled into `pooled`, or the rows' log-sum-exp into `lse_out`.
int score_impl(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
               const int32_t* cu_seqlens_host, const float* lse_opt, float* pooled, float* lse_out, int32_t* status,
               void* workspace, size_t workspace_bytes, void* stream, bool cleared = false) {
  g_last_launches = 0;
  if (!q_win || !k || !cu_seqlens_dev || (!pooled && !lse_out)) return SLKV_ERR_NULL_PTR;
  Problem pb;
  int rc = describe(p, cu_seqlens_host, &pb);
  if (rc != SLKV_OK) return rc;
  if (!aligned16(q_win) || !aligned16(k)) return SLKV_ERR_BAD_ALIGN;
  int path = 0;
  rc = resolve_path(pb, &path);
  if (rc != SLKV_OK) return rc;
  rc = bind_workspace(&pb, workspace, workspace_bytes);
  if (rc != SLKV_OK) return rc;
  pb.cu = cu_seqlens_dev; pb.q = q_win; pb.k = k; pb.v = nullptr;
  pb.tab.cu_ptr = cu_seqlens_dev;
  pb.lse_opt = lse_opt;
  if (p->history_only) cu_seqlens_host = pb.cu_virtual;      // one sequence: the tables are inline, cu_seqlens_dev unread
  cudaStream_t st = (cudaStream_t)stream;
  int launches = 0;
  cudaError_t e = join_lists(st, &launches);  // the workspace may still serve an overlapped call
  if (e != cudaSuccess) return cuda_fail(e);
  if (pb.tab.n_inline == 0) {
    e = launch_setup(pb, nullptr, nullptr, 0, nullptr, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
  }
  if (lse_out) {
    // row statistics only: pass 1, the window keys' share where the domain has one, then the merge
    rc = enqueue_window_stats(pb, path, st, &launches);
    if (rc != SLKV_OK) return rc;
    e = path == SLKV_PATH_TENSOR ? launch_score_tensor(pb, cu_seqlens_host, status, 1, lse_out, cleared, st, &launches)
                                 : launch_score_simt(pb, status, 1, st, &launches);
    if (e == cudaSuccess && path != SLKV_PATH_TENSOR) e = launch_merge_lse_simt(pb, lse_out, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
    g_last_launches = launches;
    return SLKV_OK;
  }
  if (const int cs = layer_cluster(pb, path, false)) {
    e = launch_layer(pb, path, cs, nullptr, pooled, status, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e);
    g_last_launches = launches;
    return SLKV_OK;
  }
  rc = enqueue_votes(pb, path, cu_seqlens_host, status, st, &launches);
  if (rc != SLKV_OK) return rc;
  e = launch_pool(pb, pooled, st, &launches);
  if (e != cudaSuccess) return cuda_fail(e);
  g_last_launches = launches;
  return SLKV_OK;
}
}  // namespace

int slkv_score(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
               const int32_t* cu_seqlens_host, const float* lse_opt, float* pooled, int32_t* status, void* workspace,
               size_t workspace_bytes, void* stream) {
  if (!pooled) return SLKV_ERR_NULL_PTR;
  return score_impl(p, q_win, k, cu_seqlens_dev, cu_seqlens_host, lse_opt, pooled, nullptr, status, workspace,
                    workspace_bytes, stream);
}

int slkv_row_lse(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
                 const int32_t* cu_seqlens_host, float* lse_out, int32_t* status, void* workspace,
                 size_t workspace_bytes, void* stream) {
  if (!lse_out) return SLKV_ERR_NULL_PTR;
  return score_impl(p, q_win, k, cu_seqlens_dev, cu_seqlens_host, nullptr, nullptr, lse_out, status, workspace,
                    workspace_bytes, stream);
}

int slkv_cp_row_lse(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
                    const int32_t* cu_seqlens_host, float* lse_out, int32_t* status, void* zeroed_workspace,
                    size_t workspace_bytes, void* stream) {
  if (!lse_out) return SLKV_ERR_NULL_PTR;
  return score_impl(p, q_win, k, cu_seqlens_dev, cu_seqlens_host, nullptr, nullptr, lse_out, status, zeroed_workspace,
                    workspace_bytes, stream, true);
}

}  // extern "C"

// Host-side validation of slkv_score's arguments without a workspace (for entry points that bring their own).
int slkv::check_score_args(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
                           const int32_t* cu_seqlens_host, const float* pooled) {
  if (!q_win || !k || !cu_seqlens_dev || !pooled) return SLKV_ERR_NULL_PTR;
  Problem pb;
  int rc = describe(p, cu_seqlens_host, &pb);
  if (rc != SLKV_OK) return rc;
  if (!aligned16(q_win) || !aligned16(k)) return SLKV_ERR_BAD_ALIGN;
  int path = 0;
  return resolve_path(pb, &path);
}

extern "C" {

int slkv_compress(const slkv_params* p, const void* q_win, const void* k, const void* v,
                  const int32_t* cu_seqlens_dev, const int32_t* cu_seqlens_host, const int32_t* budgets,
                  const float* lse_opt, void* k_out, void* v_out, int64_t out_capacity_rows, int32_t* offsets,
                  int32_t* kept_idx, float* pooled_opt, int32_t* status, void* workspace, size_t workspace_bytes,
                  void* stream) {
  return compress_impl(p, q_win, k, v, cu_seqlens_dev, cu_seqlens_host, budgets, lse_opt, k_out, v_out,
                       out_capacity_rows, offsets, kept_idx, pooled_opt, status, workspace, workspace_bytes,
                       (cudaStream_t)stream);
}

// ---- host-buffer variant ---------------------------------------------------------------------------
namespace {
struct HostArena {
  size_t q, k, v, cu, budgets, k_out, v_out, offsets, kept, status, ws, total;
};
bool host_arena_layout(const Problem& pb, int64_t capacity, HostArena* A) {
  const slkv_params& p = pb.p;
  const size_t e = pb.elem, d = p.head_dim;
  size_t o = 0;
  A->q = o; o = align_up(o + (size_t)p.n_seqs * p.window * p.n_q_heads * d * e);
  A->k = o; o = align_up(o + (size_t)pb.total_tokens * p.n_kv_heads * d * e);
  A->v = o; o = align_up(o + (size_t)pb.total_tokens * p.n_kv_heads * d * e);
  A->cu = o; o = align_up(o + (size_t)(p.n_seqs + 1) * 4);
  A->budgets = o; o = align_up(o + (size_t)p.n_kv_heads * 4);
  A->k_out = o; o = align_up(o + (size_t)capacity * d * e);
  A->v_out = o; o = align_up(o + (size_t)capacity * d * e);
  A->offsets = o; o = align_up(o + (size_t)(pb.n_seg + 1) * 4);
  A->kept = o; o = align_up(o + (size_t)capacity * 4);
  A->status = o; o = align_up(o + 4);
  A->ws = o; o = align_up(o + layout_of(pb).total);
  A->total = o;
  return true;
}
// The device address of [ptr, ptr + bytes) where that is page-locked host memory the device can reach, else null.
void* pinned_address(const void* ptr, size_t bytes) {
  typedef CUresult (*GetFn)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
  static const GetFn get = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
    return reinterpret_cast<GetFn>(f);
  }();
  if (!get || bytes == 0) return nullptr;
  unsigned type = 0;
  CUdeviceptr dev = 0, start = 0;
  size_t size = 0;
  CUpointer_attribute attr[4] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                 CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* out[4] = {&type, &dev, &start, &size};
  if (get(4, attr, out, (CUdeviceptr)(uintptr_t)ptr) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || !dev) return nullptr;
  const uintptr_t p = (uintptr_t)ptr, s0 = (uintptr_t)start;
  return p >= s0 && bytes <= size && p - s0 <= size - bytes && dev % 16 == 0 ? reinterpret_cast<void*>(dev) : nullptr;
}
bool dense_strides(const slkv_params& p) {
  const int64_t d = p.head_dim;
  return p.k_stride_head == d && p.k_stride_tok == d * p.n_kv_heads && p.v_stride_head == d &&
         p.v_stride_tok == d * p.n_kv_heads && p.q_stride_head == d && p.q_stride_row == d * p.n_q_heads &&
         p.q_stride_seq == d * p.n_q_heads * p.window;
}
}  // namespace

size_t slkv_compress_host_arena_bytes(const slkv_params* p, const int32_t* cu_seqlens_host,
                                      int64_t out_capacity_rows) {
  Problem pb;
  if (describe(p, cu_seqlens_host, &pb) != SLKV_OK || out_capacity_rows < 0) return 0;
  HostArena A;
  host_arena_layout(pb, out_capacity_rows, &A);
  return A.total;
}

int slkv_compress_host(const slkv_params* p, const void* q_win, const void* k, const void* v,
                       const int32_t* cu_seqlens_host, const int32_t* budgets, void* k_out, void* v_out,
                       int64_t out_capacity_rows, int32_t* offsets, int32_t* kept_idx, int64_t* rows_out,
                       void* arena, size_t arena_bytes, void* stream) {
  g_last_launches = 0;
  if (!q_win || !k || !v || !budgets || !k_out || !v_out || !offsets || !kept_idx || !arena)
    return SLKV_ERR_NULL_PTR;
  Problem pb;
  int rc = describe(p, cu_seqlens_host, &pb);
  if (rc != SLKV_OK) return rc;
  if (!dense_strides(*p) || p->history_only) return SLKV_ERR_BAD_SHAPE;
  if (out_capacity_rows < 0) return SLKV_ERR_CAPACITY;
  if (reinterpret_cast<uintptr_t>(arena) % kAlign != 0) return SLKV_ERR_BAD_ALIGN;
  HostArena A;
  host_arena_layout(pb, out_capacity_rows, &A);
  if (arena_bytes < A.total) return SLKV_ERR_WORKSPACE;
  // rows that will be written, known on the host because the budgets are (Algorithm 3 l.1-4, l.7)
  int64_t rows = 0;
  for (int s = 0; s < p->n_seqs; ++s) {
    const int64_t len = cu_seqlens_host[s + 1] - cu_seqlens_host[s];
    for (int h = 0; h < p->n_kv_heads; ++h) {
      int64_t c = budgets[h] > p->window ? budgets[h] : p->window;
      rows += len < c ? len : c;
    }
  }
  if (rows_out) *rows_out = rows;
  if (rows > out_capacity_rows) return SLKV_ERR_CAPACITY;

  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* b = static_cast<unsigned char*>(arena);
  const size_t e = pb.elem, d = p->head_dim;
  cudaError_t ce;
#define SLKV_CP(dst, src, n, kind)                                  \
  do {                                                              \
    if ((n) > 0) {                                                  \
      ce = cudaMemcpyAsync((dst), (src), (n), (kind), st);          \
      if (ce != cudaSuccess) return cuda_fail(ce);                  \
    }                                                               \
  } while (0)
  // What bounds this call is the host link.  Only the keys have to cross it: of V, page-locked memory is read by the gather
  // kernel where it lies, kept rows only, and page-locked outputs are written by that kernel directly (one launch instead of
  // four copies; 32k tokens, 8 heads, 512 rows kept per head: 2585 -> 1350 us, the keys alone 1210).  Pageable buffers are
  // copied as a whole.  However much is kept, reading page-locked V in place is faster than copying it (us, in place / copied,
  // 32k tokens, d = 128: 1/16 kept 1529 / 2678, 1/4 2121 / 3170, 1/2 2878 / 3834, everything 4312 / 5129; d = 64, everything
  // 2248 / 2605; 4k tokens, d = 128, everything 655 / 691).
  const size_t kv_bytes = (size_t)pb.total_tokens * p->n_kv_heads * d * e, out_bytes = (size_t)rows * d * e;
  const void* v_dev = pinned_address(v, kv_bytes);
  void* k_dst = pinned_address(k_out, out_bytes);
  void* v_dst = pinned_address(v_out, out_bytes);
  int32_t* off_dst = static_cast<int32_t*>(pinned_address(offsets, (size_t)(pb.n_seg + 1) * 4));
  int32_t* kept_dst = static_cast<int32_t*>(pinned_address(kept_idx, (size_t)rows * 4));
  SLKV_CP(b + A.q, q_win, (size_t)p->n_seqs * p->window * p->n_q_heads * d * e, cudaMemcpyHostToDevice);
  if (pb.tab.n_inline == 0) SLKV_CP(b + A.cu, cu_seqlens_host, (size_t)(p->n_seqs + 1) * 4, cudaMemcpyHostToDevice);
  SLKV_CP(b + A.budgets, budgets, (size_t)p->n_kv_heads * 4, cudaMemcpyHostToDevice);
  SLKV_CP(b + A.k, k, kv_bytes, cudaMemcpyHostToDevice);
  if (!v_dev) SLKV_CP(b + A.v, v, kv_bytes, cudaMemcpyHostToDevice);
  rc = compress_impl(p, b + A.q, b + A.k, v_dev ? v_dev : b + A.v, reinterpret_cast<int32_t*>(b + A.cu), cu_seqlens_host,
                     reinterpret_cast<int32_t*>(b + A.budgets), nullptr, k_dst ? k_dst : b + A.k_out,
                     v_dst ? v_dst : b + A.v_out, rows, reinterpret_cast<int32_t*>(b + A.offsets),
                     reinterpret_cast<int32_t*>(b + A.kept), nullptr, nullptr, b + A.ws, arena_bytes - A.ws, st, false,
                     kept_dst, off_dst);
  if (rc != SLKV_OK) return rc;
  if (!off_dst || rows == 0) SLKV_CP(offsets, b + A.offsets, (size_t)(pb.n_seg + 1) * 4, cudaMemcpyDeviceToHost);
  if (!kept_dst) SLKV_CP(kept_idx, b + A.kept, (size_t)rows * 4, cudaMemcpyDeviceToHost);
  if (!k_dst) SLKV_CP(k_out, b + A.k_out, out_bytes, cudaMemcpyDeviceToHost);
  if (!v_dst) SLKV_CP(v_out, b + A.v_out, out_bytes, cudaMemcpyDeviceToHost);
#undef SLKV_CP
  ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return cuda_fail(ce);
  return SLKV_OK;
}

}  // extern "C"

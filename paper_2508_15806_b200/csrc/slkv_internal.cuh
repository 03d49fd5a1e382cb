// Internal declarations shared by the translation units of libslkv (not part of the public ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "slkv.h"

namespace slkv {

constexpr double kLayerFloor = 0.01;   // minimum layer budget (Sec. 3.3)
constexpr float kLog2e = 1.4426950408889634f;

constexpr int kInlineSeqs = 64;
constexpr int kMaxSplit = 160;         // CTAs the tensor-core score kernel uses at most (one per SM)

// Per-sequence tables: token starts (cu), exclusive prefixes of the history lengths n_hist_s and of the
// 128-key tile counts.  Batches of up to kInlineSeqs sequences carry them inside the kernel parameters
// (filled on the host from cu_seqlens_host); larger batches read the arrays a set-up kernel wrote.
struct SeqTables {
  int32_t n_inline;                       // n_seqs when the inline arrays are valid, else 0
  int32_t cu[kInlineSeqs + 1];
  int32_t tile_off[kInlineSeqs + 1];
  long long hist_off[kInlineSeqs + 1];
  const int32_t* cu_ptr;
  const int32_t* tile_ptr;
  const long long* hist_ptr;
#ifdef __CUDACC__
  __device__ __forceinline__ int cu_at(int i) const { return n_inline ? cu[i] : cu_ptr[i]; }
  __device__ __forceinline__ int tile_at(int i) const { return n_inline ? tile_off[i] : tile_ptr[i]; }
  __device__ __forceinline__ long long hist_at(int i) const { return n_inline ? hist_off[i] : hist_ptr[i]; }
#endif
};

// Where a vote pass takes the window rows' log-sum-exp from, besides the row sums of the statistics pass: the caller's array (lse_opt of the public entry points), and / or the statistics of the
// window keys (softmax over all causally visible keys).  Row r of a segment is query head g*G + hh, window row i with
// r = i*G + hh (head_inner) or r = hh*window + i.
struct LseSource {
  const float* lse_opt;     // [n_seqs][n_q_heads][window], or null
  const float* win_m;       // [n_seg][R] maxima (log2 units) over the window keys a row sees, or null
  const float* win_z;       // [n_seg][R] sums of 2^(x - max) over them
  float to_log2;            // lse_opt * to_log2 is in log2 units
  int n_q_heads;
#ifdef __CUDACC__
  __device__ __forceinline__ float caller_lse(int s, int g, int r, int G, int window, bool head_inner) const {
    const int hh = head_inner ? r % G : r / window;
    const int i = head_inner ? r / G : r - hh * window;
    return lse_opt[((long long)s * n_q_heads + g * G + hh) * window + i] * to_log2;
  }
#endif
};

// Programmatic dependent launch: a kernel may start while its predecessor in the stream drains; it must
// not touch global memory the predecessor may write before pdl_wait() returns.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

constexpr int kListMaxLayers = 32;          // layers one launch of the score, selection and gather kernels takes
constexpr int kListMaxGroups = 64;          // groups of segments a layer is walked in

// What the CTAs of a launch tell one another lies in the caller's workspace, which belongs to one call at a time, so launches
// on other streams -- other threads' calls, replays of captured graphs -- never meet there.  Nobody zeroes a workspace: the
// CTAs clear what has to start at zero, their counts included, and touch none of it before all have said that they are done.
// They say so in words that carry the launch's own tag (WordSync, FlagSync in the two score kernels), which whatever a
// workspace held before does not, and leave the words without it, so that a replay, which brings the same tag, starts as the
// first launch did.  (A memset in front of the launch would do as well, for 2.6 us a call: it cuts the dependent launch.)
constexpr int kSyncFlags = 320;             // tagged words: two CTAs per SM
constexpr int kSyncCounts = kListMaxLayers * kListMaxGroups;
constexpr size_t kSyncBytes = sizeof(unsigned long long) * kSyncFlags + sizeof(unsigned) * kSyncCounts;
unsigned long long next_launch_tag();

// Launches `kernel` with the programmatic-serialisation attribute (and optionally a cluster shape).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              int cluster_x, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  if (cluster_x > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster_x;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Everything a score / select / gather launch needs, resolved by the host entry points.
struct Problem {
  slkv_params p;
  int G;                  // query heads per KV head
  int R;                  // score rows per KV head = G * window
  int elem;               // bytes per element
  int max_hist;           // max_s n_hist_s
  int64_t total_tokens;   // rows of K / V that exist (the extent of the K tensor map)
  int32_t cu_virtual[2];  // history_only: {0, rows + window}, the sequence the kernels are told about
  int64_t total_hist;     // sum_s n_hist_s
  int n_seg;              // n_seqs * n_kv_heads
  const int32_t* cu;      // dev
  SeqTables tab;          // per-sequence tables (inline or pointing into the workspace)
  const void* q;          // dev
  const void* k;          // dev
  const void* v;          // dev
  // workspace carve-up (dev)
  int64_t* hist_off;      // [n_seqs+1] exclusive prefix of n_hist_s
  int32_t* tile_off;      // [n_seqs+1] exclusive prefix of ceil(n_hist_s / 128)
  float* vote;            // [n_kv_heads * total_hist] ragged, same layout as pooled
  void* part;             // row statistics; layout of the score path (StatView, SimtStats)
  int64_t n_tiles128;     // 128-key tiles of all segments
  float* pooled_ws;       // [n_kv_heads * total_hist] used when the caller wants no pooled output
  int32_t* gather_src;    // [n_kv_heads * total_tokens] per packed row: token * n_kv_heads + head of its source
  unsigned long long* sync;   // kSyncBytes: what the CTAs of a launch tell one another (WordSync, FlagSync)
  float* win_m;           // [n_seg][R] row statistics over the window keys (SLKV_ALL_CAUSAL without lse_opt)
  float* win_z;
  const float* lse_opt;   // the caller's row log-sum-exps, or null
};

// kernel ids for launch accounting / per-kernel timing
enum KernelId { KID_SETUP = 0, KID_SCORE_LSE, KID_SCORE_VOTE, KID_POOL, KID_SELECT, KID_GATHER, KID_ALLOC, KID_SCORE_FUSED, KID_SCORE_LIST, KID_WINDOW_STATS, KID_MERGE_LSE, KID_BEHAVIOR, KID_CP, KID_LAYER, KID_SCORE_BOUND, KID_COUNT };

// Brackets one kernel launch: counts it and, when per-kernel timing is on for this thread, records a
// CUDA event pair around it on the launch stream.
struct LaunchScope {
  LaunchScope(int kid, cudaStream_t st, int* launches);
  ~LaunchScope();
  int kid_; cudaStream_t st_; int slot_;
};

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_scoped(int kid, void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st,
                                     int* launches, Args&... args) {
  LaunchScope scope(kid, st, launches);
  return launch_pdl<KArgs...>(kernel, dim3((unsigned)grid), dim3((unsigned)block), smem, st, 1, args...);
}

// slkv_score's host-side argument checks, without a workspace: SLKV_OK or the status slkv_score would return
int check_score_args(const slkv_params* p, const void* q_win, const void* k, const int32_t* cu_seqlens_dev,
                     const int32_t* cu_seqlens_host, const float* pooled);

// host-side launchers; each returns a cudaError_t and adds to *launches
cudaError_t launch_alloc(const float* inf, int n_layers, int n_heads, int fixed, long long total, int within_layer,
                         int paper_rounding, long long cap, int32_t* budgets, int32_t* status, cudaStream_t st);
cudaError_t launch_behavior(const float* attn, long long row_stride, int row_len, long long n_rows,
                            const int32_t* needle_idx, int n_needle, long long needle_stride, const int32_t* topk_idx,
                            int n_topk, long long topk_stride, float* sf, float* lg, float* inf, cudaStream_t st);
// context-parallel selection (slkv_cp.cu)
cudaError_t launch_cp_merge_lse(const float* parts, int n_parts, long long n, float to_log2, float* out,
                                cudaStream_t st, int* launches);
constexpr int kCpBins = 2048;           // of a head's histogram
struct CpStep {                          // one launch of k_cp_step; see there
  const int32_t* budgets;                // not null: start from them
  const unsigned* prefix_in;             // else from this state,
  const int32_t* need_in;
  const int32_t* hist_sum;               // not null: taken down level level_in
  unsigned* prefix_out;                  // may be null
  int32_t* need_out;
  const float* pooled;
  int32_t* hist;                         // not null: histogram of level level_out added here
  int32_t *cnt_gt, *cnt_eq, *tot_gt, *tot_eq;   // not null: slices counted against the complete prefix
  void* clear;                           // 16-byte aligned; clear_bytes a multiple of 16
  long long seq_len, row_stride, clear_bytes;
  int n_kv_heads, window, level_in, level_out, own_begin, own_count;
  int n_blk, ctas_per_head;              // set by launch_cp_step
};
cudaError_t launch_cp_step(CpStep a, cudaStream_t st, int* launches);
cudaError_t launch_cp_local_ties(const int32_t* hist_local, const unsigned* prefix, int n_kv_heads, int32_t* ties,
                                 cudaStream_t st, int* launches);
struct CpEmit {                          // one launch of k_cp_emit; see there
  const float* pooled;
  const unsigned* threshold;
  const int32_t *need, *ties_all, *cnt_gt, *cnt_eq, *tot_gt, *tot_eq;
  int32_t *offsets, *kept_idx, *gather_src, *status;
  long long row_stride, pos0, window_row0, window_pos0, capacity;
  int n_kv_heads, part, window_rows, own_begin, own_count;
  int fill_tail;                         // 1: kept_idx of the rows behind the last one is set to -1
  int n_blk;                             // set by launch_cp_emit
};
cudaError_t launch_cp_emit(CpEmit a, cudaStream_t st, int* launches);
int cp_slices(int own_count);            // slices of the owned range that are counted and packed together
cudaError_t launch_setup(const Problem& pb, const int32_t* budgets, int32_t* offsets, int64_t capacity,
                         int32_t* status, cudaStream_t st, int* launches);
size_t simt_part_bytes(const Problem& pb);
// passes: 1 = row statistics only, 2 = votes only (the log-sum-exps come from lse_source_of), 3 = both
cudaError_t launch_score_simt(const Problem& pb, int32_t* status, int passes, cudaStream_t st, int* launches);
// Row statistics of the window keys each window row sees causally (SLKV_ALL_CAUSAL) -> pb.win_m / pb.win_z, rows in
// the order of the score path (head_inner: r = i*G + hh).
cudaError_t launch_window_stats(const Problem& pb, bool head_inner, cudaStream_t st, int* launches);
// lse_out[n_seqs][n_q_heads][window] in the problem's lse_units from the row sums and the window statistics, if any.
cudaError_t launch_merge_lse_simt(const Problem& pb, float* lse_out, cudaStream_t st, int* launches);
LseSource lse_source_of(const Problem& pb);
float lse_out_scale(const Problem& pb);          // log2 units -> the problem's lse_units
bool tensor_q_head_inner(const slkv_params& p);
bool tensor_path_supported(const slkv_params& p);
int tensor_slot_stride(const Problem& pb);        // split ranges a segment may be shared by, at most
void set_tensor_trace(void* dev_buf, size_t bytes);
// passes as launch_score_simt; lse_out (optional, with passes == 1): the rows' log-sum-exps in the problem's lse_units;
// cleared: the workspace is zero (the row sums of a launch of the statistics alone have to be)
cudaError_t launch_score_tensor(const Problem& pb, const int32_t* cu_host, int32_t* status, int passes, float* lse_out, bool cleared,
                                cudaStream_t st, int* launches);
cudaError_t launch_pool(const Problem& pb, float* pooled, cudaStream_t st, int* launches);
cudaError_t launch_select(const Problem& pb, const float* pooled, const int32_t* budgets, const int32_t* offsets,
                          int32_t* kept_idx, int64_t capacity, cudaStream_t st, int* launches);
// ---- selection and gather over a list of layers of one shape ------------------------------------------------------
struct TailLayer {
  const float* vote;
  const int32_t* budgets;
  int32_t* offsets;
  int32_t* kept_idx;
  int32_t* gather_src;          // per packed row: token * n_kv_heads + head of its source row
  float* pooled_out;            // optional
  int32_t* status;              // optional
  const void* k;
  const void* v;
  void* k_out;
  void* v_out;
  int32_t* kept_copy;           // optional: kept_idx and offsets once more, written by the gather
  int32_t* offsets_copy;
  long long capacity;
};
bool select_list_supported(const Problem& pb);
int select_list_cluster(const Problem& pb);      // CTAs per segment
cudaError_t launch_select_list(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches);
bool select_cluster_supported(const Problem& pb);
cudaError_t launch_select_cluster(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches);
cudaError_t launch_gather(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches);

// ---- tensor-core score kernel: arguments and launch plans ----------------------------------------------------
// What the layers of a launch share.  A layer's history keys form a flat list of 128-key tiles, segment after segment;
// consecutive whole segments form groups, and the CTAs of a launch share a group's tiles evenly.
struct ScoreShape {
  SeqTables tab;
  int n_seqs, n_kv_heads, G, window;
  int R, Rp, MT;                // score rows per KV head: G * window; rounded up to 32; 128-row blocks of them
  int halves;                   // 64-element halves of a key row (head_dim / 64)
  int n_stages, slot_stride;        // K tiles in flight; split ranges that may share a segment (stride of the statistics)
  int q_head_inner, k_head_inner;   // tensor-map dimension order: 1 = the head axis comes before the row axis
  int total_tiles, n_cta;       // of one layer; CTAs
  // The groups the tiles of a list are walked in: group_layers = 0: a layer's n_groups groups, group_tile their first
  // tiles; else that many whole layers together.
  int n_groups, group_layers;
  float scale_log2;
  int group_tile[kListMaxGroups + 1];
};
struct ScoreLayer {
  alignas(64) CUtensorMap tm_q;
  alignas(64) CUtensorMap tm_k;
  void* part;                   // row statistics (see StatView)
  float* vote;
  LseSource lse;                // where the vote pass takes the rows' log-sum-exp from besides the statistics pass
  int32_t* status;
  const int32_t* budgets;       // launches for bounds alone
};
// One layer's score problem, ready to launch.
struct ScorePlan {
  ScoreShape sh;
  ScoreLayer lay;
};
// Fills a plan for a problem whose workspace is bound; sh.n_cta = 0 when there is no history to score.
// cudaErrorNotSupported when the driver has no tensor-map encoder.
cudaError_t plan_score_tensor(const Problem& pb, const int32_t* cu_host, int32_t* status, ScorePlan* plan);
cudaError_t plan_score_layer(const Problem& pb, int32_t* status, ScoreLayer* lay);    // the layer's part alone
int sm_count();
int score_list_stages(int MT, int halves);
// The score kernel over a list of layers of one shape: passes 1 = row statistics, 2 = votes from the callers' row
// statistics, 3 = both, kScoreBound = row statistics and estimated votes (slkv_bound.cu), kScoreWide = both with the same row sums
// as those bit for bit; sync: Problem's.
constexpr int kScoreBound = 4, kScoreWide = 5;
// A list for bounds computes every vote of a segment that keeps so many positions and that share of them.
constexpr int kEveryVoteCount = 512, kEveryVoteShare = 64;
#ifdef __CUDACC__
__device__ __forceinline__ bool every_vote(int len, int budget, int window) {
  const int n = len - window, k = min(len, max(budget, window)) - window;
  return k >= kEveryVoteCount && k < n && (long long)k * kEveryVoteShare >= n;
}
#endif
cudaError_t launch_score_list(const ScoreShape& sh, const ScoreLayer* lay, int n_layers, int passes,
                              unsigned long long* sync, cudaStream_t st, int* launches, bool cleared = false);
// Scores and selection of a list in one product with every key (slkv_bound.cu).  cudaErrorNotSupported: nothing is launched.
bool bound_possible(const Problem& pb);
bool bound_shape(const Problem& pb);              // shapes of which some lists go that way: both passes then take the same row sums
bool bound_list_supported(const Problem& pb, const TailLayer* tail, int n_layers);
void set_list_way(int way);                       // of this thread: 0 by rule, 1 one product wherever it can be, 2 two
cudaError_t launch_bound_list(const Problem& pb, const ScoreShape& sh, const ScoreLayer* lay, const TailLayer* tail, int n_layers,
                              cudaStream_t st, int* launches);
// lse_out null: into the layer's own statistics area
cudaError_t launch_merge_lse_tensor(const ScoreShape& sh, const ScoreLayer& lay, float* lse_out, float out_scale,
                                    cudaStream_t st, int* launches);
// ---- a whole layer in one launch (slkv_layer_tc.cu, slkv_layer_fma.cu) ---------------------------------------------
// CTAs per segment, or 0 where the shape is not taken; select false, tail null: the pooled scores alone.  pooled may be null with a
// tail.
int layer_tc_clusters_for(int n_seg);
int layer_tc_cluster(const Problem& pb, bool select);
int layer_fma_cluster(const Problem& pb, bool select);
cudaError_t launch_layer_fma(const Problem& pb, int cs, const TailLayer* tail, float* pooled, int32_t* status, cudaStream_t st,
                             int* launches);
cudaError_t launch_layer_tc(const Problem& pb, int cs, const TailLayer* tail, float* pooled, int32_t* status, cudaStream_t st,
                            int* launches);
// Timeline buffer of this thread (diagnostics), or null: kTraceSlots words per CTA.
unsigned long long* tensor_trace_buffer(int n_cta);
// Diagnostics: arm / consume the one-shot switches that make an inter-CTA wait of this thread's next launch run out: a wait for words
// in memory (slkv_score_pipe.cu, slkv_score_simt.cu; 1, 2), one of the kernels that do a whole layer (1 for the row sums, where the
// launch forms them, 2 for the votes).
void expire_next_wait(int on);
int take_expire_next_wait();
bool next_wait_expires();                        // armed
void expire_next_layer_wait(int on);
int take_expire_next_layer_wait(bool sums);

}  // namespace slkv

// Window relevance scores on the 5th-generation tensor cores (Sec. 3.4, Eq. 7; Algorithm 3; Eq. 3-4), a list of layers
// per launch.  bf16, head_dim 64 or 128, up to 256 query rows per KV head.
//
// Two passes over a layer's keys, in 128-key tiles (one where all that is asked for is what is kept: slkv_bound.cu):
//   statistics  S = Q K^T with the G*w query rows as the M dimension: a TMEM lane -- one thread -- owns a query row and
//               sums 2^s over a tile's keys in fp32, over a run of tiles in fp64, and adds the run's sum to the row's;
//   votes       S^T = K Q^T with the keys as the M dimension: a thread owns a key, and
//               vote[j] = (1/G) sum_rows 2^(s_rj - lse_r) is a thread-local sum and a coalesced store.
// The votes of a segment need its rows' statistics over all keys, i.e. from other CTAs.  The layers of a list and the
// groups of segments inside a layer are independent, so every CTA (one per SM) walks one stream of phases
//   S(0) .. S(lag-1), S(lag), V(0), S(lag+1), V(1), ..., V(last)
// over groups of about 32 MB of keys (1024 tiles at head_dim 128): by the time V(g) is due, the others have published S(g),
// nobody waits, and its keys are still in L2.
//
// Roles (640 threads, one CTA per SM; a twenty-first warp would cost every thread 16 registers):
//   warp 0     TMA loads of K tiles (ring of 2-4 x 32 KB, or more of 16 KB) and Q tiles; it never waits for Q while K stages are free
//   warp 1     tcgen05.mma, 128 x 128 products into four 128-column TMEM accumulators ("units")
//   warp 2     works out the runs (consecutive tiles of one segment) and hands them to the others through shared memory;
//              announces a group's statistics to the other CTAs once this CTA's share is out
//   warp 3     fetches a segment's statistics as log-sum-exps for the vote phase, ahead of its start
//   warps 4-19 four warpgroups, unit u belongs to warpgroup u % 4: TMEM -> registers -> exponentials
// so that the warps that do the arithmetic -- what bounds the kernel -- meet no other CTA, no global latency, no CTA-wide
// barrier and no launch parameters: with every role walking the phases by itself, divisions and constant-cache misses
// (the parameters of a list are kilobytes) took 3600 cycles per run and 1000 per tile of the MMA thread.
//
// What bounds it and why this shape (one B200, tiles of 128 keys x 128 rows, clock cycles per tile and SM):
//   - exponentials: 16384 per tile at 16 per clock on the special-function unit = 1024; one in eight (statistics, but for the
//     shapes of one product, see TileSum) or sixteen (votes) goes to the FMA pipe, and scale / subtract / sum run on packed pairs;
//   - shared memory: an MMA with both operands there reads 64 KB per tile at 128 B per clock, the K tile is 32 KB more:
//     730 measured for loads and MMAs alone;
//   - two epilogue warpgroups instead of four: 1250; sums over the keys across lanes instead of a lane per row: 1255;
//   - power: held for more than some milliseconds the part runs at its 1 kW limit, with every tile from HBM at 1.05 GHz
//     (0.98 us per tile, MMAs alone 0.78), with tiles from L2 at 1.5 GHz (0.68 us).  Hence the groups.
// Against the kernels before it (two streams with two accumulators and two warpgroups each on 128 SMs for up to 128 rows,
// one launch per layer with a grid-wide barrier for more), a step of 32 layers, held: 32k tokens, 128 rows: 1120 -> 870 us;
// eight ragged sequences of 147k tokens, 256 rows: 9890 -> 6640 us; 131k tokens, 256 rows: 9210 -> 5820 us.
// Every wait is bounded (1 s): SLKV_ERR_DEVICE_TIMEOUT in the status words, TMEM freed, return.
#include <cuda.h>

#include <cstdlib>
#include <cstring>

#include "slkv_internal.cuh"
#include "slkv_tc_device.cuh"

namespace slkv {
namespace {

constexpr int kWgs = 4;                              // epilogue warpgroups = TMEM units
constexpr int kListThreads = 128 + kWgs * 128;
constexpr int kMaxStages = 6;
constexpr int kPlain = 0, kWide = 1, kBound = 2;      // kinds of k_score_list
// Shared memory behind the Q tile and the K ring: mbarriers and flags, far row statistics [2][kWgs][128] (sum, reference),
// log-sum-exps [2][256], half votes [2][4][128], runs.
constexpr int kBarBytes = 640;
constexpr int kStatBytes = 2 * kWgs * 128 * 8;
constexpr int kLseBytes = 2 * 256 * 4;
constexpr int kHalfVoteBytes = 2 * 4 * 128 * 4;
constexpr int kPartBytes = kWgs * 2 * 4 * 128 * 4;      // bounds: per warpgroup two slots of its warps' shares, see bound_run; half votes there, too
// Two Q tiles, also where that leaves the ring no more than two K tiles (R > 128, d = 128): the next run's queries are
// there when its keys are.  One Q tile and four K tiles cost a pause of 1.6 us in every run of about 25: 128k positions
// 5935 -> 5810 us, eight sequences of 4k - 32k 6830 -> 6690 us (32 layers each).
constexpr int kQTiles = 2;
constexpr int kRunSlots = 8;                         // runs handed out ahead
constexpr int kFirstBytes = 2 * kWgs * 128 * 4;      // bounds: [2][kWgs][128] sums over the first tiles of a run, see bound_run
constexpr int kRunsAt = kBarBytes + kStatBytes + kLseBytes + kHalfVoteBytes, kRunsAtBound = kBarBytes + kStatBytes + kLseBytes + kPartBytes + kFirstBytes;
constexpr int kTail = kRunsAt + kRunSlots * 128, kTailBound = kRunsAtBound + kRunSlots * 128;

// The clearing of the statistics and the groups' counts: one word with the launch's tag (40 bits) above two counts of 12 bits,
// CTAs that are done and CTAs that have cleared their share.  A CTA that finds another value puts the tag first; the last CTA
// out puts the word back to zero.  (A flag per CTA, as the FMA kernel has it, saves that round trip, but here it is hidden
// behind the first tiles, and 148 CTAs polling 148 flags are not: 32 layers of 4001 tokens 127.4 -> 130.4 us.)
struct WordSync {
  unsigned long long* word;    // the counts begin kSyncFlags words further on
  unsigned long long tag;
  unsigned expect;             // CTAs to wait for: all of them
  __device__ __forceinline__ unsigned* counts() const { return reinterpret_cast<unsigned*>(word + kSyncFlags); }
  // This CTA has cleared its share (one thread, behind a barrier with those that did).
  __device__ __forceinline__ void arrive() const {
    unsigned long long seen = 0;                             // what a launch leaves behind
    for (int i = 0; i < 3; ++i) {                            // the word changes once, from whatever it was to the tag
      unsigned long long old;
      asm volatile("atom.acq_rel.gpu.global.cas.b64 %0, [%1], %2, %3;"
                   : "=l"(old) : "l"(word), "l"(seen), "l"(tag << 24 | 1u) : "memory");
      if (old == seen) return;
      if (old >> 24 == tag) break;
      seen = old;
    }
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(word) : "memory");
  }
  __device__ __forceinline__ bool all_arrived() const {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(word) : "memory");
    return v >> 24 == tag && (unsigned)(v & 0xfffu) >= expect;
  }
  // This CTA, which has arrived, will not touch the counts any more.
  __device__ __forceinline__ void leave() const {
    unsigned long long old;
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], 4096;" : "=l"(old) : "l"(word) : "memory");
    if ((unsigned)(old >> 12 & 0xfffu) == gridDim.x - 1) *word = 0;
  }
};

struct ListArgs {
  ScoreShape sh;
  ScoreLayer lay[kListMaxLayers];
  int n_layers, passes, lag;
  int group_layers, n_groups;  // as in ScoreShape; groups of the whole list
  int first_layers;            // layers whose statistics are cleared before any CTA adds to some (see fetch_lse)
  WordSync sync;               // counts [n_groups]: CTAs that have published the group's statistics
  unsigned target;             // value a group's count reaches when every CTA has published
  unsigned long long* trace;
};

// A run as warp 2 hands it out: consecutive tiles of one segment, in one pass.
struct alignas(16) RunDesc {
  int kind;                    // 0 statistics, 1 votes, 2 the end; count = 0: a phase in which this CTA has no tiles
  int count;                   // tiles
  int n_valid;                 // history keys from the run's first one to the segment's end
  int tok;                     // token of the run's first key
  int s, g;
  int gg;                      // group of the list; statistics: published with this run when last != 0
  int last;
  int n_slots;                 // split ranges that share the segment
  int seg;
  int q_y, q_z;                // coordinates of the Q tile
  const CUtensorMap* tm_q;
  const CUtensorMap* tm_k;
  int slot;                    // this CTA's place among the segment's split ranges
  float* vote;                 // of the run's first key
  float* weight;               // bounds: where the run's row weights go, the second ones `second` floats further on
  int second;
  double* acc;                 // the segment's row sums ...
  const unsigned* far;         // ... and far bits
  int sums, win;               // votes: the log-sum-exps come from the sums, with window statistics
  int layer;
};
static_assert(sizeof(RunDesc) <= 128, "run descriptor");

// What the roles keep in registers: copied through shared memory, so that no launch parameter is read in a loop.
struct Smem {
  uint32_t q, k, bar0, tmem;
  int q_half, q_bytes, stage_bytes, n_stages;
  int R, Rp, k_head_inner, both;
  float sc, inv_g;
  volatile int* abort_flag;
  RunDesc* runs;               // [kRunSlots]
  float* stat_z;               // [2][kWgs][128]: far parts (see StatView) on their way out
  float* stat_m;               // likewise
  unsigned* stat_far;          // [2]: warps that have any
  float* lse;                  // [2][256], negated
  float* half_vote;            // [2][4][128]; bounds: see bound_run
  float* first;                // [2][kWgs][128]
  __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * (uint32_t)i; }
  __device__ __forceinline__ uint32_t full(int st) const { return bar(st); }
  __device__ __forceinline__ uint32_t empty(int st) const { return bar(kMaxStages + st); }
  __device__ __forceinline__ uint32_t unit_full(int u) const { return bar(2 * kMaxStages + u); }
  __device__ __forceinline__ uint32_t unit_empty(int u) const { return bar(2 * kMaxStages + 4 + u); }
  // run k's Q tile: slot and phase
  __device__ __forceinline__ int q_slot(int k) const { return k & (kQTiles - 1); }
  __device__ __forceinline__ uint32_t q_phase(int k) const { return (uint32_t)(k / kQTiles) & 1u; }
  __device__ __forceinline__ uint32_t q_full(int k) const { return bar(2 * kMaxStages + 8 + q_slot(k)); }
  __device__ __forceinline__ uint32_t q_empty(int k) const { return bar(2 * kMaxStages + 10 + q_slot(k)); }
  __device__ __forceinline__ uint32_t stat_full(int s) const { return bar(2 * kMaxStages + 12 + s); }
  __device__ __forceinline__ uint32_t stat_empty(int s) const { return bar(2 * kMaxStages + 14 + s); }
  __device__ __forceinline__ uint32_t lse_full(int s) const { return bar(2 * kMaxStages + 16 + s); }
  __device__ __forceinline__ uint32_t lse_empty(int s) const { return bar(2 * kMaxStages + 18 + s); }
  __device__ __forceinline__ uint32_t half_full(int pair, int turn) const { return bar(2 * kMaxStages + 20 + 4 * pair + turn); }
  __device__ __forceinline__ uint32_t run_full(int k) const { return bar(2 * kMaxStages + 28 + (k & (kRunSlots - 1))); }
  __device__ __forceinline__ uint32_t run_empty(int k) const { return bar(2 * kMaxStages + 28 + kRunSlots + (k & (kRunSlots - 1))); }
  __device__ __forceinline__ uint32_t cleared() const { return bar(2 * kMaxStages + 29 + 2 * kRunSlots); }
  __device__ __forceinline__ uint32_t drain() const { return bar(2 * kMaxStages + 28 + 2 * kRunSlots); }   // a wait ran out
  __device__ __forceinline__ uint32_t rest_cleared() const { return bar(2 * kMaxStages + 30 + 2 * kRunSlots); }
  __device__ __forceinline__ uint32_t part_full(int i) const { return bar(2 * kMaxStages + 33 + 2 * kRunSlots + i); }   // [sharers][2]
  __device__ __forceinline__ uint32_t again_full() const { return bar(2 * kMaxStages + 41 + 2 * kRunSlots); }
  __device__ __forceinline__ uint32_t first_full(int s) const { return bar(2 * kMaxStages + 31 + 2 * kRunSlots + s); }
};
constexpr int kNumBars = 2 * kMaxStages + 42 + 2 * kRunSlots;
constexpr int kHeadInts = 7;
static_assert(kNumBars * 8 + kHeadInts * 4 + 16 <= kBarBytes, "mbarriers");
constexpr int kRunReaders = 4 + 4 * kWgs;              // arrivals that free a run slot: one per reading thread or warp

// The runs of this CTA, one after the other.  A group's tiles are counted through its layers.
struct GroupShare {
  int layer0, base, T, n, idx, begin, end;                 // begin, end: this CTA's tiles, counted through the group
};
__device__ __forceinline__ GroupShare group_share(const ListArgs& a, int gg) {
  const ScoreShape& sh = a.sh;
  GroupShare g;
  if (a.group_layers == 0) {
    g.layer0 = gg / sh.n_groups;
    const int grp = gg - g.layer0 * sh.n_groups;
    g.base = sh.group_tile[grp];
    g.T = sh.group_tile[grp + 1] - g.base;
  } else {
    g.layer0 = gg * a.group_layers;
    g.base = 0;
    g.T = min(a.group_layers, a.n_layers - g.layer0) * sh.total_tiles;
  }
  // the split index moves on by one CTA per group, so that the larger shares go round
  const int i = (int)blockIdx.x + gg % sh.n_cta;
  g.idx = i >= sh.n_cta ? i - sh.n_cta : i;
  g.n = min(sh.n_cta, g.T);
  const bool takes_part = g.idx < g.n;
  g.begin = takes_part ? split_begin(g.idx, g.T, g.n) : 0;
  g.end = takes_part ? split_begin(g.idx + 1, g.T, g.n) : 0;
  return g;
}
template <bool BOUND>
struct RunWalk {
  int step, pos, kind, gg;
  GroupShare s;
  __device__ __forceinline__ void start() { step = 0; pos = s.end = 0; }
  // The next run into d (shared memory); kind 2 behind the last one.
  __device__ __forceinline__ void next(const ListArgs& a, RunDesc& d) {
    const ScoreShape& sh = a.sh;
    const int NG = a.n_groups;
    while (pos >= s.end) {                                   // the next phase
      if (!BOUND && a.passes == 3) {
        const int p = step >> 1;
        if (p >= NG + a.lag) { d.kind = kind = 2; return; }
        kind = step & 1;
        gg = kind ? p - a.lag : p;
      } else {
        if (step >= NG) { d.kind = kind = 2; return; }
        kind = !BOUND && a.passes == 2;
        gg = step;
      }
      ++step;
      if (gg < 0 || gg >= NG) continue;
      s = group_share(a, gg);
      pos = s.begin;
      if (pos >= s.end && kind == 0) {
        d.kind = 0;
        d.gg = gg;
        d.count = 0;
        d.last = 1;
        return;
      }
    }
    const int in_group = a.group_layers == 0 ? 0 : pos / sh.total_tiles;
    const int layer = s.layer0 + in_group, before = in_group * sh.total_tiles - s.base;  // group tile = layer tile + before
    const ScoreLayer& L = a.lay[layer];
    d.kind = kind;
    d.gg = gg;
    d.layer = layer;
    d.tm_q = &L.tm_q;
    d.tm_k = &L.tm_k;
    const Run r = locate(sh, pos - before, s.end - before);
    pos += r.count;
    d.count = r.count;
    d.n_valid = r.n_hist - r.t0 * kTileKeys;
    d.tok = sh.tab.cu_at(r.s) + r.t0 * kTileKeys;
    d.s = r.s;
    d.g = r.g;
    d.last = pos >= s.end;
    const int first = split_index(r.seg_tile0 + before, s.T, s.n);
    d.n_slots = split_index(r.seg_tile0 + r.tiles_seg - 1 + before, s.T, s.n) - first + 1;
    d.slot = s.idx - first;
    d.vote = L.vote + sh.tab.hist_at(r.s) * sh.n_kv_heads + (long long)r.g * r.n_hist + r.t0 * kTileKeys;
    const int seg = r.s * sh.n_kv_heads + r.g;
    d.seg = seg;
    d.acc = static_cast<double*>(L.part) + (long long)seg * sh.R;
    d.far = reinterpret_cast<unsigned*>(static_cast<double*>(L.part) + (long long)sh.n_seqs * sh.n_kv_heads * sh.R) + seg * kFarWords;
    d.second = sh.n_seqs * sh.n_kv_heads * sh.slot_stride * sh.R;
    // the places of this CTA's far part, which a segment with estimates does not use
    d.weight = const_cast<float*>(reinterpret_cast<const float*>(d.far + (sh.n_seqs * sh.n_kv_heads - seg) * kFarWords)) + ((long long)seg * sh.slot_stride + d.slot) * sh.R;
    d.sums = a.passes == 3;
    d.win = L.lse.win_m != nullptr;
    d.q_y = sh.q_head_inner ? r.g * sh.G : 0;
    d.q_z = sh.q_head_inner ? 0 : r.g * sh.G;
  }
};
// The segments of a list all of whose votes are computed: warp 2's way through their tiles, which the CTAs share evenly.
struct FullWalk {
  int pos, end;
  // Segment i of the list: tiles that count.
  static __device__ __forceinline__ int tiles(const ListArgs& a, int i) {
    const ScoreShape& sh = a.sh;
    const int n_seg = sh.n_seqs * sh.n_kv_heads, layer = i / n_seg, seg = i - layer * n_seg, s = seg / sh.n_kv_heads;
    if (layer >= a.n_layers) return 0;
    const int len = sh.tab.cu_at(s + 1) - sh.tab.cu_at(s);
    return every_vote(len, __ldcg(a.lay[layer].budgets + (seg - s * sh.n_kv_heads)), sh.window) ? sh.tab.tile_at(s + 1) - sh.tab.tile_at(s) : 0;
  }
  // The segment that holds tile x, and the tiles before it; with no such tile, -1 and the number of tiles.
  static __device__ __forceinline__ int find(const ListArgs& a, int x, int& before) {
    const int lane = threadIdx.x & 31, n = a.n_layers * a.sh.n_seqs * a.sh.n_kv_heads;
    before = 0;
    for (int base = 0; base < n; base += 32) {
      const int t = tiles(a, base + lane);
      int inc = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, x >= before + inc - t && x < before + inc);
      if (hit) {
        const int l = __ffs(hit) - 1;
        before += __shfl_sync(0xffffffffu, inc - t, l);
        return base + l;
      }
      before += __shfl_sync(0xffffffffu, inc, 31);
    }
    return -1;
  }
  __device__ __forceinline__ void start(const ListArgs& a) {
    int all;
    find(a, 0x7fffffff, all);
    pos = split_begin((int)blockIdx.x, all, (int)gridDim.x);
    end = split_begin((int)blockIdx.x + 1, all, (int)gridDim.x);
  }
  // The next run into d (lane 0); its kind.
  __device__ __forceinline__ int next(const ListArgs& a, RunDesc& d) {
    if (pos >= end) {
      if ((threadIdx.x & 31) == 0) d.kind = 2;
      return 2;
    }
    int before;
    const int i = find(a, pos, before);
    const ScoreShape& sh = a.sh;
    const int n_seg = sh.n_seqs * sh.n_kv_heads, layer = i / n_seg, seg = i - layer * n_seg, s = seg / sh.n_kv_heads, g = seg - s * sh.n_kv_heads;
    const int tiles_seg = sh.tab.tile_at(s + 1) - sh.tab.tile_at(s), t0 = pos - before, count = min(end - pos, tiles_seg - t0);
    pos += count;
    if ((threadIdx.x & 31) == 0) {
      const ScoreLayer& L = a.lay[layer];
      const int n_hist = sh.tab.cu_at(s + 1) - sh.tab.cu_at(s) - sh.window;
      d.kind = 1;
      d.gg = 0;
      d.layer = layer;
      d.tm_q = &L.tm_q;
      d.tm_k = &L.tm_k;
      d.count = count;
      d.n_valid = n_hist - t0 * kTileKeys;
      d.tok = sh.tab.cu_at(s) + t0 * kTileKeys;
      d.s = s;
      d.g = g;
      d.last = 0;
      d.n_slots = list_slots(sh, a.n_layers, layer, s, g).n;
      d.slot = 0;
      d.vote = L.vote + sh.tab.hist_at(s) * sh.n_kv_heads + (long long)g * n_hist + t0 * kTileKeys;
      d.seg = seg;
      d.acc = static_cast<double*>(L.part) + (long long)seg * sh.R;
      d.far = reinterpret_cast<unsigned*>(static_cast<double*>(L.part) + (long long)n_seg * sh.R) + seg * kFarWords;
      d.weight = nullptr;
      d.second = 0;
      d.sums = 1;
      d.win = L.lse.win_m != nullptr;
      d.q_y = sh.q_head_inner ? g * sh.G : 0;
      d.q_z = sh.q_head_inner ? 0 : g * sh.G;
    }
    return 1;
  }
};
// Run k, read by a single thread or by a whole warp; kind 2 when there is none left (or a wait ran out).
template <bool WARP>
__device__ __forceinline__ RunDesc take_run(const Smem& c, int k) {
  bool ok = mbar_wait(c.run_full(k), (k / kRunSlots) & 1, c.abort_flag);
  if (WARP) ok = __all_sync(0xffffffffu, ok) != 0;
  RunDesc d;
  d.kind = 2;
  if (ok) d = c.runs[k & (kRunSlots - 1)];
  if (WARP) __syncwarp();
  if (!WARP || (threadIdx.x & 31) == 0) mbar_arrive(c.run_empty(k));
  return d;
}

// ---- warp 0, one thread: TMA loads ------------------------------------------------------------------------------
template <int MT, int HALVES, bool BOUND>
__device__ __forceinline__ void producer(const Smem& c) {
  int st = 0, it = 0, n = 0;                                 // stage, tiles so far, runs so far
  uint32_t st_phase = 0;
  bool ok = true, q_due = false;
  const CUtensorMap* q_map = nullptr;
  // the statistics pass asks L2 to keep its keys for the vote pass, which lets them go
  const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
  int q_y = 0, q_z = 0, q_s = 0;
  // Q of run number n - 1
  auto load_q = [&]() {
    const uint32_t bar = c.q_full(n - 1), dst = c.q + (uint32_t)(c.q_slot(n - 1) * c.q_bytes);
    mbar_expect_tx(bar, (uint32_t)(HALVES * c.R * 128));
    for (int h = 0; h < HALVES; ++h) tma_load_4d(dst + h * c.q_half, q_map, 64 * h, q_y, q_z, q_s, bar);
    q_due = false;
  };
  auto q_free = [&](bool wait) {
    const uint32_t bar = c.q_empty(n - 1), phase = c.q_phase(n - 1) ^ 1u;
    return wait ? mbar_wait(bar, phase, c.abort_flag) : mbar_test(bar, phase);
  };
  for (int k = 0; ok; ++k) {
    const RunDesc r = take_run<false>(c, k);
    if (r.kind == 2) break;
    if (r.count == 0) continue;
    if (q_due) {                                             // the run before is shorter than the ring: its Q first
      ok = q_free(true);
      if (!ok) break;
      load_q();
    }
    q_map = r.tm_q; q_y = r.q_y; q_z = r.q_z; q_s = r.s;
    q_due = true;
    ++n;
    const uint64_t policy = !BOUND && r.kind == 0 && c.both ? keep : drop;
    const Spread<MT> order(BOUND && r.kind == 0 ? r.count : 0);
    for (int i = 0; i < r.count; ++i, ++it) {
      const int tok = r.tok + (BOUND && r.kind == 0 ? order.tile(i) : i) * kTileKeys;
      // a stage of the ring, and Q as soon as the MMAs of the run that had its slot are through with it
      bool got = false;
      unsigned long long t0 = 0;
      for (unsigned spin = 0; !got; ++spin) {
        if (q_due && q_free(false)) load_q();
        got = q_due ? mbar_test(c.empty(st), st_phase ^ 1u) : mbar_try(c.empty(st), st_phase ^ 1u);
        if (got) break;
        if (spin == 0) t0 = now_ns();
        if ((spin & 63u) == 63u) {
          if (*c.abort_flag) break;
          if (now_ns() - t0 > kWaitLimitNs) { *c.abort_flag = 1; break; }
        }
        if (q_due) __nanosleep(32);
      }
      if (!got) { ok = false; break; }
      const uint32_t fb = c.full(st), dst = c.k + (uint32_t)(st * c.stage_bytes);
      mbar_expect_tx(fb, (uint32_t)c.stage_bytes);
      const int ky = c.k_head_inner ? r.g : tok, kz = c.k_head_inner ? tok : r.g;
      for (int h = 0; h < HALVES; ++h) tma_load_3d_hint(dst + h * kHalfBytes, r.tm_k, 64 * h, ky, kz, fb, policy);
      if (++st == c.n_stages) { st = 0; st_phase ^= 1u; }
    }
  }
  if (ok && q_due) {
    ok = q_free(true);
    if (ok) load_q();
  }
  if (!ok || *c.abort_flag) {
    // give loads already in flight a bounded chance to land before the CTA's shared memory goes away
    const unsigned long long t0 = now_ns();
    for (int s2 = 0; s2 < c.n_stages; ++s2) {
      const int last = it - 1 - ((it - 1 - s2) % c.n_stages + c.n_stages) % c.n_stages;   // last issue into stage s2
      if (it == 0 || last < 0) continue;
      while (!mbar_try(c.full(s2), (last / c.n_stages) & 1) && now_ns() - t0 < kWaitLimitNs) {}
    }
    const int loaded = n - (q_due ? 1 : 0);                  // Q tiles asked for; the last kQTiles may be in flight
    for (int k = loaded - kQTiles < 0 ? 0 : loaded - kQTiles; k < loaded; ++k)
      while (!mbar_try(c.q_full(k), c.q_phase(k)) && now_ns() - t0 < kWaitLimitNs) {}
  }
}

// ---- warp 1, one thread: MMAs -------------------------------------------------------------------------------------
template <int MT, int HALVES>
__device__ __forceinline__ void issuer(const Smem& c) {
  // statistics: D[row, key] = Q K^T (A = Q, B = K); votes: D[key, row] = K Q^T (A = K, B = Q); a unit per 128-row block
  // of Q (one 256-column product for the votes would read less shared memory, but it takes two units at once and makes
  // both wait for the slower one's warpgroup)
  const uint32_t idesc_s = instr_desc(128, kTileKeys), idesc_v0 = instr_desc(kTileKeys, min(c.Rp, 128)),
                 idesc_v1 = instr_desc(kTileKeys, max(c.Rp - 128, 32));
  const uint64_t q_desc0 = smem_desc(c.q), k_desc0 = smem_desc(c.k);
  const uint64_t q_hi = (uint64_t)(c.q_half >> 4), k_hi = (uint64_t)(kHalfBytes >> 4);
  constexpr bool two_halves = HALVES == 2;
  int st = 0, uc = 0, n = 0;                                  // stage, units so far, runs so far
  uint32_t st_phase = 0;
  bool ok = true;
  auto product = [&](uint32_t d, uint64_t ad, uint64_t a_hi, uint64_t bd, uint64_t b_hi, uint32_t idesc) {
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) tc_mma(d, ad + (uint64_t)(ks * 2), bd + (uint64_t)(ks * 2), idesc, ks > 0);
    if (two_halves) {
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) tc_mma(d, ad + a_hi + (uint64_t)(ks * 2), bd + b_hi + (uint64_t)(ks * 2), idesc, 1);
    }
  };
  auto unit_free = [&](int u_count) {
    return mbar_wait(c.unit_empty(u_count & 3), ((u_count >> 2) & 1) ^ 1, c.abort_flag);
  };
  for (int k = 0; ok; ++k) {
    const RunDesc r = take_run<false>(c, k);
    if (r.kind == 2) break;
    if (r.count == 0) continue;
    ok = mbar_wait(c.q_full(n), c.q_phase(n), c.abort_flag);
    const uint64_t q_desc = q_desc0 + (uint64_t)((c.q_slot(n) * c.q_bytes) >> 4);
    for (int i = 0; i < r.count && ok; ++i) {
      ok = mbar_wait(c.full(st), st_phase, c.abort_flag);
      if (!ok) break;
      const uint64_t kd = k_desc0 + (uint64_t)((st * c.stage_bytes) >> 4);
      for (int mt = 0; mt < MT && ok; ++mt, ++uc) {
        ok = unit_free(uc);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = c.tmem + (uint32_t)((uc & 3) * 128);
        const uint64_t qd = q_desc + (uint64_t)(mt * ((128 * 128) >> 4));
        if (r.kind == 0) product(d, qd, q_hi, kd, k_hi, idesc_s);
        else product(d, kd, k_hi, qd, q_hi, mt == 0 ? idesc_v0 : idesc_v1);
        if (mt == MT - 1) tc_commit(c.empty(st));            // K stage free once these MMAs have read it
        tc_commit(c.unit_full(uc & 3));
      }
      if (++st == c.n_stages) { st = 0; st_phase ^= 1u; }
    }
    tc_commit(c.q_empty(n));              // Q tile free once the run's MMAs are done
    ++n;
  }
  if (!ok || *c.abort_flag) {
    // gave up: the MMAs this thread has issued must be through before the accumulators are released
    tc_commit(c.drain());
    const unsigned long long t0 = now_ns();
    while (!mbar_try(c.drain(), 0) && now_ns() - t0 < kWaitLimitNs) {}
  }
}

// ---- warp 2: hands out the runs; announces statistics -----------------------------------------------------------------
// Whatever is possible next is done: a run slot that has come free is filled, statistics that are out are announced.
template <int MT, bool BOUND>
__device__ __forceinline__ void scheduler_publisher(const Smem& c, const ListArgs& a) {
  const int lane = threadIdx.x & 31;
  int k_out = 0, k_in = 0;                 // runs handed out, runs done with as publisher
  int n = 0;                               // statistics runs so far
  bool all_out = false;
  const int n_seg = a.sh.n_seqs * a.sh.n_kv_heads, stride = a.sh.slot_stride;
  RunWalk<BOUND> w;
  w.start();
  FullWalk full;
  bool votes = false;                      // bounds: behind the statistics' last run
  unsigned long long t0 = 0;
  unsigned idle = 0;
  while (true) {
    bool moved = false;
    if (!all_out && __any_sync(0xffffffffu, mbar_test(c.run_empty(k_out), ((k_out / kRunSlots) & 1) ^ 1))) {
      int kind = 0;
      RunDesc& d = c.runs[k_out & (kRunSlots - 1)];
      if (lane == 0 && !(BOUND && votes)) {
        w.next(a, d);
        kind = w.kind;
      }
      if constexpr (BOUND) {
        kind = __shfl_sync(0xffffffffu, kind, 0);
        if (kind == 2 && !votes) {
          votes = true;
          pdl_wait();                                        // budgets may come from a kernel before this one
          full.start(a);
        }
        if (votes) kind = full.next(a, d);
      }
      if (lane == 0) mbar_arrive(c.run_full(k_out));
      all_out = __shfl_sync(0xffffffffu, kind, 0) == 2;    // also orders the lanes behind lane 0's stores
      ++k_out;
      moved = true;
    }
    if (k_in < k_out) {
      const RunDesc& r = c.runs[k_in & (kRunSlots - 1)];
      if (r.kind == 2) break;
      const int slot = n & 1;
      const bool stats = r.kind == 0 && r.count > 0, publish = r.kind == 0 && r.last && c.both;
      // the epilogue warps have waited for the clearing before their statistics are out; an empty share waits here
      bool ready = stats ? mbar_test(c.stat_full(slot), (n >> 1) & 1) : !publish || mbar_test(c.cleared(), 0);
      if (publish && r.gg == 0) ready = ready && mbar_test(c.rest_cleared(), 0);
      if (__any_sync(0xffffffffu, ready)) {
        if (stats) {
          const unsigned far = c.stat_far[slot];
          if (far) {                                           // rare: scores beyond fp64's range
            const StatView st = stat_view(a.lay[r.layer].part, n_seg, c.R, stride);
            const size_t at0 = ((size_t)r.seg * stride + r.slot) * c.R;
            for (int row = lane; row < c.R; row += 32) {
              float Z = 0.f, M = 0.f;
              for (int wg = MT == 1 ? 0 : row >> 7; wg < kWgs; wg += MT)
                if (far >> (wg * 4 + ((row & 127) >> 5)) & 1u) {
                  const int at = (slot * kWgs + wg) * 128 + (row & 127);
                  stat_add(Z, M, c.stat_z[at], c.stat_m[at]);
                }
              __stcg(st.far_z + at0 + row, Z);
              __stcg(st.far_m + at0 + row, M);
            }
            if (lane == 0) {
              atomicOr(st.far + (size_t)r.seg * kFarWords + (r.slot >> 5), 1u << (r.slot & 31));
              c.stat_far[slot] = 0;
            }
          }
          ++n;
        }
        const int gg = r.gg;
        __syncwarp();
        if (lane == 0) {
          if (stats) mbar_arrive(c.stat_empty(slot));
          if (publish) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.sync.counts() + gg) : "memory");
          mbar_arrive(c.run_empty(k_in));
        }
        ++k_in;
        moved = true;
      }
    }
    if (moved) { idle = 0; continue; }
    if (idle == 0) t0 = now_ns();
    if ((++idle & 63u) == 0 && (*c.abort_flag || now_ns() - t0 > kWaitLimitNs)) { *c.abort_flag = 1; break; }
    __nanosleep(50);
  }
}

// ---- warp 3: the rows' log-sum-exps (log2 units, negated) of the segments the vote phases take, ahead of them ------
// From a CTA's last tile of a group to the log-sum-exps in every other CTA's shared memory there is one hop: add to the
// rows' sums, release, acquire, load.  (Per-CTA partial sums that the consumers merge took 14 us at 37 shares, merged by
// their owners in equal parts and fetched 11 us -- twice what the phases in between cover: beside warps that saturate the
// issue slots every dependent step costs several times its latency.)
__device__ __forceinline__ void fetch_lse(const Smem& c, const ListArgs& a) {
  const int lane = threadIdx.x & 31;
  const int G = a.sh.G, window = a.sh.window, q_head_inner = a.sh.q_head_inner;
  const int n_seg = a.sh.n_seqs * a.sh.n_kv_heads, stride = a.sh.slot_stride;
  // until all CTAs have cleared their part (group = -1), or have published the group
  auto wait_count = [&](int group) {
    if (lane == 0) {
      unsigned long long t0 = 0;
      for (unsigned spin = 0;; ++spin) {
        if (group < 0) {
          if (a.sync.all_arrived()) break;
        } else {
          unsigned v;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.sync.counts() + group) : "memory");
          if (v >= a.target) break;
        }
        if (spin == 0) t0 = now_ns();
        if ((spin & 15u) == 15u && (*c.abort_flag || now_ns() - t0 > kWaitLimitNs)) { *c.abort_flag = 1; break; }
        __nanosleep(20);
      }
    }
    __syncwarp();
    return __all_sync(0xffffffffu, *c.abort_flag == 0) != 0;
  };
  if (c.both) {
    // This CTA's part of the groups' counts and the layers' statistics areas is cleared; nobody adds to them before all are.
    // The layers that come before the first vote phase first: that the others are cleared, too, a CTA says as it publishes
    // group 0, which its vote phase waits for in every other.  (All layers first: the first sums of 32 layers waited
    // until 12 us into the launch, a phase and a half.  32 layers of 4001 tokens 129 -> 127 us, of 8000 236 -> 232.)
    for (int i = blockIdx.x + lane * gridDim.x; i < a.n_groups; i += 32 * gridDim.x) __stcg(a.sync.counts() + i, 0u);
    const int words = (int)(stat_clear_bytes(n_seg, c.R) / 4);       // < 2^30; times the CTAs it takes more than 32 bits
    const int w0 = (int)((long long)blockIdx.x * words / gridDim.x), w1 = (int)((long long)(blockIdx.x + 1) * words / gridDim.x);
    // The areas' addresses in one load, a lane each, through the generic address of the parameters: read one by one from
    // the constant bank, where each is a miss, they took 15 us for 32 layers, and every CTA's first sums waited for that.
    static_assert(kListMaxLayers <= 32, "a lane per layer");
    const ListArgs* args;
    asm volatile("mov.u64 %0, %1;" : "=l"(args) : "l"(&a));
    const unsigned long long part = lane < a.n_layers ? reinterpret_cast<unsigned long long>(args->lay[lane].part) : 0ull;
    auto clear = [&](int l0, int l1) {
      for (int l = l0; l < l1; ++l) {
        unsigned* p = reinterpret_cast<unsigned*>(__shfl_sync(0xffffffffu, part, l));
        for (int i = w0 + lane; i < w1; i += 32) __stcg(p + i, 0u);
      }
      __syncwarp();
    };
    clear(0, a.first_layers);
    if (lane == 0) a.sync.arrive();
    clear(a.first_layers, a.n_layers);
    if (lane == 0) mbar_arrive(c.rest_cleared());
    if (!wait_count(-1)) return;
  }
  if (lane == 0) mbar_arrive(c.cleared());
  int n = 0, seen = -1;                    // vote runs so far; the last group known to be published
  for (int k = 0;; ++k) {
    const RunDesc r = take_run<true>(c, k);
    if (r.kind == 2) break;
    if (r.kind == 0) continue;
    // every CTA has published its share of the group (all CTAs are resident, and a statistics phase waits for nothing
    // but vote phases that are due before it, so the count gets there; bounded all the same)
    if (c.both && r.gg != seen) {
      if (!wait_count(r.gg)) break;
      seen = r.gg;
    }
    // The common case, straight through: the sums are on their way while the slot comes free, and no launch parameter is
    // touched.
    double Z[8];
    unsigned far = 0;
    if (r.sums) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (u * 32 < c.R) Z[u] = u * 32 + lane < c.R ? __ldcg(r.acc + u * 32 + lane) : 1.0;
      if (lane < kFarWords) far = __ldcg(r.far + lane);
    }
    const bool plain = r.sums && !r.win && !__any_sync(0xffffffffu, far != 0);
    const bool ok = mbar_wait(c.lse_empty(n & 1), ((n >> 1) & 1) ^ 1, c.abort_flag);
    if (!__all_sync(0xffffffffu, ok)) break;
    float* lse = c.lse + (n & 1) * 256;
    if (plain) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (u * 32 < c.R) lse[u * 32 + lane] = u * 32 + lane < c.R ? -log2_of(Z[u]) : -INFINITY;
    } else {
      const LseSource& src = a.lay[r.layer].lse;
      const StatView st = stat_view(a.lay[r.layer].part, n_seg, c.R, stride);
#pragma unroll 1
      for (int row = lane; row < c.Rp; row += 32) {
        float l2 = INFINITY;                                    // rows of padding: 2^(0 - inf) = 0
        if (row < c.R) {
          const size_t at = (size_t)r.seg * c.R + row;
          if (src.lse_opt) l2 = src.caller_lse(r.s, r.g, row, G, window, q_head_inner != 0);
          else if (!r.sums) l2 = __ldcg(st.lse + at);
          else l2 = row_lse(st, __ldcg(st.acc + at), true, r.seg, row, c.R, stride, r.n_slots, r.win != 0,
                            r.win ? src.win_m[at] : 0.f, r.win ? src.win_z[at] : 0.f);
        }
        lse[row] = -l2;
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(c.lse_full(n & 1));
    if (n == 0 && lane == 0) trace_mark(a.trace, 3);
    ++n;
  }
}

// ---- warps 4-19: the arithmetic ---------------------------------------------------------------------------------------
template <int MT, int KIND>
__device__ __forceinline__ void epilogue(const Smem& c) {
  constexpr bool BOUND = KIND == kBound;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wg = (threadIdx.x - 128) >> 7, row = threadIdx.x & 127;
  Unit u;
  u.tcol = c.tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(wg * 128);
  u.full = c.unit_full(wg);
  u.empty = c.unit_empty(wg);
  u.abort_flag = c.abort_flag;
  // MT = 1: unit u = tile u, this warpgroup's tiles are wg, wg + 4, ...; MT = 2: tile t has the units 2t (rows 0-127,
  // or the votes' first 128 rows) and 2t + 1
  constexpr int every = MT == 1 ? kWgs : kWgs / 2, log_every = MT == 1 ? 2 : 1;
  const int mine = MT == 1 ? wg : wg >> 1, mt = MT == 1 ? 0 : wg & 1;
  const bool rows_here = mt * 128 + (warp & 3) * 32 < c.R;                // some row of this warp's lanes exists
  const int own = BOUND ? (row & ~31) + quad_row() : row;                // the row whose statistics this thread ends up with
  int it = 0, units = 0, n_stat = 0, n_vote = 0, n_half = 0, n_part = 0, n_again = 0;
  for (int k = 0;; ++k) {
    const RunDesc r = take_run<true>(c, k);
    if (r.kind == 2) break;
    if (r.count == 0) continue;
    const int i0 = (mine - it) & (every - 1);                             // this warpgroup's first tile of the run
    it += r.count;
    const int n_mine = i0 < r.count ? ((r.count - 1 - i0) >> log_every) + 1 : 0;
    bool ok;
    if (r.kind == 0) {
      double z;
      float far_z, far_m;
      if constexpr (BOUND) {
        const int sharers = MT == 1 ? wg : mine;               // the warpgroups that share a tile share a buffer and its barriers
        BoundRun b;
        b.sums = c.first + (n_stat & 1) * (kWgs * 128);
        b.sums_bar = c.first_full(n_stat & 1);
        b.sums_parity = (uint32_t)(n_stat >> 1) & 1u;
        b.part = c.half_vote + sharers * (MT * 1024);
        b.part_bars = c.part_full(2 * sharers);
        b.n_part = n_part;
        b.again_bar = c.again_full();
        b.again_parity = (uint32_t)n_again & 1u;
        n_again += second_weights(r.count) < r.count;
        b.weight = r.weight;
        b.second = r.second;
        b.est = r.vote;
        b.rows = c.R;
        b.n_warps = (c.R + 31) >> 5;
        ok = bound_run<MT>(u, units, c.sc, i0, every, r.count, r.n_valid, rows_here, wg, b, z, far_z, far_m);
        n_part += n_mine;
      } else {
        ok = stats_run<KIND != kPlain>(u, units, c.sc, i0, every, r.count, r.n_valid, rows_here, z, far_z, far_m);
      }
      const int slot = n_stat & 1;
      ok = ok && mbar_wait(c.stat_empty(slot), ((n_stat >> 1) & 1) ^ 1, c.abort_flag) && mbar_wait(c.cleared(), 0, c.abort_flag);
      ++n_stat;
      if (!__all_sync(0xffffffffu, ok)) break;
      if (z > 0.0 && mt * 128 + own < c.R)
        asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(r.acc + mt * 128 + own), "d"(z) : "memory");
      if (__any_sync(0xffffffffu, far_z > 0.f)) {
        c.stat_z[(slot * kWgs + wg) * 128 + own] = far_z;
        c.stat_m[(slot * kWgs + wg) * 128 + own] = far_m;
        if (lane == 0) atomicOr(c.stat_far + slot, 1u << (wg * 4 + (warp & 3)));
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(c.stat_full(slot));
    } else {
      const int slot = n_vote & 1;
      ok = mbar_wait(c.lse_full(slot), (n_vote >> 1) & 1, c.abort_flag);
      ++n_vote;
      if (!__all_sync(0xffffffffu, ok)) break;
      ok = votes_run(u, units, c.sc, i0, every, r.count, r.n_valid, smem_u32(c.lse + slot * 256 + mt * 128), min(c.Rp - mt * 128, 128),
                     MT == 2 ? mt : -1, c.half_vote + mine * 512, c.half_full(mine, 0), n_half, c.inv_g,
                     [&](int key, float v) { r.vote[key] = v; });
      n_half += n_mine;
      if (!__all_sync(0xffffffffu, ok)) break;
      if (lane == 0) mbar_arrive(c.lse_empty(slot));
    }
    units += n_mine;
  }
}

// MT: blocks of 128 query rows (1 or 2); HALVES: 64-element halves of head_dim (1 or 2).  A kernel for each: the code of the warps
// that do the arithmetic is what the instruction caches have to hold, and a row block's constants are folded into it.  With one
// kernel for all, 32 layers of 4001 / 8000 / 32k tokens, 128 rows: 123.7 / 225 / 838 us, now 121.1 / 220 / 812; 16000 tokens, 64 rows
// 376 -> 353; four sequences of 5k - 10k 689 -> 658; 256 rows as before.
// kBound: statistics and estimated votes in one pass over the list, then the votes of the segments that need them all
// (slkv_bound.cu); a kernel of its own, so that neither kind's loops grow.  kWide: both passes with kBound's row sums (TileSum), for
// every call of a shape that kBound's lists have, so that what is kept depends neither on the list nor on who asks for pooled scores.
template <int MT, int HALVES, int KIND>
__global__ void __launch_bounds__(kListThreads, 1)
k_score_list(const __grid_constant__ ListArgs a) {
  constexpr bool BOUND = KIND == kBound;
  // Shared memory, all dynamic and 1024-byte aligned (the swizzled tiles need it):
  //   [kQTiles Q tiles: halves x MT x 16 KB][K ring: n_stages x halves x 16 KB][mbarriers, flags][statistics][log-sum-exps][half votes]
  extern __shared__ __align__(1024) unsigned char smem[];
  const ScoreShape& sh = a.sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if ((smem_u32(smem) & 1023u) != 0) {                      // never run on a skewed layout (uniform over the CTA)
    if (tid == 0)
      for (int j = 0; j < a.n_layers; ++j)
        if (a.lay[j].status) atomicExch(a.lay[j].status, (int)SLKV_ERR_BAD_ALIGN);
    return;
  }
  // the tail's place follows from launch parameters; everything the roles use in their loops goes through shared memory
  unsigned char* tail = smem + HALVES * (kQTiles * MT * 128 * 128 + sh.n_stages * kHalfBytes);
  uint32_t& tmem_base_sh = *reinterpret_cast<uint32_t*>(tail + kBarBytes - 16);
  int& abort_sh = *reinterpret_cast<int*>(tail + kBarBytes - 12);
  volatile int* head = reinterpret_cast<volatile int*>(tail + kBarBytes - 16 - kHeadInts * 4);
  Smem c;
  c.bar0 = smem_u32(tail);
  c.abort_flag = &abort_sh;
  c.stat_z = reinterpret_cast<float*>(tail + kBarBytes);
  c.stat_m = c.stat_z + 2 * kWgs * 128;
  c.stat_far = reinterpret_cast<unsigned*>(tail + kBarBytes - 8);
  c.lse = reinterpret_cast<float*>(tail + kBarBytes + kStatBytes);
  c.half_vote = reinterpret_cast<float*>(tail + kBarBytes + kStatBytes + kLseBytes);
  c.first = reinterpret_cast<float*>(tail + kBarBytes + kStatBytes + kLseBytes + kPartBytes);       // bounds
  c.runs = reinterpret_cast<RunDesc*>(tail + (BOUND ? kRunsAtBound : kRunsAt));

  if (tid == 0) {
    trace_mark(a.trace, 0);
    if (a.trace) a.trace[(size_t)blockIdx.x * kTraceSlots + 60] = (unsigned long long)clock64();
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&a.lay[0].tm_k)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&a.lay[0].tm_q)) : "memory");
    abort_sh = 0;
    c.stat_far[0] = c.stat_far[1] = 0;
    mbar_init(c.cleared(), 1);
    mbar_init(c.rest_cleared(), 1);
    mbar_init(c.again_full(), 4 * kWgs);
    for (int st = 0; st < kMaxStages; ++st) { mbar_init(c.full(st), 1); mbar_init(c.empty(st), 1); }
    for (int u = 0; u < 4; ++u) { mbar_init(c.unit_full(u), 1); mbar_init(c.unit_empty(u), 4); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(c.stat_full(s), 4 * kWgs);
      mbar_init(c.stat_empty(s), 1);
      mbar_init(c.lse_full(s), 1);
      mbar_init(c.lse_empty(s), 4 * kWgs);
      for (int t = 0; t < 4; ++t) { mbar_init(c.half_full(s, t), 4); mbar_init(c.part_full(4 * s + t), 4 * MT); }
      mbar_init(c.first_full(s), 4 * kWgs);
    }
    for (int k = 0; k < kQTiles; ++k) { mbar_init(c.q_full(k), 1); mbar_init(c.q_empty(k), 1); }
    for (int k = 0; k < kRunSlots; ++k) { mbar_init(c.run_full(k), 1); mbar_init(c.run_empty(k), kRunReaders); }
    head[0] = sh.R; head[1] = sh.Rp;
    head[2] = sh.n_stages; head[3] = sh.k_head_inner;
    head[4] = a.passes == 3; head[5] = __float_as_int(sh.scale_log2); head[6] = __float_as_int(1.0f / (float)sh.G);
    mbar_init(c.drain(), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of the Q tile beyond R are never written by TMA: keep them zero
  if (sh.R != MT * 128) {
    for (int i = tid; i < kQTiles * HALVES * MT * 128 * 128 / 16; i += kListThreads) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  c.tmem = tmem_base_sh;
  c.R = head[0]; c.Rp = head[1];
  c.n_stages = head[2]; c.k_head_inner = head[3];
  c.both = head[4]; c.sc = __int_as_float(head[5]); c.inv_g = __int_as_float(head[6]);
  c.q_half = MT * 128 * 128;
  c.q_bytes = HALVES * c.q_half;
  c.stage_bytes = HALVES * kHalfBytes;
  c.q = smem_u32(smem);
  c.k = c.q + (uint32_t)(kQTiles * c.q_bytes);
  // Everything above touched only this CTA's own resources, and so does all that follows up to the first load of a tile and
  // the clearing of the statistics area: those two roles wait for the kernels before this one, the others get their work
  // from them.  The first runs are worked out meanwhile.
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      pdl_wait();
      trace_mark(a.trace, 1);
      producer<MT, HALVES, BOUND>(c);
    }
  } else if (warp == 1) {
    if (lane == 0) issuer<MT, HALVES>(c);
  } else if (warp == 2) {
    if (sh.tab.n_inline == 0) pdl_wait();              // a kernel before this one writes the tables
    scheduler_publisher<MT, BOUND>(c, a);
  } else if (warp == 3) {
    pdl_wait();
    fetch_lse(c, a);
  } else {
    epilogue<MT, KIND>(c);
  }

  tc_fence_before();
  __syncthreads();
  if (abort_sh && tid == 0)
    for (int j = 0; j < a.n_layers; ++j)
      if (a.lay[j].status) atomicExch(a.lay[j].status, (int)SLKV_ERR_DEVICE_TIMEOUT);
  if (tid == 0) {
    trace_mark(a.trace, 4);
    if (a.trace) a.trace[(size_t)blockIdx.x * kTraceSlots + 61] = (unsigned long long)clock64();
  }
  if (tid == 0 && a.passes == 3) a.sync.leave();     // every thread is past its last use of the counts (the barrier above)
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(512u) : "memory");
  }
}

// One-shot diagnostic: the next launch of this thread whose CTAs wait for one another expects one arrival too many.
thread_local int g_expire_next_wait = 0;

// Timeline tracing (diagnostics): a caller-owned device buffer.
thread_local unsigned long long* g_trace = nullptr;
thread_local size_t g_trace_bytes = 0;

// A phase should last about this many tiles-times-row-blocks per CTA before the phase that needs its results is due:
// publishing, the other CTAs' counters and the merge take about 5 us, a unit about 0.6 us.
constexpr int kLagUnits = 10;

typedef void (*Kern)(const ListArgs);

// A launch of the statistics pass alone finds the row sums cleared.
cudaError_t clear_stats(const ScoreShape& sh, const ScoreLayer* lay, int n_layers, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < n_layers && e == cudaSuccess; ++i)
    e = cudaMemsetAsync(lay[i].part, 0, stat_clear_bytes(sh.n_seqs * sh.n_kv_heads, sh.R), st);
  return e;
}

}  // namespace

bool next_wait_expires() { return g_expire_next_wait != 0; }
void expire_next_wait(int on) { g_expire_next_wait = on; }
int take_expire_next_wait() { const int v = g_expire_next_wait; g_expire_next_wait = 0; return v; }

void set_tensor_trace(void* dev_buf, size_t bytes) {
  g_trace = static_cast<unsigned long long*>(dev_buf);
  g_trace_bytes = bytes;
}
unsigned long long* tensor_trace_buffer(int n_cta) {
  return g_trace && g_trace_bytes >= (size_t)n_cta * kTraceSlots * sizeof(unsigned long long) ? g_trace : nullptr;
}

// K tiles of the ring beside the Q tiles.
int score_list_stages(int MT, int halves) {
  const int n = (kSmemLimit - kTailBound - kQTiles * halves * MT * 128 * 128) / (halves * kHalfBytes);
  return n < kMaxStages ? n : kMaxStages;
}

cudaError_t launch_score_list(const ScoreShape& sh, const ScoreLayer* lay, int n_layers, int passes,
                              unsigned long long* sync, cudaStream_t st, int* launches, bool cleared) {
  if (n_layers < 1 || sh.n_cta == 0) return cudaSuccess;             // no history: nothing to score
  if (n_layers > kListMaxLayers) return cudaErrorInvalidValue;
  const bool bound = passes == kScoreBound;
  const int kind = bound ? kBound : passes == kScoreWide ? kWide : kPlain;
  if (kind != kPlain) passes = 3;
#define SLKV_LIST(MT, HALVES) {k_score_list<MT, HALVES, kPlain>, k_score_list<MT, HALVES, kWide>, k_score_list<MT, HALVES, kBound>}
  static const Kern kernels[2][2][3] = {{SLKV_LIST(1, 1), SLKV_LIST(1, 2)}, {SLKV_LIST(2, 1), SLKV_LIST(2, 2)}};
#undef SLKV_LIST
  const Kern kernel = kernels[sh.MT - 1][sh.halves - 1][kind];
  static thread_local int configured_on[2][2][3] = {{{-1, -1, -1}, {-1, -1, -1}}, {{-1, -1, -1}, {-1, -1, -1}}};
  int& configured_dev = configured_on[sh.MT - 1][sh.halves - 1][kind];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    configured_dev = dev;
  }
  ListArgs a;
  a.sh = sh;
  std::memcpy(a.lay, lay, sizeof(ScoreLayer) * (size_t)n_layers);
  a.n_layers = n_layers;
  a.passes = passes;
  // A single product needs no groups: the whole list is one (its tiles are counted in 32 bits times the CTAs).
  const bool one_group = (bound || passes != 3) && (long long)sh.total_tiles * n_layers < (1 << 24);
  if (bound && !one_group) return cudaErrorNotSupported;
  a.group_layers = one_group ? n_layers : (n_layers > 1 ? sh.group_layers : 0);
  a.n_groups = a.group_layers == 0 ? n_layers * sh.n_groups : (n_layers + a.group_layers - 1) / a.group_layers;
  // units per CTA and phase, about
  const int per_phase = (int)((long long)sh.total_tiles * n_layers * sh.MT / ((long long)a.n_groups * sh.n_cta));
  a.lag = kLagUnits / (per_phase > 0 ? per_phase : 1);
  if (a.lag > a.n_groups - 1) a.lag = a.n_groups - 1;
  if (a.lag < 1) a.lag = 1;
  // Layers of the phases S(0) .. S(lag); all of them where a CTA may have no share of V(0) to wait for.
  a.first_layers = n_layers;
  const long long tiles0 = a.group_layers == 0 ? sh.group_tile[1] : (long long)a.group_layers * sh.total_tiles;
  if (tiles0 >= sh.n_cta) {
    const int before = a.group_layers == 0 ? a.lag / sh.n_groups + 1 : (a.lag + 1) * a.group_layers;
    if (before < n_layers) a.first_layers = before;
  }
  a.sync.word = sync;
  a.sync.tag = next_launch_tag() & ((1ull << 40) - 1);
  const bool waits_inside = passes == 3;
  const int expire = waits_inside ? take_expire_next_wait() : 0;
  a.target = (unsigned)sh.n_cta + (expire == 1);
  a.sync.expect = (unsigned)sh.n_cta + (expire == 2);
  a.trace = tensor_trace_buffer(sh.n_cta);
  const size_t smem = (size_t)(kQTiles * sh.halves * sh.MT * 128 * 128 + sh.n_stages * sh.halves * kHalfBytes + (bound ? kTailBound : kTail));

  // CTAs that wait for one another must all be resident: cooperative launch, with dependent launch on top where the
  // device takes both.  Where it takes no cooperative launch, or the environment says so (tests), the two passes go out
  // as two launches.
  static const bool env_no_coop = [] {
    const char* v = std::getenv("SLKV_NO_COOPERATIVE");
    return v && v[0] == '1';
  }();
  static thread_local int coop_state[64] = {};        // per device: 0 untried, 1 with dependent launch, 2 without, -1 refused
  int& cs = coop_state[dev < 64 ? dev : 0];
  if (waits_inside && (env_no_coop || cs == -1 || sh.n_cta > sm_count())) {
    if (bound) return cudaErrorNotSupported;
    a.passes = 1;
    e = clear_stats(sh, lay, n_layers, st);
    if (e != cudaSuccess) return e;
    e = launch_pdl_scoped(KID_SCORE_LSE, kernel, sh.n_cta, kListThreads, smem, st, launches, a);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < n_layers && e == cudaSuccess; ++i) e = launch_merge_lse_tensor(sh, lay[i], nullptr, 1.f, st, launches);
    if (e != cudaSuccess) return e;
    a.passes = 2;
    return launch_pdl_scoped(KID_SCORE_VOTE, kernel, sh.n_cta, kListThreads, smem, st, launches, a);
  }
  if (passes == 1 && !cleared) {
    e = clear_stats(sh, lay, n_layers, st);
    if (e != cudaSuccess) return e;
  }
  const int kid = bound ? KID_SCORE_BOUND : passes == 1 ? KID_SCORE_LSE : (n_layers > 1 ? KID_SCORE_LIST : (passes == 2 ? KID_SCORE_VOTE : KID_SCORE_FUSED));
  if (!waits_inside) return launch_pdl_scoped(kid, kernel, sh.n_cta, kListThreads, smem, st, launches, a);
  for (int attempt = 0; attempt < 2; ++attempt) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sh.n_cta);
    cfg.blockDim = dim3(kListThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cs == 2 ? 1 : 2;
    cudaError_t le;
    {
      LaunchScope scope(kid, st, launches);
      le = cudaLaunchKernelEx(&cfg, kernel, a);
    }
    if (le == cudaSuccess) {
      if (cs == 0) cs = 1;
      return cudaSuccess;
    }
    (void)cudaGetLastError();                         // not a sticky error: the launch was refused
    --*launches;
    if (cs == 2 || cs == 1) { cs = -1; break; }
    cs = 2;                                           // once more without dependent launch
  }
  cs = -1;
  if (bound) return cudaErrorNotSupported;
  return launch_score_list(sh, lay, n_layers, kind == kWide ? kScoreWide : passes, sync, st, launches);
}

}  // namespace slkv

// What the kernels that do a whole layer in one launch (slkv_layer_tc.cu, slkv_layer_fma.cu) share: a cluster of CTAs per
// (sequence, KV head) segment, whose first CTA selects and whose CTAs all copy rows (Sec. 3.4, Eq. 8; Algorithm 3 lines 1-10).
// Everything here has internal linkage.
#pragma once
#include "slkv_select_device.cuh"

namespace slkv {
namespace {

constexpr int kLayerThreads = 512;            // threads that select and copy
constexpr int kLayerMaxCluster = 10;          // above eight: where the device has room for such clusters

// Pooling, selection and gather of a launch.
struct LayerTail {
  SeqTables tab;
  int n_seqs, n_kv_heads, window, pool_mode, radius;
  int select;                  // 0: the pooled scores are all that is wanted
  int row_bytes;
  float* pooled;               // may be null
  const int32_t* budgets;
  int32_t *offsets, *kept_idx, *status;
  const void *k, *v;
  void *k_out, *v_out;
  long long capacity, k_tok_bytes, k_head_bytes, v_tok_bytes, v_head_bytes;
};
inline LayerTail layer_tail(const Problem& pb, const TailLayer* t, float* pooled) {
  LayerTail a = {};
  const slkv_params& p = pb.p;
  a.tab = pb.tab;
  a.n_seqs = p.n_seqs; a.n_kv_heads = p.n_kv_heads; a.window = p.window; a.pool_mode = p.pool_mode;
  a.radius = p.pool_kernel >> 1;
  a.pooled = pooled;
  if (!t) return a;
  a.select = 1;
  a.row_bytes = p.head_dim * pb.elem;
  a.budgets = t->budgets; a.offsets = t->offsets; a.kept_idx = t->kept_idx; a.status = t->status;
  a.k = t->k; a.v = t->v; a.k_out = t->k_out; a.v_out = t->v_out; a.capacity = t->capacity;
  a.k_tok_bytes = p.k_stride_tok * pb.elem; a.k_head_bytes = p.k_stride_head * pb.elem;
  a.v_tok_bytes = p.v_stride_tok * pb.elem; a.v_head_bytes = p.v_stride_head * pb.elem;
  return a;
}

struct Segment { int seg, s, g, t0, len, n, n_win; long long base; };      // base: of its scores
__device__ __forceinline__ Segment segment_of(const LayerTail& a, int seg) {
  Segment x;
  x.seg = seg;
  x.s = seg / a.n_kv_heads;
  x.g = seg - x.s * a.n_kv_heads;
  x.t0 = a.tab.cu_at(x.s);
  x.len = a.tab.cu_at(x.s + 1) - x.t0;
  x.n = max(x.len - a.window, 0);
  x.n_win = min(x.len, a.window);
  x.base = a.tab.hist_at(x.s) * a.n_kv_heads + (long long)x.g * x.n;
  return x;
}

struct SegmentRows { int out0, k_keep; };     // its first packed row; history rows kept
// One warp.
__device__ __forceinline__ SegmentRows segment_rows(const LayerTail& a, const Segment& x) {
  SegmentRows r = {0, 0};
  if (!a.select) return r;
  const int lane = threadIdx.x & 31;
  r.k_keep = kept_rows(x.len, __ldg(a.budgets + x.g), a.window) - x.n_win;       // C_H = C - window, clamped
  unsigned before = 0;                          // < 2^31: the host checks n_kv_heads * total_tokens
  for (int i = lane; i < x.seg; i += 32) {
    const int s2 = i / a.n_kv_heads, h2 = i - s2 * a.n_kv_heads;
    before += (unsigned)kept_rows(a.tab.cu_at(s2 + 1) - a.tab.cu_at(s2), __ldg(a.budgets + h2), a.window);
  }
  r.out0 = (int)__reduce_add_sync(kAll, before);
  return r;
}

// The first CTA, kLayerThreads threads (numbered tid, named barrier BAR): pools the segment's votes (place p at
// votes[vote_at<IT>(p)], places -4 .. -1 and n .. n + 3 hold the padding), writes the scores where they are wanted and leaves
// the kept history positions in ascending order at the start of votes' memory (votes - kLead).  gave_up, in shared
// memory: set where a wait of these threads has run out; nothing is selected then (sh may lie where loads still land).
template <int IT>
__device__ __forceinline__ int vote_at(int p) { return (p >> kLogItems<IT>) * (IT + 4) + (p & (IT - 1)); }
template <int IT, int BAR>
__device__ __forceinline__ void layer_select(const LayerTail& a, const Segment& x, int k_keep, float* votes, SelShared& sh, int tid,
                                             const volatile int* gave_up) {
  constexpr int kPer = kBins / kLayerThreads;
  const bool choose = a.select && k_keep > 0 && k_keep < x.n, max_mode = a.pool_mode == SLKV_POOL_MAX;
  if (choose) {
    if (tid == 0) { sh.n_list = 0; sh.sure = 0; }
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      reinterpret_cast<int2*>(sh.hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
      if (IT > 8) reinterpret_cast<int2*>(sh.sample)[(tid * kPer + i) / 2] = make_int2(0, 0);
    }
  }
  const int i0 = tid * IT;
  const bool mine = i0 < x.n;
  unsigned valid = 0, key[IT];
  if (mine) {
    const int have = min(x.n - i0, IT);
    valid = have >= 32 ? kAll : (1u << have) - 1u;
    const float *src = votes + vote_at<IT>(i0), *before = votes + vote_at<IT>(i0 - 4);
    switch (a.radius) {
      case 0: pool_places<0>(src, before, max_mode, key); break;
      case 1: pool_places<1>(src, before, max_mode, key); break;
      case 2: pool_places<2>(src, before, max_mode, key); break;
      case 3: pool_places<3>(src, before, max_mode, key); break;
      default: pool_places<4>(src, before, max_mode, key); break;
    }
    if (a.pooled) store_scores(a.pooled + x.base + i0, key, valid);
  }
  if (!choose) return;
  asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(kLayerThreads) : "memory");
  if (*gave_up) return;                         // written in front of the barrier, if at all
  int o;
  unsigned tau;
  const unsigned kept = select_places<kLayerThreads, IT, false, BAR>(sh, tid, key, valid, mine, reinterpret_cast<uint4*>(votes + vote_at<IT>(i0)),
                                                                     x.n, k_keep, 0, 1, o, tau);
  int* dst = reinterpret_cast<int*>(votes - kLead) + o;
  for (unsigned m = kept; m != 0; m &= m - 1) *dst++ = i0 + __ffs(m) - 1;
}

// Every CTA, kLayerThreads threads: its share of the segment's rows.  stage: the first CTA's list of kept positions; where that CTA
// has given up there is none, and whatever lies there is held inside the sequence.
template <int LANES>
__device__ __forceinline__ void layer_gather_rows(const LayerTail& a, const Segment& x, const SegmentRows r, const int* stage, int tid, int rank,
                                                  int CS) {
  constexpr int kRows = kLayerThreads / LANES, kFly = 2;
  const int lane = tid & (LANES - 1), sub = tid / LANES;
  const bool choose = r.k_keep > 0 && r.k_keep < x.n;
  const int rows = (int)min((long long)r.k_keep + x.n_win, a.capacity - r.out0);
  const unsigned char *k = static_cast<const unsigned char*>(a.k) + x.t0 * a.k_tok_bytes + x.g * a.k_head_bytes + lane * 16,
                      *v = static_cast<const unsigned char*>(a.v) + x.t0 * a.v_tok_bytes + x.g * a.v_head_bytes + lane * 16;
  unsigned char *ko = static_cast<unsigned char*>(a.k_out) + (long long)r.out0 * a.row_bytes + lane * 16,
                *vo = static_cast<unsigned char*>(a.v_out) + (long long)r.out0 * a.row_bytes + lane * 16;
  for (int i0 = rank * kRows + sub; i0 < rows; i0 += CS * kRows * kFly) {
    uint4 kv[kFly], vv[kFly];
    int pos[kFly];
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int i = i0 + u * CS * kRows;
      if (i < rows) pos[u] = i >= r.k_keep ? x.len - x.n_win + (i - r.k_keep) : (choose ? (int)min((unsigned)stage[i], (unsigned)x.len - 1u) : i);
    }
#pragma unroll
    for (int u = 0; u < kFly; ++u)
      if (i0 + u * CS * kRows < rows) {
        kv[u] = *reinterpret_cast<const uint4*>(k + pos[u] * a.k_tok_bytes);
        vv[u] = *reinterpret_cast<const uint4*>(v + pos[u] * a.v_tok_bytes);
      }
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const long long i = i0 + u * CS * kRows;
      if (i < rows) {
        *reinterpret_cast<uint4*>(ko + i * a.row_bytes) = kv[u];
        *reinterpret_cast<uint4*>(vo + i * a.row_bytes) = vv[u];
        if (lane == 0) a.kept_idx[r.out0 + i] = pos[u];
      }
    }
  }
}
__device__ __forceinline__ void layer_gather(const LayerTail& a, const Segment& x, const SegmentRows r, const int* stage, int tid, int rank, int CS) {
  if (rank == 0 && tid == 0) {
    a.offsets[x.seg] = r.out0;
    if (x.seg == a.n_seqs * a.n_kv_heads - 1) {
      const long long all = (long long)r.out0 + r.k_keep + x.n_win;
      a.offsets[x.seg + 1] = (int32_t)all;
      if (all > a.capacity && a.status) *a.status = SLKV_ERR_CAPACITY;
    }
  }
  switch (a.row_bytes >> 4) {
    case 8: layer_gather_rows<8>(a, x, r, stage, tid, rank, CS); break;
    case 16: layer_gather_rows<16>(a, x, r, stage, tid, rank, CS); break;
    default: layer_gather_rows<32>(a, x, r, stage, tid, rank, CS); break;
  }
}

// Between the CTAs of a cluster data goes in bulk copies: plain stores to another CTA's shared memory move some 7 bytes per
// clock (32 KB of votes into one CTA: 1.5-2 us).
__device__ __forceinline__ uint32_t in_cta(const void* p, int rank) {           // p's place in another CTA's shared memory
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
// 16-byte aligned, a multiple of 16 bytes; completes on bar in the CTA that receives.  The writers of src have made their
// writes visible to such copies (publish_for_copy) in front of a barrier with this thread.
__device__ __forceinline__ void copy_to_cta(const void* dst, const void* src, int bytes, const void* bar, int rank) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(in_cta(dst, rank)), "r"((uint32_t)__cvta_generic_to_shared(src)), "r"(bytes), "r"(in_cta(bar, rank)) : "memory");
}
__device__ __forceinline__ void publish_for_copy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A cluster's barrier in two halves; whole warps.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace
}  // namespace slkv

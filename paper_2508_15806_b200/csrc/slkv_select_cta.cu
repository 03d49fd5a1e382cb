// Pooling + per-head variable-k selection for a list of layers (Sec. 3.4, Eq. 8; Algorithm 3 lines 1-4, 7-8): one CTA per
// (sequence, KV head) segment of up to 32768 history positions, a cluster of up to eight for longer ones.
//
// The votes come into shared memory with asynchronous 16-byte copies (from an aligned start, whatever the segment's), a
// thread pools 8, 16 or 32 consecutive positions of them and works with the scores' bit patterns (scores are >= 0, so
// unsigned order = float order).  The k-th largest:
//   1. with 16 or 32 positions per thread, a histogram of every 16th or 32nd score: the ranks that the k-th largest has among
//      these, give or take four standard deviations, bound it from both sides (where there are none, nothing bounds it);
//   2. a histogram of the scores between the bounds, 2048 bins, 64 to an octave; the bin with the k-th largest;
//   3. where that bin's scores fit a list of 512, or of a score for each of 256 threads (mostly), they are ranked by counting,
//      else a histogram of that bin, and so on.
// Then an ordered compaction from bit masks.  Integer counters only: the result does not depend on timing, and not on the
// sample either.
// What bounds it: a chain of some ten CTA-wide steps of 0.2-0.6 us, and at 32 positions per thread instructions.  Bracketing
// the k-th largest by 128 ranked samples and a descent over the bracket took as many steps again, and its loops an atomic
// with a result per score: whole layers of 8 segments 21.7 -> 16.9 us at 1024 positions, 26.4 -> 22.7 at 4096, 29.9 -> 26.4 at
// 8192, 33.5 -> 30.1 at 12000, 32 layers of 4001 129.5 -> 118 (all in a graph).  With a bound from below alone and every position
// looked at in each step 30.6 at 12000, 44.9 at 32000 (now 42.6), 78.1 at 64000 (75.4).
#include "slkv_select_device.cuh"

namespace slkv {
namespace {

constexpr int kMaxThreads = 1024;
constexpr int kMaxItems = 32;                         // consecutive positions per thread
constexpr int kMaxSlice = kMaxThreads * kMaxItems;    // 32768 positions per CTA
constexpr int kMaxCluster = 8;

struct SelArgs {
  SeqTables tab;
  int n_seqs, n_kv_heads, window, pool_mode;
  TailLayer lay[kListMaxLayers];
};

// T threads with IT consecutive positions each.  CLUSTER: a segment is shared by the CTAs of a cluster (else every pointer
// below is known to be this CTA's own memory).
template <int T, int IT, int RAD, bool CLUSTER>
__global__ void __launch_bounds__(T, T == 1024 ? 1 : 1024 / T)
k_select_list(const __grid_constant__ SelArgs args) {
  constexpr int kWarps = T / 32, kPitch = IT + 4, kPer = kBins / T;
  extern __shared__ __align__(16) float votes_sh[];
  __shared__ SelShared sh;

  cg::cluster_group cluster = cg::this_cluster();
  const int CS = CLUSTER ? (int)cluster.num_blocks() : 1, rank = CLUSTER ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  pdl_launch_dependents();
  const TailLayer& a = args.lay[blockIdx.y];
  const int seg = blockIdx.x / CS, s = seg / args.n_kv_heads, h = seg - s * args.n_kv_heads;
  const int t0 = args.tab.cu_at(s), len = args.tab.cu_at(s + 1) - t0;
  const int n = max(len - args.window, 0), n_win = min(len, args.window);
  const int n_seg = args.n_seqs * args.n_kv_heads;
  const long long seg_base = args.tab.hist_at(s) * args.n_kv_heads + (long long)h * n;
  const float* vote = a.vote + seg_base;
  const bool max_mode = args.pool_mode == SLKV_POOL_MAX;
  const float pad = max_mode ? -INFINITY : 0.f;
  // this CTA's slice: places 0 .. own - 1, place i is position base + i (the first slice's first places may lie in the
  // segment before: base <= 0)
  const int shift = (int)(seg_base & 3);
  const int slice = ((n + shift + CS - 1) / CS + 3) & ~3;
  const int own = min(max(n + shift - rank * slice, 0), slice), base = rank * slice - shift;
  const int my_end = min(base + own, n);
  float* votes = votes_sh + kLead;
  auto at = [&](int i) { return (i >> kLogItems<IT>) * kPitch + (i & (IT - 1)); };    // a place's index (i >= -4)
  // read here, where the kernel before this one is waited for anyway: a parameter's first read is a cache miss
  const long long capacity = a.capacity;
  int32_t* const kept_idx = a.kept_idx;
  int32_t* const gather_src = a.gather_src;
  float* const pooled_out = a.pooled_out;
  asm volatile("" ::"l"(capacity), "l"(kept_idx), "l"(gather_src), "l"(pooled_out), "l"(a.offsets));
  if (tid == 0) { sh.n_list = 0; sh.sure = 0; }
#pragma unroll
  for (int i = 0; i < kPer; i += 2) {
    reinterpret_cast<int2*>(sh.hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
    reinterpret_cast<int2*>(sh.sample)[(tid * kPer + i) / 2] = make_int2(0, 0);
  }
  pdl_wait();                                           // budgets and votes may come from the kernels before this one

  // ---- the votes on their way, four places at a time, with one group on either side
  for (int q = tid - 1; 4 * q <= own + 3; q += T) {
    const int p = base + 4 * q;
    float* dst = votes + at(4 * q);
    if (p >= 0 && p + 3 < n) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(vote + p) : "memory");
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) dst[e] = p + e >= 0 && p + e < n ? __ldg(vote + p + e) : pad;
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int budget = __ldg(a.budgets + h);
  {
    unsigned part = 0;                                  // < 2^31: the host checks n_kv_heads * total_tokens
    for (int g = tid; g < seg; g += T) {
      const int s2 = g / args.n_kv_heads, h2 = g - s2 * args.n_kv_heads;
      part += (unsigned)kept_rows(args.tab.cu_at(s2 + 1) - args.tab.cu_at(s2), a.budgets[h2], args.window);
    }
    part = __reduce_add_sync(kAll, part);
    if (lane == 0) sh.wsum[0][wid] = part;
  }
  const int k_keep = kept_rows(len, budget, args.window) - n_win;             // C_H = C - window, clamped
  const bool choose = k_keep > 0 && k_keep < n;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // packed row where this segment starts = kept rows of all earlier segments (Algorithm 3 l.1-4 per head)
  const long long out0 = __reduce_add_sync(kAll, lane < kWarps ? sh.wsum[0][lane] : 0u);
  const int src_base = t0 * args.n_kv_heads + h;         // source row of position j: src_base + j * n_kv_heads
  auto put = [&](long long o, int position) {
    if (o < capacity) {
      kept_idx[o] = position;
      gather_src[o] = src_base + position * args.n_kv_heads;
    }
  };
  if (rank == 0) {
    if (tid == 0) {
      a.offsets[seg] = (int32_t)out0;
      if (seg == n_seg - 1) {
        const long long all = out0 + k_keep + n_win;
        a.offsets[n_seg] = (int32_t)all;
        if (all > capacity && a.status) *a.status = SLKV_ERR_CAPACITY;
      }
    }
    for (int t = tid; t < n_win; t += T) put(out0 + k_keep + t, len - n_win + t);    // window rows: always kept
  }
  if (!choose) {                                         // uniform over the cluster: keep all of the history, or none
    if (k_keep > 0)
      for (int j = base + tid; j < my_end; j += T)
        if (j >= 0) put(out0 + j, j);
    if (pooled_out == nullptr) return;
  }

  // ---- pooling: the thread's scores as bit patterns; bit e of the masks is its place e
  const int i0 = tid * IT;
  const bool mine = i0 < own;
  unsigned valid = 0, key[IT];
  if (mine) {
    const int p0 = base + i0, v_lo = max(-p0, 0), v_hi = min(my_end - p0, IT);            // valid places of the thread
    valid = (v_hi >= 32 ? kAll : (1u << max(v_hi, 0)) - 1u) & (v_lo >= 32 ? 0u : kAll << v_lo);
    pool_places<RAD>(votes + tid * kPitch, votes + at(i0 - 4), max_mode, key);
    if (pooled_out) store_scores(pooled_out + seg_base + p0, key, valid);
  }
  if (!choose) return;

  // (0: a barrier of all T threads)
  int o_mine;
  unsigned tau;
  const unsigned kept = select_places<T, IT, CLUSTER, 0>(sh, tid, key, valid, mine, reinterpret_cast<uint4*>(votes + tid * kPitch), n,
                                                         k_keep, rank, CS, o_mine, tau);
  // the kept positions, in shared memory first (where the votes were): whole lines then go out
  int* const stage = reinterpret_cast<int*>(votes_sh);
  int o0 = 0, o1 = k_keep;                                 // the CTA's rows among the segment's
  if (CLUSTER) {
    if (tid == 0) sh.above = o_mine;
    if (tid == T - 1) sh.m = o_mine + __popc(kept);
    __syncthreads();
    o0 = sh.above;
    o1 = sh.m;
  }
  int* dst = stage + (o_mine - o0);
  for (unsigned m = kept; m != 0; m &= m - 1) *dst++ = base + i0 + __ffs(m) - 1;
  __syncthreads();
  for (int i = o0 + tid; i < o1; i += T) put(out0 + i, stage[i - o0]);
  if (CLUSTER) cluster.sync();                             // nobody leaves while its shared memory may still be read
}

// CTAs per segment: one wherever it can hold the segment's scores, however many SMs that leaves idle -- the exchanges of a
// cluster cost as much as the smaller slices save (one layer of 8 segments, the whole call in us with 1, 2, 4 and 8 CTAs of an
// earlier selection per segment: 1024 tokens 26.6, 30.7, 30.8, 32.7; 8192 tokens 32.8, 35.4, 36.8, 38.6; 32768 tokens 48.6, 49.2,
// 48.2, 49.3).
}  // namespace
int select_list_cluster(const Problem& pb) {
  int cs = 1;
  while (cs < kMaxCluster && (pb.max_hist + 3 + cs - 1) / cs + 3 > kMaxSlice) cs *= 2;
  return cs;
}

// up to 262116 history positions
bool select_list_supported(const Problem& pb) {
  return (pb.p.pool_kernel >> 1) <= kMaxRadius && (pb.max_hist + 3) / kMaxCluster + 4 <= kMaxSlice;
}

namespace {
typedef void (*SelKern)(const SelArgs);
struct SelVariant {
  int threads, items;
  SelKern kern[kMaxRadius + 1];
};
#define SLKV_SEL(T, IT, C) \
  {T, IT, {k_select_list<T, IT, 0, C>, k_select_list<T, IT, 1, C>, k_select_list<T, IT, 2, C>, k_select_list<T, IT, 3, C>, k_select_list<T, IT, 4, C>}}
const SelVariant kVariants[] = {SLKV_SEL(256, 8, false), SLKV_SEL(512, 8, false), SLKV_SEL(1024, 8, false),
                                SLKV_SEL(512, 16, false), SLKV_SEL(1024, 16, false), SLKV_SEL(1024, 32, false), SLKV_SEL(1024, 32, true)};
#undef SLKV_SEL
// The smallest variant that holds a slice.  CTAs that have an SM each are quickest with eight positions per thread, where
// there are more of them two to an SM are: one layer of 8 segments / 32 layers in a graph, us, with 512 x 8, 1024 x 8, 512 x 16,
// 1024 x 16 threads x positions: 1024 positions 17.9 17.7 18.9 19.1 / 67.9 72.0 69.5 74.2, 2048: 20.7 21.0 22.7 22.3 / 79.3 83.3
// 80.4 84.0, 4096: 23.4 22.7 24.1 23.8 / 125 129 126 131, 8192: - 26.4 28.7 27.1 / - 210 205 210.  With 256 x 8 at 1024: 17.8 /
// 70.0, and behind the FMA scores 16.9 instead of 18.0.
const SelVariant& variant_for(int cs, int slice, long long ctas) {
  if (cs > 1) return kVariants[6];
  const bool alone = ctas <= sm_count();
  if (alone && slice <= 1024) return kVariants[0];
  if (slice <= (alone ? 2048 : 4096)) return kVariants[1];
  if (slice <= 8192) return kVariants[alone ? 2 : 3];
  return kVariants[slice <= 16384 ? 4 : 5];
}
}  // namespace

cudaError_t launch_select_list(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches) {
  const int cs = select_list_cluster(pb);
  const int slice = ((pb.max_hist + 3 + cs - 1) / cs + 3) & ~3;
  const SelVariant& var = variant_for(cs, slice, (long long)pb.n_seg * n_layers);
  const size_t smem = (size_t)vote_floats(var.threads, var.items) * sizeof(float);
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    for (const SelVariant& x : kVariants)
      for (SelKern k : x.kern) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, vote_floats(x.threads, x.items) * (int)sizeof(float));
        if (e != cudaSuccess) return e;
      }
    configured_dev = dev;
  }
  SelArgs a;
  a.tab = pb.tab;
  a.n_seqs = pb.p.n_seqs; a.n_kv_heads = pb.p.n_kv_heads; a.window = pb.p.window; a.pool_mode = pb.p.pool_mode;
  for (int i = 0; i < n_layers; ++i) a.lay[i] = lay[i];
  LaunchScope scope(KID_SELECT, st, launches);
  return launch_pdl(var.kern[pb.p.pool_kernel >> 1], dim3((unsigned)(pb.n_seg * cs), (unsigned)n_layers), dim3(var.threads), smem, st, cs, a);
}

}  // namespace slkv

// Pooling + per-head variable-k selection for a list of layers (Sec. 3.4, Eq. 8; Algorithm 3 lines 1-4, 7-8): one CTA per
// (sequence, KV head) segment of up to 32768 history positions, a cluster of up to eight for longer ones.
//
// The votes come into shared memory with asynchronous 16-byte copies (from an aligned start, whatever the segment's), a
// thread pools 8, 16 or 32 consecutive positions of them and works with the scores' bit patterns (scores are >= 0, so
// unsigned order = float order).  The k-th largest:
//   1. 128 scores sampled evenly over the segment, ranked by counting: two of them bracket the k-th largest with four
//      standard deviations to spare on either side;
//   2. while pooling, every thread notes in bit masks which scores lie above and inside the bracket; their numbers tell
//      whether the k-th lies inside (else the bracket becomes everything);
//   3. a radix descent over the scores inside alone -- 2048 bins over the bracket's range -- until a bin's scores fit a list
//      of 512 (mostly after one level), which is ranked by counting.
// Then an ordered compaction from the masks.  Integer counters only: the result does not depend on timing, and not on the
// sample either.
// What bounds it: instructions.  A CTA's 32 warps on one SM pay eight cycles for each instruction per thread (about 1900 at
// 32 positions per thread, half of the time), the rest is a dozen CTA-wide steps.  Against a descent from the top over all
// scores: 16 layers of 8 segments of 131008 positions 290 -> 91 us, one segment per CTA of 1008 positions 13 -> 9 us.
#include <cooperative_groups.h>

#include "slkv_internal.cuh"

namespace cg = cooperative_groups;

namespace slkv {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxItems = 32;                         // consecutive positions per thread: 8, 16 or 32
constexpr int kMaxSlice = kThreads * kMaxItems;       // 32768 positions per CTA
constexpr int kMaxCluster = 8;
constexpr int kMaxRadius = 4;                         // pool_kernel <= 9: four values on either side are enough
constexpr int kBins = 2048;
constexpr int kSamples = 128;
constexpr int kList = 512;
constexpr unsigned kAll = 0xffffffffu;
// Shared memory of the votes: a thread's positions are `items` floats, then four unused ones -- the pitch makes the 16-byte
// accesses of neighbouring threads conflict-free -- behind eight floats that hold the four before the first.
constexpr int kLead = 8;
__host__ __device__ __forceinline__ int vote_floats(int log_items) {
  return kLead + (kThreads + 1) * ((1 << log_items) + 4);
}

struct SelArgs {
  SeqTables tab;
  int n_seqs, n_kv_heads, window, pool_mode;
  TailLayer lay[kListMaxLayers];
};

__device__ __forceinline__ int kept_rows(int len, int budget, int window) { return min(len, max(budget, window)); }

// Pooled values at x[4 .. 11] of 16 consecutive votes.
template <int RAD>
__device__ __forceinline__ void pool8(const float (&x)[16], bool max_mode, float (&y)[8]) {
  constexpr int W = 2 * RAD + 1, F = 4 - RAD;          // window of y[e]: x[F + e .. F + e + W - 1]
  if (max_mode) {
    float m[16];
    int have = 1;                                      // m[i] = max of x[i .. i + have - 1]
#pragma unroll
    for (int i = 0; i < 16; ++i) m[i] = x[i];
#pragma unroll
    for (int step = 1; 2 * step <= W; step *= 2) {
#pragma unroll
      for (int i = F; i + step < 16; ++i) m[i] = fmaxf(m[i], m[i + step]);
      have = 2 * step;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) y[e] = have < W ? fmaxf(m[F + e], m[F + e + W - have]) : m[F + e];
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float acc = x[F + e];
#pragma unroll
      for (int t = 1; t < W; ++t) acc += x[F + e + t];
      y[e] = acc / (float)W;
    }
  }
}

// CLUSTER: a segment is shared by the CTAs of a cluster (else every pointer below is known to be this CTA's own memory).
template <int RAD, bool CLUSTER>
__global__ void __launch_bounds__(kThreads, 1)
k_select_list(const __grid_constant__ SelArgs args) {
  extern __shared__ __align__(16) float votes_sh[];
  __shared__ __align__(16) int hist[kBins];
  __shared__ __align__(16) unsigned samp[kSamples];
  __shared__ __align__(16) unsigned list[kList];
  __shared__ unsigned wsum[3][kWarps];
  __shared__ int2 cta_tot;                              // read by the cluster's other CTAs
  __shared__ unsigned sh_lo, sh_hi, sh_top, sh_tau, sh_bin, sh_n;
  __shared__ int sh_above, sh_m, sh_need, sh_r[2];

  cg::cluster_group cluster = cg::this_cluster();
  const int CS = CLUSTER ? (int)cluster.num_blocks() : 1, rank = CLUSTER ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  auto sync_all = [&]() { if (CLUSTER) cluster.sync(); else __syncthreads(); };
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
  const int log_items = own <= 8 * kThreads ? 3 : (own <= 16 * kThreads ? 4 : 5);
  const int items = 1 << log_items, pitch = items + 4;
  float* votes = votes_sh + kLead;
  auto at = [&](int i) { return (i >> log_items) * pitch + (i & (items - 1)); };      // a place's index (i >= -4)
  const long long capacity = a.capacity;
  if (tid == 0) { sh_lo = 0; sh_hi = 0x7f800000u; sh_n = 0; }
  reinterpret_cast<int2*>(hist)[tid] = make_int2(0, 0);
  pdl_wait();                                           // budgets and votes may come from the kernels before this one

  // ---- the votes on their way, four places at a time, with one group on either side
  for (int q = tid - 1; 4 * q <= own + 3; q += kThreads) {
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
  if (n > 0 && tid < kSamples) {
    const int p = (int)(((long long)(2 * tid + 1) * n) / (2 * kSamples));
    float w[2 * RAD + 1];
#pragma unroll
    for (int t = 0; t <= 2 * RAD; ++t) {
      const int q = p - RAD + t;
      w[t] = q >= 0 && q < n ? __ldg(vote + q) : pad;
    }
    float v = w[0];
#pragma unroll
    for (int t = 1; t <= 2 * RAD; ++t) v = max_mode ? fmaxf(v, w[t]) : v + w[t];
    if (!max_mode) v /= (float)(2 * RAD + 1);
    samp[tid] = (__float_as_uint(v) & ~(kSamples - 1u)) | (unsigned)tid;       // all different; the bracket is widened by it
  }
  {
    unsigned part = 0;                                  // < 2^31: the host checks n_kv_heads * total_tokens
    for (int g = tid; g < seg; g += kThreads) {
      const int s2 = g / args.n_kv_heads, h2 = g - s2 * args.n_kv_heads;
      part += (unsigned)kept_rows(args.tab.cu_at(s2 + 1) - args.tab.cu_at(s2), a.budgets[h2], args.window);
    }
    part = __reduce_add_sync(kAll, part);
    if (lane == 0) wsum[0][wid] = part;
  }
  const int k_keep = kept_rows(len, budget, args.window) - n_win;             // C_H = C - window, clamped
  const bool choose = k_keep > 0 && k_keep < n;
  if (wid == kWarps - 1 && choose) {
    // sample ranks that bracket the k-th score; outside 0 .. kSamples - 1: no bound there
    const float f = __fdividef((float)k_keep, (float)n), q = (float)kSamples * f;
    const float dev = 4.f * sqrtf(q * (1.f - f)) + 1.f;
    if (lane == 0) { sh_r[0] = (int)floorf(q - dev) - 1; sh_r[1] = (int)ceilf(q + dev); }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // packed row where this segment starts = kept rows of all earlier segments (Algorithm 3 l.1-4 per head)
  const long long out0 = __reduce_add_sync(kAll, wsum[0][lane]);
  const int src_base = t0 * args.n_kv_heads + h;         // source row of position j: src_base + j * n_kv_heads
  auto put = [&](long long o, int position) {
    if (o < capacity) {
      a.kept_idx[o] = position;
      a.gather_src[o] = src_base + position * args.n_kv_heads;
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
    for (int t = tid; t < n_win; t += kThreads) put(out0 + k_keep + t, len - n_win + t);    // window rows: always kept
  }
  if (!choose) {                                         // uniform over the cluster: keep all of the history, or none
    if (k_keep > 0)
      for (int j = base + tid; j < my_end; j += kThreads)
        if (j >= 0) put(out0 + j, j);
    if (a.pooled_out == nullptr) return;
  }

  // ---- the bracket: ranks of the samples by counting, eight lanes per sample
  if (choose) {
    const int r_hi = sh_r[0], r_lo = sh_r[1];
    const int i = tid >> 3, part = tid & 7;
    const unsigned x = samp[i];
    int above = 0;
#pragma unroll
    for (int j = 0; j < kSamples / 8; j += 4) {
      const uint4 y = *reinterpret_cast<const uint4*>(samp + part * (kSamples / 8) + j);
      above += (y.x > x) + (y.y > x) + (y.z > x) + (y.w > x);
    }
    above += __shfl_xor_sync(kAll, above, 1);
    above += __shfl_xor_sync(kAll, above, 2);
    above += __shfl_xor_sync(kAll, above, 4);
    if (part == 0 && above == 0) sh_top = x | (kSamples - 1u);
    if (part == 0 && above == r_hi) sh_hi = x | (kSamples - 1u);
    if (part == 0 && above == r_lo) sh_lo = x & ~(kSamples - 1u);
  }
  __syncthreads();
  unsigned lo = sh_lo, hi = sh_hi;                       // every CTA of the cluster finds the same

  // ---- pooling; bit j of the masks is the thread's place j
  const int i0 = tid << log_items;
  const bool mine = i0 < own;
  unsigned gt = 0, cand = 0, valid = 0;
  float4 keep[kMaxItems / 4];
  if (mine) {
    const int p0 = base + i0, v_lo = max(-p0, 0), v_hi = min(my_end - p0, items);         // valid places of the thread
    valid = (v_hi >= 32 ? kAll : (1u << max(v_hi, 0)) - 1u) & (v_lo >= 32 ? 0u : kAll << v_lo);
    const float* src = votes + tid * pitch;
    float x[16];
    auto load4 = [&](const float* f, int k) {
      const float4 v = *reinterpret_cast<const float4*>(f);
      x[k] = v.x; x[k + 1] = v.y; x[k + 2] = v.z; x[k + 3] = v.w;
    };
    load4(votes + at(i0 - 4), 8);
    load4(src, 12);
#pragma unroll
    for (int g = 0; g < kMaxItems / 8; ++g) {
      if (8 * g < items) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = x[k + 8];
        load4(src + 8 * g + 4, 8);
        load4(8 * g + 8 < items ? src + 8 * g + 8 : src + pitch, 12);      // the next thread's first four
        float y[8];
        pool8<RAD>(x, max_mode, y);
        unsigned b_gt = 0, b_ge = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const unsigned v = __float_as_uint(y[e]);
          b_gt |= v > hi ? 1u << e : 0u;
          b_ge |= v >= lo ? 1u << e : 0u;
        }
        gt |= b_gt << (8 * g);
        cand |= b_ge << (8 * g);
        keep[2 * g] = make_float4(y[0], y[1], y[2], y[3]);
        keep[2 * g + 1] = make_float4(y[4], y[5], y[6], y[7]);
      }
    }
    gt &= valid;
    cand &= valid & ~gt;
  }
  {
    const unsigned both = __reduce_add_sync(kAll, (unsigned)__popc(gt) | ((unsigned)__popc(cand) << 16));
    if (lane == 0) wsum[1][wid] = both;
  }
  __syncthreads();                                       // everybody has read the votes: the scores take their places
  unsigned* keys = reinterpret_cast<unsigned*>(votes) + tid * pitch;
  if (mine) {
#pragma unroll
    for (int g = 0; g < kMaxItems / 4; ++g)
      if (4 * g < items) *reinterpret_cast<float4*>(keys + 4 * g) = keep[g];
  }
  if (a.pooled_out) {
    __syncthreads();
    for (int i = tid; i < own; i += kThreads)
      if (base + i >= 0 && base + i < my_end) a.pooled_out[seg_base + base + i] = votes[at(i)];
  }
  if (!choose) return;
  int need = k_keep;
  {
    const unsigned tot = __reduce_add_sync(kAll, wsum[1][lane]);
    int n_gt = (int)(tot & 0xffffu), n_cand = (int)(tot >> 16);
    if (CLUSTER) {
      if (tid == 0) cta_tot = make_int2(n_gt, n_cand);
      cluster.sync();
      int2 o = make_int2(0, 0);
      if (lane < CS) o = *cluster.map_shared_rank(&cta_tot, lane);
      n_gt = (int)__reduce_add_sync(kAll, (unsigned)o.x);
      n_cand = (int)__reduce_add_sync(kAll, (unsigned)o.y);
      // cta_tot is written again only behind the cluster-wide barriers of the descent
    }
    if (n_gt < k_keep && k_keep <= n_gt + n_cand) {
      need = k_keep - n_gt;
    } else {
      lo = 0; hi = kAll;
      gt = 0; cand = valid;
    }
  }

  // ---- radix descent inside [lo, hi]: `need` of the scores there, the largest, are kept
  // the bins divide lo .. top, the last one takes what lies above; at first top is four times the largest sample
  unsigned tau, top = max(min(sh_top + (2u << 23), hi), lo);
  while (true) {
    const unsigned span = top - lo;
    const int sh = span < (unsigned)kBins ? 0 : 21 - __clz(span);
    for (unsigned m = cand; m != 0; m &= m - 1) atomicAdd(&hist[min((keys[__ffs(m) - 1] - lo) >> sh, kBins - 1u)], 1);
    sync_all();
    int2 c2 = reinterpret_cast<const int2*>(hist)[tid];
    if (CLUSTER)
      for (int o = 1; o < CS; ++o) {
        const int2 x = reinterpret_cast<const int2*>(cluster.map_shared_rank(hist, (rank + o) % CS))[tid];
        c2.x += x.x;
        c2.y += x.y;
      }
    const unsigned sum = __reduce_add_sync(kAll, (unsigned)(c2.x + c2.y));
    if (lane == 0) wsum[0][wid] = sum;
    __syncthreads();
    const int above_w = (int)__reduce_add_sync(kAll, lane > wid ? wsum[0][lane] : 0u);
    if (above_w < need && need <= above_w + (int)sum) {   // the bin is one of this warp's 64
      int inc = c2.x + c2.y;                              // suffix sum over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_down_sync(kAll, inc, o);
        if (lane + o < 32) inc += v;
      }
      const int above = above_w + inc - (c2.x + c2.y);
      if (above < need && need <= above + c2.y) { sh_bin = 2 * tid + 1; sh_above = above; sh_m = c2.y; }
      else if (above + c2.y < need && need <= above + c2.y + c2.x) { sh_bin = 2 * tid; sh_above = above + c2.y; sh_m = c2.x; }
    }
    sync_all();                                           // in a cluster also: nobody reads the others' bins any more
    const int m_bin = sh_m;
    need -= sh_above;
    lo += sh_bin << sh;
    if (sh_bin < kBins - 1u) hi = min(hi, lo + ((1u << sh) - 1u));
    top = hi;
    if (lo == hi) { tau = lo; break; }
    // the bin's scores go on; where they fit, in a list of the cluster's first CTA (their order does not matter)
    const bool listed = m_bin <= kList;
    unsigned* list0 = CLUSTER ? cluster.map_shared_rank(list, 0) : nullptr;
    unsigned* n0 = CLUSTER ? cluster.map_shared_rank(&sh_n, 0) : nullptr;
    unsigned in_bin = 0;
    for (unsigned m = cand; m != 0; m &= m - 1) {
      const unsigned v = keys[__ffs(m) - 1], bit = m & (0u - m);
      if (v > hi) gt |= bit;
      else if (v >= lo) {
        in_bin |= bit;
        if (listed) {
          if (CLUSTER) list0[atomicAdd(n0, 1u)] = v;
          else list[atomicAdd(&sh_n, 1u)] = v;
        }
      }
    }
    cand = in_bin;
    if (listed) {                                         // ranked by counting
      sync_all();
      if (CLUSTER && rank > 0) {
        for (int i = tid; i < m_bin; i += kThreads) list[i] = list0[i];
        __syncthreads();
      }
      int log_p = 5;                                      // 2^log_p lanes per score
      while ((m_bin << log_p) > kThreads) --log_p;
      const int i = tid >> log_p, P = 1 << log_p, part = tid & (P - 1);
      if (wid << 5 >> log_p < m_bin) {                    // some score for this warp
        const unsigned x = list[min(i, m_bin - 1)];
        int above = 0, at_least = 0;
        for (int j = part; j < m_bin; j += P) { const unsigned y = list[j]; above += y > x; at_least += y >= x; }
        for (int o = 1; o < P; o <<= 1) {
          above += __shfl_xor_sync(kAll, above, o);
          at_least += __shfl_xor_sync(kAll, at_least, o);
        }
        if (i < m_bin && part == 0 && above < need && need <= at_least) { sh_tau = x; sh_need = need - above; }
      }
      __syncthreads();
      tau = sh_tau;
      need = sh_need;
      break;
    }
    reinterpret_cast<int2*>(hist)[tid] = make_int2(0, 0);
    __syncthreads();
  }

  // ---- ordered compaction: the scores above tau, and the first `need` equal to it; threads own consecutive positions
  unsigned eq = 0;
  for (unsigned m = cand; m != 0; m &= m - 1) {
    const unsigned v = keys[__ffs(m) - 1], bit = m & (0u - m);
    if (v > tau) gt |= bit;
    else if (v == tau) eq |= bit;
  }
  const unsigned cnt = (unsigned)__popc(gt) | ((unsigned)__popc(eq) << 16);
  unsigned inc = cnt;                                     // both totals are <= 32768
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(kAll, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) wsum[2][wid] = inc;
  __syncthreads();
  const unsigned before = __reduce_add_sync(kAll, lane < wid ? wsum[2][lane] : 0u) + inc - cnt;
  int gt_before = (int)(before & 0xffffu), eq_before = (int)(before >> 16);
  if (CLUSTER) {
    if (tid == kThreads - 1) cta_tot = make_int2(gt_before + __popc(gt), eq_before + __popc(eq));
    cluster.sync();
    int2 o = make_int2(0, 0);
    if (lane < rank) o = *cluster.map_shared_rank(&cta_tot, lane);
    gt_before += (int)__reduce_add_sync(kAll, (unsigned)o.x);
    eq_before += (int)__reduce_add_sync(kAll, (unsigned)o.y);
  }
  // of the thread's scores equal to tau, the first `take`
  const int take = min(max(need - eq_before, 0), __popc(eq));
  unsigned kept = gt;
  for (int t = 0; t < take; ++t) { kept |= eq & (0u - eq); eq &= eq - 1; }
  long long o = out0 + gt_before + min(eq_before, need);
  for (unsigned m = kept; m != 0; m &= m - 1, ++o) put(o, base + i0 + __ffs(m) - 1);
  if (CLUSTER) cluster.sync();                             // nobody leaves while its shared memory may still be read
}

// CTAs per segment: one wherever it can hold the segment's scores, however many SMs that leaves idle -- the exchanges of a
// cluster cost as much as the smaller slices save.  One layer of 8 segments, the whole call in us with 1, 2, 4 and 8 CTAs per
// segment: 1024 tokens 26.6, 30.7, 30.8, 32.7; 8192 tokens 32.8, 35.4, 36.8, 38.6; 16384 tokens 39.0, 41.2, 41.1, 43.1; 32768
// tokens 48.6, 49.2, 48.2, 49.3.
int cluster_size(const Problem& pb) {
  int cs = 1;
  while (cs < kMaxCluster && (pb.max_hist + 3 + cs - 1) / cs + 3 > kMaxSlice) cs *= 2;
  return cs;
}

}  // namespace

// up to 262116 history positions
bool select_list_supported(const Problem& pb) {
  return (pb.p.pool_kernel >> 1) <= kMaxRadius && (pb.max_hist + 3) / kMaxCluster + 4 <= kMaxSlice;
}

cudaError_t launch_select_list(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches) {
  typedef void (*Kern)(const SelArgs);
  static const Kern kerns[2][kMaxRadius + 1] = {
      {k_select_list<0, false>, k_select_list<1, false>, k_select_list<2, false>, k_select_list<3, false>, k_select_list<4, false>},
      {k_select_list<0, true>, k_select_list<1, true>, k_select_list<2, true>, k_select_list<3, true>, k_select_list<4, true>}};
  const int cs = cluster_size(pb);
  const int slice = ((pb.max_hist + 3 + cs - 1) / cs + 3) & ~3;
  const size_t smem = (size_t)vote_floats(slice <= 8 * kThreads ? 3 : (slice <= 16 * kThreads ? 4 : 5)) * sizeof(float);
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    for (int r = 0; r < 2 * (kMaxRadius + 1); ++r) {
      e = cudaFuncSetAttribute(kerns[r & 1][r >> 1], cudaFuncAttributeMaxDynamicSharedMemorySize, vote_floats(5) * (int)sizeof(float));
      if (e != cudaSuccess) return e;
    }
    configured_dev = dev;
  }
  SelArgs a;
  a.tab = pb.tab;
  a.n_seqs = pb.p.n_seqs; a.n_kv_heads = pb.p.n_kv_heads; a.window = pb.p.window; a.pool_mode = pb.p.pool_mode;
  for (int i = 0; i < n_layers; ++i) a.lay[i] = lay[i];
  LaunchScope scope(KID_SELECT, st, launches);
  return launch_pdl(kerns[cs > 1][pb.p.pool_kernel >> 1], dim3((unsigned)(pb.n_seg * cs), (unsigned)n_layers), dim3(kThreads), smem, st, cs, a);
}

}  // namespace slkv

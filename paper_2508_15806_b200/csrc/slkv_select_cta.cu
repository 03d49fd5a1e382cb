// Pooling + per-head variable-k selection for a list of layers (Sec. 3.4, Eq. 8; Algorithm 3 lines 1-4, 7-8): one CTA per
// (sequence, KV head) segment of up to 32768 history positions, a cluster of up to eight for longer ones.
//
// The votes come into shared memory with asynchronous 16-byte copies (from an aligned start, whatever the segment's), a
// thread pools 8, 16 or 32 consecutive positions of them and works with the scores' bit patterns (scores are >= 0, so
// unsigned order = float order).  The k-th largest:
//   1. with 16 or 32 positions per thread, a histogram of every 16th or 32nd score: the rank that the k-th largest has among
//      these, plus four standard deviations, bounds it from below (else the bound is zero);
//   2. a histogram of the scores above the bound, 2048 bins, 64 to an octave; the bin with the k-th largest;
//   3. where that bin's scores fit a list of 512 (mostly), they are ranked by counting, else a histogram of that bin, and so on.
// Then an ordered compaction from bit masks.  Integer counters only: the result does not depend on timing, and not on the
// sample either.
// What bounds it: a chain of some ten CTA-wide steps of 0.2-0.6 us, and at 32 positions per thread instructions.  Bracketing
// the k-th largest by 128 ranked samples and a descent over the bracket took as many steps again, and its loops an atomic
// with a result per score: whole layers of 8 segments 21.7 -> 16.9 us at 1024 positions, 26.4 -> 22.7 at 4096, 29.9 -> 26.4 at
// 8192, 33.7 -> 30.7 at 12000, 32 layers of 4001 129.5 -> 118 (all in a graph).
#include <cooperative_groups.h>

#include "slkv_internal.cuh"

namespace cg = cooperative_groups;

namespace slkv {
namespace {

constexpr int kMaxThreads = 1024;
constexpr int kMaxItems = 32;                         // consecutive positions per thread
constexpr int kMaxSlice = kMaxThreads * kMaxItems;    // 32768 positions per CTA
constexpr int kMaxCluster = 8;
constexpr int kMaxRadius = 4;                         // pool_kernel <= 9: four values on either side are enough
constexpr int kBins = 2048;
constexpr unsigned kAll = 0xffffffffu;
// First level's bins: 64 to an octave from 2^-24 up to 2^8 (a vote is at most the window, 256), the scores below in bin 0,
// whatever lies above in the last.
constexpr unsigned kFloorBits = (127u - 24u) << 23;
constexpr int kFirstShift = 17;
__device__ __forceinline__ unsigned first_bin(unsigned v) {
  const unsigned base = kFloorBits - (1u << kFirstShift);
  return min((max(v, base) - base) >> kFirstShift, kBins - 1u);
}
// Shared memory of the votes: a thread's positions are `items` floats, then four unused ones -- the pitch makes the 16-byte
// accesses of neighbouring threads conflict-free -- behind eight floats that hold the four before the first.
constexpr int kLead = 8;
template <int IT> constexpr int kLogItems = IT == 8 ? 3 : (IT == 16 ? 4 : 5);
constexpr int vote_floats(int threads, int items) { return kLead + (threads + 1) * (items + 4); }

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

// T threads with IT consecutive positions each.  CLUSTER: a segment is shared by the CTAs of a cluster (else every pointer
// below is known to be this CTA's own memory).
template <int T, int IT, int RAD, bool CLUSTER>
__global__ void __launch_bounds__(T, T == 1024 ? 1 : 1024 / T)
k_select_list(const __grid_constant__ SelArgs args) {
  constexpr int kWarps = T / 32, kPitch = IT + 4, kPer = kBins / T;     // bins per thread
  constexpr int kList = 512;
  constexpr bool kSample = IT > 8;
  extern __shared__ __align__(16) float votes_sh[];
  __shared__ __align__(16) int hist[kBins + 1];        // the last one: places that do not count
  __shared__ __align__(16) int sample[kSample ? kBins : 2];
  __shared__ __align__(16) unsigned list[kList];
  __shared__ unsigned wsum[3][32];
  __shared__ int2 cta_tot;                              // read by the cluster's other CTAs
  __shared__ unsigned sh_tau, sh_bin, sh_n;
  __shared__ int sh_above, sh_m, sh_need;

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
  float* votes = votes_sh + kLead;
  auto at = [&](int i) { return (i >> kLogItems<IT>) * kPitch + (i & (IT - 1)); };    // a place's index (i >= -4)
  // read here, where the kernel before this one is waited for anyway: a parameter's first read is a cache miss
  const long long capacity = a.capacity;
  int32_t* const kept_idx = a.kept_idx;
  int32_t* const gather_src = a.gather_src;
  float* const pooled_out = a.pooled_out;
  asm volatile("" ::"l"(capacity), "l"(kept_idx), "l"(gather_src), "l"(pooled_out), "l"(a.offsets));
  if (tid == 0) sh_n = 0;
#pragma unroll
  for (int i = 0; i < kPer; i += 2) {
    reinterpret_cast<int2*>(hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
    if (kSample) reinterpret_cast<int2*>(sample)[(tid * kPer + i) / 2] = make_int2(0, 0);
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
    if (lane == 0) wsum[0][wid] = part;
  }
  const int k_keep = kept_rows(len, budget, args.window) - n_win;             // C_H = C - window, clamped
  const bool choose = k_keep > 0 && k_keep < n;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // packed row where this segment starts = kept rows of all earlier segments (Algorithm 3 l.1-4 per head)
  const long long out0 = __reduce_add_sync(kAll, lane < kWarps ? wsum[0][lane] : 0u);
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
    const float* src = votes + tid * kPitch;
    float x[16];
    auto load4 = [&](const float* f, int k) {
      const float4 v = *reinterpret_cast<const float4*>(f);
      x[k] = v.x; x[k + 1] = v.y; x[k + 2] = v.z; x[k + 3] = v.w;
    };
    load4(votes + at(i0 - 4), 8);
    load4(src, 12);
#pragma unroll
    for (int g = 0; g < IT / 8; ++g) {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = x[k + 8];
      load4(src + 8 * g + 4, 8);
      load4(8 * g + 8 < IT ? src + 8 * g + 8 : src + kPitch, 12);          // the next thread's first four
      float y[8];
      pool8<RAD>(x, max_mode, y);
#pragma unroll
      for (int e = 0; e < 8; ++e) key[8 * g + e] = __float_as_uint(y[e]);
    }
    if (pooled_out) {
      float* dst = pooled_out + seg_base + p0;           // 16-byte aligned where the array is
      const bool wide = (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
#pragma unroll
      for (int g = 0; g < IT; g += 4) {
        if (wide && (valid >> g & 15u) == 15u) {
          *reinterpret_cast<uint4*>(dst + g) = make_uint4(key[g], key[g + 1], key[g + 2], key[g + 3]);
        } else {
#pragma unroll
          for (int e = g; e < g + 4; ++e)
            if (valid >> e & 1u) dst[e] = __uint_as_float(key[e]);
        }
      }
    }
  }
  if (!choose) return;

  // ---- the k-th largest by histograms.  bin_of: the bin that holds the `want` largest score of `bins` (more than that are
  // counted there), how many lie above it and in it; with no such bin, sh_bin = kBins.
  auto bin_of = [&](int* bins, int want) {
    if (tid == 0) sh_bin = kBins;
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      int2 v = reinterpret_cast<const int2*>(bins)[(tid * kPer + i) / 2];
      if (CLUSTER)
        for (int o = 1; o < CS; ++o) {
          const int2 w = reinterpret_cast<const int2*>(cluster.map_shared_rank(bins, (rank + o) % CS))[(tid * kPer + i) / 2];
          v.x += w.x;
          v.y += w.y;
        }
      c[i] = v.x;
      c[i + 1] = v.y;
      sum += v.x + v.y;
    }
    const int warp_sum = (int)__reduce_add_sync(kAll, (unsigned)sum);
    if (lane == 0) wsum[1][wid] = (unsigned)warp_sum;
    __syncthreads();
    const int above_w = (int)__reduce_add_sync(kAll, lane > wid && lane < kWarps ? wsum[1][lane] : 0u);
    if (above_w < want && want <= above_w + warp_sum) {   // the bin is one of this warp's
      int inc = sum;                                      // suffix sum over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_down_sync(kAll, inc, o);
        if (lane + o < 32) inc += v;
      }
      int above = above_w + inc - sum;
#pragma unroll
      for (int i = kPer - 1; i >= 0; --i) {
        if (above < want && want <= above + c[i]) { sh_bin = kPer * tid + i; sh_above = above; sh_m = c[i]; }
        above += c[i];
      }
    }
    sync_all();                                           // in a cluster also: nobody reads the others' bins any more
  };
  // Long slices: one place in IT is counted first.  Of these, the rank that the k-th largest has among them, plus four
  // standard deviations, bounds it from below, and only the scores above that bound are counted (an atomic on shared memory
  // takes seven cycles of the SM per warp, whether one lane adds or 32).
  unsigned bound = 0;
  uint4* const shelf = reinterpret_cast<uint4*>(votes + tid * kPitch);
  if (kSample) {
    if (mine && valid >> (IT / 2) & 1u) atomicAdd(&sample[first_bin(key[IT / 2])], 1);
    sync_all();                                          // everybody has read the votes, too: the scores take their places
    if (mine)
#pragma unroll
      for (int g = 0; g < IT; g += 4) shelf[g / 4] = make_uint4(key[g], key[g + 1], key[g + 2], key[g + 3]);
    const float f = __fdividef((float)k_keep, (float)n), q = f * (float)(n / IT);
    bin_of(sample, (int)(q + 4.f * sqrtf(q * (1.f - f))) + 2);
    const unsigned bin = sh_bin;
    if (bin > 0 && bin < (unsigned)kBins) bound = kFloorBits + ((bin - 1) << kFirstShift);
  }
  // f(e, score) for the thread's places
  auto each = [&](auto f) {
#pragma unroll
    for (int g = 0; g < IT; g += 4) {
      const uint4 v = kSample ? shelf[g / 4] : make_uint4(key[g], key[g + 1], key[g + 2], key[g + 3]);
      f(g, v.x); f(g + 1, v.y); f(g + 2, v.z); f(g + 3, v.w);
    }
  };
  int need = k_keep;
  unsigned lo = 0, hi = kAll, gt = 0, cand = valid, tau;
  int sh = kFirstShift;
  bool first = true;
  while (true) {
    auto index = [&](unsigned v) { return (int)(first ? first_bin(v) : min((v - lo) >> sh, kBins - 1u)); };
    // equal neighbours are added at once: a maximum holds for up to pool_kernel positions
    if (kSample && mine) {
      unsigned ends = 0, counted = 0, next = 0;           // places whose right neighbour's score is another; those that count
      each([&](int e, unsigned v) {
        if (e > 0) ends |= v != next ? 1u << (e - 1) : 0u;
        counted |= v >= bound ? 1u << e : 0u;
        next = v;
      });
      counted &= cand;
      ends = (ends | ~(counted >> 1)) & counted;
      const unsigned* keys = reinterpret_cast<const unsigned*>(shelf);
      int from = -1;                                      // the last place before the run
      for (unsigned m = ends, c = counted; m != 0; m &= m - 1) {
        const int e = __ffs(m) - 1;
        from = __ffs(c) - 2;
        atomicAdd(&hist[index(keys[e])], e - from);
        c &= e == 31 ? 0u : kAll << (e + 1);
      }
    } else if (mine) {
      int bin = kBins, run = 0;
      each([&](int e, unsigned v) {
        const int b = cand >> e & 1u ? index(v) : kBins;
        if (e > 0 && b != bin) { atomicAdd(&hist[bin], run); run = 0; }
        bin = b;
        ++run;
      });
      atomicAdd(&hist[bin], run);
    }
    sync_all();
    bin_of(hist, need);
    const unsigned bin = sh_bin;
    if (kSample && bin == (unsigned)kBins) {              // the bound was too high: everything counts
      bound = 0;
#pragma unroll
      for (int i = 0; i < kPer; i += 2) reinterpret_cast<int2*>(hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
      __syncthreads();
      continue;
    }
    const int m_bin = sh_m;
    need -= sh_above;
    if (first) {
      if (bin > 0) lo = kFloorBits + ((bin - 1) << kFirstShift);
      if (bin < kBins - 1u) hi = kFloorBits + (bin << kFirstShift) - 1u;
    } else {
      lo += bin << sh;
      if (bin < kBins - 1u) hi = min(hi, lo + ((1u << sh) - 1u));
    }
    first = false;
    // the bin's scores go on; where they fit, in a list of the cluster's first CTA (their order does not matter)
    const bool listed = m_bin <= kList && lo != hi;
    if (mine) {
      unsigned in_bin = 0;
      each([&](int e, unsigned v) {
        const unsigned bit = cand & 1u << e;
        gt |= v > hi ? bit : 0u;
        in_bin |= v >= lo && v <= hi ? bit : 0u;
      });
      cand = in_bin;
      if (listed && in_bin) {
        unsigned* dst = (CLUSTER ? cluster.map_shared_rank(list, 0) : list) +
                        atomicAdd(CLUSTER ? cluster.map_shared_rank(&sh_n, 0) : &sh_n, (unsigned)__popc(in_bin));
        if (kSample) {
          const unsigned* keys = reinterpret_cast<const unsigned*>(shelf);
          for (unsigned m = in_bin; m != 0; m &= m - 1) *dst++ = keys[__ffs(m) - 1];
        } else {
          each([&](int e, unsigned v) { if (in_bin >> e & 1u) *dst++ = v; });
        }
      }
    }
    if (lo == hi) { tau = lo; break; }
    if (listed) {                                         // ranked by counting
      sync_all();
      if (CLUSTER && rank > 0) {
        const unsigned* list0 = cluster.map_shared_rank(list, 0);
        for (int i = tid; i < m_bin; i += T) list[i] = list0[i];
        __syncthreads();
      }
      int log_p = 5;                                      // 2^log_p lanes per score
      while ((m_bin << log_p) > T) --log_p;
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
    const unsigned span = hi - lo;
    sh = span < (unsigned)kBins ? 0 : 21 - __clz(span);
    bound = lo;
#pragma unroll
    for (int i = 0; i < kPer; i += 2) reinterpret_cast<int2*>(hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
    __syncthreads();
  }

  // ---- ordered compaction: the scores above tau, and the first `need` equal to it; threads own consecutive positions
  unsigned eq = 0;
  if (mine)
    each([&](int e, unsigned v) {
      const unsigned bit = cand & 1u << e;
      gt |= v > tau ? bit : 0u;
      eq |= v == tau ? bit : 0u;
    });
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
    if (tid == T - 1) cta_tot = make_int2(gt_before + __popc(gt), eq_before + __popc(eq));
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
  // the kept positions, in shared memory first (where the votes were): whole lines then go out
  int* const stage = reinterpret_cast<int*>(votes_sh);
  const int o_mine = gt_before + min(eq_before, need);
  int o0 = 0, o1 = k_keep;                                 // the CTA's rows among the segment's
  if (CLUSTER) {
    if (tid == 0) sh_above = o_mine;
    if (tid == T - 1) sh_m = o_mine + __popc(kept);
    __syncthreads();
    o0 = sh_above;
    o1 = sh_m;
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
  const int cs = cluster_size(pb);
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

// Selection of the k largest of a segment's pooled scores (Sec. 3.4, Eq. 8; Algorithm 3 lines 7-8), device side: shared by the
// list selection (slkv_select_cta.cu) and the kernels that do a whole layer in one launch (slkv_layer_tc.cu,
// slkv_layer_fma.cu).  Everything here has internal linkage.
#pragma once
#include <cooperative_groups.h>

#include "slkv_internal.cuh"

namespace slkv {
namespace {

namespace cg = cooperative_groups;

constexpr int kMaxRadius = 4;                         // pool_kernel <= 9: four values on either side are enough
constexpr int kBins = 2048;
constexpr int kList = 512;                            // scores that are ranked by counting, at most; a thread for each
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
__host__ __device__ constexpr int vote_floats(int threads, int items) { return kLead + (threads + 1) * (items + 4); }

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

// Shared memory of a selection.
struct alignas(16) SelShared {
  int hist[kBins + 4];         // the last ones: places that do not count
  int sample[kBins];
  unsigned list[kList];
  unsigned wsum[3][32];
  int2 cta_tot;                // read by the cluster's other CTAs
  unsigned tau, bin, bin2, n_list;
  int above, m, need, sure;
};

// A thread's kept places of a segment: T threads (numbered tid) with IT consecutive places each, their scores' bit patterns
// in key (scores are >= 0: unsigned order = float order), those that exist in valid.  k_keep of the n scores are kept, the
// largest, ties to the lower place.  CLUSTER: the segment is shared by the CTAs of a cluster (rank, CS).  BAR: the named
// barrier of the T threads.  shelf: the thread's row of the votes' shared memory, which the scores take over once all T
// threads are past their pooling (IT > 8 only).  sh.hist, sh.sample, sh.n_list and sh.sure are zero, for all to see.
// Returns the kept places as a mask and, in o_mine, how many of the segment's lie before the thread's; tau: the k-th largest score.
template <int T, int IT, bool CLUSTER, int BAR>
__device__ __forceinline__ unsigned select_places(SelShared& sh_, int tid, unsigned (&key)[IT], unsigned valid, bool mine,
                                                  uint4* shelf, int n, int k_keep, int rank, int CS, int& o_mine, unsigned& tau) {
  constexpr int kWarps = T / 32, kPer = kBins / T;      // bins per thread
  constexpr int kRanked = kList < T ? kList : T;        // a bin of more scores goes through another level of bins
  static_assert(kRanked <= T && kRanked <= kList && kPer % 2 == 0 && kWarps <= 32, "a thread per listed score, whole int2 of bins");
  constexpr bool kSample = IT > 8;
  const int lane = tid & 31, wid = tid >> 5;
  auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(T) : "memory"); };
  auto sync_all = [&]() { if (CLUSTER) cg::this_cluster().sync(); else sync(); };
  int* const hist = sh_.hist;
  auto clear_hist = [&]() {
#pragma unroll
    for (int i = 0; i < kPer; i += 2) reinterpret_cast<int2*>(hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
  };
  // ---- the k-th largest by histograms.  bin_of: the bin that holds the `want` largest score of `bins` (more than that are
  // counted there), how many lie above it and in it; with no such bin, sh_.bin = kBins.  want2: likewise, the bin alone.
  auto bin_of = [&](int* bins, int want, int want2) {
    if (tid == 0) sh_.bin = sh_.bin2 = kBins;
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      int2 v = reinterpret_cast<const int2*>(bins)[(tid * kPer + i) / 2];
      if (CLUSTER)
        for (int o = 1; o < CS; ++o) {
          const int2 w = reinterpret_cast<const int2*>(cg::this_cluster().map_shared_rank(bins, (rank + o) % CS))[(tid * kPer + i) / 2];
          v.x += w.x;
          v.y += w.y;
        }
      c[i] = v.x;
      c[i + 1] = v.y;
      sum += v.x + v.y;
    }
    const int warp_sum = (int)__reduce_add_sync(kAll, (unsigned)sum);
    if (lane == 0) sh_.wsum[1][wid] = (unsigned)warp_sum;
    sync();
    const int above_w = (int)__reduce_add_sync(kAll, lane > wid && lane < kWarps ? sh_.wsum[1][lane] : 0u);
    if ((above_w < want && want <= above_w + warp_sum) || (above_w < want2 && want2 <= above_w + warp_sum)) {   // one of this warp's
      int inc = sum;                                      // suffix sum over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_down_sync(kAll, inc, o);
        if (lane + o < 32) inc += v;
      }
      int above = above_w + inc - sum;
#pragma unroll
      for (int i = kPer - 1; i >= 0; --i) {
        if (above < want && want <= above + c[i]) { sh_.bin = kPer * tid + i; sh_.above = above; sh_.m = c[i]; }
        if (above < want2 && want2 <= above + c[i]) sh_.bin2 = kPer * tid + i;
        above += c[i];
      }
    }
    sync_all();                                           // in a cluster also: nobody reads the others' bins any more
  };
  // Long slices: one place in IT is counted first.  Of these, the rank that the k-th largest has among them, give or take four
  // standard deviations, bounds it from below and above: only the scores between the bounds, an eighth of them at most, go
  // through the bins (an atomic on shared memory takes seven cycles of the SM per warp, whether one lane adds or 32, and a loop
  // over the bits of a mask as many turns as the warp's fullest lane), those above are counted together.
  unsigned bound = 0, sure_above = kAll;
  if (kSample) {
    if (mine && valid >> (IT / 2) & 1u) atomicAdd(&sh_.sample[first_bin(key[IT / 2])], 1);
    sync_all();                                          // everybody has read the votes, too: the scores take their places
    if (mine)
#pragma unroll
      for (int g = 0; g < IT; g += 4) shelf[g / 4] = make_uint4(key[g], key[g + 1], key[g + 2], key[g + 3]);
    const float f = __fdividef((float)k_keep, (float)n), q = f * (float)(n / IT);
    const float dev = 4.f * sqrtf(q * (1.f - f));
    bin_of(sh_.sample, (int)(q + dev) + 2, (int)floorf(q - dev) - 1);
    const unsigned bin = sh_.bin, bin2 = sh_.bin2;
    if (bin > 0 && bin < (unsigned)kBins) bound = kFloorBits + ((bin - 1) << kFirstShift);
    if (bin2 < kBins - 1u) sure_above = kFloorBits + (bin2 << kFirstShift) - 1u;
  }
  // f(e, score) for the thread's places
  auto each = [&](auto f) {
#pragma unroll
    for (int g = 0; g < IT; g += 4) {
      const uint4 v = kSample ? shelf[g / 4] : make_uint4(key[g], key[g + 1], key[g + 2], key[g + 3]);
      f(g, v.x); f(g + 1, v.y); f(g + 2, v.z); f(g + 3, v.w);
    }
  };
  const unsigned* keys = reinterpret_cast<const unsigned*>(shelf);
  // of the thread's places, those between the bounds, and the last ones of each run of equal scores among them (a maximum holds
  // for up to pool_kernel positions); runs: f(score, the run's places)
  unsigned between = 0, ends = 0;
  auto runs = [&](auto f) {
    for (unsigned m = ends, left = between; m != 0; m &= m - 1) {
      const unsigned last = m & (0u - m), run = left & (last | (last - 1));
      left ^= run;
      f(keys[__ffs(m) - 1], run);
    }
  };
  int need = k_keep;
  unsigned lo = 0, hi = kAll, gt = 0, cand = valid;
  int sh = kFirstShift;
  bool first = true;
  while (true) {
    auto index = [&](unsigned v) { return (int)(first ? first_bin(v) : min((v - lo) >> sh, kBins - 1u)); };
    // neighbours of one bin, or of one score, are added at once
    if (kSample && mine) {
      unsigned sure = 0, next = 0;
      between = ends = 0;
      each([&](int e, unsigned v) {
        if (e > 0) ends |= v != next ? 1u << (e - 1) : 0u;
        between |= v >= bound ? 1u << e : 0u;
        sure |= v > sure_above ? 1u << e : 0u;
        next = v;
      });
      between &= cand & ~sure;
      gt |= sure & cand;
      ends = (ends | ~(between >> 1)) & between;
      runs([&](unsigned v, unsigned run) { atomicAdd(&hist[index(v)], __popc(run)); });
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
    int n_sure = 0;
    if (kSample && first) {
      const unsigned w = __reduce_add_sync(kAll, (unsigned)__popc(gt));
      if (lane == 0 && w) atomicAdd(&sh_.sure, (int)w);
    }
    sync_all();
    if (kSample && first) {
      n_sure = sh_.sure;
      if (CLUSTER) n_sure = (int)__reduce_add_sync(kAll, lane < CS ? (unsigned)*cg::this_cluster().map_shared_rank(&sh_.sure, lane) : 0u);
    }
    bin_of(hist, need - n_sure, 0);
    const unsigned bin = sh_.bin;
    if (kSample && bin == (unsigned)kBins) {              // the k-th largest lies outside: everything goes through the bins
      bound = 0;
      sure_above = kAll;
      gt = 0;
      if (tid == 0) sh_.sure = 0;
      clear_hist();
      sync();
      continue;
    }
    const int m_bin = sh_.m;
    need -= n_sure;
    need -= sh_.above;
    if (first) {
      if (bin > 0) lo = kFloorBits + ((bin - 1) << kFirstShift);
      if (bin < kBins - 1u) hi = kFloorBits + (bin << kFirstShift) - 1u;
    } else {
      lo += bin << sh;
      if (bin < kBins - 1u) hi = min(hi, lo + ((1u << sh) - 1u));
    }
    first = false;
    // the bin's scores go on; where they fit, in a list of the cluster's first CTA (their order does not matter)
    const bool listed = m_bin <= kRanked && lo != hi;
    if (mine) {
      unsigned in_bin = 0;
      if (kSample) {
        runs([&](unsigned v, unsigned run) {
          if (v > hi) gt |= run; else if (v >= lo) in_bin |= run;
        });
      } else {
        each([&](int e, unsigned v) {
          const unsigned bit = cand & 1u << e;
          gt |= v > hi ? bit : 0u;
          in_bin |= v >= lo && v <= hi ? bit : 0u;
        });
      }
      cand = in_bin;
      if (listed && in_bin) {
        unsigned* dst = (CLUSTER ? cg::this_cluster().map_shared_rank(sh_.list, 0) : sh_.list) +
                        atomicAdd(CLUSTER ? cg::this_cluster().map_shared_rank(&sh_.n_list, 0) : &sh_.n_list, (unsigned)__popc(in_bin));
        if (kSample) {
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
        const unsigned* list0 = cg::this_cluster().map_shared_rank(sh_.list, 0);
        for (int i = tid; i < m_bin; i += T) sh_.list[i] = list0[i];
        sync();
      }
      int log_p = 5;                                      // 2^log_p lanes per score; m_bin <= T: one at least
      while ((m_bin << log_p) > T) --log_p;
      const int i = tid >> log_p, P = 1 << log_p, part = tid & (P - 1);
      if (wid << 5 >> log_p < m_bin) {                    // some score for this warp
        const unsigned x = sh_.list[min(i, m_bin - 1)];
        int above = 0, at_least = 0;
        for (int j = part; j < m_bin; j += P) { const unsigned y = sh_.list[j]; above += y > x; at_least += y >= x; }
        for (int o = 1; o < P; o <<= 1) {
          above += __shfl_xor_sync(kAll, above, o);
          at_least += __shfl_xor_sync(kAll, at_least, o);
        }
        if (i < m_bin && part == 0 && above < need && need <= at_least) { sh_.tau = x; sh_.need = need - above; }
      }
      sync();
      tau = sh_.tau;
      need = sh_.need;
      break;
    }
    const unsigned span = hi - lo;
    sh = span < (unsigned)kBins ? 0 : 21 - __clz(span);
    bound = lo;
    sure_above = kAll;
    clear_hist();
    sync();
  }

  // ---- ordered compaction: the scores above tau, and the first `need` equal to it; threads own consecutive positions
  unsigned eq = 0;
  if (kSample) {
    for (unsigned m = cand; m != 0; m &= m - 1) {
      const unsigned v = keys[__ffs(m) - 1], bit = m & (0u - m);
      if (v > tau) gt |= bit; else if (v == tau) eq |= bit;
    }
  } else if (mine) {
    each([&](int e, unsigned v) {
      const unsigned bit = cand & 1u << e;
      gt |= v > tau ? bit : 0u;
      eq |= v == tau ? bit : 0u;
    });
  }
  const unsigned cnt = (unsigned)__popc(gt) | ((unsigned)__popc(eq) << 16);
  unsigned inc = cnt;                                     // both totals are <= 32768
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(kAll, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) sh_.wsum[2][wid] = inc;
  sync();
  const unsigned before = __reduce_add_sync(kAll, lane < wid ? sh_.wsum[2][lane] : 0u) + inc - cnt;
  int gt_before = (int)(before & 0xffffu), eq_before = (int)(before >> 16);
  if (CLUSTER) {
    if (tid == T - 1) sh_.cta_tot = make_int2(gt_before + __popc(gt), eq_before + __popc(eq));
    cg::this_cluster().sync();
    int2 o = make_int2(0, 0);
    if (lane < rank) o = *cg::this_cluster().map_shared_rank(&sh_.cta_tot, lane);
    gt_before += (int)__reduce_add_sync(kAll, (unsigned)o.x);
    eq_before += (int)__reduce_add_sync(kAll, (unsigned)o.y);
  }
  // of the thread's scores equal to tau, the first `take`
  const int take = min(max(need - eq_before, 0), __popc(eq));
  unsigned kept = gt;
  for (int t = 0; t < take; ++t) { kept |= eq & (0u - eq); eq &= eq - 1; }
  o_mine = gt_before + min(eq_before, need);
  return kept;
}

// The scores of IT places from shared memory (the votes of place i at votes[at(i)], four readable on either side).
template <int RAD, int IT>
__device__ __forceinline__ void pool_places(const float* src, const float* before, bool max_mode, unsigned (&key)[IT]) {
  float x[16];
  auto load4 = [&](const float* f, int k) {
    const float4 v = *reinterpret_cast<const float4*>(f);
    x[k] = v.x; x[k + 1] = v.y; x[k + 2] = v.z; x[k + 3] = v.w;
  };
  load4(before, 8);
  load4(src, 12);
#pragma unroll
  for (int g = 0; g < IT / 8; ++g) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = x[k + 8];
    load4(src + 8 * g + 4, 8);
    load4(8 * g + 8 < IT ? src + 8 * g + 8 : src + IT + 4, 12);            // the next thread's first four
    float y[8];
    pool8<RAD>(x, max_mode, y);
#pragma unroll
    for (int e = 0; e < 8; ++e) key[8 * g + e] = __float_as_uint(y[e]);
  }
}

// A thread's scores into the caller's array (dst: place 0).
template <int IT>
__device__ __forceinline__ void store_scores(float* dst, const unsigned (&key)[IT], unsigned valid) {
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

}  // namespace
}  // namespace slkv

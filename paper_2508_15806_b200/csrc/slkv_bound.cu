// Lists of layers whose votes nobody asked for, only what is kept (Sec. 3.4, Eq. 7-8; Algorithm 3): one product with every key
// instead of two.  Max pooling, everything the list score kernel takes, no log-sum-exps handed in.
//
// A vote needs its rows' sums over all keys, so a kernel that computes all votes goes over the keys twice.  Few of them decide
// what is kept.  Here k_score_list (kBound; slkv_score_pipe.cu, bound_run) adds up the rows' sums as ever and from the same
// exponentials, run by run, estimates the keys' votes with the rows' sums over the run's first tiles: est[j] = sum_r w_r 2^s_rj.
// k_select_bound then knows how far every weight is off.  With rho the largest w_r^-1 / sum_r of the run,
// vote[j] <= rho * est[j] / G: the keys whose bound is above a threshold get their exact vote, on the tensor cores as in the vote
// pass and bit for bit the same (kWide's, whose row sums these are), the others none.  With T the k-th largest pooled score of what is there, a position whose score is
// T or more has it from a key whose vote is T or more; if the threshold is below T, no key without its vote is such a one, so the
// kept positions are those of all votes, ties included.  If not, every key whose bound is T or more is added, and then it
// holds: T can only have grown.
// Segments that keep a large share of their positions (every_vote) have all their votes computed by the score kernel, behind
// the statistics, as ever.  Wherever the bounds cannot be relied on -- weights or sums outside a range in which fp32 neither over-
// nor underflows, anything that is not finite -- every key of the segment gets its exact vote here.
#include <cuda.h>

#include "slkv_internal.cuh"
#include "slkv_select_device.cuh"
#include "slkv_tc_device.cuh"

namespace slkv {
namespace {

struct BoundArgs {
  ScoreShape sh;
  ScoreLayer lay[kListMaxLayers];
  TailLayer tail[kListMaxLayers];
  long long k_stride_tok, k_stride_head;       // elements
  int k_tiles, n_layers;                       // tiles of keys in shared memory at a time
};

// ---- selection ----------------------------------------------------------------------------------------------------------
// Bins of the estimated scores: 32 to an octave from 2^-52 up to 2^12.
constexpr unsigned kEstFloor = (127u - 52u) << 23;
constexpr int kEstShift = 18;
__device__ __forceinline__ int est_bin(unsigned v) {
  const unsigned base = kEstFloor - (1u << kEstShift);
  return (int)min((max(v, base) - base) >> kEstShift, kBins - 1u);
}
// The estimates are sums of bf16 values (four roundings of 2^-9), votes and estimates have exponentials of arguments below 2^7
// (2^-16): together under a hundredth.
constexpr float kSlack = 1.02f;
// The first threshold: where T is expected, at the rows' mean error, and a little lower.
constexpr float kMargin = 0.8f, kFewMargin = 0.45f;
constexpr int kFew = 64;                     // up to this many positions the lower one: a second round costs more than some keys
// Logarithms (base 2) of sums, and of errors, with which the bounds hold: see bound_run.
constexpr float kLowLog = -48.f, kHighLog = 110.f, kMaxError = 60.f;
// A threshold below this proves nothing: an estimate takes scores below 2^-126 for zero, which in the vote are up to 2^(-126 - kLowLog)
// of a row each, 2^-70 over 256 rows.  That is a thousandth of this, well within kSlack; the first threshold lies above 2^-54.
constexpr float kTinyScore = 0x1p-60f;

struct alignas(16) BoundShared {
  unsigned long long q_full, mma_done;
  uint32_t tmem;
  int abort_flag, bad, bin, halo;
  alignas(16) float lse[256];                // negated
  float half[2][128];
  float mid[2 * kMaxSplit], reach[2 * kMaxSplit];      // per run and set of weights: expected vote and bound, over the estimate
  float beside[8];                           // exact votes of the four places on either side of a cluster's slice
};

constexpr int kThreads = 1024;

// IT consecutive positions a thread.  CLUSTER: a segment is shared by the CTAs of a cluster.
template <int IT, int RAD, bool CLUSTER>
__global__ void __launch_bounds__(kThreads, 1)
k_select_bound(const __grid_constant__ BoundArgs args) {
  constexpr int T = kThreads;
  constexpr int kWarps = T / 32, kPitch = IT + 4, kPer = kBins / T;
  // [votes] or [Q][keys][list of places]
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ SelShared sh;
  __shared__ BoundShared b;
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = CLUSTER ? (int)cluster.num_blocks() : 1, rank = CLUSTER ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const ScoreShape& shp = args.sh;
  const TailLayer& a = args.tail[blockIdx.y];
  const ScoreLayer& L = args.lay[blockIdx.y];
  if ((smem_u32(smem) & 1023u) != 0) {                  // the swizzled tiles need it (uniform over the launch)
    if (tid == 0 && a.status) atomicExch(a.status, (int)SLKV_ERR_BAD_ALIGN);
    return;
  }
  const int n_kv = shp.n_kv_heads, window = shp.window, R = shp.R, MT = shp.MT, halves = shp.halves;
  const int seg = blockIdx.x / CS, s = seg / n_kv, h = seg - s * n_kv;
  const int t0 = shp.tab.cu_at(s), len = shp.tab.cu_at(s + 1) - t0;
  const int n = max(len - window, 0), n_win = min(len, window);
  const int n_seg = shp.n_seqs * n_kv;
  const long long seg_base = shp.tab.hist_at(s) * n_kv + (long long)h * n;
  float* const vote = L.vote + seg_base;
  // the CTA's slice, as in k_select_list: place i is position base + i
  const int shift = (int)(seg_base & 3);
  const int slice = ((n + shift + CS - 1) / CS + 3) & ~3;
  const int own = min(max(n + shift - rank * slice, 0), slice), base = rank * slice - shift;
  const int my_end = min(base + own, n);
  float* const votes = reinterpret_cast<float*>(smem) + kLead;
  auto at = [&](int i) { return (i >> kLogItems<IT>) * kPitch + (i & (IT - 1)); };
  const int q_half = MT * 128 * 128, q_bytes = halves * q_half, stage = halves * kHalfBytes;
  unsigned short* const list = reinterpret_cast<unsigned short*>(smem + q_bytes + args.k_tiles * stage);      // a place + 4
  const uint32_t q_sh = smem_u32(smem), k_sh = q_sh + (uint32_t)q_bytes;
  auto clear_bins = [&]() {
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      reinterpret_cast<int2*>(sh.hist)[(tid * kPer + i) / 2] = make_int2(0, 0);
      reinterpret_cast<int2*>(sh.sample)[(tid * kPer + i) / 2] = make_int2(0, 0);
    }
    if (tid == 0) { sh.n_list = 0; sh.sure = 0; sh.hist[kBins + 1] = 0; }      // the last: estimates that are not finite
  };
  auto sync_all = [&]() { if (CLUSTER) cluster.sync(); else __syncthreads(); };
  const uint32_t tmem_cols = 128u * (uint32_t)(args.k_tiles * MT);
  clear_bins();
  if (tid == 0) {
    b.abort_flag = 0;
    b.bad = 0;
    mbar_init(smem_u32(&b.q_full), 1);
    mbar_init(smem_u32(&b.mma_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();
  // TMEM is asked for behind the wait, and the next kernel let go behind that: a CTA that holds columns waits for no other
  // kernel, and one of a kernel that takes its columns before it waits comes only when these are given out.
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&b.tmem)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // ---- the estimates on their way, with one group of four places on either side
  for (int q = tid - 1; 4 * q <= own + 3; q += T) {
    const int p = base + 4 * q;
    float* dst = votes + at(4 * q);
    if (p >= 0 && p + 3 < n) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(vote + p) : "memory");
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) dst[e] = p + e >= 0 && p + e < n ? __ldcg(vote + p + e) : 0.f;
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int budget = __ldg(a.budgets + h);
  {
    unsigned part = 0;                                  // < 2^31: the host checks n_kv_heads * total_tokens
    for (int g = tid; g < seg; g += T) {
      const int s2 = g / n_kv, h2 = g - s2 * n_kv;
      part += (unsigned)kept_rows(shp.tab.cu_at(s2 + 1) - shp.tab.cu_at(s2), a.budgets[h2], window);
    }
    part = __reduce_add_sync(kAll, part);
    if (lane == 0) sh.wsum[0][wid] = part;
  }
  const int k_keep = kept_rows(len, budget, window) - n_win;             // C_H = C - window, clamped
  const bool choose = k_keep > 0 && k_keep < n;
  const bool every = every_vote(len, budget, window);   // votes, not estimates
  // ---- the rows' log-sum-exps
  const StatView st = stat_view(L.part, n_seg, R, shp.slot_stride);
  bool far_off = false;                                  // a row with which the bounds do not hold
  if (tid < 256) {
    float l2 = INFINITY;
    if (tid < R && choose && !every) {
      const size_t row = (size_t)seg * R + tid;
      bool far = false;
      for (int w = 0; w < kFarWords; ++w) far |= __ldcg(st.far + (size_t)seg * kFarWords + w) != 0;
      const bool win = L.lse.win_m != nullptr;
      l2 = row_lse(st, __ldcg(st.acc + row), far, seg, tid, R, shp.slot_stride, min(shp.slot_stride, kMaxSplit), win,
                   win ? L.lse.win_m[row] : 0.f, win ? L.lse.win_z[row] : 0.f);
      far_off = far || !(l2 >= kLowLog && l2 <= kHighLog);
    }
    b.lse[tid] = -l2;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  tc_fence_before();
  const bool rows_off = __syncthreads_or(far_off) != 0;
  tc_fence_after();
  pdl_launch_dependents();
  const uint32_t tmem = b.tmem;
  const long long capacity = a.capacity;
  int32_t* const kept_idx = a.kept_idx;
  int32_t* const gather_src = a.gather_src;
  // packed row where this segment starts = kept rows of all earlier segments (Algorithm 3 l.1-4 per head)
  const long long out0 = __reduce_add_sync(kAll, lane < kWarps ? sh.wsum[0][lane] : 0u);
  const int src_base = t0 * n_kv + h;                    // source row of position j: src_base + j * n_kv
  auto put = [&](long long o, int position) {
    if (o < capacity) {
      kept_idx[o] = position;
      gather_src[o] = src_base + position * n_kv;
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
  if (!choose && k_keep > 0)                             // uniform over the cluster: keep all of the history, or none
    for (int j = base + tid; j < my_end; j += T)
      if (j >= 0) put(out0 + j, j);

  if (choose) {
    const int i0 = tid * IT;
    const bool mine = i0 < own;
    unsigned valid = 0;
    const float inv_g = 1.0f / (float)shp.G;
    // ---- per run of the score kernel: how far its weights are off, the largest and the mean of the rows'
    const SegmentSlots runs = list_slots(shp, args.n_layers, blockIdx.y, s, h);
    if (!every) {
      for (int c = wid; c < 2 * runs.n; c += kWarps) {
        const int count = runs.count(c >> 1);
        if (c & 1 && second_weights(count) >= count) continue;         // of a run with one set of weights
        const float* weight = (c & 1 ? st.far_m : st.far_z) + ((size_t)seg * shp.slot_stride + (c >> 1)) * R;
        float m = -INFINITY, sum = 0.f;
        bool bad = false;
        for (int r = lane; r < R; r += 32) {
          const float err = b.lse[r] - log2f(__ldcg(weight + r));
          bad |= !(fabsf(err) <= kMaxError);
          m = fmaxf(m, err);
          sum += err;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
          sum += __shfl_xor_sync(kAll, sum, o);
        }
        if (__any_sync(kAll, bad) && lane == 0) b.bad = 1;
        if (lane == 0) {
          b.mid[c] = exp2f(sum / (float)R) * inv_g;
          b.reach[c] = exp2f(m) * kSlack * inv_g;
        }
      }
      __syncthreads();
    }
    const bool safe_rows = !rows_off && b.bad == 0;
    auto run_of = [&](int p) {
      const int tile = p >> 7, c = runs.slot(tile), count = runs.count(c), t = tile - runs.begin(c);
      const int nth = MT == 1 ? Spread<1>(count).tile(t) : Spread<2>(count).tile(t);       // its own inverse
      return 2 * c + (nth >= second_weights(count));
    };
    // the thread's places lie in one tile or two: from place `cut` on in the second
    int run_a = 0, run_b = 0, cut = IT;
    if (!every && mine) {
      const int p0 = max(base + i0, 0), p1 = min(base + i0 + IT, my_end) - 1;
      run_a = run_b = run_of(p0);
      if (p1 >> 7 != p0 >> 7) { run_b = run_of(p1); cut = (p1 & ~127) - base - i0; }
      const float mid_a = b.mid[run_a], mid_b = b.mid[run_b];
#pragma unroll
      for (int e = 0; e < IT; ++e)
        if (i0 + e < own) votes[tid * kPitch + e] *= e < cut ? mid_a : mid_b;
    }
    if (!every && wid == 0 && lane < 8) {                // the four places on either side
      const int place = lane < 4 ? lane - 4 : own + lane - 4, p = base + place;
      if (own > 0 && p >= 0 && p < n) votes[at(place)] *= b.mid[run_of(p)];
    }
    __syncthreads();
    // ---- the bin of the k-th largest pooled expected vote
    if (mine) {
      const int p0 = base + i0, v_lo = max(-p0, 0), v_hi = min(my_end - p0, IT);
      valid = (v_hi >= 32 ? kAll : (1u << max(v_hi, 0)) - 1u) & (v_lo >= 32 ? 0u : kAll << v_lo);
    }
    if (mine && !every) {
      unsigned key[IT];
      pool_places<RAD>(votes + tid * kPitch, votes + at(i0 - 4), true, key);
      int bin = kBins, run = 0;
      bool bad = false;
#pragma unroll
      for (int e = 0; e < IT; ++e) {
        const int x = valid >> e & 1u ? est_bin(key[e]) : kBins;
        bad |= (valid >> e & 1u) && __float_as_uint(votes[tid * kPitch + e]) >= 0x7f800000u;
        if (x != bin) {
          if (run) atomicAdd(&sh.hist[bin], run);
          run = 0;
        }
        bin = x;
        ++run;
      }
      atomicAdd(&sh.hist[bin], run);
      if (bad) atomicAdd(&sh.hist[kBins + 1], 1);
    }
    bool safe = false;
    if (!every) {
      if (tid == 0) b.bin = 0;
      sync_all();
      int c[kPer], sum = 0, bad = sh.hist[kBins + 1];
#pragma unroll
      for (int i = 0; i < kPer; ++i) c[i] = sh.hist[tid * kPer + i];
      if (CLUSTER)
        for (int o = 1; o < CS; ++o) {
          const int* other = cluster.map_shared_rank(sh.hist, (rank + o) % CS);
          bad += other[kBins + 1];
#pragma unroll
          for (int i = 0; i < kPer; ++i) c[i] += other[tid * kPer + i];
        }
      safe = safe_rows && bad == 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) sum += c[i];
      const int warp_sum = (int)__reduce_add_sync(kAll, (unsigned)sum);
      if (lane == 0) sh.wsum[1][wid] = (unsigned)warp_sum;
      __syncthreads();
      const int above_w = (int)__reduce_add_sync(kAll, lane > wid && lane < kWarps ? sh.wsum[1][lane] : 0u);
      if (above_w < k_keep && k_keep <= above_w + warp_sum) {
        int inc = sum;                                   // suffix sum over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_down_sync(kAll, inc, o);
          if (lane + o < 32) inc += v;
        }
        int above = above_w + inc - sum;
#pragma unroll
        for (int i = kPer - 1; i >= 0; --i) {
          if (above < k_keep && k_keep <= above + c[i]) b.bin = kPer * tid + i;
          above += c[i];
        }
      }
      sync_all();                                        // nobody reads the others' bins any more
    }
    float bound = 0.f;                                   // a key whose vote may be this large gets it
    if (safe && b.bin > 0) bound = __uint_as_float(kEstFloor + ((unsigned)(b.bin - 1) << kEstShift)) * (k_keep <= kFew ? kFewMargin : kMargin);

    unsigned done = 0, halo_done = 0, kept = 0;
    float beside = 0.f;                                  // warp 0, a lane each: the bounds of the places beside the slice
    int o_mine = 0, n_mma = 0, n_q = 0;
    for (int round = 0;; ++round) {
      if (!every) {
        // ---- the places that get their exact vote now; in a cluster also the four on either side of the slice, for the pooling
        unsigned want = valid, halo = 0;
        if (bound > 0.f && mine) {
          // from the expected vote, later from the estimate itself, to the bound
          const float f_a = round == 0 ? b.reach[run_a] / b.mid[run_a] : b.reach[run_a], f_b = round == 0 ? b.reach[run_b] / b.mid[run_b] : b.reach[run_b];
          want = 0;
#pragma unroll 2
          for (int e = 0; e < IT; e += 4) {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (round == 0) {
              x = *reinterpret_cast<const float4*>(votes + tid * kPitch + e);
            } else if ((valid >> e & 15u) == 15u) {
              x = __ldcg(reinterpret_cast<const float4*>(vote + base + i0 + e));
            } else {
              const float* f = vote + base + i0 + e;
              if (valid >> e & 1u) x.x = __ldcg(f);
              if (valid >> e & 2u) x.y = __ldcg(f + 1);
              if (valid >> e & 4u) x.z = __ldcg(f + 2);
              if (valid >> e & 8u) x.w = __ldcg(f + 3);
            }
            want |= (!(x.x * (e < cut ? f_a : f_b) < bound) ? 1u : 0u) << e | (!(x.y * (e + 1 < cut ? f_a : f_b) < bound) ? 2u : 0u) << e |
                    (!(x.z * (e + 2 < cut ? f_a : f_b) < bound) ? 4u : 0u) << e | (!(x.w * (e + 3 < cut ? f_a : f_b) < bound) ? 8u : 0u) << e;
          }
          want = (want & valid) | done;
        }
        if (CLUSTER && wid == 0) {
          const int place = lane < 4 ? lane - 4 : own + lane - 4, p = base + place;
          bool hit = lane < 8 && own > 0 && (lane < 4 ? rank > 0 : p < n);
          if (hit && bound > 0.f && !(halo_done >> lane & 1u)) {
            const int c = run_of(p);
            if (round == 0) beside = votes[at(place)] * (b.reach[c] / b.mid[c]);
            hit = !(beside < bound);
          }
          halo = __ballot_sync(kAll, hit);
        }
        const unsigned fresh = want & ~done;
        int inc = __popc(fresh);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(kAll, inc, o);
          if (lane >= o) inc += x;
        }
        if (lane == 31) sh.wsum[2][wid] = (unsigned)inc;
        __syncthreads();                                   // also: nobody reads the estimates any more
        int o = (int)__reduce_add_sync(kAll, lane < wid ? sh.wsum[2][lane] : 0u) + inc - __popc(fresh);
        int total = (int)__reduce_add_sync(kAll, lane < kWarps ? sh.wsum[2][lane] : 0u);
        for (unsigned m = fresh; m != 0; m &= m - 1) list[o++] = (unsigned short)(i0 + __ffs(m) - 1 + 4);
        if (CLUSTER && wid == 0) {
          const unsigned now = halo & ~halo_done;
          if (now >> lane & 1u)
            list[total + __popc(now & ((1u << lane) - 1u))] = (unsigned short)((lane < 4 ? lane - 4 : own + lane - 4) + 4);
          if (lane == 0) b.halo = (int)now;
        }
        // rows of the Q tile that TMA does not write
        if (R != MT * 128)
          for (int i = tid; i < q_bytes / 16; i += T) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (CLUSTER) total += __popc(b.halo);
        // ---- their votes, 128 keys at a time: as in the vote pass, key by key the same
        if (total > 0) {
          if (tid == 0) {
            const uint32_t bar = smem_u32(&b.q_full);
            mbar_expect_tx(bar, (uint32_t)(halves * R * 128));
            for (int hf = 0; hf < halves; ++hf)
              tma_load_4d(q_sh + hf * q_half, &L.tm_q, 64 * hf, shp.q_head_inner ? h * shp.G : 0, shp.q_head_inner ? 0 : h * shp.G, s, bar);
          }
          const int per_row = 8 * halves, NB = args.k_tiles, batch = NB * kTileKeys, n_batches = (total + batch - 1) / batch;
          const unsigned char* k_seg = static_cast<const unsigned char*>(a.k) + ((long long)(t0 + base - 4) * args.k_stride_tok + h * args.k_stride_head) * 2;
          auto load = [&](int i) {
            const int rows = min(total - i * batch, batch);
            for (int x = tid; x < rows * per_row; x += T) {
              const int r = halves == 2 ? x >> 4 : x >> 3, c = x & (per_row - 1);
              const unsigned char* src = k_seg + (long long)list[i * batch + r] * args.k_stride_tok * 2 + c * 16;
              const uint32_t dst = k_sh + (uint32_t)((r >> 7) * stage + (c >> 3) * kHalfBytes + (r & 127) * 128 + (((c & 7) ^ (r & 7)) << 4));
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            }
          };
          const float scale = shp.scale_log2;
          const int Rp = shp.Rp, units = NB * MT;          // unit: a tile's rows of one block
          load(0);
          bool ok = true;
          for (int i = 0; i < n_batches; ++i) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            const int tiles_here = (min(total - i * batch, batch) + kTileKeys - 1) / kTileKeys;
            if (tid == 0) {
              if (i == 0) ok = mbar_wait(smem_u32(&b.q_full), (uint32_t)n_q & 1u, &b.abort_flag);
              if (ok) {
                tc_fence_after();
                for (int x = 0; x < tiles_here * MT; ++x) {
                  const int kt = x / MT, mt = x - kt * MT;
                  const uint32_t idesc = instr_desc(kTileKeys, min(Rp - mt * 128, 128));
                  const uint64_t kd = smem_desc(k_sh + (uint32_t)(kt * stage)), qd = smem_desc(q_sh + (uint32_t)(mt * 128 * 128));
                  for (int ks = 0; ks < 4 * halves; ++ks)
                    tc_mma(tmem + (uint32_t)(x * 128), kd + (uint64_t)((ks >> 2) * (kHalfBytes >> 4) + (ks & 3) * 2),
                           qd + (uint64_t)((ks >> 2) * (q_half >> 4) + (ks & 3) * 2), idesc, ks > 0);
                }
                tc_commit(smem_u32(&b.mma_done));
              }
            }
            __syncwarp();
            ok = mbar_wait(smem_u32(&b.mma_done), (uint32_t)n_mma & 1u, &b.abort_flag);
            ok = __all_sync(kAll, ok);
            ++n_mma;
            float acc = 0.f;
            const int unit = wid >> 2, kt = unit / MT, mt = unit - kt * MT;
            if (ok) {
              if (i + 1 < n_batches) load(i + 1);          // the products have read the keys
              tc_fence_after();
              if (unit < units && kt < tiles_here) {
                acc = key_vote(tmem + ((uint32_t)((wid & 3) * 32) << 16) + (uint32_t)(unit * 128), min(Rp - mt * 128, 128), scale, smem_u32(b.lse + mt * 128));
                if (MT == 2 && mt == 0) b.half[kt][tid & 127] = acc;
              }
            }
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (b.abort_flag) break;                       // uniform: written before the barrier
            const int key = i * batch + kt * kTileKeys + (tid & 127);
            if (unit < units && mt == MT - 1 && key < min(total, (i + 1) * batch)) {
              if (MT == 2) acc += b.half[kt][tid & 127];
              const int place = (int)list[key] - 4;
              if (CLUSTER && (place < 0 || place >= own)) b.beside[place < 0 ? place + 4 : place - own + 4] = acc * inv_g;
              else __stcg(vote + base + place, acc * inv_g);
            }
          }
          asm volatile("cp.async.wait_all;" ::: "memory");
          if (tid == 0 && b.abort_flag) {                  // a load in flight, for a bounded time
            const unsigned long long w0 = now_ns();
            while (!mbar_try(smem_u32(&b.q_full), (uint32_t)n_q & 1u) && now_ns() - w0 < kWaitLimitNs) {}
          }
          ++n_q;
        }
        done = want;
        halo_done |= halo;
        // ---- the votes that are there, none elsewhere; pooled, and the k largest
        __syncthreads();
        clear_bins();
#pragma unroll
        for (int e = 0; e < IT; e += 4) *reinterpret_cast<float4*>(votes + tid * kPitch + e) = make_float4(0.f, 0.f, 0.f, 0.f);
        for (unsigned m = done; m != 0; m &= m - 1) {
          const int e = __ffs(m) - 1;
          votes[tid * kPitch + e] = __ldcg(vote + base + i0 + e);
        }
      }
      __syncthreads();
      // Outside the segment minus infinity, as in k_select_list: it differs from zero where votes are not finite.
      if (wid == 0 && lane < 11) {
        const int place = lane < 4 ? lane - 4 : (lane < 8 ? own + lane - 4 : lane - 8), p = base + place;
        if (p < 0 || p >= n) votes[at(place)] = -INFINITY;
        else if (!every && lane < 8) votes[at(place)] = CLUSTER && (halo_done >> lane & 1u) ? b.beside[lane] : 0.f;
      }
      __syncthreads();
      unsigned key[IT], tau;
      if (mine) pool_places<RAD>(votes + tid * kPitch, votes + at(i0 - 4), true, key);
      kept = select_places<T, IT, CLUSTER, 0>(sh, tid, key, valid, mine, reinterpret_cast<uint4*>(votes + tid * kPitch), n, k_keep, rank,
                                              CS, o_mine, tau);
      const float score = __uint_as_float(tau);
      if (bound <= 0.f || round > 0 || (bound < score && score > kTinyScore)) break;
      bound = score > kTinyScore ? score * 0.999f : 0.f;
      sync_all();
    }
    // the kept positions, in shared memory first; whole lines then go out
    int* const stage_idx = reinterpret_cast<int*>(smem);
    int o0 = 0, o1 = k_keep;                             // the CTA's rows among the segment's
    __syncthreads();
    if (CLUSTER) {
      if (tid == 0) sh.above = o_mine;
      if (tid == T - 1) sh.m = o_mine + __popc(kept);
      __syncthreads();
      o0 = sh.above;
      o1 = sh.m;
    }
    int* dst = stage_idx + (o_mine - o0);
    for (unsigned m = kept; m != 0; m &= m - 1) *dst++ = base + i0 + __ffs(m) - 1;
    __syncthreads();
    for (int i = o0 + tid; i < o1; i += T) put(out0 + i, stage_idx[i - o0]);
  }
  tc_fence_before();
  if (CLUSTER) cluster.sync(); else __syncthreads();     // nobody leaves while its shared memory may still be read
  if (b.abort_flag && tid == 0 && a.status) atomicExch(a.status, (int)SLKV_ERR_DEVICE_TIMEOUT);
  if (wid == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
  }
}

// ---- host side ----------------------------------------------------------------------------------------------------------
typedef void (*Kern)(const BoundArgs);
struct Variant {
  int items;
  Kern kern[kMaxRadius + 1];
};
#define SLKV_SEL(IT, C) \
  {IT, {k_select_bound<IT, 0, C>, k_select_bound<IT, 1, C>, k_select_bound<IT, 2, C>, k_select_bound<IT, 3, C>, k_select_bound<IT, 4, C>}}
const Variant kVariants[] = {SLKV_SEL(16, false), SLKV_SEL(32, false), SLKV_SEL(32, true)};
#undef SLKV_SEL

size_t select_bytes(const ScoreShape& sh, const Variant& v, int k_tiles) {
  const size_t product = (size_t)sh.halves * (sh.MT * 128 * 128 + k_tiles * kHalfBytes);
  const size_t votes = (size_t)vote_floats(kThreads, v.items) * sizeof(float);
  const size_t list = (size_t)(kThreads * v.items + 16) * sizeof(unsigned short);
  return product + list > votes ? product + list : votes;
}

thread_local int g_list_way = 0;

}  // namespace

void set_list_way(int way) { g_list_way = way; }

bool bound_possible(const Problem& pb) {
  if (pb.p.pool_mode != SLKV_POOL_MAX || !select_list_supported(pb) || pb.R <= 64) return false;
  return (int64_t)pb.n_seg * tensor_slot_stride(pb) * pb.R < (1ll << 31);                    // places of the weights: 32-bit
}
bool bound_shape(const Problem& pb) {
  if (!bound_possible(pb)) return false;
  const int64_t mean = pb.total_hist / pb.p.n_seqs;
  return mean >= 32000 || (pb.R > 128 ? mean >= 12000 && pb.n_tiles128 >= 3000 : mean >= 16000);
}

// Where the second product is worth more than the longer selection.  It saves some 3.5 ns for every product of 128 keys x 128 rows; the
// selection takes 50-90 us longer whatever the list's length, for 256 rows twice that.  With it come the segments that need all their votes
// (every_vote): both products, the second one from HBM.  The budgets are on the device, but what a layer keeps at most is known
// here.  Were its budgets even, the share of its segments that need all votes would be 0 or 1, were they as uneven as can be, up to
// `most`, here the mean over the layers.  Lists, us, two products / one, budgets lognormal with a standard deviation of 1.5:
//   128 rows  16384 tokens, 20 layers (20480 products): most 0.4 235 / 221, 0.6 259 / 282;  28 (28672): 0.4 323 / 289, 0.6 357 / 360
//             32768 tokens, 10 (20480): 0.3 227 / 233;  14 (28672): 0.3 310 / 272, 0.6 328 / 342;  16 (32768): 0.6 364 / 342, 0.75 375 / 371, 0.83 385 / 414
//             65536 tokens, 5 (20480): 0.4 231 / 228, 0.7 252 / 267;  8 (32768): 0.73 385 / 375, 0.82 400 / 417
//             131072 tokens, 8 (65520): 0.74 856 / 720, even 0.98 774 / 642, 1.00 809 / 867
//             four of 12000 to 24000, 4 (18016): 0.3 205 / 216;  5 (22520): 0.3 256 / 238, 0.74 277 / 277;  8 (36032): 0.74 435 / 426, 0.83 461 / 468
//   256 rows  33000 tokens, 5 (20640): 0.35 210 / 207;  7 (28896): 0.35 283 / 268, 0.7 293 / 304;  8 (33024): 0.54 318 / 301, 0.71 328 / 342
//             in clusters of two, 45000 tokens, 5 (28160): 0.27 281 / 249;  6 (33792): 0.73 342 / 341;  60000, 4 (30016): 0.4 295 / 305;  5 (37520): 0.4 361 / 328,
//             0.7 375 / 404;  48000 tokens, 8 (48000): 0.63 472 / 451, 0.95 510 / 526;  65536 tokens, 8 (65536): 0.81 659 / 650, 0.88 667 / 692
//             in clusters of four, 100000 tokens, 3 (37488): 0.25 363 / 377;  131072 tokens, 4 (65536): 611 / 521;  8 (131072): 0.67 1270 / 1261
//             eight of 16384 to 32768, 8 (98304): 0.87 2124 / 1820
//   64 rows   one sequence of 20000 tokens 428 / 446
// The line lies between the two; shapes differ by some 10 % about it, and a list on the wrong side loses that much.  48 models of 8 to 32 layers with
// lengths over the range and budgets lognormal or most of them in six heads: 0.58 to 1.04 of the time with two products, 0.87 to 1.07 of that with one
// wherever the lengths allow it.
bool bound_list_supported(const Problem& pb, const TailLayer* tail, int n_layers) {
  if (g_list_way != 0) return g_list_way == 1 && bound_possible(pb);
  if (!bound_shape(pb)) return false;
  const int64_t mean = pb.total_hist / pb.p.n_seqs;
  const int64_t line = mean / kEveryVoteShare > kEveryVoteCount ? mean / kEveryVoteShare : kEveryVoteCount;
  const int64_t window_rows = (int64_t)pb.p.n_kv_heads * (pb.total_tokens - pb.total_hist);
  // Room for every row says nothing of what is kept: few positions, which is what a cache is compressed for.
  const int64_t all_rows = (int64_t)pb.p.n_kv_heads * pb.total_tokens;
  double most = 0.0;
  for (int i = 0; i < n_layers; ++i) {
    const double share = tail[i].capacity >= all_rows ? 0.5 : (double)(tail[i].capacity - window_rows) / (double)(line * pb.n_seg);
    most += share < 1.0 ? (share > 0.0 ? share : 0.0) : 1.0;
  }
  most /= n_layers;
  const double products = (double)pb.n_tiles128 * n_layers * (pb.R > 128 ? 2 : 1);
  auto above = [&](double least, double at0, double slope, double steep) {
    const double x = at0 + slope * most;
    return products >= (x > least ? x : least) + (most > steep ? 24000 : 0);
  };
  if (pb.R <= 128) return most < 0.99 && above(13000, 6400, 30000, 0.78);
  const double clusters = pb.max_hist < 32764 ? 0.0 : 10000 * (pb.max_hist / 32764.0 - 1.0);        // beyond what one CTA holds
  return most < 0.96 && above(18000, 8500 + (clusters < 16000 ? clusters : 16000), 35000, 0.85);
}

cudaError_t launch_bound_list(const Problem& pb, const ScoreShape& sh, const ScoreLayer* lay, const TailLayer* tail, int n_layers,
                              cudaStream_t st, int* launches) {
  if (n_layers < 1 || n_layers > kListMaxLayers || sh.n_cta == 0) return cudaErrorInvalidValue;
  BoundArgs a;
  a.sh = sh;
  for (int i = 0; i < n_layers; ++i) { a.lay[i] = lay[i]; a.lay[i].budgets = tail[i].budgets; a.tail[i] = tail[i]; }
  a.k_stride_tok = pb.p.k_stride_tok;
  a.k_stride_head = pb.p.k_stride_head;
  // One CTA per segment wherever it can hold the segment: in a cluster of four with 512 threads each the two searches for a k-th
  // largest took 10 and 16 us instead of 3 and 8.
  const int cs = select_list_cluster(pb);
  const int slice = ((pb.max_hist + 3 + cs - 1) / cs + 3) & ~3;
  const Variant& var = kVariants[cs > 1 ? 2 : slice <= 16384 ? 0 : 1];
  constexpr size_t kStatic = sizeof(SelShared) + sizeof(BoundShared) + 1024;
  // two tiles of keys at a time where shared memory holds them
  a.k_tiles = select_bytes(sh, var, 2) <= kSmemLimit - kStatic ? 2 : 1;
  a.n_layers = n_layers;
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    for (const Variant& v : kVariants)
      for (Kern k : v.kern) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmemLimit - kStatic));
        if (e != cudaSuccess) return e;
      }
    configured_dev = dev;
  }
  e = launch_score_list(sh, a.lay, n_layers, kScoreBound, pb.sync, st, launches);
  if (e != cudaSuccess) return e;
  LaunchScope scope(KID_SELECT, st, launches);
  return launch_pdl(var.kern[pb.p.pool_kernel >> 1], dim3((unsigned)(pb.n_seg * cs), (unsigned)n_layers), dim3(kThreads),
                    select_bytes(sh, var, a.k_tiles), st, cs, a);
}

}  // namespace slkv

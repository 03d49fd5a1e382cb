// Context-parallel selection (Sec. 3.4, Eq. 8; Algorithm 3 with one sequence's history keys split over ranks).
//
// Each rank holds a contiguous range of the history keys (plus pool_kernel / 2 rows of its neighbours' on each side, so
// that pooling needs nothing from them) and scores it with the ordinary score kernels against row log-sum-exps merged
// over all ranks.  What is left is one top-k per KV head over scores that live on different ranks: a radix descent over
// the scores' bit patterns (11 + 11 + 10 bits) whose histograms are summed across ranks between the levels, the ties at
// the threshold handed out in rank order (lower positions first, as on one GPU), then every rank packs the rows it owns.
// Integer counters only: the kept set does not depend on timing or on the number of ranks.
#include "slkv_internal.cuh"

namespace slkv {
namespace {

constexpr int kCpThreads = 1024;
constexpr int kCpItems = 4;                 // consecutive positions per thread of k_cp_emit
constexpr int kCpSlice = kCpThreads * kCpItems;       // positions counted, and packed, together
constexpr int kCpStepThreads = 256;
static_assert(kCpSlice == kCpStepThreads * 16 && kCpBins == kCpStepThreads * 8, "k_cp_step's shares of a thread");

__device__ __forceinline__ unsigned cp_digit(unsigned bits, int level) {
  return level == 0 ? bits >> 21 : (level == 1 ? (bits >> 10) & 2047u : bits & 1023u);
}
__device__ __forceinline__ bool cp_match(unsigned bits, unsigned prefix, int level) {
  return level == 0 || (level == 1 ? (bits >> 21) == (prefix >> 21) : (bits >> 10) == (prefix >> 10));
}

// lse_out[i] = log-sum-exp over the parts of lse_parts[r][i], all in the units `to_log2` converts to base 2.
__global__ void k_cp_merge_lse(const float* __restrict__ parts, int n_parts, long long n, float to_log2,
                               float* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float m = -INFINITY;
  for (int r = 0; r < n_parts; ++r) m = fmaxf(m, parts[(long long)r * n + i] * to_log2);
  if (!(m > -INFINITY)) { out[i] = -INFINITY; return; }       // no rank has a key for this row
  float z = 0.f;
  for (int r = 0; r < n_parts; ++r) z += exp2f(parts[(long long)r * n + i] * to_log2 - m);
  out[i] = (m + log2f(z)) / to_log2;
}

// One step of the descent, with everything between two exchanges in one launch: per head
//   start   from the budgets (level 0: need = the history rows the head keeps of the whole sequence, Algorithm 3 l.1-3,
//           l.7; no prefix yet), or from a state, or from a state taken one level down on the histogram summed over all
//           ranks: the digit d with count(digits > d) < need <= count(digits >= d) joins the prefix, need drops by the
//           count above it (d = 0 if the counts above it never reach need; need == 0: the prefix becomes all ones --
//           nothing lies above it -- and stays);
//   count   the own positions by their digit of the next level, hist[h][d] += those whose bits agree with the prefix
//           above it; or, with the threshold complete, by slice those above it and those equal to it, and their totals;
//   clear   a share of the output buffers, by CTAs behind those that count.
// Every CTA of a head repeats the start: 8 KB of bins from L2, less than a launch of its own (2.6 us).  The clearing is
// what the memory is free for meanwhile: scores of 32k positions and 8 heads are 1 MB, the rows to clear 134 MB.
// Streaming stores: plain ones leave L2 full of zeros to be written back under the next layer's loads of K (111 -> 106 us
// per layer of 32k positions).
// A thread takes 16 consecutive positions and adds a run of equal digits at once: pooled scores come in runs (a
// maximum holds for pool_kernel positions), and neighbouring threads adding to the same bin one by one serialise.
__global__ void __launch_bounds__(kCpStepThreads) k_cp_step(const __grid_constant__ CpStep a) {
  __shared__ int sh[kCpBins];
  __shared__ long long wtot[8];
  __shared__ unsigned sh_prefix;
  __shared__ int sh_need;
  pdl_launch_dependents();
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int n_work = a.n_kv_heads * a.ctas_per_head;
  if ((int)blockIdx.x >= n_work) {
    pdl_wait();
    const long long n16 = a.clear_bytes >> 4, step = (long long)(gridDim.x - n_work) * kCpStepThreads;
    uint4* dst = static_cast<uint4*>(a.clear);
#pragma unroll 4
    for (long long i = (long long)(blockIdx.x - n_work) * kCpStepThreads + t; i < n16; i += step)
      __stcs(dst + i, make_uint4(0u, 0u, 0u, 0u));
    return;
  }
  const int h = blockIdx.x / a.ctas_per_head, part = blockIdx.x - h * a.ctas_per_head;
  if (a.hist)
    for (int b = t; b < kCpBins; b += kCpStepThreads) sh[b] = 0;
  pdl_wait();

  unsigned prefix;
  int need;
  if (a.budgets) {
    const long long kept = min(a.seq_len, max((long long)a.budgets[h], (long long)a.window));
    prefix = 0u;
    need = (int)(kept - min(a.seq_len, (long long)a.window));
  } else {
    prefix = a.prefix_in[h];
    need = a.need_in ? a.need_in[h] : 0;
  }
  if (a.hist_sum && need <= 0) {
    prefix = 0xffffffffu;
    need = 0;
  } else if (a.hist_sum) {
    const int from = a.level_in, bins = from == 2 ? 1024 : kCpBins;
    const int shift = from == 0 ? 21 : (from == 1 ? 10 : 0);
    // thread t holds the 8 digits from bins - 1 - 8 t downwards; digit 0 is where the search ends anyway
    int c[8];
    long long s = 0;
    const int top = bins - 1 - 8 * t;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      c[q] = top - q >= 1 ? a.hist_sum[h * kCpBins + top - q] : 0;
      s += c[q];
    }
    long long inc = s;
    for (int o = 1; o < 32; o <<= 1) {
      const long long n = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += n;
    }
    if (lane == 31) wtot[wid] = inc;
    __syncthreads();
    long long above = inc - s, total = 0;
    for (int w2 = 0; w2 < 8; ++w2) {
      if (w2 < wid) above += wtot[w2];
      total += wtot[w2];
    }
    if (t == 0 && total < need) {                        // the counts above digit 0 do not reach need: digit 0
      sh_prefix = prefix;
      sh_need = (int)(need - total);
    }
    if (above < need && above + s >= need) {             // the digit lies among this thread's eight
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (above + c[q] >= need) {
          sh_prefix = prefix | (unsigned)(top - q) << shift;
          sh_need = (int)(need - above);
          break;
        }
        above += c[q];
      }
    }
    __syncthreads();
    prefix = sh_prefix;
    need = sh_need;
  }
  if (part == 0 && t == 0 && a.prefix_out) {             // in place only with one CTA per head
    a.prefix_out[h] = prefix;
    a.need_out[h] = need;
  }
  if (!a.hist && !a.cnt_gt) return;

  __syncthreads();                                       // sh cleared
  const unsigned* row = reinterpret_cast<const unsigned*>(a.pooled + (long long)h * a.row_stride + a.own_begin);
  const int level = a.level_out;
  for (int blk = part; blk < a.n_blk; blk += a.ctas_per_head) {
    const long long j0 = (long long)blk * kCpSlice + t * 16;
    unsigned bits[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) bits[q] = j0 + q < a.own_count ? row[j0 + q] : 0u;
    if (a.hist) {
      int run_digit = -1, run = 0;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int dg = j0 + q < a.own_count && cp_match(bits[q], prefix, level) ? (int)cp_digit(bits[q], level) : -1;
        if (dg != run_digit) {
          if (run_digit >= 0) atomicAdd(&sh[run_digit], run);
          run_digit = dg; run = 0;
        }
        ++run;
      }
      if (run_digit >= 0) atomicAdd(&sh[run_digit], run);
    } else {
      unsigned n = 0;                                    // equal ones in the high half, those above in the low half
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (j0 + q < a.own_count) n += (bits[q] > prefix ? 1u : 0u) + (bits[q] == prefix ? 65536u : 0u);
      n = __reduce_add_sync(0xffffffffu, n);
      __syncthreads();
      if (lane == 0) sh[wid] = (int)n;
      __syncthreads();
      if (t == 0) {
        unsigned all = 0;
        for (int w2 = 0; w2 < 8; ++w2) all += (unsigned)sh[w2];
        const int gt = (int)(all & 65535u), eq = (int)(all >> 16);
        a.cnt_gt[h * a.n_blk + blk] = gt;
        a.cnt_eq[h * a.n_blk + blk] = eq;
        if (gt) atomicAdd(&a.tot_gt[h], gt);
        if (eq) atomicAdd(&a.tot_eq[h], eq);
      }
    }
  }
  if (!a.hist) return;
  __syncthreads();
  for (int b = t; b < kCpBins; b += kCpStepThreads)
    if (sh[b]) atomicAdd(&a.hist[h * kCpBins + b], sh[b]);
}

// ties[h] = this rank's positions whose score equals the threshold = its last-level histogram at the threshold's digit.
__global__ void k_cp_local_ties(const int32_t* __restrict__ hist_local, const unsigned* __restrict__ prefix,
                                int n_kv_heads, int32_t* __restrict__ ties) {
  pdl_launch_dependents();
  pdl_wait();
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= n_kv_heads) return;
  ties[h] = prefix[h] == 0xffffffffu ? 0 : hist_local[h * kCpBins + (prefix[h] & 1023u)];
}

// Packs slice blk of head h's kept positions in ascending order: kept_idx = position in the whole sequence,
// gather_src = row of this rank's K / V (token * n_kv_heads + head); slice 0 also writes the window rows on the rank
// that holds them, and the head's offset.  A head takes of its ties what the ranks before this one have left of need,
// within [0, own ties]; its rows = scores above the threshold + ties taken + window rows.  A kept position's packed row
// = the rows of the heads before + (scores above the threshold before it) + min(ties before it, ties taken).
// Every CTA adds up the heads' rows and its own head's slices by itself: a few hundred counters from L2 instead of a
// launch between the counting and the packing (5 us in a single CTA).
__global__ void __launch_bounds__(kCpThreads) k_cp_emit(const __grid_constant__ CpEmit a) {
  __shared__ unsigned wtot[kCpThreads / 32];
  __shared__ int red[kCpThreads / 32][4];
  pdl_launch_dependents();
  pdl_wait();
  const int h = blockIdx.y, blk = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  auto take_of = [&](int g) {
    long long t = a.need[g];
    for (int r = 0; r < a.part; ++r) t -= a.ties_all[(long long)r * a.n_kv_heads + g];
    const int own = a.tot_eq[g];
    return t < 0 ? 0 : (t > own ? own : (int)t);
  };
  const unsigned tau = a.threshold[h];
  const int tk = take_of(h), rows_h = a.tot_gt[h] + tk + a.window_rows;
  const unsigned* row = reinterpret_cast<const unsigned*>(a.pooled + (long long)h * a.row_stride + a.own_begin);
  const long long first = (long long)blk * kCpSlice + tid * kCpItems;
  unsigned bits[kCpItems];
  unsigned packed = 0;                           // ties in the high half, scores above the threshold in the low half
#pragma unroll
  for (int q = 0; q < kCpItems; ++q) {
    bits[q] = first + q < a.own_count ? row[first + q] : 0u;
    if (first + q < a.own_count) packed += (bits[q] > tau ? 1u : 0u) + (bits[q] == tau ? 65536u : 0u);
  }
  int before = 0, all = 0, gt0 = 0, eq0 = 0;     // rows of the heads before h, of all; the head's counts before the slice
  for (int g = tid; g < a.n_kv_heads; g += kCpThreads) {
    const int r = a.tot_gt[g] + take_of(g) + a.window_rows;
    all += r;
    if (g < h) before += r;
  }
  for (int b = tid; b < blk; b += kCpThreads) {
    gt0 += a.cnt_gt[h * a.n_blk + b];
    eq0 += a.cnt_eq[h * a.n_blk + b];
  }
  before = __reduce_add_sync(0xffffffffu, before);
  all = __reduce_add_sync(0xffffffffu, all);
  gt0 = __reduce_add_sync(0xffffffffu, gt0);
  eq0 = __reduce_add_sync(0xffffffffu, eq0);
  unsigned inc = packed;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) wtot[wid] = inc;
  if (lane == 0) { red[wid][0] = before; red[wid][1] = all; red[wid][2] = gt0; red[wid][3] = eq0; }
  __syncthreads();
  if (wid == 0) {
    unsigned w = wtot[lane], winc = w;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += n;
    }
    wtot[lane] = winc - w;                       // exclusive over the warps
  } else if (wid <= 4) {
    const int v = __reduce_add_sync(0xffffffffu, red[lane][wid - 1]);
    if (lane == 0) red[0][wid - 1] = v;          // the only warp that reads or writes this column
  }
  __syncthreads();
  const long long out0 = red[0][0], total = red[0][1];
  const unsigned excl = wtot[wid] + inc - packed;
  unsigned gb = (unsigned)red[0][2] + (excl & 65535u), eb = (unsigned)red[0][3] + (excl >> 16);
#pragma unroll
  for (int q = 0; q < kCpItems; ++q) {
    if (first + q >= a.own_count) break;
    const bool gt = bits[q] > tau, eq = bits[q] == tau;
    if (gt || (eq && (int)eb < tk)) {
      const long long o = out0 + gb + min(eb, (unsigned)tk);
      if (o < a.capacity) {
        a.kept_idx[o] = (int32_t)(a.pos0 + first + q);
        a.gather_src[o] = (int32_t)((a.own_begin + first + q) * a.n_kv_heads + h);
      }
    }
    gb += gt;
    eb += eq;
  }
  // window rows (Algorithm 3 l.4, l.10): always kept, behind the history rows, on the rank that holds them
  if (blk == 0) {
    const long long w0 = out0 + rows_h - a.window_rows;
    for (int i = tid; i < a.window_rows; i += kCpThreads)
      if (w0 + i < a.capacity) {
        a.kept_idx[w0 + i] = (int32_t)(a.window_pos0 + i);
        a.gather_src[w0 + i] = (int32_t)((a.window_row0 + i) * a.n_kv_heads + h);
      }
    if (tid == 0) {
      a.offsets[h] = (int32_t)out0;
      if (h == 0) {
        a.offsets[a.n_kv_heads] = (int32_t)total;
        if (total > a.capacity && a.status) atomicCAS(a.status, 0, (int)SLKV_ERR_CAPACITY);
      }
    }
  }
  if (a.fill_tail)                               // positions of the rows nobody fills: -1
    for (long long o = total + ((long long)h * gridDim.x + blk) * kCpThreads + tid; o < a.capacity;
         o += (long long)gridDim.x * gridDim.y * kCpThreads)
      a.kept_idx[o] = -1;
}

}  // namespace

cudaError_t launch_cp_merge_lse(const float* parts, int n_parts, long long n, float to_log2, float* out,
                                cudaStream_t st, int* launches) {
  LaunchScope scope(KID_CP, st, launches);
  return launch_pdl(k_cp_merge_lse, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, 1, parts, n_parts, n, to_log2, out);
}

cudaError_t launch_cp_step(CpStep a, cudaStream_t st, int* launches) {
  a.n_blk = cp_slices(a.own_count);
  // up to 64 CTAs per head to count: they repeat the start, and each adds its bins to the head's
  a.ctas_per_head = a.hist || a.cnt_gt ? (a.hist && a.n_blk > 64 ? 64 : a.n_blk) : 1;
  if (a.clear_bytes <= 0) a.clear_bytes = 0;
  const long long want = (a.clear_bytes + kCpStepThreads * 64 - 1) / (kCpStepThreads * 64);     // 4 stores per thread
  const int most = sm_count() * 4;                       // with the counting CTAs resident at once
  const unsigned n_clear = (unsigned)(want < most ? want : most);
  LaunchScope scope(KID_CP, st, launches);
  return launch_pdl(k_cp_step, dim3((unsigned)a.n_kv_heads * a.ctas_per_head + n_clear), dim3(kCpStepThreads), 0, st, 1, a);
}

cudaError_t launch_cp_local_ties(const int32_t* hist_local, const unsigned* prefix, int n_kv_heads, int32_t* ties,
                                 cudaStream_t st, int* launches) {
  LaunchScope scope(KID_CP, st, launches);
  return launch_pdl(k_cp_local_ties, dim3((n_kv_heads + 127) / 128), dim3(128), 0, st, 1, hist_local, prefix,
                    n_kv_heads, ties);
}

int cp_slices(int own_count) { return own_count > 0 ? (own_count + kCpSlice - 1) / kCpSlice : 1; }

cudaError_t launch_cp_emit(CpEmit a, cudaStream_t st, int* launches) {
  a.n_blk = cp_slices(a.own_count);
  LaunchScope scope(KID_CP, st, launches);
  return launch_pdl(k_cp_emit, dim3(a.n_blk, a.n_kv_heads), dim3(kCpThreads), 0, st, 1, a);
}

}  // namespace slkv

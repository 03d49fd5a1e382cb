// Sequence tables, pooling, per-head variable-k selection and the packed K/V gather
// (Sec. 3.4, Eq. 8; Algorithm 3 lines 1-4 and 7-10).
#include "slkv_internal.cuh"

namespace slkv {
namespace {

constexpr int kScanThreads = 1024;

// Exclusive scan of one value per thread across the CTA; returns the exclusive prefix, *total = CTA sum.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* warp_tot /*[32]*/, T* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    T n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  __syncthreads();                       // warp_tot may still be read from a previous call
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  T base = 0, tot = 0;
  for (int w = 0; w < nw; ++w) {
    T t = warp_tot[w];
    if (w < wid) base += t;
    tot += t;
  }
  *total = tot;
  return base + inc - v;
}

__device__ __forceinline__ int kept_rows(int len, int budget, int window) {
  // Algorithm 3 l.1-3 (keep all when the length fits the budget) and the always-kept window
  return min(len, max(budget, window));
}

// hist_off[s] = sum_{s'<s} max(len_s' - w, 0); with budgets: offsets[seg] = packed row where segment
// seg = s*Hkv + h starts.
__global__ void __launch_bounds__(kScanThreads, 1)
k_setup(const int32_t* __restrict__ cu, int n_seqs, int n_kv_heads, int window, const int32_t* __restrict__ budgets,
        int64_t* __restrict__ hist_off, int32_t* __restrict__ tile_off, int32_t* __restrict__ offsets,
        long long capacity, int32_t* __restrict__ status) {
  __shared__ long long wt[32];
  const int tid = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  long long run = 0, run_tiles = 0;
  for (int s0 = 0; s0 < n_seqs; s0 += kScanThreads) {
    int s = s0 + tid;
    long long nh = 0;
    if (s < n_seqs) nh = max(cu[s + 1] - cu[s] - window, 0);
    long long tot, ex = block_excl_scan<long long>(nh, wt, &tot);
    if (s < n_seqs) hist_off[s] = run + ex;
    run += tot;
    ex = block_excl_scan<long long>((nh + 127) >> 7, wt, &tot);     // 128-key tiles of the tensor-core path
    if (s < n_seqs) tile_off[s] = (int32_t)(run_tiles + ex);
    run_tiles += tot;
  }
  if (tid == 0) { hist_off[n_seqs] = run; tile_off[n_seqs] = (int32_t)run_tiles; }
  if (budgets == nullptr) return;
  const int n_seg = n_seqs * n_kv_heads;
  run = 0;
  for (int g0 = 0; g0 < n_seg; g0 += kScanThreads) {
    int seg = g0 + tid;
    long long kept = 0;
    if (seg < n_seg) {
      int s = seg / n_kv_heads, h = seg - s * n_kv_heads;
      kept = kept_rows(cu[s + 1] - cu[s], budgets[h], window);
    }
    long long tot, ex = block_excl_scan<long long>(kept, wt, &tot);
    if (seg < n_seg) offsets[seg] = (int32_t)(run + ex);
    run += tot;
  }
  if (tid == 0) {
    offsets[n_seg] = (int32_t)run;
    if (run > capacity && status) *status = SLKV_ERR_CAPACITY;
  }
}

// pooled[j] = max (or zero-padded mean) of vote[j-r .. j+r] inside the segment's history.
__global__ void __launch_bounds__(256)
k_pool(const float* __restrict__ vote, float* __restrict__ pooled, const __grid_constant__ SeqTables tab,
       int n_kv_heads, int window, int pool_kernel, int pool_mode) {
  pdl_launch_dependents();
  pdl_wait();
  const int s = blockIdx.z, h = blockIdx.y;
  const int n_hist = max(tab.cu_at(s + 1) - tab.cu_at(s) - window, 0);
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_hist) return;
  const long long base = tab.hist_at(s) * n_kv_heads + (long long)h * n_hist;
  const float* src = vote + base;
  const int r = pool_kernel >> 1;
  const int lo = max(j - r, 0), hi = min(j + r, n_hist - 1);
  float acc;
  if (pool_mode == SLKV_POOL_MAX) {
    acc = src[lo];
    for (int t = lo + 1; t <= hi; ++t) acc = fmaxf(acc, src[t]);
  } else {
    acc = 0.f;
    for (int t = lo; t <= hi; ++t) acc += src[t];
    acc = acc / (float)pool_kernel;
  }
  pooled[base + j] = acc;
}

// One CTA per segment.  Finds the k-th largest pooled score by a 4 x 8-bit radix descent over the
// float bit patterns (scores are >= 0, so unsigned order = float order), then writes the positions of
// the k best in ascending order (equal scores: lower position first) followed by the window positions.
__global__ void __launch_bounds__(kScanThreads, 1)
k_select(const float* __restrict__ pooled, const __grid_constant__ SeqTables tab,
         const int32_t* __restrict__ budgets, const int32_t* __restrict__ offsets, int32_t* __restrict__ kept_idx,
         int32_t* __restrict__ gather_src, int n_kv_heads, int window, long long capacity) {
  __shared__ int hist[256];
  __shared__ int wt[32];
  __shared__ unsigned sh_prefix;
  __shared__ int sh_need;
  const int tid = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  const int seg = blockIdx.x;
  const int s = seg / n_kv_heads, h = seg - s * n_kv_heads;
  const int len = tab.cu_at(s + 1) - tab.cu_at(s);
  const int n_hist = max(len - window, 0);
  const int n_win = min(len, window);
  const int k = kept_rows(len, budgets[h], window) - n_win;      // history rows to keep (C_H = C - window)
  const long long out0 = offsets[seg];
  const int src_base = tab.cu_at(s) * n_kv_heads + h;           // source row of position j: src_base + j * n_kv_heads
  const unsigned* src = reinterpret_cast<const unsigned*>(pooled + tab.hist_at(s) * n_kv_heads + (long long)h * n_hist);

  // window rows (Algorithm 3 l.4, l.10): always kept, appended after the history rows
  for (int t = tid; t < n_win; t += kScanThreads) {
    long long o = out0 + k + t;
    if (o < capacity) {
      kept_idx[o] = len - n_win + t;
      gather_src[o] = src_base + (len - n_win + t) * n_kv_heads;
    }
  }
  if (k <= 0) return;
  if (k >= n_hist) {                                             // nothing to drop
    for (int j = tid; j < n_hist; j += kScanThreads)
      if (out0 + j < capacity) {
        kept_idx[out0 + j] = j;
        gather_src[out0 + j] = src_base + j * n_kv_heads;
      }
    return;
  }

  unsigned prefix = 0, mask = 0;
  int need = k;
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (int j = tid; j < n_hist; j += kScanThreads) {
      unsigned v = src[j];
      if ((v & mask) == prefix) atomicAdd(&hist[(v >> shift) & 255u], 1);
    }
    __syncthreads();
    if (tid == 0) {
      int cum = 0, b = 255;
      for (; b > 0; --b) {
        int c = hist[b];
        if (cum + c >= need) break;
        cum += c;
      }
      sh_prefix = prefix | ((unsigned)b << shift);
      sh_need = need - cum;
    }
    __syncthreads();
    prefix = sh_prefix;
    need = sh_need;
    mask |= 255u << shift;
    __syncthreads();
  }
  const unsigned tau = prefix;      // k-th largest value; `need` of the elements equal to it are kept

  int gt_seen = 0, eq_seen = 0;
  for (int j0 = 0; j0 < n_hist; j0 += kScanThreads) {
    const int j = j0 + tid;
    unsigned v = (j < n_hist) ? src[j] : 0u;
    const int gt = (j < n_hist) && (v > tau);
    const int eq = (j < n_hist) && (v == tau);
    int tot, ex = block_excl_scan<int>(gt | (eq << 16), wt, &tot);
    const int gt_before = gt_seen + (ex & 0xffff), eq_before = eq_seen + (ex >> 16);
    if (gt || (eq && eq_before < need)) {
      long long o = out0 + gt_before + min(eq_before, need);
      if (o < capacity) {
        kept_idx[o] = j;
        gather_src[o] = src_base + j * n_kv_heads;
      }
    }
    gt_seen += tot & 0xffff;
    eq_seen += tot >> 16;
  }
}

// Copies the kept rows of K and V of a list of layers into the packed caches: 16 bytes per lane, a row per lane group, two
// rows of K and of V in flight per group.  The selection left the source row (token * n_kv_heads + head) of every packed row
// in gather_src.  What bounds it: HBM, where there are enough rows.  The rows of all layers are one flat list of chunks that
// the CTAs share evenly, however skewed the layers' row counts are (16 layers of which one keeps most rows, 130k in all:
// 145 us with an equal number of CTAs per layer, 60 now).
constexpr int kGatherThreads = 256;
struct GatherArgs {
  int n_seg, n_kv_heads, row_bytes, n_layers;
  long long k_tok_bytes, k_head_bytes, v_tok_bytes, v_head_bytes, all_rows;
  TailLayer lay[kListMaxLayers];
};
__global__ void __launch_bounds__(kGatherThreads)
k_gather(const __grid_constant__ GatherArgs g) {
  __shared__ int chunks_up_to[32];                          // of layers 0 .. l
  __shared__ long long rows_of[32];
  pdl_launch_dependents();
  const int tid = threadIdx.x, wlane = tid & 31;
  const int lanes = g.row_bytes >> 4;                       // 16-byte lanes per row (power of two <= 32)
  const int rows_per_cta = kGatherThreads / lanes, chunk_rows = 2 * rows_per_cta;
  const int lane = tid % lanes, sub = tid / lanes;
  pdl_wait();
  if (g.n_layers > 1 && tid < 32) {
    long long n_rows = 0;
    if (tid < g.n_layers) n_rows = min((long long)g.lay[tid].offsets[g.n_seg], min(g.lay[tid].capacity, g.all_rows));
    int inc = (int)((n_rows + chunk_rows - 1) / chunk_rows);
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, inc, o);
      if (tid >= o) inc += x;
    }
    chunks_up_to[tid] = inc;
    rows_of[tid] = n_rows;
  }
  if (g.n_layers > 1) __syncthreads();
  const long long rows0 = g.n_layers > 1 ? 0 : min((long long)g.lay[0].offsets[g.n_seg], min(g.lay[0].capacity, g.all_rows));
  if (blockIdx.x == 0 && g.lay[0].offsets_copy)
    for (int i = tid; i <= g.n_seg; i += kGatherThreads) g.lay[0].offsets_copy[i] = g.lay[0].offsets[i];
  const int up_to = g.n_layers > 1 ? chunks_up_to[wlane] : 0x7fffffff;
  const int total = g.n_layers > 1 ? chunks_up_to[31] : (int)((rows0 + chunk_rows - 1) / chunk_rows);
  for (int c = blockIdx.x; c < total; c += gridDim.x) {
    const int l = __popc(__ballot_sync(0xffffffffu, up_to <= c));            // the layer the chunk lies in
    const TailLayer& a = g.lay[l];
    const int c0 = c - (l > 0 ? chunks_up_to[l - 1] : 0);
    const long long n_rows = g.n_layers > 1 ? rows_of[l] : rows0, r0 = (long long)c0 * chunk_rows + sub;
    uint4 kv[2], vv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long r = r0 + u * rows_per_cta;
      if (r >= n_rows) continue;
      const int src = a.gather_src[r];
      if (a.kept_copy && lane == 0) a.kept_copy[r] = a.kept_idx[r];
      const int tok = src / g.n_kv_heads, h = src - tok * g.n_kv_heads;
      kv[u] = *reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(a.k) + tok * g.k_tok_bytes + h * g.k_head_bytes + lane * 16);
      vv[u] = *reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(a.v) + tok * g.v_tok_bytes + h * g.v_head_bytes + lane * 16);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long r = r0 + u * rows_per_cta;
      if (r >= n_rows) continue;
      *reinterpret_cast<uint4*>(static_cast<unsigned char*>(a.k_out) + r * g.row_bytes + lane * 16) = kv[u];
      *reinterpret_cast<uint4*>(static_cast<unsigned char*>(a.v_out) + r * g.row_bytes + lane * 16) = vv[u];
    }
  }
}

}  // namespace

cudaError_t launch_setup(const Problem& pb, const int32_t* budgets, int32_t* offsets, int64_t capacity,
                         int32_t* status, cudaStream_t st, int* launches) {
  LaunchScope scope(KID_SETUP, st, launches);
  return launch_pdl(k_setup, dim3(1), dim3(kScanThreads), 0, st, 1, pb.cu, pb.p.n_seqs, pb.p.n_kv_heads,
                    pb.p.window, budgets, pb.hist_off, pb.tile_off, offsets, (long long)capacity, status);
}

cudaError_t launch_pool(const Problem& pb, float* pooled, cudaStream_t st, int* launches) {
  if (pb.max_hist <= 0) return cudaSuccess;
  dim3 grid((pb.max_hist + 255) / 256, pb.p.n_kv_heads, pb.p.n_seqs);
  LaunchScope scope(KID_POOL, st, launches);
  return launch_pdl(k_pool, grid, dim3(256), 0, st, 1, (const float*)pb.vote, pooled, pb.tab, pb.p.n_kv_heads,
                    pb.p.window, pb.p.pool_kernel, pb.p.pool_mode);
}

cudaError_t launch_select(const Problem& pb, const float* pooled, const int32_t* budgets, const int32_t* offsets,
                          int32_t* kept_idx, int64_t capacity, cudaStream_t st, int* launches) {
  LaunchScope scope(KID_SELECT, st, launches);
  return launch_pdl(k_select, dim3(pb.n_seg), dim3(kScanThreads), 0, st, 1, pooled, pb.tab, budgets, offsets,
                    kept_idx, pb.gather_src, pb.p.n_kv_heads, pb.p.window, (long long)capacity);
}

cudaError_t launch_gather(const Problem& pb, const TailLayer* lay, int n_layers, cudaStream_t st, int* launches) {
  GatherArgs g;
  g.n_seg = pb.n_seg; g.n_kv_heads = pb.p.n_kv_heads;
  g.row_bytes = pb.p.head_dim * pb.elem;
  g.k_tok_bytes = pb.p.k_stride_tok * pb.elem; g.k_head_bytes = pb.p.k_stride_head * pb.elem;
  g.v_tok_bytes = pb.p.v_stride_tok * pb.elem; g.v_head_bytes = pb.p.v_stride_head * pb.elem;
  g.all_rows = (long long)pb.p.n_kv_heads * pb.total_tokens;
  g.n_layers = n_layers;
  const int chunk_rows = 2 * kGatherThreads / (g.row_bytes >> 4);
  long long chunks = 0;
  for (int i = 0; i < n_layers; ++i) {
    g.lay[i] = lay[i];
    const long long m = lay[i].capacity < g.all_rows ? lay[i].capacity : g.all_rows;
    chunks += (m + chunk_rows - 1) / chunk_rows;
  }
  if (chunks <= 0) return cudaSuccess;
  const int most = sm_count() * 6;                          // resident at a time
  LaunchScope scope(KID_GATHER, st, launches);
  return launch_pdl(k_gather, dim3((unsigned)(chunks < most ? chunks : most)), dim3(kGatherThreads), 0, st, 1, g);
}

}  // namespace slkv

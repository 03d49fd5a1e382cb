// Host side of the tensor-core score kernel (Sec. 3.4, Eq. 7; Algorithm 3 l.6; Eq. 3-4): tensor maps, the split of a
// layer's key tiles into groups and over CTAs, and the kernel that turns the row statistics into log-sum-exps for
// slkv_row_lse.
#include <cuda.h>

#include <atomic>

#include "slkv_internal.cuh"
#include "slkv_tc_device.cuh"

namespace slkv {
namespace {

constexpr int kMergeThreads = 256;
// Keys per group of a two-pass launch, in bytes: 1024 tiles at head_dim 128, 2048 at 64.  At 32 MB the vote pass finds its
// keys in L2, given that it lets them go itself: 68 MB from HBM per layer of 32k tokens and 8 heads instead of 134, and HBM
// reads are what the part's power goes into (a 32 KB tile costs 4.9 uJ from HBM, 1.3 from L2; its MMAs 3.3, its exponentials
// 1.9).  A phase costs a CTA about 1.2 us beside its tiles, so smaller groups lose more than they save.  Steps of 32 layers
// (16 for the last two), held, us:
//   head_dim 128, 128 rows            16 MB   24 MB   32 MB   48 MB   64 MB
//     4001 tokens                       154     144     136     138     137
//     32768 tokens                     1059     960     866     952     931
//     8 x 4k-32k tokens, 256 rows      3631    3437    3394    3480    3538
//     131072 tokens, 256 rows          2940    2945    2950    3025    3088
//   head_dim 64, 128 rows                      16 MB   24 MB   32 MB   40 MB
//     8192 tokens                               195     187     184     183
//     32768 tokens                              663     641     644     644
//     8 x 4k-32k tokens, 256 rows              2605    2572    2561    2554
//     131072 tokens, 256 rows                  2257    2226    2223    2282
constexpr long long kGroupBytes = 32ll << 20;

// The rows' log-sum-exps from the statistics of a launch over one layer: lse_out[s][h][i], in the units out_scale converts
// to, or (null) the layer's own array, which a vote pass reads.
__global__ void __launch_bounds__(kMergeThreads)
k_merge_lse_tensor(const __grid_constant__ ScoreShape a, void* part, const LseSource lse, float* __restrict__ lse_out,
                   float out_scale) {
  pdl_launch_dependents();
  pdl_wait();
  const int seg = blockIdx.x, s = seg / a.n_kv_heads, g = seg - s * a.n_kv_heads;
  const int n_hist = a.tab.cu_at(s + 1) - a.tab.cu_at(s) - a.window;
  if (n_hist <= 0) return;
  const StatView st = stat_view(part, a.n_seqs * a.n_kv_heads, a.R, a.slot_stride);
  bool any_far = false;
  for (int w = 0; w < kFarWords; ++w) any_far |= st.far[(size_t)seg * kFarWords + w] != 0;
  const int row = threadIdx.x;
  if (row >= a.R) return;
  const bool has_win = lse.win_m != nullptr;
  const size_t at = (size_t)seg * a.R + row;
  const float l2 = row_lse(st, st.acc[at], any_far, seg, row, a.R, a.slot_stride, min(a.slot_stride, kMaxSplit), has_win,
                           has_win ? lse.win_m[at] : 0.f, has_win ? lse.win_z[at] : 0.f);
  if (!lse_out) { st.lse[at] = l2; return; }
  const int hh = a.q_head_inner ? row % a.G : row / a.window;
  const int i = a.q_head_inner ? row / a.G : row - hh * a.window;
  lse_out[((long long)s * lse.n_q_heads + g * a.G + hh) * a.window + i] = l2 * out_scale;
}

// ---- host side ----------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static std::atomic<EncodeTiledFn> known{nullptr};             // several threads may be the first
  EncodeTiledFn fn = known.load(std::memory_order_relaxed);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      known.store(fn = reinterpret_cast<EncodeTiledFn>(p), std::memory_order_relaxed);
  }
  return fn;
}

}  // namespace

int sm_count() {
  static thread_local int dev_cached = -1, n = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (dev != dev_cached) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 148;
    dev_cached = dev;
  }
  return n;
}

bool tensor_path_supported(const slkv_params& p) {
  if (p.dtype != SLKV_BF16) return false;
  const int G = p.n_q_heads / p.n_kv_heads, R = G * p.window;
  if (R > 256) return false;
  return encode_fn() != nullptr;
}

// Row order inside the Q tile: the query heads of a group next to each other (r = i*G + hh) when the head stride is
// the smaller one, else the window rows (r = hh*window + i).
bool tensor_q_head_inner(const slkv_params& p) { return p.q_stride_head <= p.q_stride_row; }

int tensor_slot_stride(const Problem& pb) {
  const int tiles = (pb.max_hist + kTileKeys - 1) / kTileKeys, n = kMaxSplit;
  return (tiles < n ? tiles : n) + 1;
}

cudaError_t plan_score_layer(const Problem& pb, int32_t* status, ScoreLayer* lay) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const slkv_params& p = pb.p;
  CUtensorMap& tm_q = lay->tm_q;
  CUtensorMap& tm_k = lay->tm_k;
  // Tensor-map dimensions go from the smallest stride to the largest.  The order of the G*w query rows
  // inside the Q tile follows from it (head-fastest or window-row-fastest); the scores do not depend on it.
  const int q_head_inner = tensor_q_head_inner(p) ? 1 : 0;
  const int k_head_inner = p.k_stride_head <= p.k_stride_tok;
  {
    cuuint64_t dims[4] = {(cuuint64_t)p.head_dim, (cuuint64_t)p.window, (cuuint64_t)p.n_q_heads, (cuuint64_t)p.n_seqs};
    cuuint64_t strides[3] = {(cuuint64_t)p.q_stride_row * 2, (cuuint64_t)p.q_stride_head * 2, (cuuint64_t)p.q_stride_seq * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)p.window, (cuuint32_t)pb.G, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    if (q_head_inner) {
      cuuint64_t t = dims[1]; dims[1] = dims[2]; dims[2] = t;
      t = strides[0]; strides[0] = strides[1]; strides[1] = t;
      cuuint32_t b = box[1]; box[1] = box[2]; box[2] = b;
    }
    if (enc(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pb.q), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  {
    cuuint64_t dims[3] = {(cuuint64_t)p.head_dim, (cuuint64_t)p.n_kv_heads, (cuuint64_t)pb.total_tokens};
    cuuint64_t strides[2] = {(cuuint64_t)p.k_stride_head * 2, (cuuint64_t)p.k_stride_tok * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)kTileKeys};
    cuuint32_t estr[3] = {1, 1, 1};
    if (!k_head_inner) {
      cuuint64_t t = dims[1]; dims[1] = dims[2]; dims[2] = t;
      t = strides[0]; strides[0] = strides[1]; strides[1] = t;
      cuuint32_t b = box[1]; box[1] = box[2]; box[2] = b;
    }
    if (enc(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(pb.k), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }

  lay->part = pb.part;
  lay->vote = pb.vote;
  lay->lse = lse_source_of(pb);
  lay->status = status;
  return cudaSuccess;
}

cudaError_t plan_score_tensor(const Problem& pb, const int32_t* cu_host, int32_t* status, ScorePlan* plan) {
  ScoreShape& a = plan->sh;
  const slkv_params& p = pb.p;
  a.n_cta = 0;
  if (pb.max_hist <= 0) return cudaSuccess;
  cudaError_t e = plan_score_layer(pb, status, &plan->lay);
  if (e != cudaSuccess) return e;
  a.tab = pb.tab;
  a.n_seqs = p.n_seqs; a.n_kv_heads = p.n_kv_heads; a.G = pb.G; a.window = p.window;
  a.R = pb.R;
  a.Rp = (pb.R + 31) / 32 * 32;
  a.MT = (pb.R + 127) / 128;
  a.halves = p.head_dim / 64;
  a.n_stages = score_list_stages(a.MT, a.halves);
  a.slot_stride = tensor_slot_stride(pb);
  a.q_head_inner = tensor_q_head_inner(p) ? 1 : 0;
  a.k_head_inner = p.k_stride_head <= p.k_stride_tok;
  a.scale_log2 = kLog2e / sqrtf((float)p.head_dim);

  auto tiles_of = [&](int s) {
    const long long nh = (long long)cu_host[s + 1] - cu_host[s] - p.window;
    return nh > 0 ? (nh + kTileKeys - 1) / kTileKeys : 0ll;
  };
  long long total = 0;
  for (int s = 0; s < p.n_seqs; ++s) total += tiles_of(s) * p.n_kv_heads;
  a.total_tiles = (int)total;
  int n_cta = sm_count();
  if (n_cta > kMaxSplit) n_cta = kMaxSplit;
  a.n_cta = total < n_cta ? (int)total : n_cta;
  // groups of whole segments, of about equal size
  const long long group_tiles = kGroupBytes / (a.halves * kHalfBytes);
  long long want = (total + group_tiles / 2) / group_tiles;
  if (want > kListMaxGroups) want = kListMaxGroups;
  if (want < 1) want = 1;
  long long acc = 0;
  int ng = 0;
  a.group_tile[0] = 0;
  for (int s = 0; s < p.n_seqs; ++s) {
    const long long t = tiles_of(s);
    if (t == 0) continue;
    for (int g = 0; g < p.n_kv_heads; ++g) {
      acc += t;
      if (ng < (int)want - 1 && acc * want >= (ng + 1) * total && acc < total) a.group_tile[++ng] = (int)acc;
    }
  }
  a.group_tile[++ng] = (int)total;
  a.n_groups = ng;
  a.group_layers = 0;
  if (total < group_tiles * 3 / 4) {                     // short layers: several of a list together
    a.group_layers = (int)((group_tiles + total / 2) / total);
    if (a.group_layers > kListMaxLayers) a.group_layers = kListMaxLayers;
  }
  return cudaSuccess;
}

cudaError_t launch_merge_lse_tensor(const ScoreShape& sh, const ScoreLayer& lay, float* lse_out, float out_scale,
                                    cudaStream_t st, int* launches) {
  if (sh.n_cta == 0) return cudaSuccess;
  LaunchScope scope(KID_MERGE_LSE, st, launches);
  return launch_pdl(k_merge_lse_tensor, dim3(sh.n_seqs * sh.n_kv_heads), dim3(kMergeThreads), 0, st, 1, sh, lay.part,
                    lay.lse, lse_out, out_scale);
}

cudaError_t launch_score_tensor(const Problem& pb, const int32_t* cu_host, int32_t* status, int passes, float* lse_out, bool cleared,
                                cudaStream_t st, int* launches) {
  ScorePlan plan;
  cudaError_t e = plan_score_tensor(pb, cu_host, status, &plan);
  if (e != cudaSuccess || plan.sh.n_cta == 0) return e;
  e = launch_score_list(plan.sh, &plan.lay, 1, passes, pb.sync, st, launches, cleared);
  if (e != cudaSuccess || !lse_out) return e;
  return launch_merge_lse_tensor(plan.sh, plan.lay, lse_out, lse_out_scale(pb), st, launches);
}

}  // namespace slkv

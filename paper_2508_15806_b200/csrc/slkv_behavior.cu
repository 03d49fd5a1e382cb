// Attention behaviour analysis (Sec. 3.2, Algorithm 1): SF_sc, LG_sc and INF_sc of a batch of attention rows.
//
// One warp per row.  A row's needle positions N and top-k positions T arrive as index lists; the kernels read only the
// weights at those positions (the rest of the row never matters), so a batch over [layers x heads x prompts] moves a
// few hundred bytes per row however long the context is.  Sets are sets: an index that occurs twice in a list counts
// once.  Sums are fp64 over at most a few hundred terms; 0 / 0 counts as 0.
// What bounds it: two dependent reads from DRAM per row (a list's entry, the weight there), and next to no bytes.
#include "slkv_internal.cuh"

namespace slkv {
namespace {

constexpr int kRowsPerCta = 8;          // warps per CTA

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct Lists {
  const float* attn;
  const int32_t *needle_idx, *topk_idx;
  float *sf, *lg, *inf;
  long long row_stride, n_rows, needle_stride, topk_stride;
  int row_len, n_needle, n_topk;
};

// tnw: weight of all needle positions, wo / wd: of the top-k positions that are / are not needles (lane shares)
__device__ __forceinline__ void scores(const Lists& a, long long row, int lane, double tnw, double wo, double wd) {
  tnw = warp_sum(tnw); wo = warp_sum(wo); wd = warp_sum(wd);
  if (lane == 0) {
    const double ws = fmax(0.0, tnw - wo);                         // needle weight outside the top-k set
    const double s = wo + wd > 0.0 ? wo / (wo + wd) : 0.0;         // SF_sc: surface focus
    const double l = wo + ws > 0.0 ? wo / (wo + ws) : 0.0;         // LG_sc: logic grasp
    const double h = s + l > 0.0 ? 2.0 * s * l / (s + l) : 0.0;    // INF_sc: their harmonic mean
    a.sf[row] = (float)s; a.lg[row] = (float)l; a.inf[row] = (float)h;
  }
}

// Lists of up to 32 E entries: a lane holds entries lane + 32 e of both and reads their weights at once, duplicates or
// not; which of them count is found out meanwhile, against the lists in shared memory, four entries per (broadcast) read.
template <int E>
__global__ void __launch_bounds__(kRowsPerCta * 32) k_behavior_short(const __grid_constant__ Lists a) {
  __shared__ int4 lists[kRowsPerCta][2][8 * E];
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long row = (long long)blockIdx.x * kRowsPerCta + warp;
  if (row >= a.n_rows) return;
  const float* W = a.attn + row * a.row_stride;
  const int32_t* list[2] = {a.needle_idx + row * a.needle_stride, a.topk_idx + row * a.topk_stride};
  const int n[2] = {a.n_needle, a.n_topk};
  int idx[2][E];
  float weight[2][E];
  bool counts[2][E], on_needle[E];
#pragma unroll
  for (int l = 0; l < 2; ++l)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = lane + 32 * e < n[l] ? list[l][lane + 32 * e] : -1;
      idx[l][e] = i;
      counts[l][e] = i >= 0 && i < a.row_len;                      // entries outside the row are padding
    }
#pragma unroll
  for (int l = 0; l < 2; ++l)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      weight[l][e] = counts[l][e] ? W[idx[l][e]] : 0.0f;
      reinterpret_cast<int*>(lists[warp][l])[lane + 32 * e] = idx[l][e];
    }
#pragma unroll
  for (int e = 0; e < E; ++e) on_needle[e] = false;
  __syncwarp();
#pragma unroll
  for (int l = 0; l < 2; ++l)
    for (int q = 0; 4 * q < n[l]; ++q) {
      const int4 v = lists[warp][l][q];
      const int x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (x[j] == idx[l][e] && 4 * q + j < lane + 32 * e) counts[l][e] = false;        // not its first occurrence
          if (l == 0 && x[j] == idx[1][e]) on_needle[e] = true;
        }
    }
  double tnw = 0.0, wo = 0.0, wd = 0.0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    if (counts[0][e]) tnw += (double)weight[0][e];
    if (counts[1][e]) { if (on_needle[e]) wo += (double)weight[1][e]; else wd += (double)weight[1][e]; }
  }
  scores(a, row, lane, tnw, wo, wd);
}

// Lists of any length, read where they are.
__global__ void __launch_bounds__(kRowsPerCta * 32) k_behavior(const __grid_constant__ Lists a) {
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * kRowsPerCta + (threadIdx.x >> 5);
  if (row >= a.n_rows) return;
  const float* W = a.attn + row * a.row_stride;
  const int32_t* Nn = a.needle_idx + row * a.needle_stride;
  const int32_t* Tt = a.topk_idx + row * a.topk_stride;
  auto valid = [&](int i) { return i >= 0 && i < a.row_len; };    // entries outside the row are padding
  // total needle weight TNW: every distinct needle position once
  double tnw = 0.0;
  for (int p = lane; p < a.n_needle; p += 32) {
    const int i = Nn[p];
    if (!valid(i)) continue;
    bool first = true;
    for (int b = 0; b < p; ++b) first = first && Nn[b] != i;
    if (first) tnw += (double)W[i];
  }
  // top-k positions: on a needle (WO, weight on target) or not (WD, weight that distracts)
  double wo = 0.0, wd = 0.0;
  for (int p = lane; p < a.n_topk; p += 32) {
    const int i = Tt[p];
    if (!valid(i)) continue;
    bool first = true;
    for (int b = 0; b < p; ++b) first = first && Tt[b] != i;
    if (!first) continue;
    bool on_needle = false;
    for (int b = 0; b < a.n_needle; ++b) on_needle = on_needle || Nn[b] == i;
    if (on_needle) wo += (double)W[i]; else wd += (double)W[i];
  }
  scores(a, row, lane, tnw, wo, wd);
}

}  // namespace

cudaError_t launch_behavior(const float* attn, long long row_stride, int row_len, long long n_rows,
                            const int32_t* needle_idx, int n_needle, long long needle_stride, const int32_t* topk_idx,
                            int n_topk, long long topk_stride, float* sf, float* lg, float* inf, cudaStream_t st) {
  if (n_rows == 0) return cudaSuccess;
  int launches = 0;
  LaunchScope scope(KID_BEHAVIOR, st, &launches);
  const dim3 grid((unsigned)((n_rows + kRowsPerCta - 1) / kRowsPerCta)), block(kRowsPerCta * 32);
  const Lists a = {attn, needle_idx, topk_idx, sf, lg, inf, row_stride, n_rows, needle_stride, topk_stride,
                   row_len, n_needle, n_topk};
  const int most = n_needle > n_topk ? n_needle : n_topk;
  if (most <= 32) return launch_pdl(k_behavior_short<1>, grid, block, 0, st, 1, a);
  if (most <= 64) return launch_pdl(k_behavior_short<2>, grid, block, 0, st, 1, a);
  if (most <= 128) return launch_pdl(k_behavior_short<4>, grid, block, 0, st, 1, a);
  return launch_pdl(k_behavior, grid, block, 0, st, 1, a);        // a lane's registers would not hold its entries
}

}  // namespace slkv

// A whole fp32 layer in one launch (Sec. 3.4, Eq. 7-8; Algorithm 3): scores with fp32 FMA arithmetic, pooling, selection and
// gather, a cluster of CTAs per (sequence, KV head) segment.  Up to 128 query rows per KV head; single calls of few segments whose
// scores fit in the cluster's shared memory; k_score_simt takes the rest.
//
// As slkv_layer_tc.cu: row sums, votes and kept positions go from CTA to CTA in bulk copies, nothing is cleared, nothing
// polled.  A CTA takes whole blocks of 32 keys, forms their scores 32 keys x 8 or 16 rows per warp out of shared memory (the
// same operations in the same order as k_score_simt: a row's statistics and a key's vote are the same bit for bit) and keeps them
// for the votes.
// What bounds it: latency at the small sizes (8 heads, 1024 positions, 16 rows, head_dim 64: 24.6 us from a stream as three
// launches with two meetings of all CTAs, 12.0 here: keys 0.7, products 1.0, exchange 1, log-sum-exps 0.9, votes 1.4, selection
// 2.4, rows 1.5), shared-memory reads of the operands beyond: a clock per register of a warp, twice what the FMAs take.
#include <type_traits>

#include "slkv_fma_device.cuh"
#include "slkv_layer_device.cuh"

namespace slkv {
namespace {

constexpr int kBlock = 32;                     // keys
constexpr int kMaxRows = 128;
constexpr int kMaxScores = 16384;              // of a CTA
constexpr float kTiny = 1e-30f;                // as k_score_simt: a block's sum outside (kTiny, inf) goes the far way

struct LayerFmaArgs {
  LayerTail tail;
  LseSource lse;
  WindowArgs win;              // Q, K and their strides, too
  int all_causal, stats;       // stats 0: the caller's log-sum-exps
  int expire;                  // diagnostics: 1 the wait for the row sums runs out, 2 the one for the votes
  int G, R, q_rows, s_pitch;   // rows of Q's and pitch of the scores' shared memory
  int chunk;                   // keys that are loaded together, whole blocks; two chunks fit, or one that is all of a CTA's
  int32_t* status;
};

__device__ __forceinline__ unsigned long long now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Bounded (1 s): *gave_up is set, and the status, when the wait ran out.
__device__ __forceinline__ void bar_wait(const void* bar, volatile int* gave_up, int32_t* status) {
  const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0, 100;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(b) : "memory");
    if (ok) return;
    if (it == 0) t0 = now();
    if ((it & 63u) == 63u && now() - t0 > 1000ull * 1000ull * 1000ull) {
      *gave_up = 1;
      if (status) atomicExch(status, (int)SLKV_ERR_DEVICE_TIMEOUT);
      return;
    }
  }
}

template <int D, int IT> struct FmaShared {
  static constexpr int kPitch = D + 4;
  static constexpr int kVotes = vote_floats(kLayerThreads, IT) > window_floats(D) ? vote_floats(kLayerThreads, IT) : window_floats(D);
  struct alignas(16) Sums { double z[kMaxRows]; int far, unused[3]; };
  alignas(16) float votes_mem[(kVotes + 3) & ~3];
  Sums all[kLayerMaxCluster];
  alignas(16) float2 win[kMaxRows];            // the window keys' share (maximum, sum)
  float lse[kMaxRows];
  float part[kMaxScores / kBlock];             // sums of a block's keys [block][row]; the votes' row groups
  unsigned long long sums_bar, votes_bar, max_bar, far_bar;
  SegmentRows rows;
  int far_here, gave_up;
  // then Q [q_rows][kPitch], the scores [R][s_pitch] and the keys [chunk or 2 chunk][kPitch], whose memory is later used by
  union Later {
    struct alignas(16) { double z[kLayerMaxCluster][kMaxRows]; float row_max[kLayerMaxCluster][kMaxRows]; } beyond;   // scores beyond fp32's range
    SelShared select;                                                                                  // the first CTA
  };
};

template <int D, int IT>
__global__ void __launch_bounds__(kLayerThreads, 1)
k_layer_fma(const __grid_constant__ LayerFmaArgs a) {
  using F = FmaShared<D, IT>;
  constexpr int kPitch = F::kPitch, kPerRow = D / 4;
  const int chunk = a.chunk;
  extern __shared__ __align__(16) unsigned char smem[];
  F& f = *reinterpret_cast<F*>(smem);
  float* const qs = reinterpret_cast<float*>(smem + sizeof(F));
  float* const sc = qs + a.q_rows * kPitch;
  float* const ks = sc + a.R * a.s_pitch;
  typename F::Later& later = *reinterpret_cast<typename F::Later*>(ks);
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kLayerThreads / 32;
  auto sync = [&]() { __syncthreads(); };
  const Segment x = segment_of(a.tail, blockIdx.x / CS);
  const int blocks = (x.n + kBlock - 1) / kBlock;
  const int first = blocks * rank / CS, n_b = blocks * (rank + 1) / CS - first;        // this CTA's blocks
  const int key0 = first * kBlock, n_here = max(min(x.n - key0, n_b * kBlock), 0);     // ... and keys
  const int window_blocks = (a.R + kWinRows - 1) / kWinRows, my_blocks = rank < window_blocks ? (window_blocks - rank - 1) / CS + 1 : 0;
  const bool win = a.stats && a.all_causal && x.n > 0;
  constexpr int vote_bytes = kBlock / IT * (IT + 4) * 4;       // of a block, as they lie in shared memory
  float* votes = f.votes_mem + kLead;
  auto expect = [&](const void* b, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(b)), "r"(bytes) : "memory");
  };
  pdl_launch_dependents();
  if (tid == 0) {
    f.far_here = f.gave_up = 0;
    auto init = [&](const void* b, int count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(b)), "r"(count) : "memory");
    };
    init(&f.sums_bar, 1 + (a.expire == 1));
    init(&f.votes_bar, 1 + (a.expire == 2));
    init(&f.max_bar, 1);
    init(&f.far_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    expect(&f.sums_bar, (CS - 1) * (int)sizeof(typename F::Sums) + (win ? (window_blocks - my_blocks) * kWinRows * 8 : 0));
    if (rank == 0) expect(&f.votes_bar, (blocks - n_b) * vote_bytes);
  }
  sync();
  cluster_arrive();                                            // everybody is there (waited for before the first copy)
  pdl_wait();

  // ---- queries and the first keys on their way
  const float* q = static_cast<const float*>(a.win.q) + x.s * a.win.q_stride_seq;
  const float* k = static_cast<const float*>(a.win.k) + (long long)(x.t0 + key0) * a.win.k_stride_tok + (long long)x.g * a.win.k_stride_head;
  auto copy16 = [&](float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
  };
  auto load_k = [&](int c) {                                   // chunk c
    const int from = c * chunk, n = min(chunk, n_here - from);
    for (int i = tid; i < n * kPerRow; i += kLayerThreads) {
      const int r = i / kPerRow, e = (i - r * kPerRow) * 4;
      copy16(ks + ((c & 1) * chunk + r) * kPitch + e, k + (long long)(from + r) * a.win.k_stride_tok + e);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int i = tid; i < a.R * kPerRow; i += kLayerThreads) {   // row r = hh*window + i
    const int r = i / kPerRow, e = (i - r * kPerRow) * 4, hh = r / a.tail.window, wi = r - hh * a.tail.window;
    copy16(qs + r * kPitch + e, q + wi * a.win.q_stride_row + (long long)(x.g * a.G + hh) * a.win.q_stride_head + e);
  }
  load_k(0);
  load_k(1);
  if (warp == kWarps - 1) {
    const SegmentRows r = segment_rows(a.tail, x);
    if (lane == 0) f.rows = r;
  }
  if (!a.stats && tid < a.R) f.lse[tid] = a.lse.caller_lse(x.s, x.g, tid, a.G, a.tail.window, false);
  if (win && tid < 128)
    for (int b = rank; b < window_blocks; b += CS) {
      window_rows<float, D, 2>(a.win, f.votes_mem, tid, x.s, x.g, x.t0 + x.n, b * kWinRows,
                               [&](int r, float m, float z) { f.win[r] = make_float2(m, z); });
      asm volatile("bar.sync 2, 128;" ::: "memory");
    }

  // ---- scores, and the sums of 2^score over blocks of keys
  auto unit = [&](auto rows_per_lane, const float* kb, int blk, int row0) {
    constexpr int J = decltype(rows_per_lane)::value;          // lane: keys kl + 8 i, rows rl + 4 j
    const int kl = lane & 7, rl = lane >> 3;
    const float* kp = kb + kl * kPitch;
    const float* qp = qs + (row0 + rl) * kPitch;
    f32x2 acc[4][J];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < J; ++j) acc[i][j] = 0;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      ulonglong2 kv[4], qv[J];
#pragma unroll
      for (int i = 0; i < 4; ++i) kv[i] = *reinterpret_cast<const ulonglong2*>(kp + i * 8 * kPitch + c);
#pragma unroll
      for (int j = 0; j < J; ++j) qv[j] = *reinterpret_cast<const ulonglong2*>(qp + j * 4 * kPitch + c);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) {
          acc[i][j] = fma2(kv[i].x, qv[j].x, acc[i][j]);
          acc[i][j] = fma2(kv[i].y, qv[j].y, acc[i][j]);
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int row = row0 + rl + 4 * j;
      float v = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int key = blk * kBlock + kl + 8 * i;
        const float s = sum_of(acc[i][j]) * a.win.scale_log2;
        if (row < a.R) sc[row * a.s_pitch + key] = s;
        if (key < n_here) v += exp2f(s);
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(kAll, v, o);
      if (kl == 0 && row < a.R) f.part[blk * a.R + row] = v;
    }
  };
  const int chunks = (n_here + chunk - 1) / chunk;
  for (int c = 0; c < chunks; ++c) {
    if (c + 1 < chunks || c == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    sync();
    const int blks = (min(chunk, n_here - c * chunk) + kBlock - 1) / kBlock, blk0 = c * (chunk / kBlock);
    const float* kc = ks + (c & 1) * chunk * kPitch;
    // What bounds this is shared memory: an operand register of a warp takes a clock, a step of four dimensions 24 of them for
    // 32 x 8 scores, 32 for 32 x 16.
    const int wide = (a.R + 15) / 16, narrow = (a.R + 7) / 8;
    if (a.R > 8) {
      for (int u = warp; u < blks * wide; u += kWarps) unit(std::integral_constant<int, 4>(), kc + (u / wide) * kBlock * kPitch, blk0 + u / wide, u % wide * 16);
    } else {
      for (int u = warp; u < blks * narrow; u += kWarps) unit(std::integral_constant<int, 2>(), kc + (u / narrow) * kBlock * kPitch, blk0 + u / narrow, u % narrow * 8);
    }
    sync();
    if (c + 2 < chunks) load_k(c + 2);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");

  // ---- row sums of the cluster, log-sum-exps
  if (a.stats) {
    const int row = tid;
    if (row < kMaxRows) {
      double z = 0.0;
      if (row < a.R)
        for (int b = 0; b < n_b; ++b) {
          const float v = f.part[b * a.R + row];
          if (v < INFINITY && v > kTiny) z += (double)v;
          else f.far_here = 1;
        }
      f.all[rank].z[row] = z;
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (row == 0) f.all[rank].far = f.far_here;
      publish_for_copy();
      cluster_wait();
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (tid < CS && tid != rank) {
        copy_to_cta(&f.all[rank], &f.all[rank], sizeof(f.all[0]), &f.sums_bar, tid);
        if (win)
          for (int b = rank; b < window_blocks; b += CS) copy_to_cta(&f.win[b * kWinRows], &f.win[b * kWinRows], kWinRows * 8, &f.sums_bar, tid);
      }
    } else {
      cluster_wait();
    }
    bar_wait(&f.sums_bar, &f.gave_up, a.status);
    sync();
    // The same in every CTA, and without meetings of them all, which a CTA that gives up would have to come to as well.
    bool far = false;
    for (int c = 0; c < CS; ++c) far |= f.all[c].far != 0;
    far = far && f.gave_up == 0;                               // else they need not all be there
    auto to_all = [&](const void* row, int bytes, const void* bar) {
      publish_for_copy();
      sync();
      if (tid == rank) expect(bar, (CS - 1) * bytes);
      else if (tid < CS) copy_to_cta(row, row, bytes, bar, tid);
      bar_wait(bar, &f.gave_up, a.status);
    };
    if (far) {
      // some block's sum left fp32's range: the rows' maxima, then sums relative to them
      for (int r = warp; r < a.R; r += kWarps) {
        float m = -INFINITY;
        for (int j = lane; j < n_here; j += 32) m = fmaxf(m, sc[r * a.s_pitch + j]);
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
        if (lane == 0) later.beyond.row_max[rank][r] = m;
      }
      to_all(later.beyond.row_max[rank], sizeof(later.beyond.row_max[0]), &f.max_bar);
      for (int u = warp; u < n_b * ((a.R + 3) / 4); u += kWarps) {           // a block and four rows per warp
        const int b = u / ((a.R + 3) / 4), r = u % ((a.R + 3) / 4) * 4 + (lane >> 3);
        float m = -INFINITY, v = 0.f;
        for (int c = 0; c < CS; ++c) m = fmaxf(m, later.beyond.row_max[c][min(r, a.R - 1)]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int key = b * kBlock + (lane & 7) + 8 * i;
          if (key < n_here && r < a.R) v += exp2f(sc[r * a.s_pitch + key] - m);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(kAll, v, o);
        if ((lane & 7) == 0 && r < a.R) f.part[b * a.R + r] = v;
      }
      sync();
      if (row < a.R) {
        double z = 0.0;
        for (int b = 0; b < n_b; ++b) z += (double)f.part[b * a.R + row];
        later.beyond.z[rank][row] = z;
      }
      to_all(later.beyond.z[rank], sizeof(later.beyond.z[0]), &f.far_bar);
    }
    if (row < a.R) {
      float M = 0.f;
      double Z = 0.0;
      if (far) {
        M = -INFINITY;
        for (int c = 0; c < CS; ++c) { M = fmaxf(M, later.beyond.row_max[c][row]); Z += later.beyond.z[c][row]; }
      } else {
        for (int c = 0; c < CS; ++c) Z += f.all[c].z[row];
      }
      if (win) {                                               // as simt_row_lse
        const float wm = f.win[row].x, Mn = fmaxf(M, wm);
        Z = __dadd_rn(__dmul_rn(Z, (double)exp2f(M - Mn)), __dmul_rn((double)f.win[row].y, (double)exp2f(wm - Mn)));
        M = Mn;
      }
      f.lse[row] = __fadd_rn(M, (float)log2(Z));
    }
  } else {
    cluster_wait();
  }
  const float pad = a.tail.pool_mode == SLKV_POOL_MAX ? -INFINITY : 0.f;
  if (rank == 0 && tid >= 128 && tid < 136) {
    const int p = tid < 132 ? tid - 132 : x.n + tid - 132;
    votes[vote_at<IT>(p)] = pad;
  }
  sync();

  // ---- votes.  A key's rows are added up in one order whatever CTA it lies in, and that of k_score_simt: four rows 4 apart to a
  // part, the parts in a binary tree.  A key per thread, or a subtree of it where there are threads left (1008 keys of 16 rows: as
  // quick as rows dealt out to the threads in turn, whose sums depended on how many keys a CTA has).
  {
    const int span = n_b * kBlock;                             // keys and padding
    int parts = 4, groups = 1;                                 // parts: 16 rows have four
    while (4 * parts < a.R) parts *= 2;
    while (2 * groups * span <= kLayerThreads && groups < min(parts, 8)) groups *= 2;
    const int per = parts / groups;
    for (int j0 = 0; j0 < span; j0 += kLayerThreads / groups) {
      const int grp = groups > 1 ? tid / span : 0, key = groups > 1 ? tid - grp * span : j0 + tid;
      const bool on = key < span && grp < groups;
      float v = 0.f;
      if (on && key < n_here) {
        float left[5];                                         // level l: the sum of 2^l parts that waits for its right half
        for (int i = 0; i < per; ++i) {
          const int part = grp * per + i, r0 = (part >> 2) * 16 + (part & 3);
          float e[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int r = min(r0 + 4 * j, a.R - 1);
            e[j] = exp2f(sc[r * a.s_pitch + key] - f.lse[r]);
          }
          v = r0 < a.R ? e[0] : 0.f;
#pragma unroll
          for (int j = 1; j < 4; ++j) v += r0 + 4 * j < a.R ? e[j] : 0.f;
          if (per == 1) break;
          bool carry = true;
#pragma unroll
          for (int l = 0; l < 5; ++l) {
            if (carry && (i >> l & 1)) v = left[l] + v;
            else if (carry) { left[l] = v; carry = false; }
          }
        }
      }
      if (groups > 1) {
        if (on && grp > 0) f.part[(grp - 1) * span + key] = v;
        sync();
        if (on && grp == 0) {
          auto p = [&](int g) { return f.part[(g - 1) * span + key]; };
          v += p(1);
          if (groups > 2) v += p(2) + p(3);
          if (groups > 4) v += (p(4) + p(5)) + (p(6) + p(7));
        }
      }
      if (on && grp == 0) votes[vote_at<IT>(key0 + key)] = key < n_here ? v / (float)a.G : pad;
      if (groups > 1) break;
    }
    publish_for_copy();
  }
  sync();
  if (rank == 0) {
    bar_wait(&f.votes_bar, &f.gave_up, a.status);
  } else if (tid == 0 && n_b > 0) {
    float* mine = votes + vote_at<IT>(key0);
    copy_to_cta(mine, mine, n_b * vote_bytes, &f.votes_bar, 0);
  }
  const SegmentRows r = f.rows;
  if (rank == 0) layer_select<IT, 0>(a.tail, x, r.k_keep, votes, later.select, tid, &f.gave_up);
  cluster_arrive();
  cluster_wait();
  if (a.tail.select) layer_gather(a.tail, x, r, reinterpret_cast<const int*>(cluster.map_shared_rank(f.votes_mem, 0)), tid, rank, CS);
  cluster_arrive();                                            // nobody reads another CTA's memory any more
  cluster_wait();
}

// Keys of a CTA, in whole blocks; the pitch of its scores' rows puts eight keys of four rows into different banks.
int keys_per_cta(const Problem& pb, int cs) {
  const int blocks = (pb.max_hist + kBlock - 1) / kBlock;
  return (blocks + cs - 1) / cs * kBlock;
}
int score_pitch(const Problem& pb, int cs) { return keys_per_cta(pb, cs) + 8; }
int query_rows(const Problem& pb) { return (pb.R + 15) / 16 * 16; }
template <int D, int IT> size_t smem_fixed(const Problem& pb, int cs) {
  return sizeof(FmaShared<D, IT>) + sizeof(float) * ((size_t)query_rows(pb) * (D + 4) + (size_t)pb.R * score_pitch(pb, cs));
}
// All keys of a CTA at once where they fit -- with 16 query rows each block of them is work for one warp --, else two chunks
// in turn; 0: there is no room.  8 heads, 16 rows, head_dim 128, the whole call in us with chunks of 64 keys / as here: 2000
// positions 23.0 / 16.2, 4000 33.7 / 25.2.
template <int D, int IT> int chunk_of(const Problem& pb, int cs) {
  const long long room = 227 * 1024 - (long long)smem_fixed<D, IT>(pb, cs);
  const int keys = keys_per_cta(pb, cs), fit = room > 0 ? (int)(room / ((D + 4) * 4)) / kBlock * kBlock : 0;
  const int least = ((int)sizeof(typename FmaShared<D, IT>::Later) / ((D + 4) * 4) + kBlock) / kBlock * kBlock;
  const int all = keys > least ? keys : least;
  if (all <= fit) return all;
  const int half = fit / 2 / kBlock * kBlock;
  return 2 * half >= least ? half : 0;
}
bool few_positions(const Problem& pb) { return pb.max_hist <= 8 * kLayerThreads; }

int chunk_for(const Problem& pb, int cs) {
  const bool small = few_positions(pb);
  if (pb.p.head_dim == 64) return small ? chunk_of<64, 8>(pb, cs) : chunk_of<64, 16>(pb, cs);
  return small ? chunk_of<128, 8>(pb, cs) : chunk_of<128, 16>(pb, cs);
}

template <int D, int IT>
cudaError_t launch(const Problem& pb, int cs, LayerFmaArgs& a, cudaStream_t st, int* launches) {
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    e = cudaFuncSetAttribute(k_layer_fma<D, IT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_layer_fma<D, IT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    configured_dev = dev;
  }
  const size_t smem = smem_fixed<D, IT>(pb, cs) + sizeof(float) * (D + 4) * (size_t)(keys_per_cta(pb, cs) <= a.chunk ? a.chunk : 2 * a.chunk);
  LaunchScope scope(KID_LAYER, st, launches);
  return launch_pdl(k_layer_fma<D, IT>, dim3((unsigned)(pb.n_seg * cs)), dim3(kLayerThreads), smem, st, cs, a);
}

}  // namespace

// CTAs per segment, 0: the shape is not taken.  The clusters are those of slkv_layer_tc.cu; their CTAs are fewer than the SMs,
// which tells where the products take most of the time.  A block of 32 keys costs a CTA half a unit of 32 keys x 16 rows beside its
// units; the general path takes a step of all SMs for every 296 tiles of 64 keys x 64 rows, the longer the more of the rows exist
// where it walks them twice.  What the general path's launches cost on top is worth a `head`, of which loading the keys in two
// chunks leaves nothing but with head_dim 64; with few segments two chunks are never taken.  Measured both ways, 199 to 502 shapes of
// each kind that are taken: slower from a stream by 0.8 us at most (layers), 1.3 (scores) and, with log-sum-exps handed in, 6.4 and
// 7.1 (40 segments of 1500-3000 tokens, head_dim 128, 16 rows, in two chunks: 52.0 against 45.6).  us in a graph / from a stream, here and on the general path (r: lengths from half to the
// whole; two chunks from * on; - not taken):
//                       1200 tokens            2300                    3000                    4000
//   2 segs, d 128, 16   13.2/14.0  18.4/21.9   16.2/16.9  20.5/22.6   -
//   8 segs, d  64, 16   11.9/12.4  18.8/20.7   13.7/14.2  19.2/22.5   14.9/15.4  23.4/26.8   16.7/17.2  24.1/26.8
//   8 segs, d 128, 16   13.9/14.7  21.1/24.1   16.8/17.7  21.8/24.7   21.8/22.7  28.9/32.9 * 25.9/26.8  29.0/32.9
//   8 segs, d 128, 32   16.1/16.9  22.1/24.8   21.0/21.8  22.8/25.5 * 29.7/30.5  30.1/33.0   35.3/36.2  31.5/35.0 -
//   8 segs, d 128, 64   20.4/21.3  26.9/29.3 * 32.6/33.5  27.8/30.9 -
//   16 r,   d 128, 32   21.1/22.0  24.5/26.8 * 32.2/33.1  31.5/34.9   40.9/41.8  31.0/34.0 -
//   40 segs, d 64, 16   17.2/18.2  31.8/35.0 * 23.9/24.7  44.8/47.4   29.5/30.4  61.4/64.3   -
int layer_fma_cluster(const Problem& pb, bool select) {
  const slkv_params& p = pb.p;
  if (p.dtype != SLKV_F32 || pb.R > kMaxRows || (p.pool_kernel >> 1) > kMaxRadius || p.history_only || pb.tab.n_inline == 0 ||
      pb.max_hist < 1 || pb.max_hist > 16 * kLayerThreads)
    return 0;
  const int cs = layer_tc_clusters_for(pb.n_seg);
  if (cs < 2 || (long long)keys_per_cta(pb, cs) * pb.R > kMaxScores) return 0;
  const int chunk = chunk_for(pb, cs), keys = keys_per_cta(pb, cs), sms = sm_count();
  const bool at_once = chunk >= keys, both = !pb.lse_opt;
  if (chunk == 0 || (!at_once && 2 * pb.n_seg * cs < sms)) return 0;
  const int units = (pb.R + 15) / 16;
  const int head = at_once ? (both && select ? 40 : both || select ? 25 : 10) : (both && select && p.head_dim == 64 ? 20 : 0);
  const long long steps = (2 * pb.n_tiles128 + 2 * sms - 1) / (2 * sms) * ((pb.R + 63) / 64);
  return keys / kBlock * (2 * units + 1) <= (both ? 20 + 5 * units : 20) * steps + head ? cs : 0;
}

cudaError_t launch_layer_fma(const Problem& pb, int cs, const TailLayer* tail, float* pooled, int32_t* status, cudaStream_t st,
                             int* launches) {
  LayerFmaArgs a;
  a.tail = layer_tail(pb, tail, pooled);
  a.lse = lse_source_of(pb);
  a.win = window_args(pb, false);
  a.stats = pb.lse_opt ? 0 : 1;
  a.all_causal = pb.p.softmax_domain == SLKV_ALL_CAUSAL;
  a.G = pb.G; a.R = pb.R;
  a.q_rows = query_rows(pb);
  a.s_pitch = score_pitch(pb, cs);
  a.chunk = chunk_for(pb, cs);
  a.status = status;
  a.expire = take_expire_next_layer_wait(a.stats != 0);
  const bool small = few_positions(pb);
  if (pb.p.head_dim == 64) return small ? launch<64, 8>(pb, cs, a, st, launches) : launch<64, 16>(pb, cs, a, st, launches);
  return small ? launch<128, 8>(pb, cs, a, st, launches) : launch<128, 16>(pb, cs, a, st, launches);
}

}  // namespace slkv

// A whole layer in one launch (Sec. 3.4, Eq. 7-8; Algorithm 3): scores on the tensor cores, pooling, selection and gather, a
// cluster of CTAs per (sequence, KV head) segment.  bf16, head_dim 64 or 128, up to 128 query rows per KV head, up to 8192 history
// positions, single calls of few segments; the list kernel (slkv_score_pipe.cu) takes the rest.
//
// The segments of a call are independent, and the CTAs of a cluster run at the same time by construction: row sums, votes and
// kept positions go from CTA to CTA through shared memory behind a cluster barrier, nothing has to be cleared, nothing is
// polled, and the launch needs neither a cooperative grid (whose start a stream puts off to the next multiple of 2 us) nor a
// workspace.
//   warp 0     TMA loads of Q and of the CTA's K tiles; the last tiles of the statistics pass stay for the vote pass, which
//              walks the tiles backwards
//   warp 1     tcgen05.mma, a 128-column TMEM unit per tile
//   warp 2     the segment's packed rows from the budgets
//   warps 4-19 the arithmetic of the list kernel, tile by tile the same (results are the same bit for bit where the fp64 sums
//              are exact); then, in the first CTA, pooling and selection; then the CTA's share of the rows
// What bounds it: latency -- keys on their way 2 us, exponentials 0.6-0.8 us per tile and pass, exchanges of 1 us, the
// selection's chain of 2-4 us, rows in and out 1.5 us (8 segments of 8192 positions, 7 tiles per CTA: statistics 6, exchange
// 1.6, votes 5.8 with their way into the first CTA, selection 5, rows 1.6).
#include <cuda.h>

#include "slkv_layer_device.cuh"
#include "slkv_tc_device.cuh"

namespace slkv {
namespace {

constexpr int kThreads = 128 + kLayerThreads;
constexpr int kMaxStages = 8;

struct LayerArgs {
  alignas(64) CUtensorMap tm_q;
  alignas(64) CUtensorMap tm_k;
  LayerTail tail;
  LseSource lse;
  WindowArgs win;
  int all_causal, passes;      // passes: 3, or 2: the caller's log-sum-exps
  int expire;                  // diagnostics: 1 the wait for the row sums runs out, 2 the one for the votes
  int G, R, Rp, halves, n_stages, q_head_inner, k_head_inner;
  float scale_log2;
  int32_t* status;
};

// Shared memory behind the Q tile and the K ring.
template <int IT> struct Far {
  alignas(16) float votes_mem[(vote_floats(kLayerThreads, IT) > window_floats(128) ? vote_floats(kLayerThreads, IT) : window_floats(128)) + 3 & ~3];
  struct alignas(16) Sums { double z[128]; int far, unused[3]; };
  Sums all[kLayerMaxCluster];                  // row sums of the cluster's CTAs; far: some of them are in far[] there
  double z_wg[4][128];                         // ... of this CTA's warpgroups
  float2 far_wg[4][128];                       // what fp64 cannot hold of them (sum, reference)
  float2 far[128];                             // the same of the CTA; read by the others
  alignas(16) float2 win[128];                 // the window keys' share (maximum, sum)
  float lse[128];                              // log-sum-exps, negated
  unsigned long long bars[2 * kMaxStages + 10], sums_bar, votes_bar;
  int far_here, abort_flag;
  uint32_t tmem;
  SegmentRows rows;
};

// Tiles first .. first + n of a segment in order, then back again: where each lies in the ring and when.
struct Ring {
  int n, stages;
  __device__ __forceinline__ int uses(int st) const { return (n - st + stages - 1) / stages; }       // tiles of a pass in a stage
};

template <int IT>
__global__ void __launch_bounds__(kThreads, 1)
k_layer_tc(const __grid_constant__ LayerArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q_half = 128 * 128, stage_bytes = a.halves * kHalfBytes;
  Far<IT>& f = *reinterpret_cast<Far<IT>*>(smem + a.halves * q_half + a.n_stages * stage_bytes);
  const uint32_t q_sh = smem_u32(smem), k_sh = q_sh + (uint32_t)(a.halves * q_half), bar0 = smem_u32(f.bars);
  auto full = [&](int st) { return bar0 + 8u * (uint32_t)st; };
  auto empty = [&](int st) { return bar0 + 8u * (uint32_t)(kMaxStages + st); };
  auto unit_full = [&](int u) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + u); };
  auto unit_empty = [&](int u) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + 4 + u); };
  const uint32_t q_full = bar0 + 8u * (2 * kMaxStages + 8), drain = q_full + 8u;
  volatile int* abort_flag = &f.abort_flag;

  const Segment x = segment_of(a.tail, blockIdx.x / CS);
  const int tiles = (x.n + kTileKeys - 1) / kTileKeys;
  const int first = tiles * rank / CS, n_t = tiles * (rank + 1) / CS - first;          // this CTA's tiles
  const bool stats = a.passes == 3;
  const Ring ring = {n_t, a.n_stages};
  const int window_blocks = (a.R + kWinRows - 1) / kWinRows, my_blocks = rank < window_blocks ? (window_blocks - rank - 1) / CS + 1 : 0;
  constexpr int vote_bytes = kTileKeys / IT * (IT + 4) * 4;                            // of a tile, as they lie in shared memory

  pdl_launch_dependents();
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&a.tm_k)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&a.tm_q)) : "memory");
    f.abort_flag = 0;
    f.far_here = 0;
    for (int st = 0; st < a.n_stages; ++st) { mbar_init(full(st), 1); mbar_init(empty(st), 1); }
    for (int u = 0; u < 4; ++u) { mbar_init(unit_full(u), 1); mbar_init(unit_empty(u), 4); }
    mbar_init(q_full, 1);
    mbar_init(drain, 1);
    mbar_init(smem_u32(&f.sums_bar), 1 + (a.expire == 1));
    mbar_init(smem_u32(&f.votes_bar), 1 + (a.expire == 2));
    if (stats) mbar_expect_tx(smem_u32(&f.sums_bar), (uint32_t)((CS - 1) * sizeof(typename Far<IT>::Sums) +
                                                                 (a.all_causal && x.n > 0 ? (window_blocks - my_blocks) * kWinRows * 8 : 0)));
    if (rank == 0) mbar_expect_tx(smem_u32(&f.votes_bar), (uint32_t)((tiles - n_t) * vote_bytes));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of the Q tile beyond R are never written by TMA: keep them zero
  if (a.R != 128) {
    for (int i = tid; i < a.halves * q_half / 16; i += kThreads) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&f.tmem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = f.tmem;
  // Barriers of the cluster, which every thread passes whatever happens: 0 everybody is there, 1 kept positions, 2 nobody reads
  // another CTA's memory any more.  Row sums and votes are waited for where they arrive.
  cluster_arrive();                                                                        // 0

  if (warp == 0) {
    // ---- loads.  Tile i of the CTA lies in stage i % n_stages; the statistics pass takes the tiles in order, the vote pass
    // backwards, so that the last n_stages tiles are there already.
    bool ok = true;
    auto load = [&](int i) {
      const int st = i % a.n_stages, tok = x.t0 + (first + i) * kTileKeys;
      const uint32_t dst = k_sh + (uint32_t)(st * stage_bytes);
      mbar_expect_tx(full(st), (uint32_t)stage_bytes);
      const int ky = a.k_head_inner ? x.g : tok, kz = a.k_head_inner ? tok : x.g;
      for (int h = 0; h < a.halves; ++h) tma_load_3d(dst + h * kHalfBytes, &a.tm_k, 64 * h, ky, kz, full(st));
    };
    if (lane == 0 && n_t > 0) {
      pdl_wait();
      mbar_expect_tx(q_full, (uint32_t)(a.halves * a.R * 128));
      const int q_y = a.q_head_inner ? x.g * a.G : 0, q_z = a.q_head_inner ? 0 : x.g * a.G;
      for (int h = 0; h < a.halves; ++h) tma_load_4d(q_sh + h * q_half, &a.tm_q, 64 * h, q_y, q_z, x.s, q_full);
      for (int j = 0; j < n_t && ok; ++j) {                  // votes alone: backwards from the start
        const int i = stats ? j : n_t - 1 - j;
        if (j >= a.n_stages) ok = mbar_wait(empty(i % a.n_stages), (stats ? i / a.n_stages - 1 : ring.uses(i % a.n_stages) - 2 - i / a.n_stages) & 1, abort_flag);
        if (ok) load(i);
      }
    }
    if (lane == 0 && n_t > 0 && stats)
      for (int i = n_t - 1 - a.n_stages; i >= 0 && ok; --i) {
        const int st = i % a.n_stages, uses = ring.uses(st), q = i / a.n_stages;
        ok = mbar_wait(empty(st), (2 * uses - q - 3) & 1, abort_flag);
        if (ok) load(i);
      }
    if (lane == 0 && n_t > 0 && (!ok || *abort_flag)) {
      // loads in flight get a bounded chance to land before the CTA's shared memory goes away
      const unsigned long long t0 = now_ns();
      while (now_ns() - t0 < 2000000ull) {}
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- products: statistics D[row, key] = Q K^T, votes D[key, row] = K Q^T
    const uint32_t idesc_s = instr_desc(128, kTileKeys), idesc_v = instr_desc(kTileKeys, a.Rp);
    const uint64_t qd = smem_desc(q_sh), kd0 = smem_desc(k_sh), q_hi = (uint64_t)(q_half >> 4), k_hi = (uint64_t)(kHalfBytes >> 4);
    bool ok = true;
    int uc = 0;
    auto product = [&](int i, int nth_fill, bool votes) {
      const int st = i % a.n_stages;
      ok = mbar_wait(full(st), nth_fill & 1, abort_flag) && mbar_wait(unit_empty(uc & 3), ((uc >> 2) & 1) ^ 1, abort_flag);
      if (!ok) return;
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)((uc & 3) * 128);
      const uint64_t kd = kd0 + (uint64_t)((st * stage_bytes) >> 4);
      const uint64_t ad = votes ? kd : qd, bd = votes ? qd : kd, a_hi = votes ? k_hi : q_hi, b_hi = votes ? q_hi : k_hi;
      const uint32_t idesc = votes ? idesc_v : idesc_s;
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) tc_mma(d, ad + (uint64_t)(ks * 2), bd + (uint64_t)(ks * 2), idesc, ks > 0);
      if (a.halves == 2) {
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) tc_mma(d, ad + a_hi + (uint64_t)(ks * 2), bd + b_hi + (uint64_t)(ks * 2), idesc, 1);
      }
      // a stage's completions are the ones its next load waits for, each before the next can come: the statistics of the
      // tiles that stay are none
      if (votes || i + a.n_stages < n_t) tc_commit(empty(st));
      tc_commit(unit_full(uc & 3));
      ++uc;
    };
    if (lane == 0 && n_t > 0) {
      ok = mbar_wait(q_full, 0, abort_flag);
      if (stats)
        for (int i = 0; i < n_t && ok; ++i) product(i, i / a.n_stages, false);
    }
    if (lane == 0 && n_t > 0) {
      for (int i = n_t - 1; i >= 0 && ok; --i) {
        const int uses = ring.uses(i % a.n_stages), q = i / a.n_stages;
        product(i, !stats ? uses - 1 - q : (q == uses - 1 ? q : 2 * uses - 2 - q), true);
      }
      if (!ok || *abort_flag) {
        // gave up: the MMAs issued must be through before the accumulators are released
        tc_commit(drain);
        const unsigned long long t0 = now_ns();
        while (!mbar_try(drain, 0) && now_ns() - t0 < kWaitLimitNs) {}
      }
    }
    __syncwarp();
  } else if (warp < 4) {
    if (warp == 2) {
      pdl_wait();
      const SegmentRows r = segment_rows(a.tail, x);
      if (lane == 0) f.rows = r;
      __syncwarp();
      asm volatile("bar.sync 3, %0;" ::"n"(kLayerThreads + 32) : "memory");
    }
  } else {
    const int t = tid - 128, wg = t >> 7, row = t & 127;
    float* votes = f.votes_mem + kLead;
    auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(kLayerThreads) : "memory"); };
    Unit u;
    u.tcol = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(wg * 128);
    u.full = unit_full(wg);
    u.empty = unit_empty(wg);
    u.abort_flag = abort_flag;
    pdl_wait();
    if (stats) {
      // the window keys' statistics, 16 rows at a time, while the keys are on their way (in the votes' memory)
      const bool win = a.all_causal && x.n > 0;
      if (win && wg == 0)
        for (int b = rank; b < window_blocks; b += CS) {
          auto out = [&](int r, float m, float z) { f.win[r] = make_float2(m, z); };
          if (a.halves == 2) window_rows<__nv_bfloat16, 128, 2>(a.win, f.votes_mem, t, x.s, x.g, x.t0 + x.n, b * kWinRows, out);
          else window_rows<__nv_bfloat16, 64, 2>(a.win, f.votes_mem, t, x.s, x.g, x.t0 + x.n, b * kWinRows, out);
          asm volatile("bar.sync 2, 128;" ::: "memory");
        }
      double z;
      float far_z, far_m;
      stats_run<false>(u, 0, a.scale_log2, wg, 4, n_t, x.n - first * kTileKeys, (warp & 3) * 32 < a.R, z, far_z, far_m);
      f.z_wg[wg][row] = z;
      f.far_wg[wg][row] = make_float2(far_z, far_m);
      if (far_z > 0.f) f.far_here = 1;
      sync();
      const bool far = f.far_here != 0;
      if (wg == 0) {
        f.all[rank].z[row] = (f.z_wg[0][row] + f.z_wg[1][row]) + (f.z_wg[2][row] + f.z_wg[3][row]);
        if (row == 0) f.all[rank].far = far;
        if (far) {
          float fz = 0.f, fm = 0.f;
          for (int w = 0; w < 4; ++w) stat_add(fz, fm, f.far_wg[w][row].x, f.far_wg[w][row].y);
          f.far[row] = make_float2(fz, fm);
          asm volatile("fence.acq_rel.cluster;" ::: "memory");                             // read by the others once they have `far`
        }
        publish_for_copy();
        cluster_wait();                                                                    // 0
        asm volatile("bar.sync 2, 128;" ::: "memory");
        if (t < CS && t != rank) {
          copy_to_cta(&f.all[rank], &f.all[rank], sizeof(f.all[0]), &f.sums_bar, t);
          if (win)
            for (int b = rank; b < window_blocks; b += CS) copy_to_cta(&f.win[b * kWinRows], &f.win[b * kWinRows], kWinRows * 8, &f.sums_bar, t);
        }
        mbar_wait(smem_u32(&f.sums_bar), 0, abort_flag);
      } else {
        cluster_wait();                                                                    // 0
      }
      if (wg == 0) {
        float l2 = INFINITY;                                   // rows of padding: 2^(0 - inf) = 0
        if (row < a.R) {
          double Z = 0.0;
          bool any_far = false;
          for (int c = 0; c < CS; ++c) { Z += f.all[c].z[row]; any_far |= f.all[c].far != 0; }
          if (!any_far && !win) {
            l2 = log2_of(Z);
          } else {                                             // as row_lse
            float sz = 0.f, sm = 0.f;
            if (Z > 0.0) {
              sm = (float)((__double2hiint(Z) >> 20) - 1023);
              sz = (float)__hiloint2double((__double2hiint(Z) & 0xfffff) | 0x3ff00000, __double2loint(Z));
            }
            for (int c = 0; c < CS; ++c)
              if (f.all[c].far) {
                const float2 o = *cluster.map_shared_rank(&f.far[row], c);
                stat_add(sz, sm, o.x, o.y);
              }
            if (win) stat_add(sz, sm, f.win[row].y, f.win[row].x);
            l2 = __fadd_rn(sm, log2f(sz));
          }
        }
        f.lse[row] = -l2;
      }
    } else {
      if (wg == 0) f.lse[row] = row < a.R ? -a.lse.caller_lse(x.s, x.g, row, a.G, a.tail.window, a.q_head_inner != 0) : -INFINITY;
      cluster_wait();                                                                      // 0
    }
    const float pad = a.tail.pool_mode == SLKV_POOL_MAX ? -INFINITY : 0.f;
    if (rank == 0 && wg == 1 && row < 8) {
      const int p = row < 4 ? row - 4 : x.n + row - 4;
      votes[vote_at<IT>(p)] = pad;
    }
    sync();
    {
      const int j0 = (wg - (stats ? n_t : 0)) & 3, nth = stats && wg < n_t ? ((n_t - 1 - wg) >> 2) + 1 : 0;
      const int n_here = x.n - first * kTileKeys;
      votes_run(u, nth, a.scale_log2, j0, 4, n_t, 0x7fffffff, smem_u32(f.lse), a.Rp, -1, nullptr, 0u, 0, 1.0f / (float)a.G,
                [&](int j, float v) {
                  const int key = (n_t - 1 - (j >> 7)) * kTileKeys + (j & 127);
                  votes[vote_at<IT>(first * kTileKeys + key)] = key < n_here ? v : pad;
                });
      publish_for_copy();
    }
    // with warp 2: a CTA without tiles may be here before the budgets are
    asm volatile("bar.sync 3, %0;" ::"n"(kLayerThreads + 32) : "memory");
    if (rank == 0) {
      mbar_wait(smem_u32(&f.votes_bar), 0, abort_flag);
    } else if (t == 0 && n_t > 0) {
      float* mine = votes + vote_at<IT>(first * kTileKeys);
      copy_to_cta(mine, mine, n_t * vote_bytes, &f.votes_bar, 0);
    }
    const SegmentRows r = f.rows;
    if (rank == 0) layer_select<IT, 1>(a.tail, x, r.k_keep, votes, *reinterpret_cast<SelShared*>(smem), t, abort_flag);
    cluster_arrive();                                                                      // 1
    cluster_wait();
    if (a.tail.select) layer_gather(a.tail, x, r, reinterpret_cast<const int*>(cluster.map_shared_rank(f.votes_mem, 0)), t, rank, CS);
  }
  if (warp < 4) {
    cluster_wait();                                                                        // 0
    cluster_arrive();                                                                      // 1
    cluster_wait();
  }
  tc_fence_before();
  cluster_arrive();                                                                        // 2
  cluster_wait();
  tc_fence_after();
  if (f.abort_flag && tid == 0 && a.status) atomicExch(a.status, (int)SLKV_ERR_DEVICE_TIMEOUT);
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

typedef void (*Kern)(const LayerArgs);
template <int IT> size_t layer_smem(int halves, int stages) { return (size_t)halves * 128 * 128 + (size_t)stages * halves * kHalfBytes + sizeof(Far<IT>); }
template <int IT> int layer_stages(int halves) {
  const int n = (int)((kSmemLimit - layer_smem<IT>(halves, 0)) / (halves * kHalfBytes));
  return n < kMaxStages ? n : kMaxStages;
}

cudaError_t configure() {
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || configured_dev == dev) return e;
  for (Kern k : {k_layer_tc<8>, k_layer_tc<16>}) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  configured_dev = dev;
  return e;
}

// Clusters of cs CTAs that run at the same time on the current device.
int clusters_at_once(int cs) {
  static thread_local int dev_known = -1, known[kLayerMaxCluster + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev != dev_known) {
    for (int c = 2; c <= kLayerMaxCluster; ++c) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)c);
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = layer_smem<16>(2, layer_stages<16>(2));
      cudaLaunchAttribute attr;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = (unsigned)c; attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&known[c], k_layer_tc<16>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();                        // not a sticky error
        known[c] = 0;
      }
    }
    dev_known = dev;
  }
  return known[cs];
}

}  // namespace

// The largest cluster, two CTAs at least, of which n_seg run at the same time, an SM for each CTA; 0: none.
int layer_tc_clusters_for(int n_seg) {
  if (configure() != cudaSuccess) return 0;
  for (int cs = kLayerMaxCluster; cs >= 2; --cs)
    if (n_seg <= clusters_at_once(cs)) return cs;
  return 0;
}

// CTAs per segment, 0: the shape is not taken.  The largest cluster of which there is one for every segment at the same time
// (eight segments: of ten CTAs; sixteen: of six), two CTAs at least: the clusters run on n_seg * CS SMs and as long as the longest
// segment's, while the general path spreads a layer's tiles over all SMs but takes three launches and exchanges through memory,
// some 8 us.  A tile costs a CTA 1.1 us here, one of an even share over all SMs 0.8 there, so as many of the first as make up for
// the launches may stand over three quarters of the second; fewer where there is less to save -- the scores alone take two launches,
// log-sum-exps handed in the exchange.  Measured both ways, 99 to 276 shapes of each kind that are taken: slower from a stream by 1.5
// us at most (layers), 1.2 (scores), 3.7 and 1.0 (with log-sum-exps: 32 heads of 7000 tokens, 16 rows, 26.9 against 23.3).  One
// layer of head_dim 128 and 128 rows, us in a graph / from a stream, here and on the general path (r: lengths from half to the
// whole; -: not taken):
//   segments   2000 tokens            4000 tokens            6000 tokens            8100 tokens
//   2          12.0/13.0  16.8/21.2   15.0/15.7  17.8/22.6   18.4/19.1  18.4/22.7   21.1/21.9  19.5/24.7
//   8          13.3/13.7  19.0/23.3   16.0/16.4  21.3/24.7   19.6/20.2  23.6/26.8   22.5/23.1  25.4/28.8
//   16         14.8/15.4  22.9/26.8   19.5/20.2  24.9/28.2   24.1/24.9  28.2/31.0   28.4/29.3  30.5/33.4
//   32         20.6/21.5  25.8/29.0   27.4/28.3  30.6/33.2   34.8/35.5  35.3/39.0   41.2/41.6  38.7/41.9
//   40         19.3/20.0  27.6/30.9   27.5/28.3  33.2/36.7   36.4/37.2  36.0/39.1   44.5/45.1  43.7/47.2
//   40 r       18.8/19.7  26.1/28.9   27.0/27.7  30.3/33.0   35.9/36.7  35.0/38.8   43.2/44.2  37.6/41.2 -
//   64         24.2/25.1  32.0/35.1   36.4/37.1  37.7/41.2   49.3/49.8  51.7/55.2   61.9/62.4  62.6/65.7 -
//   64 r       23.5/24.4  30.1/33.0   35.3/36.1  36.9/40.7   47.5/48.4  41.5/45.2 - 60.4/61.6  52.4/55.5 -
// and with 16 rows 8 x 8100 19.5/20.1 23.7/26.9, 64 x 8100 57.7/58.2 55.4/58.3 -, 64 r x 8100 55.2/56.2 45.1/48.5 -.
// More segments than clusters: two rounds (16 segments of 1000 tokens in clusters of eight 24.1, of four 14.0).
int layer_tc_cluster(const Problem& pb, bool select) {
  const slkv_params& p = pb.p;
  if (!tensor_path_supported(p) || pb.R > 128 || (p.pool_kernel >> 1) > kMaxRadius || p.history_only || pb.tab.n_inline == 0 ||
      pb.max_hist < 1 || pb.max_hist > 16 * kLayerThreads)
    return 0;
  const int cs = layer_tc_clusters_for(pb.n_seg), tiles = (pb.max_hist + kTileKeys - 1) / kTileKeys;
  const double over = pb.lse_opt ? (select ? 5.5 : 4.0) : (select ? 9.5 : 7.5);
  return cs >= 2 && (tiles + cs - 1) / cs <= over + 0.75 * (double)pb.n_tiles128 / sm_count() ? cs : 0;
}

cudaError_t launch_layer_tc(const Problem& pb, int cs, const TailLayer* tail, float* pooled, int32_t* status, cudaStream_t st,
                            int* launches) {
  cudaError_t e = configure();
  if (e != cudaSuccess) return e;
  ScoreLayer lay;
  e = plan_score_layer(pb, status, &lay);
  if (e != cudaSuccess) return e;
  const slkv_params& p = pb.p;
  LayerArgs a;
  a.tm_q = lay.tm_q; a.tm_k = lay.tm_k;
  a.tail = layer_tail(pb, tail, pooled);
  a.lse = lay.lse;
  a.q_head_inner = tensor_q_head_inner(p) ? 1 : 0;
  a.k_head_inner = p.k_stride_head <= p.k_stride_tok;
  a.win = window_args(pb, a.q_head_inner != 0);
  a.passes = pb.lse_opt ? 2 : 3;
  a.all_causal = !pb.lse_opt && p.softmax_domain == SLKV_ALL_CAUSAL;
  a.G = pb.G; a.R = pb.R; a.Rp = (pb.R + 31) / 32 * 32;
  a.halves = p.head_dim / 64;
  a.scale_log2 = kLog2e / sqrtf((float)p.head_dim);
  a.status = status;
  a.expire = take_expire_next_layer_wait(a.passes == 3);
  const bool small = pb.max_hist <= 8 * kLayerThreads;
  a.n_stages = small ? layer_stages<8>(a.halves) : layer_stages<16>(a.halves);
  const size_t smem = small ? layer_smem<8>(a.halves, a.n_stages) : layer_smem<16>(a.halves, a.n_stages);
  LaunchScope scope(KID_LAYER, st, launches);
  return launch_pdl(small ? k_layer_tc<8> : k_layer_tc<16>, dim3((unsigned)(pb.n_seg * cs)), dim3(kThreads), smem, st, cs, a);
}

}  // namespace slkv

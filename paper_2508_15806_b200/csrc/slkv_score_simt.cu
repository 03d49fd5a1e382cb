// Window relevance scores with fp32 FMA arithmetic (Sec. 3.4, Eq. 7; Algorithm 3 l.6; Eq. 3-4).
//
// Serves the fp32 configuration and every shape the tensor-core kernel does not take.  A register-tiled product: a CTA of
// 256 threads forms 64 keys x 64 rows of scores at a time, 4 x 4 per thread in packed pairs (fma.rn.f32x2) over the head
// dimension, K and Q as fp32 rows in shared memory, padded so that the 16-byte loads of a warp -- eight key groups, four row
// groups -- are one wavefront each; eight of those feed 64 multiply-adds.  Persistent CTAs walk the segments' key tiles:
//   statistics  row sums of 2^score per 32 keys, added up in fp64 with atomics (exact, whatever the order, where n such
//               sums are within a factor 2^29 / n of one another; else the same to 2^-53 times a few); nothing is subtracted unless a sum over- or underflows, in which case every CTA learns so at
//               the barrier and two more rounds find the rows' maxima and sum relative to them;
//   votes       vote[j] = (1/G) sum_rows 2^(s_rj - lse_r), rows in a fixed order.
// Both passes are one cooperative launch with a grid-wide barrier between them; score tiles that fit in shared memory are
// kept over the barrier instead of being formed again.
// What bounds it: latency at the small sizes (1024 tokens, 8 heads, 16 rows: two dot-product loops of one thread per key and
// two launches took 80 us, this takes 10), the FMA pipe at the large ones.
#include "slkv_internal.cuh"
#include "slkv_fma_device.cuh"

namespace slkv {
namespace {

constexpr int kThreads = 256;
constexpr int kKeys = 64;              // keys per tile
constexpr int kRows = 64;              // rows per step
constexpr int kSmemMost = 200 * 1024;
constexpr unsigned long long kWaitLimitNs = 1000ull * 1000ull * 1000ull;

// stages of a launch
enum { kStats = 1, kMaxima = 2, kFarSums = 4, kVotes = 8 };

// The statistics area (pb.part): per segment and row the fp64 sum, then the same over relative to the row's maximum, then
// the maxima (order-preserving integers), then one word: some sum over- or underflowed.  Cleared before use.
struct SimtStats {
  double* acc;
  double* acc_far;
  unsigned* row_max;
  unsigned* far;
};
size_t simt_stat_bytes(int n_seg, int R) { return (size_t)n_seg * R * 20 + 8; }
__host__ __device__ __forceinline__ SimtStats simt_stats(void* part, int n_seg, int R) {
  SimtStats s;
  s.acc = static_cast<double*>(part);
  s.acc_far = s.acc + (size_t)n_seg * R;
  s.row_max = reinterpret_cast<unsigned*>(s.acc_far + (size_t)n_seg * R);
  s.far = s.row_max + (size_t)n_seg * R;
  return s;
}
// order-preserving map of floats to unsigned integers; 0 is below every float
__device__ __forceinline__ unsigned ordered(float x) {
  const unsigned u = __float_as_uint(x);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unordered(unsigned u) { return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u); }

// Row log-sum-exp (log2 units), the window keys' statistics folded in when there are any (softmax over all causally
// visible keys).  The same operations in every kernel that forms it.
__device__ __forceinline__ float simt_row_lse(const SimtStats& st, size_t at, bool far, bool has_win, float wm, float wz) {
  float M = far ? unordered(__ldcg(st.row_max + at)) : 0.f;
  double Z = __ldcg((far ? st.acc_far : st.acc) + at);
  if (has_win) {
    const float Mn = fmaxf(M, wm);
    Z = __dadd_rn(__dmul_rn(Z, (double)exp2f(M - Mn)), __dmul_rn((double)wz, (double)exp2f(wm - Mn)));
    M = Mn;
  }
  return __fadd_rn(M, (float)log2(Z));
}

// The clearing of the statistics: a flag per CTA, the launch's tag once the CTA has cleared its share.  A CTA takes its flag
// back at its end: all are past barrier 1 then, and so have seen it.  One counter, as the tensor-core kernel has it, would
// have to be given its tag first, an atomic's round trip in front of a chain this short: fp32 layers of 400 - 3000 tokens took
// 23.0 instead of 21.9 us on average.
struct FlagSync {
  unsigned long long* flags;   // [kSyncFlags], 16-byte aligned, then the barriers' counts
  unsigned long long tag;
  unsigned expect;             // CTAs to wait for: all of them
  __device__ __forceinline__ unsigned* counts() const { return reinterpret_cast<unsigned*>(flags + kSyncFlags); }
  // This CTA has cleared its share (one thread, behind a barrier with those that did).
  __device__ __forceinline__ void arrive() const {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(flags + blockIdx.x), "l"(tag) : "memory");
  }
  // All CTAs have cleared theirs (a whole warp asks): all loads in flight at once.
  __device__ __forceinline__ bool all_arrived() const {
    unsigned long long f[kSyncFlags / 32];
    const unsigned n = gridDim.x, i0 = 2 * (threadIdx.x & 31);
#pragma unroll
    for (int k = 0; k < kSyncFlags / 64; ++k) {
      f[2 * k] = f[2 * k + 1] = tag;
      if (i0 + 64 * k < n)
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(f[2 * k]), "=l"(f[2 * k + 1]) : "l"(flags + i0 + 64 * k) : "memory");
    }
    bool here = expect <= n;
#pragma unroll
    for (int k = 0; k < kSyncFlags / 64; ++k) here = here && f[2 * k] == tag && (f[2 * k + 1] == tag || i0 + 64 * k + 1 == n);
    if (!__all_sync(0xffffffffu, here)) return false;
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return true;
  }
  __device__ __forceinline__ void take_back() const { flags[blockIdx.x] = 0; }
};

struct SimtArgs {
  SeqTables tab;
  const void* q;
  const void* k;
  void* part;
  float* vote;
  LseSource lse;
  int32_t* status;
  int n_seqs, n_kv_heads, G, window, R, n_tiles, keep, q_rows, stages, coop;
  unsigned barrier_target;     // arrivals that end the wait at barrier 1: the CTAs
  long long k_stride_tok, k_stride_head, q_stride_seq, q_stride_row, q_stride_head;
  float scale_log2;
  FlagSync sync;               // counts 0 .. 2: arrivals at the barriers 1 .. 3
};
constexpr int kBarriers = 3;

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Until all CTAs have cleared their part, the barriers' counts included (a whole warp waits; false when the wait ran out).
__device__ __forceinline__ bool cleared_wait(const SimtArgs& a) {
  unsigned long long t0 = 0;
  for (unsigned spin = 0; !a.sync.all_arrived(); ++spin) {
    if (spin == 0) t0 = now_ns();
    if (__any_sync(0xffffffffu, now_ns() - t0 > kWaitLimitNs)) {
      if (a.status && (threadIdx.x & 31) == 0) atomicExch(a.status, (int)SLKV_ERR_DEVICE_TIMEOUT);
      return false;
    }
    __nanosleep(20);
  }
  return true;
}
// Waits, in one thread, until a count has reached `target`.
__device__ __forceinline__ bool count_wait(const SimtArgs& a, const unsigned* count, unsigned target) {
  unsigned long long t0 = 0;
  for (unsigned spin = 0;; ++spin) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
    if (v >= target) return true;
    if (spin == 0) t0 = now_ns();
    if (now_ns() - t0 > kWaitLimitNs) {
      if (a.status) atomicExch(a.status, (int)SLKV_ERR_DEVICE_TIMEOUT);
      return false;
    }
    __nanosleep(20);
  }
}
// Arrives at barrier number b (1 .. 3) of the launch and waits for all CTAs (bounded: false when the wait ran out).
// cleared: this warp has waited for the clearing; stuck: its wait for that ran out, so that something is missing from the sums.
__device__ __forceinline__ bool grid_wait(const SimtArgs& a, int b, unsigned target, bool cleared, bool stuck) {
  __shared__ int ok_sh;
  if (__syncthreads_or(stuck)) return false;
  if (threadIdx.x < 32) {
    bool ok = cleared || cleared_wait(a);
    if (ok && threadIdx.x == 0) {
      unsigned* count = a.sync.counts() + b - 1;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
      ok = count_wait(a, count, target);
    }
    if (threadIdx.x == 0) ok_sh = ok;
  }
  __syncthreads();
  return ok_sh != 0;
}

template <typename T, int D>
struct Tiles {
  static constexpr int kVec = 16 / sizeof(T);                  // elements of a 16-byte load
  static constexpr int kPitch = D + 4;                         // floats per row in shared memory
  static constexpr int kPerRow = D / kVec;                     // 16-byte loads per row
  static constexpr int kLoads = kKeys * kPerRow / kThreads;    // ... per thread for a key tile
};

// Where a tile of the flat list lies.
struct Place { int seg, s, g, tile, n_hist, key0, t0; };
__device__ __forceinline__ Place place_of(const SimtArgs& a, int t) {
  // tile_off of the tables counts 128-key tiles; here a sequence has two of these per such tile
  int lo = 0, hi = a.n_seqs;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (2 * a.n_kv_heads * a.tab.tile_at(mid) <= t) lo = mid; else hi = mid;
  }
  Place p;
  p.s = lo;
  const int per_head = 2 * (a.tab.tile_at(lo + 1) - a.tab.tile_at(lo));
  const int rel = t - 2 * a.n_kv_heads * a.tab.tile_at(lo);
  p.g = rel / per_head;
  p.tile = rel - p.g * per_head;
  p.seg = p.s * a.n_kv_heads + p.g;
  p.t0 = a.tab.cu_at(lo);
  p.n_hist = max(a.tab.cu_at(lo + 1) - p.t0 - a.window, 0);
  p.key0 = p.tile * kKeys;                                     // may lie past the end: nothing valid then
  return p;
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads, 2)
k_score_simt(const __grid_constant__ SimtArgs a) {
  using TT = Tiles<T, D>;
  extern __shared__ __align__(16) float smem[];
  float* ks = smem;                                            // [kKeys][kPitch]
  float* qs = ks + kKeys * TT::kPitch;                         // [q_rows][kPitch]
  float* lse_sh = qs + a.q_rows * TT::kPitch;                  // [chunks * kRows]
  const int chunks = (a.R + kRows - 1) / kRows;
  float* part_sh = lse_sh + chunks * kRows;                    // [4][kKeys]
  float* kept = part_sh + 4 * kKeys;                           // [keep][chunks][16][kThreads]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kw = (warp & 1) * 32 + (lane & 7), rw = (warp >> 1) * 16 + (lane >> 3);   // keys kw + 8 i, rows rw + 4 j
  const T* q = static_cast<const T*>(a.q);
  const T* k = static_cast<const T*>(a.k);
  const int n_seg = a.n_seqs * a.n_kv_heads;
  const SimtStats st = simt_stats(a.part, n_seg, a.R);
  const int begin = (int)((long long)blockIdx.x * a.n_tiles / gridDim.x), end = (int)((long long)(blockIdx.x + 1) * a.n_tiles / gridDim.x);
  pdl_launch_dependents();
  pdl_wait();

  if (a.coop) {
    // clear the statistics area and the barriers' counts; nobody adds to them before all CTAs have done their part
    const long long words = (long long)n_seg * a.R * 5 + 2;            // may be more than 2^31
    const long long w0 = blockIdx.x * words / gridDim.x, w1 = (blockIdx.x + 1) * words / gridDim.x;
    for (long long i = w0 + tid; i < w1; i += kThreads) __stcg(static_cast<unsigned*>(a.part) + i, 0u);
    if (blockIdx.x == 0 && tid < kBarriers) __stcg(a.sync.counts() + tid, 0u);
    __syncthreads();
    if (tid == 0) a.sync.arrive();
  }

  int q_seg = -1, q_chunk = -1;                                // what qs holds (q_chunk when it holds one step's rows)
  auto load_q = [&](const Place& p, int chunk) {
    const bool all = a.q_rows >= chunks * kRows;
    if (p.seg == q_seg && (all || chunk == q_chunk)) return;
    __syncthreads();
    const int r0 = all ? 0 : chunk * kRows, n = all ? chunks * kRows : kRows;
    for (int i = tid; i < n * TT::kPerRow; i += kThreads) {
      const int rr = i / TT::kPerRow, c = i - rr * TT::kPerRow, r = r0 + rr;
      float f[TT::kVec];
#pragma unroll
      for (int e = 0; e < TT::kVec; ++e) f[e] = 0.f;
      if (r < a.R) {                                           // row r = hh*window + i: query head g*G + hh, window row i
        const int hh = r / a.window, wi = r - hh * a.window;
        const T* src = q + p.s * a.q_stride_seq + wi * a.q_stride_row + (long long)(p.g * a.G + hh) * a.q_stride_head + c * TT::kVec;
        unpack(*reinterpret_cast<const uint4*>(src), f, T());
      }
#pragma unroll
      for (int e = 0; e < TT::kVec; e += 4)
        *reinterpret_cast<float4*>(qs + rr * TT::kPitch + c * TT::kVec + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
    }
    q_seg = p.seg;
    q_chunk = chunk;
    __syncthreads();
  };
  uint4 kreg[TT::kLoads];
  auto fetch_k = [&](int t) {                                  // a tile's keys on their way into registers
    const Place p = place_of(a, t);
#pragma unroll
    for (int u = 0; u < TT::kLoads; ++u) {
      const int i = tid + u * kThreads, row = i / TT::kPerRow, c = i - row * TT::kPerRow, j = p.key0 + row;
      kreg[u] = j < p.n_hist ? *reinterpret_cast<const uint4*>(k + (long long)(p.t0 + j) * a.k_stride_tok +
                                                               (long long)p.g * a.k_stride_head + c * TT::kVec)
                             : make_uint4(0, 0, 0, 0);
    }
  };
  auto store_k = [&]() {
    __syncthreads();                                           // everybody is done with the tile before
#pragma unroll
    for (int u = 0; u < TT::kLoads; ++u) {
      const int i = tid + u * kThreads, row = i / TT::kPerRow, c = i - row * TT::kPerRow;
      float f[TT::kVec];
      unpack(kreg[u], f, T());
#pragma unroll
      for (int e = 0; e < TT::kVec; e += 4)
        *reinterpret_cast<float4*>(ks + row * TT::kPitch + c * TT::kVec + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
    }
    __syncthreads();
  };
  // scores in log2 units: s[i][j] of key kw + 8 i and row chunk * 64 + rw + 4 j
  float s[4][4];
  auto scores = [&](int chunk) {
    const float* kp = ks + kw * TT::kPitch;
    const float* qp = qs + ((a.q_rows >= chunks * kRows ? chunk * kRows : 0) + rw) * TT::kPitch;
    f32x2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      ulonglong2 kv[4], qv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) kv[i] = *reinterpret_cast<const ulonglong2*>(kp + i * 8 * TT::kPitch + c);
#pragma unroll
      for (int j = 0; j < 4; ++j) qv[j] = *reinterpret_cast<const ulonglong2*>(qp + j * 4 * TT::kPitch + c);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fma2(kv[i].x, qv[j].x, acc[i][j]);
          acc[i][j] = fma2(kv[i].y, qv[j].y, acc[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = sum_of(acc[i][j]) * a.scale_log2;
  };
  bool cleared = !a.coop, stuck = false;
  // one round over this CTA's tiles: stage is one of the enum's
  auto round = [&](int stage) {
    const bool far = stage == kVotes && !a.lse.lse_opt && __ldcg(st.far) != 0;
    int lse_seg = -1;
    for (int t = begin; t < end; ++t) {
      const Place p = place_of(a, t);
      const int slot = t - begin;
      const bool have = slot < a.keep && stage != kStats;       // the scores are still there
      if (!have) {
        if (t == begin || (slot == a.keep && stage != kStats)) fetch_k(t);
        store_k();
        if (t + 1 < end) fetch_k(t + 1);
      }
      if (p.key0 >= p.n_hist) continue;                         // the padding half of a 128-key tile
      if (stage == kVotes && p.seg != lse_seg) {
        __syncthreads();
        for (int r = tid; r < chunks * kRows; r += kThreads) {
          float l2 = INFINITY;                                  // rows of padding count nothing
          if (r < a.R) {
            const size_t at = (size_t)p.seg * a.R + r;
            const bool has_win = a.lse.win_m != nullptr;
            l2 = a.lse.lse_opt ? a.lse.caller_lse(p.s, p.g, r, a.G, a.window, false)
                               : simt_row_lse(st, at, far, has_win, has_win ? a.lse.win_m[at] : 0.f, has_win ? a.lse.win_z[at] : 0.f);
          }
          lse_sh[r] = l2;
        }
        lse_seg = p.seg;
        __syncthreads();
      }
      float vote = 0.f;                                         // threads 0..63: key tid
      for (int chunk = 0; chunk < chunks; ++chunk) {
        float* mine = kept + ((size_t)slot * chunks + chunk) * 16 * kThreads + tid;
        if (have) {
#pragma unroll
          for (int e = 0; e < 16; ++e) s[e >> 2][e & 3] = mine[e * kThreads];
        } else {
          load_q(p, chunk);
          if (chunk * kRows + (warp >> 1) * 16 < a.R) scores(chunk);      // else no row of this warp exists
          if (slot < a.keep)
#pragma unroll
            for (int e = 0; e < 16; ++e) mine[e * kThreads] = s[e >> 2][e & 3];
        }
        const int row0 = chunk * kRows + rw;
        if (stage == kVotes) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float v = 0.f;
            if (chunk * kRows + (warp >> 1) * 16 < a.R)
#pragma unroll
              for (int j = 0; j < 4; ++j) v += exp2f(s[i][j] - lse_sh[row0 + 4 * j]);
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (lane < 8) part_sh[(warp >> 1) * kKeys + kw + 8 * i] = v;
          }
          __syncthreads();
          if (tid < kKeys) vote += (part_sh[tid] + part_sh[kKeys + tid]) + (part_sh[2 * kKeys + tid] + part_sh[3 * kKeys + tid]);
          __syncthreads();
        } else if (chunk * kRows + (warp >> 1) * 16 < a.R) {
          if (!cleared) {                                       // uniform over the warp
            if (!stuck) cleared = cleared_wait(a);
            stuck = !cleared;
          }
#pragma unroll
          for (int j = 0; j < 4 && cleared; ++j) {
            const int row = row0 + 4 * j;
            const size_t at = (size_t)p.seg * a.R + min(row, a.R - 1);
            float v = stage == kMaxima ? -INFINITY : 0.f;
            const float ref = stage == kFarSums ? unordered(__ldcg(st.row_max + at)) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (p.key0 + kw + 8 * i >= p.n_hist) continue;
              v = stage == kMaxima ? fmaxf(v, s[i][j]) : v + exp2f(s[i][j] - ref);
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
              const float w = __shfl_xor_sync(0xffffffffu, v, o);
              v = stage == kMaxima ? fmaxf(v, w) : v + w;
            }
            // the keys of this half-tile may all lie past the end
            if ((lane & 7) != 0 || row >= a.R || p.key0 + (warp & 1) * 32 >= p.n_hist) continue;
            if (stage == kStats) {
              if (v < INFINITY && v > 1e-30f) atomicAdd(st.acc + at, (double)v);
              else atomicOr(st.far, 1u);
            } else if (stage == kMaxima) {
              atomicMax(st.row_max + at, ordered(v));
            } else {
              atomicAdd(st.acc_far + at, (double)v);
            }
          }
        }
      }
      if (stage == kVotes && tid < kKeys && p.key0 + tid < p.n_hist)
        a.vote[a.tab.hist_at(p.s) * a.n_kv_heads + (long long)p.g * p.n_hist + p.key0 + tid] = vote / (float)a.G;
    }
  };

  bool ok = true;
  if (a.stages & kStats) round(kStats);
  if (a.coop) ok = grid_wait(a, 1, a.barrier_target, cleared, stuck);
  if (ok && (a.stages & (kMaxima | kFarSums)) && __ldcg(st.far) != 0) {     // the same for every CTA: all sums are in
    if (a.stages & kMaxima) round(kMaxima);
    if (a.coop) ok = grid_wait(a, 2, gridDim.x, true, false);
    if (ok && (a.stages & kFarSums)) round(kFarSums);
    if (a.coop && ok) ok = grid_wait(a, 3, gridDim.x, true, false);
  }
  if (ok && (a.stages & kVotes)) round(kVotes);
  if (a.coop && tid == 0) a.sync.take_back();
}

// Row statistics over the window keys a window row sees causally (its own position and the window keys before it).
// Only the all-causal softmax domain needs them.  A CTA takes 16 rows of a segment (window_rows).  (One thread per row walking
// the keys by itself, one CTA per segment, took 24 us for 8 segments of 128 rows and 32 window keys; this takes 4.)
template <typename T, int D>
__global__ void __launch_bounds__(128)
k_window_stats(const WindowArgs a, const __grid_constant__ SeqTables tab, float* __restrict__ win_m, float* __restrict__ win_z) {
  __shared__ __align__(16) float sh[window_floats(D)];
  pdl_launch_dependents();
  pdl_wait();
  const int seg = blockIdx.x, s = seg / a.n_kv_heads, g = seg - s * a.n_kv_heads;
  const int t0 = tab.cu_at(s);
  const int n_hist = tab.cu_at(s + 1) - t0 - a.window;
  if (n_hist <= 0) return;                                     // no history: nothing is scored
  const int R = a.G * a.window;
  window_rows<T, D, 0>(a, sh, threadIdx.x, s, g, t0 + n_hist, blockIdx.y * kWinRows, [&](int r, float m, float z) {
    win_m[(long long)seg * R + r] = m;
    win_z[(long long)seg * R + r] = z;
  });
}

// lse_out[s][h][i] from the row sums (and the window statistics, if any).
__global__ void __launch_bounds__(128)
k_merge_lse_simt(void* part, const LseSource lse, const __grid_constant__ SeqTables tab, float* __restrict__ lse_out,
                 int n_seg, int n_kv_heads, int G, int window, float out_scale) {
  pdl_launch_dependents();
  pdl_wait();
  const int seg = blockIdx.x, s = seg / n_kv_heads, g = seg - s * n_kv_heads;
  const int n_hist = tab.cu_at(s + 1) - tab.cu_at(s) - window;
  if (n_hist <= 0) return;
  const int R = G * window;
  const SimtStats st = simt_stats(part, n_seg, R);
  const bool far = __ldcg(st.far) != 0, has_win = lse.win_m != nullptr;
  for (int r = threadIdx.x; r < R; r += 128) {
    const size_t at = (size_t)seg * R + r;
    const float l2 = simt_row_lse(st, at, far, has_win, has_win ? lse.win_m[at] : 0.f, has_win ? lse.win_z[at] : 0.f);
    const int hh = r / window, i = r - hh * window;
    lse_out[((long long)s * lse.n_q_heads + g * G + hh) * window + i] = l2 * out_scale;
  }
}

template <typename T, int D>
cudaError_t launch_passes(const Problem& pb, int32_t* status, int passes, cudaStream_t st, int* launches) {
  using TT = Tiles<T, D>;
  static thread_local int configured_dev = -1;
  static thread_local int coop_state = 0;                      // 0 untried, 1 with dependent launch, 2 without, -1 refused
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (configured_dev != dev) {
    e = cudaFuncSetAttribute(k_score_simt<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost);
    if (e != cudaSuccess) return e;
    coop_state = 0;
    configured_dev = dev;
  }
  const slkv_params& p = pb.p;
  SimtArgs a;
  a.tab = pb.tab;
  a.q = pb.q; a.k = pb.k; a.part = pb.part; a.vote = pb.vote; a.lse = lse_source_of(pb); a.status = status;
  a.n_seqs = p.n_seqs; a.n_kv_heads = p.n_kv_heads; a.G = pb.G; a.window = p.window; a.R = pb.R;
  a.n_tiles = (int)(2 * pb.n_tiles128);
  a.k_stride_tok = p.k_stride_tok; a.k_stride_head = p.k_stride_head;
  a.q_stride_seq = p.q_stride_seq; a.q_stride_row = p.q_stride_row; a.q_stride_head = p.q_stride_head;
  a.scale_log2 = kLog2e / sqrtf((float)p.head_dim);
  // Two CTAs per SM where there is work for them (their loads and barriers overlap), one where not; the query rows of a
  // segment stay in shared memory where they fit beside the keys, else 64 at a time.
  const int sms = sm_count(), chunks = (pb.R + kRows - 1) / kRows;
  const int limit = a.n_tiles > sms ? 110 * 1024 : kSmemMost;
  const int fixed = (kKeys * TT::kPitch + chunks * kRows + 4 * kKeys) * 4, q_all = chunks * kRows * TT::kPitch * 4;
  a.q_rows = fixed + q_all <= limit ? chunks * kRows : kRows;
  const int base = fixed + a.q_rows * TT::kPitch * 4;
  const int resident = sms * (limit == kSmemMost ? 1 : 2), most = resident < kSyncFlags ? resident : kSyncFlags;
  const int grid = a.n_tiles < most ? a.n_tiles : most;
  a.barrier_target = (unsigned)grid;
  const int per_cta = (a.n_tiles + grid - 1) / grid, kept_tile = chunks * 16 * kThreads * 4;
  a.keep = 0;
  if (passes == 3) a.keep = (limit - base) / kept_tile < per_cta ? (limit - base) / kept_tile : per_cta;
  const size_t smem = (size_t)base + (size_t)a.keep * kept_tile;

  if (passes != 2 && coop_state >= 0) {
    a.stages = passes == 3 ? kStats | kMaxima | kFarSums | kVotes : kStats | kMaxima | kFarSums;
    a.coop = 1;
    const int expire = take_expire_next_wait();
    a.barrier_target += expire == 1;
    a.sync.expect = (unsigned)grid + (expire == 2);
    a.sync.flags = pb.sync;
    a.sync.tag = next_launch_tag();
    for (int attempt = 0; attempt < 2; ++attempt) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(grid);
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = st;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = coop_state == 2 ? 1 : 2;
      {
        LaunchScope scope(passes == 3 ? KID_SCORE_FUSED : KID_SCORE_LSE, st, launches);
        e = cudaLaunchKernelEx(&cfg, k_score_simt<T, D>, a);
      }
      if (e == cudaSuccess) {
        if (coop_state == 0) coop_state = 1;
        return cudaSuccess;
      }
      (void)cudaGetLastError();                                // not a sticky error: the launch was refused
      --*launches;
      if (coop_state != 0) break;
      coop_state = 2;                                          // once more without dependent launch
    }
    coop_state = -1;
  }
  // no cooperative launch: the stages as launches of their own
  a.coop = 0;
  a.keep = 0;
  a.sync = FlagSync{};
  if (passes & 1) {
    e = cudaMemsetAsync(a.part, 0, simt_stat_bytes(pb.n_seg, pb.R), st);
    for (int stage = kStats; stage <= kFarSums && e == cudaSuccess; stage <<= 1) {
      a.stages = stage;
      e = launch_pdl_scoped(KID_SCORE_LSE, k_score_simt<T, D>, grid, kThreads, (size_t)base, st, launches, a);
    }
    if (e != cudaSuccess) return e;
  }
  if (!(passes & 2)) return cudaSuccess;
  a.stages = kVotes;
  return launch_pdl_scoped(KID_SCORE_VOTE, k_score_simt<T, D>, grid, kThreads, (size_t)base, st, launches, a);
}

template <typename T, int D>
cudaError_t launch_window(const Problem& pb, bool head_inner, cudaStream_t st, int* launches) {
  LaunchScope scope(KID_WINDOW_STATS, st, launches);
  return launch_pdl(k_window_stats<T, D>, dim3(pb.n_seg, (pb.R + kWinRows - 1) / kWinRows), dim3(128), 0, st, 1,
                    window_args(pb, head_inner), pb.tab, pb.win_m, pb.win_z);
}

}  // namespace

size_t simt_part_bytes(const Problem& pb) { return simt_stat_bytes(pb.n_seg, pb.R); }

cudaError_t launch_score_simt(const Problem& pb, int32_t* status, int passes, cudaStream_t st, int* launches) {
  if (pb.max_hist <= 0) return cudaSuccess;
  const bool bf = pb.p.dtype == SLKV_BF16;
  if (pb.p.head_dim == 64)
    return bf ? launch_passes<__nv_bfloat16, 64>(pb, status, passes, st, launches)
              : launch_passes<float, 64>(pb, status, passes, st, launches);
  return bf ? launch_passes<__nv_bfloat16, 128>(pb, status, passes, st, launches)
            : launch_passes<float, 128>(pb, status, passes, st, launches);
}

cudaError_t launch_window_stats(const Problem& pb, bool head_inner, cudaStream_t st, int* launches) {
  if (pb.max_hist <= 0) return cudaSuccess;
  const bool bf = pb.p.dtype == SLKV_BF16;
  if (pb.p.head_dim == 64)
    return bf ? launch_window<__nv_bfloat16, 64>(pb, head_inner, st, launches) : launch_window<float, 64>(pb, head_inner, st, launches);
  return bf ? launch_window<__nv_bfloat16, 128>(pb, head_inner, st, launches) : launch_window<float, 128>(pb, head_inner, st, launches);
}

// The row statistics a vote pass (or the merge) uses besides the partials of its own pass 1.
LseSource lse_source_of(const Problem& pb) {
  LseSource l;
  l.lse_opt = pb.lse_opt;
  const bool win = !pb.lse_opt && pb.p.softmax_domain == SLKV_ALL_CAUSAL;
  l.win_m = win ? pb.win_m : nullptr;
  l.win_z = win ? pb.win_z : nullptr;
  l.to_log2 = pb.p.lse_units == SLKV_LSE_LOG2 ? 1.0f : kLog2e;
  l.n_q_heads = pb.p.n_q_heads;
  return l;
}

float lse_out_scale(const Problem& pb) { return pb.p.lse_units == SLKV_LSE_LOG2 ? 1.0f : 0.6931471805599453f; }

cudaError_t launch_merge_lse_simt(const Problem& pb, float* lse_out, cudaStream_t st, int* launches) {
  if (pb.max_hist <= 0) return cudaSuccess;
  LaunchScope scope(KID_MERGE_LSE, st, launches);
  return launch_pdl(k_merge_lse_simt, dim3(pb.n_seg), dim3(128), 0, st, 1, pb.part, lse_source_of(pb), pb.tab, lse_out,
                    pb.n_seg, pb.p.n_kv_heads, pb.G, pb.p.window, lse_out_scale(pb));
}

}  // namespace slkv

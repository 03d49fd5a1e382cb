// Stage-2 KV budget allocation (Sec. 3.3, Eq. 6; Algorithm 2), one CTA, fp64 in a fixed operation order.
//
// Head (i, j) gets  fixed + share_ij  where the shares split the dynamic pool D = total - N*fixed in
// proportion to Algorithm 2's weight (0.01 + L_i/L_s) * (inf_ij/L_s) and are rounded by largest
// remainder so that they sum to D exactly.  Options: the head share over the layer's own sum (the prose under
// Eq. 6), a per-head cap whose excess is handed on to the other heads, Algorithm 2's own rounding.
// The sums over heads and layers run in index order on one thread and every product / quotient is a separately
// rounded IEEE operation (__dadd_rn / __dmul_rn / __ddiv_rn stop the compiler from fusing them), so the integers that
// come out do not depend on the launch shape.
//
// What bounds it: latency.  The order of the sums is part of the result, so one chain of N dependent fp64 additions stays
// (5 ns each); everything else runs on all threads: the weights (two fp64 divisions each) are in shared memory before the chain
// starts, and the largest remainders are found by counting them in as many parts of [0, 1) as there are threads -- of a few
// hundred remainders one or two share a part -- or, up to 96 heads, in pairs.  A thread per head up to 1024: a barrier of 1024
// threads costs a quarter of a microsecond more than one of 256.  In a graph, us, with all of it in one thread 256 heads 70.5;
// with 1024 threads and all pairs of remainders compared / 1024 threads and parts / as it is: 16 heads 4.1 / - / 3.1, 64: 4.3 / 4.8
// / 3.3, 100: 5.0 / 5.0 / 4.2, 256: 8.2 / 5.6 / 4.9, 384: 12.9 / 6.4 / 5.7, 512: 19.2 / 7.1 / 6.5, 1024: 61.1 / 10.5.
#include "slkv_internal.cuh"

namespace slkv {
namespace {

constexpr int kMost = 16384;           // heads
constexpr int kPairsMost = 96;         // heads up to which all pairs of remainders are compared: us in a graph with the pairs / counted
                                       // in parts, 256 threads, 32 heads 3.2 / 3.6, 64 3.4 / 3.8, 80 4.0 / 4.1, 96 4.1 / 4.1, 112 4.5 /
                                       // 4.3, 128 4.5 / 4.2, 160 6.1 / 4.5, 256 7.9 / 4.9
constexpr int kSmemMost = (kMost + 1024) * 8 + kMost * 5;      // 16384 heads in 1024 layers
constexpr int kListMost = 256;         // remainders of one part up to which they are ranked by counting (2 us); where more are
                                       // (nearly) equal, a radix descent over all of them takes eight levels of about 1 us

struct AllocOpts {
  int within_layer;      // head share over the layer's sum (prose under Eq. 6) instead of the grand sum (Algorithm 2)
  int paper_rounding;    // Algorithm 2's own last line instead of the normalisation
  long long cap;         // < 0: none
};

// Algorithm 2's weight of a head of influence x in a layer of H heads with sum La_i: (0.01 + L_i / L_s) * S_ij.
__device__ __forceinline__ double head_weight(double x, double La_i, double Ls, int H, bool within_layer) {
  const double lw = __dadd_rn(kLayerFloor, __ddiv_rn(La_i, Ls));       // 0.01 + L_{i,h}
  double share;
  if (within_layer) share = La_i > 0.0 ? __ddiv_rn(x, La_i) : __ddiv_rn(1.0, (double)H);
  else share = __ddiv_rn(x, Ls);                                       // S_{j,h}
  return __dmul_rn(lw, share);
}

// v[0] + v[1] + ... in index order, one thread; eight loads are in flight ahead of the additions.
__device__ __forceinline__ double ordered_sum(const double* v, int n) {
  double acc = 0.0;
  int a = 0;
  for (; a + 8 <= n; a += 8) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = v[a + u];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc = __dadd_rn(acc, x[u]);
  }
  for (; a < n; ++a) acc = __dadd_rn(acc, v[a]);
  return acc;
}

// Over a CTA of T threads.
template <int T>
__device__ long long block_sum_ll(long long v, long long* red) {
  __syncthreads();
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  long long t = (threadIdx.x & 31) < T / 32 ? red[threadIdx.x & 31] : 0;
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// COUNT: remainders counted in parts, else by pairs.  Up to MOST heads.
template <int T, bool COUNT, int MOST>
__global__ void __launch_bounds__(T, 1)
k_alloc(const float* __restrict__ inf, int L, int H, int fixed, long long total, const AllocOpts opt,
        int32_t* __restrict__ budgets, int32_t* __restrict__ status) {
  constexpr int kParts = T;              // parts of [0, 1) the remainders are counted in
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = L * H;
  double* wt = reinterpret_cast<double*>(smem_raw);        // [N] INF_sc, then the weights (0 once a head is filled), then
                                                           //     the remainders' bit patterns + 1 (0: not a candidate)
  unsigned long long* key = reinterpret_cast<unsigned long long*>(smem_raw);
  double* La = wt + N;                                     // [L] layer sums
  int* fl = reinterpret_cast<int*>(La + L);                // [N] dynamic parts
  unsigned char* active = reinterpret_cast<unsigned char*>(fl + N);   // [N] head still below the cap
  __shared__ long long red[T / 32];
  __shared__ double sh_Ls, sh_W;
  __shared__ int hist[COUNT ? 256 : 1], parts[COUNT ? kParts : 1], list[COUNT ? kListMost : 1];
  __shared__ int sh_digit, sh_above, sh_count, sh_same;
  const int tid = threadIdx.x;
  const long long D = total - (long long)N * fixed;
  const bool within = opt.within_layer != 0;
  if (COUNT) parts[tid] = 0;
  pdl_launch_dependents();
  pdl_wait();

  int bad = 0;
  for (int a = tid; a < N; a += T) {
    const float x = inf[a];
    bad |= !(x >= 0.0f) || !(x <= 3.402823466e38f);                  // negative, NaN or infinite
    wt[a] = (double)x;
    active[a] = 1;
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0 && status) *status = SLKV_ERR_NEG_INF_SC;
    return;
  }
  for (int i = tid; i < L; i += T) La[i] = ordered_sum(wt + (size_t)i * H, H);
  __syncthreads();
  if (tid == 0) sh_Ls = ordered_sum(La, L);
  __syncthreads();
  const double Ls = sh_Ls;
  const bool uniform = !(Ls > 0.0);                                   // no head has any influence: all weights 1

  if (opt.paper_rounding) {
    // Algorithm 2's own last line: C = floor(max(0, fixed + D * w) + 0.5), clipped at the cap; nothing is normalised
    for (int a = tid; a < N; a += T) {
      const double w = uniform ? __ddiv_rn(1.0, (double)N) : head_weight(wt[a], La[a / H], Ls, H, within);
      const double b = __dadd_rn((double)fixed, __dmul_rn((double)D, w));
      long long c = (long long)floor(__dadd_rn(fmax(0.0, b), 0.5));
      if (opt.cap >= 0 && c > opt.cap) c = opt.cap;
      budgets[a] = (int32_t)c;
    }
    return;
  }
  for (int a = tid; a < N; a += T) wt[a] = uniform ? 1.0 : head_weight(wt[a], La[a / H], Ls, H, within);

  // Heads that would rise above the cap are filled and taken out (their weight becomes 0, which leaves the ordered sum
  // of the others as it is), the rest share what is left, until none does (without a cap: one round, nobody is taken
  // out).
  const long long room = opt.cap >= 0 ? opt.cap - fixed : -1;
  long long d_rem = D;
  int n_active = N;
  double W;
  bool flat;
  while (true) {
    __syncthreads();
    if (tid == 0) sh_W = ordered_sum(wt, N);
    __syncthreads();
    W = sh_W;
    flat = !(W > 0.0);                                                // every weight left underflowed: share evenly
    if (flat) W = (double)n_active;
    if (room < 0 || n_active == 0) break;
    long long filled = 0;
    for (int a = tid; a < N; a += T) {
      if (!active[a]) continue;
      const double q = __ddiv_rn(__dmul_rn((double)d_rem, flat ? 1.0 : wt[a]), W);
      if (q >= (double)room) { active[a] = 0; wt[a] = 0.0; fl[a] = (int)room; ++filled; }
    }
    filled = block_sum_ll<T>(filled, red);
    if (filled == 0) break;
    d_rem -= filled * room;
    n_active -= (int)filled;
  }

  // quotas, floors, remainders of the heads still below the cap
  long long fsum = 0;
  for (int a = tid; a < N; a += T) {
    unsigned long long kk = 0;
    if (active[a]) {
      const double q = __ddiv_rn(__dmul_rn((double)d_rem, flat ? 1.0 : wt[a]), W);
      const double f = floor(q);
      kk = (unsigned long long)__double_as_longlong(__dadd_rn(q, -f)) + 1ull;    // remainders are >= 0: bit order = order
      fl[a] = (int)(long long)f;
      fsum += (long long)f;
    }
    key[a] = kk;
  }
  long long Rleft = d_rem - block_sum_ll<T>(fsum, red);                  // its barriers also publish key[] and fl[]
  if (n_active > 0 && Rleft >= n_active) {                            // not reachable in exact arithmetic
    const long long each = Rleft / n_active;
    for (int a = tid; a < N; a += T)
      if (active[a]) fl[a] += (int)each;
    Rleft -= each * n_active;
  }
  if (!COUNT && Rleft > 0) {
    // largest remainder first, ties -> lower index: head a gets +1 iff fewer than Rleft heads precede it
    int lanes = 1;                                                    // threads per head, neighbours in a warp
    while (lanes < 32 && 2 * lanes * N <= T) lanes *= 2;
    const int a = tid / lanes, sub = tid % lanes;
    const unsigned long long ka = a < N ? key[a] : 0ull;
    int rank = 0;
    if (ka)
      for (int b = sub; b < N; b += lanes) {
        const unsigned long long kb = key[b];
        rank += (kb > ka) || (kb == ka && b < a);
      }
    for (int o = 1; o < lanes; o *= 2) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (ka && sub == 0 && rank < Rleft) fl[a] += 1;
  } else if (COUNT && Rleft > 0) {
    // the Rleft-th largest remainder lies in one of kParts equal parts of [0, 1); what lies in a part above it gets +1, what lies
    // in the same part is ranked by counting
    auto part_of = [&](unsigned long long k) { return min((int)(__longlong_as_double((long long)(k - 1ull)) * (double)kParts), kParts - 1); };
    for (int a = tid; a < N; a += T)
      if (key[a]) atomicAdd(&parts[part_of(key[a])], 1);
    __syncthreads();
    const int lane0 = tid & 31, warp0 = tid >> 5, mine = parts[kParts - 1 - tid];           // from the top
    int upto = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane0 >= o) upto += n;
    }
    if (lane0 == 31) hist[warp0] = upto;
    __syncthreads();
    upto += (int)__reduce_add_sync(0xffffffffu, lane0 < warp0 ? (unsigned)hist[lane0] : 0u);
    if (upto - mine < Rleft && Rleft <= upto) { sh_digit = kParts - 1 - tid; sh_above = upto - mine; sh_count = 0; sh_same = mine; }
    __syncthreads();
    const int same = sh_same, part = sh_digit;
    if (same <= kListMost) {
      const int need = (int)Rleft - sh_above;
      for (int a = tid; a < N; a += T) {
        if (!key[a]) continue;
        const int p = part_of(key[a]);
        if (p > part) fl[a] += 1;
        else if (p == part) list[atomicAdd(&sh_count, 1)] = a;
      }
      __syncthreads();
      if (tid < same) {
        const int a = list[tid];
        const unsigned long long ka = key[a];
        int rank = 0;
        for (int j = 0; j < same; ++j) {
          const int b2 = list[j];
          const unsigned long long kb = key[b2];
          rank += (kb > ka) || (kb == ka && b2 < a);
        }
        if (rank < need) fl[a] += 1;
      }
    } else {
      // the Rleft-th largest key by a radix descent, eight bits at a time
      unsigned long long prefix = 0, mask = 0;
      int need = (int)Rleft;
      for (int shift = 56; shift >= 0; shift -= 8) {
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        for (int a = tid; a < N; a += T) {
          const unsigned long long k = key[a];
          if (k && (k & mask) == prefix) atomicAdd(&hist[(int)(k >> shift) & 255], 1);
        }
        __syncthreads();
        if (tid < 32) {                                               // lane t: the bins 255 - 8t .. 248 - 8t
          int c[8], s = 0;
#pragma unroll
          for (int u = 0; u < 8; ++u) { c[u] = hist[255 - 8 * tid - u]; s += c[u]; }
          int inc = s;
          for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, inc, o);
            if (tid >= o) inc += n;
          }
          int above = inc - s;
          if (above < need && need <= inc)
            for (int u = 0; u < 8; ++u) {
              if (need <= above + c[u]) { sh_digit = 255 - 8 * tid - u; sh_above = above; break; }
              above += c[u];
            }
        }
        __syncthreads();
        prefix |= (unsigned long long)sh_digit << shift;
        mask |= 255ull << shift;
        need -= sh_above;
        __syncthreads();
      }
      // keys above `prefix` and, in index order, the first `need` equal to it
      const int per = (N + T - 1) / T;
      const int a0 = min(tid * per, N), a1 = min(a0 + per, N);
      int eq = 0;
      for (int a = a0; a < a1; ++a) eq += key[a] == prefix;
      int inc = eq;
      const int lane = tid & 31, wid = tid >> 5;
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
      }
      if (lane == 31) hist[wid] = inc;
      __syncthreads();
      int before = inc - eq;
      for (int w2 = 0; w2 < wid; ++w2) before += hist[w2];
      for (int a = a0; a < a1; ++a) {
        if (key[a] > prefix) fl[a] += 1;
        else if (key[a] == prefix && before++ < need) fl[a] += 1;
      }
    }
  }
  while (Rleft < 0) {
    // floors overshot the pool (rounding): take one back from the smallest remainders, ties -> higher index
    __syncthreads();
    long long taken = 0;
    int dec[(MOST + T - 1) / T];
    int nd = 0;
    for (int a = tid; a < N; a += T, ++nd) {
      dec[nd] = 0;
      if (!active[a] || fl[a] <= 0) continue;
      int rank = 0;
      for (int b = 0; b < N; ++b) {
        if (!active[b] || fl[b] <= 0) continue;
        rank += (key[b] < key[a]) || (key[b] == key[a] && b > a);
      }
      if (rank < -Rleft) { dec[nd] = 1; ++taken; }
    }
    __syncthreads();
    nd = 0;
    for (int a = tid; a < N; a += T, ++nd)
      if (dec[nd]) fl[a] -= 1;
    Rleft += block_sum_ll<T>(taken, red);
  }
  __syncthreads();
  for (int a = tid; a < N; a += T) budgets[a] = fl[a] + fixed;
}

}  // namespace

cudaError_t launch_alloc(const float* inf, int n_layers, int n_heads, int fixed, long long total, int within_layer,
                         int paper_rounding, long long cap, int32_t* budgets, int32_t* status, cudaStream_t st) {
  const size_t n = (size_t)n_layers * n_heads;
  const size_t smem = (n + n_layers) * sizeof(double) + n * (sizeof(int) + 1);
  // A thread per head (below kPairsMost several); half the threads for 257-512 heads take 0.5 us longer.
  const bool many = n > 512;
  auto* const kernel = n <= kPairsMost ? k_alloc<256, false, kPairsMost>
                       : n <= 256 ? k_alloc<256, true, 256> : n <= 512 ? k_alloc<512, true, 512> : k_alloc<1024, true, kMost>;
  const int threads = n <= 256 ? 256 : n <= 512 ? 512 : 1024;
  static thread_local int configured_dev = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (many && configured_dev != dev) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMost);
    if (e != cudaSuccess) return e;
    configured_dev = dev;
  }
  AllocOpts opt;
  opt.within_layer = within_layer; opt.paper_rounding = paper_rounding; opt.cap = cap;
  int launches = 0;
  LaunchScope scope(KID_ALLOC, st, &launches);
  return launch_pdl(kernel, dim3(1), dim3(threads), smem, st, 1, inf, n_layers, n_heads, fixed, total, opt,
                    budgets, status);
}

}  // namespace slkv

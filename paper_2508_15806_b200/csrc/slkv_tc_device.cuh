// Device-side building blocks of the tensor-core score kernels (Sec. 3.4, Eq. 7; Algorithm 3): PTX wrappers for
// mbarriers, TMA loads, tcgen05 MMA / TMEM loads, the 2^x arithmetic, the tile schedule.  Included by the .cu
// files that hold the kernels; everything here has internal linkage.
#pragma once
#include <cuda.h>

#include "slkv_internal.cuh"
#include "slkv_fma_device.cuh"

namespace slkv {

namespace {

constexpr int kTileKeys = 128;                 // keys per tile (MMA N in the statistics pass, M in the vote pass)
constexpr int kHalfBytes = kTileKeys * 128;    // one 64-element (128-byte) half of a 128-row tile
constexpr int kSmemLimit = 227 * 1024;         // dynamic shared memory a CTA can have
constexpr int kTraceSlots = 64;                // timeline words per CTA (see slkv_trace_set_buffer)
// A tile's row sum that is not above this has underflowed (terms below fp32's range are flushed to zero, or clamped to
// 2^-125 on the polynomial path): the exact path then sums relative to the tile's maximum.
constexpr float kTinySum = 1e-30f;
constexpr unsigned long long kWaitLimitNs = 1000ull * 1000ull * 1000ull;   // 1 s per wait


// ---- PTX wrappers -------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(100u) : "memory");    // may sleep up to 0.1 us: a waiting thread must
                                                                   // not eat the issue slots of the epilogue warps
  return ok != 0;
}
// The same without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void trace_mark(const unsigned long long* base, int slot) {
  if (base) const_cast<unsigned long long*>(base)[(size_t)blockIdx.x * kTraceSlots + slot] = now_ns();
}
// Waits for the phase with the given parity.  false = gave up (limit reached or another thread did).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (unsigned it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63u) == 0) {
      if (*abort_flag) return false;
      if (now_ns() - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
// policy: L2 eviction policy (from createpolicy) for the lines the load touches
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, int w,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Pairs of fp32 values in one 64-bit register: fma / add on both with one instruction.
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 a, f32x2 b) {
  float x, y, z, w;
  unpack2(a, x, y);
  unpack2(b, z, w);
  return (x + y) + (z + w);
}
// 2^x of both halves on the special-function unit.
__device__ __forceinline__ f32x2 ex2_pair(f32x2 x) {
  float a, b;
  unpack2(x, a, b);
  return pack2(ex2(a), ex2(b));
}
// 2^x of both halves on the FMA and integer pipes instead of the special-function unit, which is the busiest pipe of
// both passes (one exponential per query row and key): x = n + f with n = round(x), 2^f by a degree-5 polynomial that
// is minimax in relative error on [-0.5, 0.5] (Remez exchange; 2.1e-7 evaluated in fp32, ex2.approx has 2^-22 =
// 2.4e-7), n added into the exponent field.  x is clamped at -125 (the result is then 2^-125: negligible in any sum
// that holds a term near 1) and, where CLAMP_HI, at 128.5, from where the exponent field overflows to Inf / NaN, which
// the statistics pass's overflow check catches.
template <bool CLAMP_HI>
__device__ __forceinline__ f32x2 ex2_pair_poly(f32x2 x) {
  float a, b;
  unpack2(x, a, b);
  a = fmaxf(a, -125.f);
  b = fmaxf(b, -125.f);
  if (CLAMP_HI) {
    a = fminf(a, 128.5f);
    b = fminf(b, 128.5f);
  }
  x = pack2(a, b);
  const f32x2 t = add2(x, pack2(12582912.f, 12582912.f));     // 1.5 * 2^23: round(x) lands in the low mantissa bits
  const f32x2 f = fma2(add2(t, pack2(-12582912.f, -12582912.f)), pack2(-1.f, -1.f), x);
  f32x2 p = fma2(pack2(0.0013276472454890609f, 0.0013276472454890609f), f, pack2(0.009675540961325169f, 0.009675540961325169f));
  p = fma2(p, f, pack2(0.05550713092088699f, 0.05550713092088699f));
  p = fma2(p, f, pack2(0.24022120237350464f, 0.24022120237350464f));
  p = fma2(p, f, pack2(0.6931469440460205f, 0.6931469440460205f));
  p = fma2(p, f, pack2(1.0000001192092896f, 1.0000001192092896f));
  float pa, pb, ta, tb;
  unpack2(p, pa, pb);
  unpack2(t, ta, tb);
  return pack2(__int_as_float(__float_as_int(pa) + (__float_as_int(ta) << 23)),
               __int_as_float(__float_as_int(pb) + (__float_as_int(tb) << 23)));
}
// Issues a TMEM load of 16 consecutive columns of this thread's lane; the registers are valid only after tc_ld_wait on
// the same array.
__device__ __forceinline__ void tc_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// Waits for this thread's outstanding TMEM loads; naming the registers keeps their uses behind the wait.
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
        "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) :: "memory");
}

// K-major, 128-byte-swizzled operand: rows 128 bytes apart, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// D fp32, A and B bf16, both K-major, M x N tile
__device__ __forceinline__ uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The part that share i of n takes of T items, and its inverse (the index whose
// range holds tile x of the group): shares differ by one tile at most.  The products fit 32 bits for tiles: describe() lets
// through fewer than 2^31 / 128 + 2^20 of a layer, a list of one group has fewer than 2^24, and n is 160 at most.
__device__ __forceinline__ int split_begin(int i, int T, int n) { return (int)(((unsigned)i * (unsigned)T) / (unsigned)n); }
__device__ __forceinline__ int split_index(int x, int T, int n) {
  return (int)((((unsigned)x + 1u) * (unsigned)n - 1u) / (unsigned)T);
}
// In how many parts the CTAs of a launch whose list is one group share a segment (n, from the `first` of the split on).
struct SegmentSlots {
  int before, tiles, shares, first, n;         // of the list's tiles: before the segment, all; shares they are split into
  int tiles_seg;
  __device__ __forceinline__ int slot(int tile) const { return split_index(before + tile, tiles, shares) - first; }
  // Part c: its first tile, of the segment, and how many.
  __device__ __forceinline__ int begin(int c) const { return max(split_begin(first + c, tiles, shares) - before, 0); }
  __device__ __forceinline__ int count(int c) const { return min(split_begin(first + c + 1, tiles, shares) - before, tiles_seg) - begin(c); }
};
__device__ __forceinline__ SegmentSlots list_slots(const ScoreShape& sh, int n_layers, int layer, int s, int g) {
  SegmentSlots x;
  const int tiles_seg = sh.tab.tile_at(s + 1) - sh.tab.tile_at(s);
  x.tiles = n_layers * sh.total_tiles;
  x.tiles_seg = tiles_seg;
  x.shares = min(sh.n_cta, x.tiles);
  x.before = layer * sh.total_tiles + sh.n_kv_heads * sh.tab.tile_at(s) + g * tiles_seg;
  x.first = split_index(x.before, x.tiles, x.shares);
  x.n = split_index(x.before + tiles_seg - 1, x.tiles, x.shares) - x.first + 1;
  return x;
}
// Row statistics in global memory, per segment and row: acc = the sum of 2^score over all keys, in fp64 and without a
// reference.  The terms are fp32 sums over one tile each, added atomically in whatever order they come.  n of them within a
// factor 2^29 / n of one another fit one 53-bit window, the additions are exact and the order shows nowhere; else the sum is
// the same to 2^-53 times a few, and about one fp32 logarithm in 10^8 differs in its last bit.
// Scores beyond fp64's range (above 900 or below -900 in log2 units) go elsewhere: share `slot` then holds such a part of
// the row's sum as z * 2^m, and its bit in far[] is set.
constexpr float kFarScore = 900.f;
constexpr int kFarWords = kMaxSplit / 32;
struct StatView {
  double* acc;                 // [n_seg][R]
  unsigned* far;               // [n_seg][kFarWords]; acc and far are cleared before use
  float* far_z;                // [n_seg][stride][R]
  float* far_m;                // likewise
  float* lse;                  // [n_seg][R], where a kernel of its own merges (log2 units)
};
__host__ __device__ __forceinline__ size_t stat_clear_bytes(int n_seg, int R) {
  return (size_t)n_seg * R * sizeof(double) + (size_t)n_seg * kFarWords * sizeof(unsigned);
}
__device__ __forceinline__ StatView stat_view(void* part, int n_seg, int R, int stride) {
  StatView v;
  v.acc = static_cast<double*>(part);
  v.far = reinterpret_cast<unsigned*>(v.acc + (size_t)n_seg * R);
  v.far_z = reinterpret_cast<float*>(v.far + (size_t)n_seg * kFarWords);
  v.far_m = v.far_z + (size_t)n_seg * stride * R;
  v.lse = v.far_m + (size_t)n_seg * stride * R;
  return v;
}
// Folds (zo, mo) into (z, m): sums of 2^(x - m) with different references.
__device__ __forceinline__ void stat_add(float& z, float& m, float zo, float mo) {
  if (!(zo > 0.f)) return;
  const float mn = z > 0.f ? fmaxf(m, mo) : mo;
  z = (z > 0.f ? z * ex2(m - mn) : 0.f) + zo * ex2(mo - mn);
  m = mn;
}
// log2 of a positive fp64 number, in fp32 arithmetic on its fraction and exponent.
__device__ __forceinline__ float log2_of(double Z) {
  const int hi = __double2hiint(Z);
  return __fadd_rn((float)((hi >> 20) - 1023), log2f((float)__hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(Z))));
}
// The log-sum-exp (log2 units) of a row from its sum Z, the far parts of its segment's n_slots shares if there are any, and
// the window keys' statistics (wm, wz), if any.  One definition for every kernel that merges.
__device__ __forceinline__ float row_lse(const StatView& st, double Z, bool any_far, int seg, int row, int R, int stride,
                                         int n_slots, bool has_win, float wm, float wz) {
  if (!any_far && !has_win) return log2_of(Z);
  float z = 0.f, m = 0.f;
  if (Z > 0.0) {
    m = (float)((__double2hiint(Z) >> 20) - 1023);
    z = (float)__hiloint2double((__double2hiint(Z) & 0xfffff) | 0x3ff00000, __double2loint(Z));
  }
  if (any_far)
    for (int c = 0; c < n_slots; ++c)
      if (__ldcg(st.far + (size_t)seg * kFarWords + (c >> 5)) >> (c & 31) & 1u) {
        const size_t at = ((size_t)seg * stride + c) * R + row;
        stat_add(z, m, __ldcg(st.far_z + at), __ldcg(st.far_m + at));
      }
  if (has_win) stat_add(z, m, wz, wm);
  return __fadd_rn(m, log2f(z));
}

// A run = consecutive tiles of one segment inside the CTA's range [begin, end) of a layer's flat tile list.
struct Run { int s, g, t0, count, n_hist, seg_tile0, tiles_seg; };

__device__ __forceinline__ Run locate(const ScoreShape& a, int pos, int end) {
  int lo = 0, hi = a.n_seqs;                       // last s with Hkv*tile_off[s] <= pos
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (a.n_kv_heads * a.tab.tile_at(mid) <= pos) lo = mid; else hi = mid;
  }
  Run r;
  r.s = lo;
  r.tiles_seg = a.tab.tile_at(lo + 1) - a.tab.tile_at(lo);
  const int rel = pos - a.n_kv_heads * a.tab.tile_at(lo);
  r.g = rel / r.tiles_seg;
  r.t0 = rel - r.g * r.tiles_seg;
  r.seg_tile0 = pos - r.t0;
  r.count = min(end - pos, r.tiles_seg - r.t0);
  r.n_hist = max(a.tab.cu_at(lo + 1) - a.tab.cu_at(lo) - a.window, 0);
  return r;
}

// Statistics pass, exact path for this thread's row of one accumulator: z * 2^m = the sum over the tile's keys
// first .. n_valid - 1 (first a multiple of 8), m a whole number.  For tiles whose sum over- or underflows on the fast path,
// and a segment's last keys.  Eight columns at a time: inlined beside the fast path, it must not need registers of its own.
__device__ __forceinline__ void tile_stats_exact(uint32_t tcol, float sc, int first, int n_valid, float& m, float& z) {
  m = 0.f;
  z = 0.f;
#pragma unroll 1
  for (int c0 = first; c0 < kTileKeys && c0 < n_valid; c0 += 8) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(tcol + c0) : "memory");
    float mx = -INFINITY;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (c0 + e < n_valid) mx = fmaxf(mx, __uint_as_float(r[e]) * sc);
    const bool any = mx > -INFINITY && mx < INFINITY;    // not only -inf scores
    const float mn = !any ? m : (z > 0.f ? fmaxf(m, ceilf(mx)) : ceilf(mx));
    z = z > 0.f ? z * ex2(m - mn) : 0.f;
    m = mn;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (any && c0 + e < n_valid) z += ex2(fmaf(__uint_as_float(r[e]), sc, -m));
  }
}

// ---- the epilogue warps' arithmetic on accumulators --------------------------------------------------------------------
// Votes: sum_e 2^(v_e * sc + off_e) over 16 accumulator values, in two pair accumulators.  POLY: the first pair's exponentials
// go to the FMA pipe, where it takes fourteen instructions instead of two.  By cycles alone two pairs of eight would go there;
// at the power limit the instructions cost more clock than they save cycles (32 layers of 32k / 128k positions, in both
// passes no pair of a chunk's eight on the FMA pipe 862 / 5866 us, one 877 / 5806, two 890 / 5905).  Here: in the votes one in
// every other chunk, in the statistics one in eight (TileSum).
// The loops around this are kept small, the statistics' one chunk at a time with the last keys of a segment outside: four
// warps on a scheduler hide a TMEM load's latency, and the epilogue warps are spread over both passes' loops, which have to
// stay in the instruction cache (4k positions: statistics loop unrolled four times 154 us, twice 144, two chunks with the
// last keys masked inside 140.9, as it is 140.1; 128k: 6147, 5865, 5868, 5820).
template <bool POLY>
__device__ __forceinline__ void exp_chunk(const uint32_t (&r)[16], f32x2 sc2, uint32_t off_sh, f32x2& s0, f32x2& s1) {
#pragma unroll
  for (int e = 0; e < 16; e += 4) {
    f32x2 o0, o1;
    // an explicit shared-memory load: a generic one takes another path
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(o0), "=l"(o1) : "r"(off_sh + 4u * e));
    const f32x2 x0 = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sc2, o0);
    const f32x2 x1 = fma2(pack2(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), sc2, o1);
    s0 = add2(s0, POLY && e == 0 ? ex2_pair_poly<false>(x0) : ex2_pair(x0));
    s1 = add2(s1, ex2_pair(x1));
  }
}
__device__ __forceinline__ float pair_sum(f32x2 v) {
  float a, b;
  unpack2(v, a, b);
  return a + b;
}
// Statistics: a row's sum of 2^(v * sc) over a tile, in two pair accumulators, one pair of eight on the FMA pipe.  WIDE: the sums of a
// launch for bounds, where eight accumulators, one for each column modulo 8, lie in the lanes as in bound_run; there a pair of
// columns is one of four lanes' and none goes to the FMA pipe.  Short lists miss that share (with / without: 32 layers of 4001 tokens, 128 rows
// 125.0 / 126.5 us, 16 of 24000, 256 rows 495 / 504, a rank's statistics and votes of 32768 111.1 / 112.1), long ones hardly (12000 tokens 302 / 302).  A chunk of
// sixteen columns on the FMA pipe, the same in both: 131.6, 505, 112.1, and the launch for bounds 623 -> 661.
template <bool WIDE>
struct TileSum {
  f32x2 s[WIDE ? 4 : 2];
  __device__ __forceinline__ TileSum() {
#pragma unroll
    for (int i = 0; i < (WIDE ? 4 : 2); ++i) s[i] = 0;
  }
  __device__ __forceinline__ void chunk(const uint32_t (&r)[16], f32x2 sc2) {
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
      const f32x2 x = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sc2, 0);
      f32x2& to = s[(e >> 1) & (WIDE ? 3 : 1)];
      to = add2(to, !WIDE && e == 0 ? ex2_pair_poly<true>(x) : ex2_pair(x));
    }
  }
  __device__ __forceinline__ float total() const {
    const float low = pair_sum(s[0]) + pair_sum(s[1]);
    if constexpr (WIDE) return low + (pair_sum(s[2]) + pair_sum(s[3]));
    else return low;
  }
};

// An epilogue thread's unit.
struct Unit {
  uint32_t tcol;               // its TMEM lane and its warpgroup's unit
  uint32_t full, empty;        // the unit's mbarriers
  volatile int* abort_flag;
};
__device__ __forceinline__ bool unit_wait(const Unit& u, int nth) {
  const bool ok = mbar_wait(u.full, nth & 1, u.abort_flag);
  if (!__all_sync(0xffffffffu, ok)) return false;                        // the TMEM loads need the whole warp
  tc_fence_after();
  return true;
}
__device__ __forceinline__ void unit_release(const Unit& u) {
  tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(u.empty);
}

// Statistics of one run for this thread's query row: tiles i0, i0 + every, ... < count.  z: the sum of 2^score, without a
// reference; (far_z, far_m): what of it fp64 cannot hold (see StatView).  A tile is summed in fp32, without a reference
// either as long as nothing overflows and not everything underflows; one whose sum is not finite and above kTinySum is
// redone exactly.  false: a wait ran out.
template <bool WIDE>
__device__ __forceinline__ bool stats_run(const Unit u, int nth, float sc, int i0, int every, int count, int n_valid0,
                                          bool rows_here, double& z, float& far_z, float& far_m) {
  z = 0.0;
  far_z = far_m = 0.f;
  const f32x2 sc2 = pack2(sc, sc);
#pragma unroll 1
  for (int i = i0; i < count; i += every, ++nth) {
    if (!unit_wait(u, nth)) return false;
    if (rows_here) {
      const int n_valid = n_valid0 - i * kTileKeys;
      const int whole = n_valid < kTileKeys ? n_valid & ~15 : kTileKeys;
      TileSum<WIDE> s;
#pragma unroll 1
      for (int c0 = 0; c0 < whole; c0 += 16) {
        uint32_t v[16];
        tc_ld16_issue(u.tcol + c0, v);
        tc_ld_wait(v);
        s.chunk(v, sc2);
      }
      float tile = s.total();
      if (n_valid < kTileKeys) {                               // the segment's last keys; those past its end count nothing
        float tm, tz;
        tile_stats_exact(u.tcol, sc, whole, n_valid, tm, tz);
        tile += tz * ex2(tm);
      }
      const bool exact = !(tile < INFINITY && tile > kTinySum);
      if (!__any_sync(0xffffffffu, exact)) {
        z += (double)tile;
      } else {                                                 // the exact path's TMEM loads need the whole warp
        float tm, tz;
        tile_stats_exact(u.tcol, sc, 0, n_valid, tm, tz);
        if (!exact) z += (double)tile;                         // the same value whatever the other rows hold
        else if (fabsf(tm) <= kFarScore) z += scalbn((double)tz, (int)tm);
        else stat_add(far_z, far_m, tz, tm);
      }
    }
    unit_release(u);
  }
  return true;
}

// ---- statistics and estimated votes from one product ------------------------------------------------------------------------
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Both halves rounded to bf16, the first in the low half.
__device__ __forceinline__ uint32_t bf16_pair(f32x2 v) {
  float a, b;
  unpack2(v, a, b);
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint32_t add_bf16(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// 16 TMEM columns of this warp's 32 lanes as a matrix operand lies in registers: thread 4 g + t has the columns 2 t and 2 t + 1 of
// the eight at 8 b for the rows g + 8 q in v[8 (q >> 1) + 4 b + 2 (q & 1)] and the one behind it.
__device__ __forceinline__ void tc_ld_quads(uint32_t taddr, uint32_t (&v)[16]) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[8 * i]), "=r"(v[8 * i + 1]), "=r"(v[8 * i + 2]), "=r"(v[8 * i + 3]), "=r"(v[8 * i + 4]), "=r"(v[8 * i + 5]),
                   "=r"(v[8 * i + 6]), "=r"(v[8 * i + 7])
                 : "r"(taddr + ((uint32_t)i << 20)) : "memory");
}
// The row, of the warp's 32, whose sum a thread has in the end.
__device__ __forceinline__ int quad_row() { return ((threadIdx.x & 31) >> 2) + 8 * (threadIdx.x & 3); }
// TileSum<true> for four rows of two columns in eight, whose sums these are bit for bit (s[q]: row g + 8 q), and the four rows'
// weight * exponential of the two columns in h[b], rounded to bf16.
__device__ __forceinline__ void bound_chunk(const uint32_t (&v)[16], f32x2 sc2, const f32x2 (&w2)[4], f32x2 (&s)[4], uint32_t* h) {
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    f32x2 est = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int at = 8 * (q >> 1) + 4 * b + 2 * (q & 1);
      const f32x2 p = ex2_pair(fma2(pack2(__uint_as_float(v[at]), __uint_as_float(v[at + 1])), sc2, 0));
      s[q] = add2(s[q], p);
      est = q == 0 ? mul2(p, w2[0]) : fma2(p, w2[q], est);
    }
    h[b] = bf16_pair(est);
  }
}
// The sum of the thread's row: of the four rows that lie in four lanes each, a lane keeps one.
__device__ __forceinline__ float quad_sum(const f32x2 (&s)[4]) {
  const bool odd = threadIdx.x & 1, high = threadIdx.x & 2;
  float a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) a[q] = pair_sum(s[q]);
  const float lo = (odd ? a[1] : a[0]) + __shfl_xor_sync(0xffffffffu, odd ? a[0] : a[1], 1);
  const float hi = (odd ? a[3] : a[2]) + __shfl_xor_sync(0xffffffffu, odd ? a[2] : a[3], 1);
  return (high ? hi : lo) + __shfl_xor_sync(0xffffffffu, high ? lo : hi, 2);
}
// The sums over the warp's rows of 64 columns (h[b]: of those at 8 b) or of 16, out[0 ..]: of two registers a lane keeps one and
// sends the other.
__device__ __forceinline__ void lane_sums(uint32_t (&h)[8], float* out) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int n = 4; n >= 1; n >>= 1)
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const uint32_t keep = lane & (4 * n) ? h[i + n] : h[i], send = lane & (4 * n) ? h[i] : h[i + n];
      h[i] = add_bf16(keep, __shfl_xor_sync(0xffffffffu, send, 4 * n));
    }
  reinterpret_cast<float2*>(out)[lane] = make_float2(__uint_as_float(h[0] << 16), __uint_as_float(h[0] & 0xffff0000u));
}
__device__ __forceinline__ void lane_sums(uint32_t (&h)[2], float* out) {
  const int lane = threadIdx.x & 31;
  uint32_t x = add_bf16(lane & 16 ? h[1] : h[0], __shfl_xor_sync(0xffffffffu, lane & 16 ? h[0] : h[1], 16));
  x = add_bf16(x, __shfl_xor_sync(0xffffffffu, x, 8));
  x = add_bf16(x, __shfl_xor_sync(0xffffffffu, x, 4));
  if ((lane & 12) == 0) reinterpret_cast<float2*>(out)[4 * (lane >> 4) + (lane & 3)] = make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
}

// The order in which a run's tiles are taken where the first kFirst are to be spread over it: tile j and tile
// j (count - 1) / (kFirst - 1) change places.
template <int MT>
struct Spread {
  static constexpr int kFirst = MT == 1 ? 4 : 2;
  int to[kFirst];                                              // where tile j lies; tile 0 stays
  __device__ __forceinline__ explicit Spread(int count) {
#pragma unroll
    for (int j = 0; j < kFirst; ++j) to[j] = count >= 16 ? j * (count - 1) / (kFirst - 1) : j;
  }
  __device__ __forceinline__ int tile(int i) const {
    int t = i;
#pragma unroll
    for (int j = 1; j < kFirst; ++j) t = i == j ? to[j] : (i == to[j] ? j : t);
    return t;
  }
};

// In the order of Spread, the first tile with the second set of weights, the reciprocals of the rows' sums over the tiles before it:
// a quarter of a long run, none of a short one.
__device__ __forceinline__ int second_weights(int count) { return count >= 64 ? count >> 2 : 0x7fffffff; }

// What the warpgroups of a CTA tell one another in a run for bounds.
struct BoundRun {
  float* sums;                 // [4][128]: the rows' sums over the warpgroup's first tile
  uint32_t sums_bar;           // every epilogue warp
  uint32_t sums_parity;
  uint32_t again_bar;          // the same for the second weights
  uint32_t again_parity;
  float* part;                 // two slots of the sharing warpgroups' warps' shares [4 MT][128]
  uint32_t part_bars;
  int n_part;                  // tiles these warpgroups have been through
  float* weight;               // where the rows' weights go; the second ones `second` floats further on
  int second;
  float* est;                  // estimated votes, of the run's first key
  int rows, n_warps;           // rows per KV head, warps that hold some
};

// Statistics of one run, as stats_run<true> (the sums are the same bit for bit, but of row quad_row() of the warp's), and with the same exponentials an estimate of every key's
// vote, est[key] = sum_rows weight_r * 2^score.  The rows' sums are not known yet: weight_r is the reciprocal of the row's sum over
// the run's first tiles in the order of Spread, one per warpgroup (two: per pair), whose accumulators are read twice for it, and from a
// quarter of the run on over that quarter (the bounds are three to five times as tight in the keys that they let through).  The
// warps' shares of a tile, 32 rows each, meet in shared memory, two slots in turn (a warp is back at a slot only once all have
// passed the barrier of the one behind, and so have read it).
template <int MT>
__device__ __forceinline__ bool bound_run(const Unit u, int nth, float sc, int i0, int every, int count, int n_valid0, bool rows_here,
                                          int wg, BoundRun b, double& z, float& far_z, float& far_m) {
  constexpr int kShare = 4 * MT * 128;
  z = 0.0;
  far_z = far_m = 0.f;
  const f32x2 sc2 = pack2(sc, sc);
  const int row = threadIdx.x & 127, lane = threadIdx.x & 31, mt = MT == 1 ? 0 : wg & 1, warp = mt * 4 + (row >> 5);
  const Spread<MT> order(count);
  float first = 0.f;
  if (i0 < count) {
    if (!unit_wait(u, nth)) return false;
    if (rows_here) {
      const int n_valid = n_valid0 - order.tile(i0) * kTileKeys, whole = n_valid < kTileKeys ? n_valid & ~15 : kTileKeys;
      TileSum<true> s;
#pragma unroll 1
      for (int c0 = 0; c0 < whole; c0 += 16) {
        uint32_t v[16];
        tc_ld16_issue(u.tcol + c0, v);
        tc_ld_wait(v);
        s.chunk(v, sc2);
      }
      first = s.total();
      if (whole < n_valid && whole < kTileKeys) {
        float tm, tz;
        tile_stats_exact(u.tcol, sc, whole, n_valid, tm, tz);
        first += tz * ex2(tm);
      }
    }
  }
  b.sums[wg * 128 + row] = first;
  __syncwarp();
  if (lane == 0) mbar_arrive(b.sums_bar);
  const bool there = mbar_wait(b.sums_bar, b.sums_parity, u.abort_flag);
  if (!__all_sync(0xffffffffu, there)) return false;
  // Sums between 2^-60 and 2^100: what fp32 flushes to zero is then 2^-66 of a row at most and nothing overflows.  A weight that is not
  // finite makes every estimate so.
  const int row0 = mt * 128 + (row & ~31), own = quad_row();
  f32x2 w2[4];
  auto weigh = [&](float* out) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = row0 + (lane >> 2) + 8 * q;
      float total = b.sums[r];                                 // of warpgroup mt, rows of block mt
#pragma unroll
      for (int w = MT; w < 4; w += MT) total += b.sums[w * 128 + r];
      float weight = total >= 0x1p-60f && total <= 0x1p100f ? __fdividef(1.f, total) : __int_as_float(0x7fffffff);
      if (r >= b.rows) weight = 0.f;
      else if (wg < MT && q == (lane & 3)) __stcg(out + r, weight);
      w2[q] = pack2(weight, weight);
    }
  };
  weigh(b.weight);
  int refresh = second_weights(count);
#pragma unroll 1
  for (int i = i0; i < count; i += every, ++nth, ++b.n_part) {
    if (i >= refresh) {
      // all warpgroups get here: a run this long has tiles for each behind that; and none still reads the first sums, for which
      // its first unit had to be given back
      refresh = 0x7fffffff;
      b.sums[wg * 128 + (row & ~31) + own] = (float)z;
      __syncwarp();
      if (lane == 0) mbar_arrive(b.again_bar);
      const bool all = mbar_wait(b.again_bar, b.again_parity, u.abort_flag);
      if (!__all_sync(0xffffffffu, all)) return false;
      weigh(b.weight + b.second);
    }
    if (!unit_wait(u, nth)) return false;
    const int tile = order.tile(i), n_valid = n_valid0 - tile * kTileKeys, slot = b.n_part & 1;
    float* const mine = b.part + slot * kShare + warp * 128;
    if (rows_here) {
      f32x2 s[4] = {0, 0, 0, 0};
      float sum;
      if (n_valid >= kTileKeys) {
#pragma unroll 1
        for (int c0 = 0; c0 < kTileKeys; c0 += 64) {
          uint32_t v[16], h[8];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            tc_ld_quads(u.tcol + c0 + 16 * c, v);
            tc_ld_wait(v);
            bound_chunk(v, sc2, w2, s, h + 2 * c);
          }
          lane_sums(h, mine + c0);
        }
        sum = quad_sum(s);
      } else {                                                 // a segment's last keys: the sums as in stats_run
        const int whole = n_valid & ~15;
        f32x2 unused[4] = {0, 0, 0, 0};
#pragma unroll 1
        for (int c0 = 0; c0 < n_valid; c0 += 16) {
          uint32_t v[16], h[2];
          tc_ld_quads(u.tcol + c0, v);
          tc_ld_wait(v);
          if (c0 < whole) bound_chunk(v, sc2, w2, s, h);
          else bound_chunk(v, sc2, w2, unused, h);
          lane_sums(h, mine + c0);
        }
        sum = quad_sum(s);
        float tm, tz;
        tile_stats_exact(u.tcol, sc, whole, n_valid, tm, tz);
        sum += __shfl_sync(0xffffffffu, tz * ex2(tm), own);
      }
      const bool exact = !(sum < INFINITY && sum > kTinySum);
      if (!__any_sync(0xffffffffu, exact)) {
        z += (double)sum;
      } else {
        float tm, tz;
        tile_stats_exact(u.tcol, sc, 0, n_valid, tm, tz);
        tm = __shfl_sync(0xffffffffu, tm, own);
        tz = __shfl_sync(0xffffffffu, tz, own);
        if (!exact) z += (double)sum;
        else if (fabsf(tm) <= kFarScore) z += scalbn((double)tz, (int)tm);
        else stat_add(far_z, far_m, tz, tm);
      }
    }
    unit_release(u);
    const uint32_t bar = b.part_bars + 8u * (uint32_t)slot;
    if (lane == 0) mbar_arrive(bar);                           // behind the whole warp's stores: unit_release's __syncwarp
    const bool ok = mbar_wait(bar, (b.n_part >> 1) & 1, u.abort_flag);
    if (!__all_sync(0xffffffffu, ok)) return false;
    if (MT == 1 || (row >> 6) == mt) {
      const float* shares = b.part + slot * kShare + row;
      float sum = shares[0];
      for (int w = 1; w < b.n_warps; ++w) sum += shares[w * 128];
      if (row < n_valid) b.est[tile * kTileKeys + row] = sum;
    }
  }
  return true;
}

// Votes of one run for this thread's key of every tile, handed to out(key, vote): the sum over this warpgroup's rows (cols of them, from its
// log-sum-exps lse on).  MT = 2: the other 128 rows are the neighbouring warpgroup's; the first one, whose unit is filled
// first, leaves its share in shared memory for the second (four slots in turn: a tile's second product waits until the
// second warpgroup has given its unit back, so the first one cannot be more than three of its tiles ahead).
// false: a wait ran out.
template <typename Out>
__device__ __forceinline__ bool votes_run(const Unit u, int nth, float sc, int i0, int every, int count, int n_keys,
                                       uint32_t lse, int cols, int half, float* half_vote, uint32_t half_bar, int n_half,
                                       float inv_g, Out out) {
  const f32x2 sc2 = pack2(sc, sc);
  const int row = threadIdx.x & 127;
#pragma unroll 1
  for (int i = i0; i < count; i += every, ++nth) {
    if (!unit_wait(u, nth)) return false;
    uint32_t ra[16], rb[16];
    f32x2 s0 = 0, s1 = 0;
    tc_ld16_issue(u.tcol, ra);
#pragma unroll 1
    for (int c0 = 0; c0 < cols; c0 += 32) {
      tc_ld_wait(ra);
      tc_ld16_issue(u.tcol + c0 + 16, rb);
      exp_chunk<true>(ra, sc2, lse + 4u * c0, s0, s1);
      tc_ld_wait(rb);
      if (c0 + 32 < cols) tc_ld16_issue(u.tcol + c0 + 32, ra); else unit_release(u);
      exp_chunk<false>(rb, sc2, lse + 4u * c0 + 64u, s0, s1);
    }
    float acc = sum2(s0, s1);
    if (half >= 0) {
      const int turn = n_half & 3;
      const uint32_t parity = (n_half >> 2) & 1;
      ++n_half;
      if (half == 0) {
        half_vote[turn * 128 + row] = acc;
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(half_bar + 8u * turn);
        continue;
      }
      const bool ok = mbar_wait(half_bar + 8u * turn, parity, u.abort_flag);
      if (!__all_sync(0xffffffffu, ok)) return false;
      acc += half_vote[turn * 128 + row];
    }
    const int key = i * kTileKeys + row;
    if (key < n_keys) out(key, acc * inv_g);
  }
  return true;
}

// A thread's key against this accumulator's rows (cols of them): votes_run's sum, bit for bit.
__device__ __forceinline__ float key_vote(uint32_t tcol, int cols, float sc, uint32_t lse) {
  const f32x2 sc2 = pack2(sc, sc);
  uint32_t v[16];
  f32x2 s0 = 0, s1 = 0;
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += 32) {
    tc_ld16_issue(tcol + c0, v);
    tc_ld_wait(v);
    exp_chunk<true>(v, sc2, lse + 4u * c0, s0, s1);
    tc_ld16_issue(tcol + c0 + 16, v);
    tc_ld_wait(v);
    exp_chunk<false>(v, sc2, lse + 4u * c0 + 64u, s0, s1);
  }
  return sum2(s0, s1);
}

}  // namespace
}  // namespace slkv

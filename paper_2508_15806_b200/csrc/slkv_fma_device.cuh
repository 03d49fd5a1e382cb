// Device-side pieces of the FMA arithmetic: packed pairs, unpacked 16-byte loads, the window keys' row statistics.  Included by
// the .cu files that need them; everything here has internal linkage.
#pragma once
#include "slkv_internal.cuh"

namespace slkv {
namespace {

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float sum_of(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a + b;
}

__device__ __forceinline__ void unpack(const uint4& u, float (&f)[4], float) {
  f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y); f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack(const uint4& u, float (&f)[8], __nv_bfloat16) {
  // a bf16 is the high half of an fp32
  f[0] = __uint_as_float(u.x << 16); f[1] = __uint_as_float(u.x & 0xffff0000u);
  f[2] = __uint_as_float(u.y << 16); f[3] = __uint_as_float(u.y & 0xffff0000u);
  f[4] = __uint_as_float(u.z << 16); f[5] = __uint_as_float(u.z & 0xffff0000u);
  f[6] = __uint_as_float(u.w << 16); f[7] = __uint_as_float(u.w & 0xffff0000u);
}

// What the window keys' statistics are formed from.
struct WindowArgs {
  const void* q;
  const void* k;
  int n_kv_heads, G, window, head_inner;         // rows r = i*G + hh (head_inner) or r = hh*window + i
  long long k_stride_tok, k_stride_head, q_stride_seq, q_stride_row, q_stride_head;
  float scale_log2;
};
inline WindowArgs window_args(const Problem& pb, bool head_inner) {
  const slkv_params& p = pb.p;
  WindowArgs a;
  a.q = pb.q; a.k = pb.k;
  a.n_kv_heads = p.n_kv_heads; a.G = pb.G; a.window = p.window; a.head_inner = head_inner ? 1 : 0;
  a.k_stride_tok = p.k_stride_tok; a.k_stride_head = p.k_stride_head;
  a.q_stride_seq = p.q_stride_seq; a.q_stride_row = p.q_stride_row; a.q_stride_head = p.q_stride_head;
  a.scale_log2 = kLog2e / sqrtf((float)p.head_dim);
  return a;
}

// 16 rows of a segment, row0 on, by 128 threads (numbered tid, named barrier BAR): key blocks of 32 in shared memory, a lane
// per key, a warp per four rows.  out(row, maximum in log2 units, sum of 2^(x - maximum)) is called by one lane per row.
constexpr int kWinRows = 16;
__host__ __device__ constexpr int window_floats(int D) { return (32 + kWinRows) * (D + 4); }
template <typename T, int D, int BAR, typename Out>
__device__ __forceinline__ void window_rows(const WindowArgs& a, float* sh, int tid, int s, int g, int tok0, int row0, Out out) {
  constexpr int kVec = 16 / sizeof(T), kPitch = D + 4, kPerRow = D / kVec;
  float *ks = sh, *qs = sh + 32 * kPitch;
  const T* q = static_cast<const T*>(a.q);
  const T* k = static_cast<const T*>(a.k);
  const int R = a.G * a.window, lane = tid & 31, warp = tid >> 5;
  auto sync = [&]() { asm volatile("bar.sync %0, 128;" ::"n"(BAR) : "memory"); };
  auto window_row = [&](int r) { return a.head_inner ? r / a.G : r % a.window; };
  auto query_head = [&](int r) { return g * a.G + (a.head_inner ? r % a.G : r / a.window); };
  auto load = [&](float* dst, const T* src) {
    float f[kVec];
    unpack(*reinterpret_cast<const uint4*>(src), f, T());
#pragma unroll
    for (int e = 0; e < kVec; e += 4) *reinterpret_cast<float4*>(dst + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
  };
  int last = 0;                                                // the last key any of the rows sees
  for (int r = row0; r < min(row0 + kWinRows, R); ++r) last = max(last, window_row(r));
  for (int i = tid; i < kWinRows * kPerRow; i += 128) {
    const int rr = i / kPerRow, c = (i - rr * kPerRow) * kVec, r = min(row0 + rr, R - 1);
    load(qs + rr * kPitch + c, q + s * a.q_stride_seq + window_row(r) * a.q_stride_row + (long long)query_head(r) * a.q_stride_head + c);
  }
  float m[4], z[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) { m[u] = -INFINITY; z[u] = 0.f; }
  for (int j0 = 0; j0 <= last; j0 += 32) {
    sync();
    for (int i = tid; i < 32 * kPerRow; i += 128) {
      const int jj = i / kPerRow, c = (i - jj * kPerRow) * kVec, j = min(j0 + jj, a.window - 1);
      load(ks + jj * kPitch + c, k + (long long)(tok0 + j) * a.k_stride_tok + (long long)g * a.k_stride_head + c);
    }
    sync();
    f32x2 acc[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      const ulonglong2 kv = *reinterpret_cast<const ulonglong2*>(ks + lane * kPitch + c);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(qs + (warp * 4 + u) * kPitch + c);
        acc[u] = fma2(kv.x, qv.x, acc[u]);
        acc[u] = fma2(kv.y, qv.y, acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = min(row0 + warp * 4 + u, R - 1);
      const bool seen = j0 + lane <= window_row(r);
      const float x = sum_of(acc[u]) * a.scale_log2;
      float mx = seen ? x : -INFINITY;
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (!(mx > -INFINITY)) continue;                         // the row sees none of these keys (uniform over the warp)
      const float mn = fmaxf(m[u], mx);
      float e = seen ? exp2f(x - mn) : 0.f;
      for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
      z[u] = z[u] * exp2f(m[u] - mn) + e;                      // exp2f(-inf) = 0 covers the first block
      m[u] = mn;
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = row0 + warp * 4 + u;
    if (lane == 0 && r < R) out(r, m[u], z[u]);
  }
}

}  // namespace
}  // namespace slkv

// whtmix_small.cuh -- fp32 / bf16 planes of 2^10 .. 2^13 elements (Section III-B map and its backward), one tile of 2^13
// elements (2^(13-M) whole planes) per CTA of 128 threads, 64 elements a thread.
//
// A tile takes the three-phase kernel's row rounds (whtmix_tri.cuh: A on bits {0, 1, 9..}, one shared-memory exchange, B on
// bits {3..8} and {2} by shuffles) forward, the gain G/L, and the same rounds back; bits from M up, which number planes, are
// left out of round A.  Round B needs 64 registers a thread for the data, so four CTAs share an SM and hide one
// another's latency; nothing but X, G and Y moves.  The generic tile engine spends five rounds of 4-byte shared-memory
// accesses each way and pads planes by copies: [200, 64, 64] f32 forward 7.4 -> 5.6 us, forward and backward 26.5 -> 14.9; [2000, 64,
// 64] bf16 35.7 -> 15.9 and 194 -> 63.6; [50, 62 of 64, 64] f32 37.1 -> 12.8.
// The backward holds the spectrum of X in registers beside dY and writes the dG terms (W X)(W dY)/L plane by plane;
// k_small_dg adds them up in ascending b.
#pragma once

#include "whtmix_tri.cuh"

namespace whtmix {
namespace sml {

using tri::bf2;
using tri::bf_in;
using tri::mul2;
constexpr int WT = 128;

// Element 4 t + 512 v of the tile as (plane, element): its place in the stored planes (lv elements each), and whether it is
// there.  M <= 13.
template <int M>
__device__ __forceinline__ bool place(const Params& P, long long tile, int t, int v, long long* at) {
  const int e = 4 * t + 512 * v, r = e & ((1 << M) - 1);
  const long long b = (tile << (13 - M)) + (e >> M);
  *at = b * P.lv + r;
  return b < P.B && r < P.lv;
}
template <int D, int M>
__device__ __forceinline__ void load(const Params& P, const void* src, long long tile, int t, float2 (&a)[16][2]) {
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    long long at;
    const bool in = place<M>(P, tile, t, v, &at);
    if constexpr (D == DT_BF16) {
      const uint2 u = in ? __ldcs(reinterpret_cast<const uint2*>(static_cast<const unsigned short*>(src) + at)) : make_uint2(0u, 0u);
      a[v][0] = make_float2(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u));
      a[v][1] = make_float2(__uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
    } else {
      const float4 q = in ? __ldcs(reinterpret_cast<const float4*>(static_cast<const float*>(src) + at)) : make_float4(0.f, 0.f, 0.f, 0.f);
      a[v][0] = make_float2(q.x, q.y);
      a[v][1] = make_float2(q.z, q.w);
    }
  }
}
template <int D, int M>
__device__ __forceinline__ void store(const Params& P, void* dst, long long tile, int t, const float2 (&a)[16][2]) {
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    long long at;
    if (!place<M>(P, tile, t, v, &at)) continue;
    if constexpr (D == DT_BF16) {
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(a[v][0].x, a[v][0].y), h1 = __floats2bfloat162_rn(a[v][1].x, a[v][1].y);
      __stcs(reinterpret_cast<uint2*>(static_cast<unsigned short*>(dst) + at),
             make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1)));
    } else {
      __stcs(reinterpret_cast<float4*>(static_cast<float*>(dst) + at), make_float4(a[v][0].x, a[v][0].y, a[v][1].x, a[v][1].y));
    }
  }
}
template <int M>
__device__ __forceinline__ void round_a(float2 (&a)[16][2]) {
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    bf_in(a[v][0]);
    bf_in(a[v][1]);
    bf2(a[v][0], a[v][1]);
  }
#pragma unroll
  for (int h = 1; h < (1 << (M - 9)); h <<= 1)
#pragma unroll
    for (int v = 0; v < 16; ++v)
      if ((v & h) == 0) {
        bf2(a[v][0], a[v + h][0]);
        bf2(a[v][1], a[v + h][1]);
      }
}
// quads (round A) <-> round B's layout through the exchange buffer
__device__ __forceinline__ void to_b(float* buf, int t, const tri::RowB& rb, const float2 (&a)[16][2], float2 (&b)[32]) {
#pragma unroll
  for (int v = 0; v < 16; ++v)
    *reinterpret_cast<float4*>(buf + tri::quad_word(t, v)) = make_float4(a[v][0].x, a[v][0].y, a[v][1].x, a[v][1].y);
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 32; ++s) b[s] = make_float2(buf[rb.word(s)], buf[rb.word(s + 32)]);
}
__device__ __forceinline__ void to_a(float* buf, int t, const tri::RowB& rb, const float2 (&b)[32], float2 (&a)[16][2]) {
#pragma unroll
  for (int s = 0; s < 32; ++s) {
    buf[rb.word(s)] = b[s].x;
    buf[rb.word(s + 32)] = b[s].y;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const float4 q = *reinterpret_cast<const float4*>(buf + tri::quad_word(t, v));
    a[v][0] = make_float2(q.x, q.y);
    a[v][1] = make_float2(q.z, q.w);
  }
}
// round B's element s of thread t: tile element b_base(t) + 8 s
__device__ __forceinline__ int b_base(int t) { return (t & 7) + 512 * (t >> 3); }

template <int M>
__device__ __forceinline__ void apply_gain(const Params& P, int t, float2 (&b)[32]) {
  const float* g = static_cast<const float*>(P.g) + (b_base(t) & ((1 << M) - 1));
  const float2 sc = make_float2(P.scale, P.scale);
#pragma unroll
  for (int s = 0; s < 32; ++s) b[s] = mul2(b[s], mul2(make_float2(__ldg(g + 8 * s), __ldg(g + 8 * (s + 32))), sc));
}

template <int D, int M>
__global__ void __launch_bounds__(WT, 4) k_forward_small(Params P) {
  __shared__ __align__(16) float buf[tri::TILE];
  pdl_wait();
  const int t = threadIdx.x;
  const tri::RowB rb(t);
  float2 a[16][2], b[32];
  load<D, M>(P, P.x, blockIdx.x, t, a);
  round_a<M>(a);
  to_b(buf, t, rb, a, b);
  tri::round_b(b);
  apply_gain<M>(P, t, b);
  tri::round_b(b);
  to_a(buf, t, rb, b, a);  // (each thread writes only the words it read)
  round_a<M>(a);
  store<D, M>(P, P.y, blockIdx.x, t, a);
  pdl_trigger();
}

// Planes b0 .. of the batch, P.gp of them (P.x, P.dy, P.dx and P.B already moved to b0): dX, and the dG terms of plane b at
// P.ws[b << M].
template <int D, int M>
__global__ void __launch_bounds__(WT, 2) k_backward_small(Params P) {
  __shared__ __align__(16) float buf[tri::TILE];
  pdl_wait();
  const int t = threadIdx.x;
  const tri::RowB rb(t);
  float2 a[16][2], xh[32], b[32];
  load<D, M>(P, P.x, blockIdx.x, t, a);
  round_a<M>(a);
  to_b(buf, t, rb, a, xh);
  load<D, M>(P, P.dy, blockIdx.x, t, a);
  tri::round_b(xh);
  round_a<M>(a);
  __syncthreads();
  to_b(buf, t, rb, a, b);
  tri::round_b(b);
  const int e = b_base(t);
  if ((static_cast<long long>(blockIdx.x) << (13 - M)) + (e >> M) < P.B) {
    float* part = static_cast<float*>(P.ws) + (static_cast<long long>(blockIdx.x) << 13) + e;
    const float2 sc = make_float2(P.scale, P.scale);
#pragma unroll
    for (int s = 0; s < 32; ++s) {
      const float2 p = mul2(mul2(xh[s], b[s]), sc);
      __stcg(part + 8 * s, p.x);
      __stcg(part + 8 * (s + 32), p.y);
    }
  }
  apply_gain<M>(P, t, b);
  tri::round_b(b);
  to_a(buf, t, rb, b, a);
  round_a<M>(a);
  store<D, M>(P, P.dx, blockIdx.x, t, a);
  pdl_trigger();
}

// dG = (first ? 0 : dG) + the terms of planes 0 .. nb - 1, in ascending order, 32 positions a CTA: the warps stage 128
// planes at a time in shared memory (read plane after plane from L2 by the summing thread, the sum took the latency of
// one load per few planes), one warp adds them.
constexpr int DG_PLANES = 128;
constexpr int DG_THREADS = 256;
static __global__ void __launch_bounds__(DG_THREADS) k_small_dg(float* dg, const float* part, int m, long long nb, int first) {
  __shared__ float st[2][DG_PLANES][32];
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* p = part + 32ll * blockIdx.x + lane;
  float* out = dg + 32ll * blockIdx.x + lane;
  float acc = warp == 0 && !first ? __ldcg(out) : 0.f;
  constexpr int PER = DG_PLANES / (DG_THREADS / 32);
  int buf = 0;
  for (long long b0 = 0; b0 < nb; b0 += DG_PLANES, buf ^= 1) {
    float v[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const long long b = b0 + warp * PER + i;
      v[i] = b < nb ? __ldcg(p + (b << m)) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) st[buf][warp * PER + i][lane] = v[i];
    __syncthreads();  // (the other buffer's reads lie before the barrier of the round in between)
    if (warp == 0) {
      const int n = static_cast<int>(nb - b0 < DG_PLANES ? nb - b0 : DG_PLANES);
#pragma unroll 16
      for (int i = 0; i < n; ++i) acc += st[buf][i][lane];
    }
  }
  if (warp == 0) __stcg(out, acc);
  pdl_trigger();
}

}  // namespace sml
}  // namespace whtmix

// whtmix_plane.cuh -- forward for planes of 2^14 <= N*C <= 2^16 elements, one plane per CTA, the whole fp32 plane held in the
// SM's tensor memory between its two ends (Section III-B, Eq. 2-3: Y = H_N (G o (H_N X H_C)) H_C / (N C), flattened to one
// 2^m-point transform).
//
// Element r = l + 128 n of the plane lives in tensor-memory lane l (bits 0..6), column n (bits 7..m-1); a worker of 128
// threads (thread t of worker i is lane t) takes blocks i, i + 4 of 64 columns, NB = 2^(m-13) of them.
//   in      the low seven bits.  bf16: on the tensor cores, D[l, n] = sum_k H_128[l, k] x[128 n + k] (bf16 times +-1 is
//           exact, fp32 accumulation).  fp32: in registers, 64 consecutive elements a thread (bits 0..5) and one shuffle
//           stage (bit 6), then through shared memory to lane = bits 0..6.
//   middle  per lane: bits 7..12 of each block, the block bits 13.. with the gain G/L between their two passes, and bits
//           7..12 again, all between registers and tensor memory (the warps of a lane quarter share its lanes).
//   out     the low seven bits again, as fp32 in, and out through the same shared memory in coalesced stores.
// Nothing but X, G and Y crosses HBM and nothing crosses L2 twice; a batch of B planes is B CTAs.
//
// What bounds it: the additions and the shared-memory data path of one SM (for a 2^16-element plane about 6.7 and 6 us of
// the 15.6 that 128 of them take, [128, 512, 128] bf16) and, for a single small plane, the chain of launch, load, rounds and
// store.  Measured against the previous kernel (rows of 2^14 in two workers of 128 elements a thread):
// [128, 512, 128] bf16 23.4 -> 15.6 us, [1, 256, 64] f32 10.5 -> 6.2, [300, 256, 64] f32 24.0 -> 11.7, bf16 18.8 -> 9.4,
// [128, 512, 64] f32 18.9 -> 11.8, [96, 512, 128] f32 33.4 -> 22.8.
#pragma once

#include "whtmix_tri.cuh"

namespace whtmix {
namespace pln {

using tri::bf_in;
using tri::bf2;
using tri::mul2;
constexpr int WT = 128;

// These kernels use no workspace: a wait that gives up sets this header's error word (read by whtmix_sync).
static __device__ GridBarrier plane_barrier;

template <int D, int M>
struct Plane {
  static constexpr int NB = 1 << (M - 13);                 // blocks of 64 columns
  static constexpr int WORKERS = NB < 4 ? NB : 4;
  static constexpr int THREADS = WT * WORKERS;
  static constexpr int BPW = NB / WORKERS;                 // blocks per worker
  static constexpr int COLS = 64 * NB;                     // tensor-memory columns
  static constexpr int SLOT_BYTES = WORKERS * 32768;       // a 2^13-element block per worker; bf16 X before that
  static constexpr bool MMA = D == DT_BF16;
  static constexpr size_t SMEM = SLOT_BYTES + (MMA ? tri::H_BYTES : 0);
  static constexpr int W = 32 / NB, WP = W / 2;            // rows of each block per pass of the block bits
  static constexpr int PASSES = 64 / WORKERS / W;
  static constexpr int MMAS = MMA ? (COLS + 255) / 256 : 1;
  static_assert(!MMA || COLS * 256 <= SLOT_BYTES, "X fits the slots");
};

// Block layout in a slot: element e = 64 R + 4 c + i (R = bits 6..12, chunk c) at float 64 R + 4 (c ^ (R mod 8)) + i, so that 64
// consecutive elements per thread, 128 consecutive lanes per warp and linear 16-byte chunks are all conflict-free.
// Thread t's 64 consecutive elements: R = t.
__device__ __forceinline__ float4* chunk_of(float* slot, int R, int c) {
  return reinterpret_cast<float4*>(slot + 64 * R + 4 * (c ^ (R & 7)));
}
// lane order: element t + 128 n
struct LaneWord {
  int q[4];
  __device__ __forceinline__ explicit LaneWord(int t) {
    const int b = t ^ (((t >> 6) & 1) << 2);
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = b ^ (k << 3);
  }
  __device__ __forceinline__ int operator()(int n) const { return q[n & 3] + 128 * n; }
};

// bits 0..5 of 64 consecutive elements in registers, bit 6 across lanes l, l ^ 1
__device__ __forceinline__ void low_bits(float2 (&a)[16][2]) {
  tri::round_a(a);
  const float2 sgn = (threadIdx.x & 1) ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
#pragma unroll
  for (int v = 0; v < 16; ++v)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, a[v][i].x, 1), __shfl_xor_sync(0xffffffffu, a[v][i].y, 1));
      a[v][i] = fast::fma2(a[v][i], sgn, p);
    }
}
__device__ __forceinline__ void read_chunks(float* slot, int t, float2 (&a)[16][2]) {
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const float4 q = *chunk_of(slot, t, c);
    a[c][0] = make_float2(q.x, q.y);
    a[c][1] = make_float2(q.z, q.w);
  }
}
__device__ __forceinline__ void write_chunks(float* slot, int t, const float2 (&a)[16][2]) {
#pragma unroll
  for (int c = 0; c < 16; ++c) *chunk_of(slot, t, c) = make_float4(a[c][0].x, a[c][0].y, a[c][1].x, a[c][1].y);
}
// bits 7..12 of 64 columns
__device__ __forceinline__ void column_bits(float2 (&v)[32]) {
#pragma unroll
  for (int j = 0; j < 32; ++j) bf_in(v[j]);
  tri::bfly32<0>(v);
}
__device__ __forceinline__ void to_tmem(uint32_t ta, const float2 (&v)[32]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) tri::st_pairs<8>(ta + 16 * q, v + 8 * q);
}

template <int D, int M>
__global__ void __launch_bounds__(Plane<D, M>::THREADS, 512 / Plane<D, M>::THREADS) k_forward_plane(Params P) {
  using C = Plane<D, M>;
  constexpr int NB = C::NB, W = C::W, WP = C::WP;
  extern __shared__ __align__(1024) unsigned char pl_smem[];
  __shared__ uint64_t mma_done[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int dead;
  const int worker = threadIdx.x / WT, t = threadIdx.x % WT, quarter = (threadIdx.x >> 5) & 3;
  float* slot = reinterpret_cast<float*>(pl_smem) + worker * tri::TILE;
  const uint32_t smem = tc::smem_u32(pl_smem);
  if (threadIdx.x < 32) tc::tmem_alloc(&tmem_slot, C::COLS);
  if constexpr (C::MMA) {
    tri::build_h<C::THREADS>(pl_smem + C::SLOT_BYTES);
    if (threadIdx.x == 0) {
      dead = 0;
      for (int i = 0; i < 2; ++i) tc::mbar_init(&mma_done[i], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tri::fence_async();
  }
  fast::tmem_fence_before();
  __syncthreads();
  fast::tmem_fence_after();
  pdl_wait();
  const uint32_t ta = tmem_slot + (static_cast<uint32_t>(32 * quarter) << 16);
  const long long e0 = static_cast<long long>(blockIdx.x) * P.lv;
  const int lv = static_cast<int>(P.lv);
  const float2 sc = make_float2(P.scale, P.scale);
  auto warps_sync = [&] {  // the warps of this lane quarter
    fast::tmem_wait_st();
    fast::tmem_fence_before();
    asm volatile("bar.sync %0, %1;" ::"r"(quarter + 5), "r"(32 * C::WORKERS) : "memory");
    fast::tmem_fence_after();
  };
  // in, and bits 7..12
  if constexpr (C::MMA) {
    constexpr int ROWS = C::COLS, PANEL = ROWS * 128;           // 128 elements a row, two panels of 64
    constexpr int PART = (ROWS < 256 ? ROWS : 256) * 16;        // 16-byte chunks per product
    const unsigned short* x = static_cast<const unsigned short*>(P.x) + e0;
#pragma unroll
    for (int j = 0; j < C::MMAS; ++j) {
#pragma unroll
      for (int i = 0; i < PART / C::THREADS; ++i) {
        const int q = PART * j + C::THREADS * i + threadIdx.x, n = q >> 4, c = q & 15;
        tri::cp_async16z(smem + (c >> 3) * PANEL + n * 128 + (((c & 7) ^ (n & 7)) << 4), x + (8 * q < lv ? 8 * q : 0), 8 * q < lv);
      }
      fast::cp_async_commit();
    }
#pragma unroll
    for (int j = 0; j < C::MMAS; ++j) {
      if (j + 1 < C::MMAS) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 0;" ::: "memory");
      tri::fence_async();
      __syncthreads();
      if (threadIdx.x == 0) {
        constexpr int N = ROWS < 256 ? ROWS : 256;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          tc::mma_bf16(tmem_slot + 256 * j, tc::sw128_desc(smem + C::SLOT_BYTES + (k >> 2) * 16384 + (k & 3) * 32),
                       tc::sw128_desc(smem + (k >> 2) * PANEL + 256 * 128 * j + (k & 3) * 32), tc::instr_desc(128, N), k > 0);
        tc::mma_commit(&mma_done[j]);
      }
    }
#pragma unroll 1
    for (int k = 0; k < C::BPW; ++k) {
      const int b = worker + C::WORKERS * k;
      tri::wait_bar(&mma_done[b >> 2], 0, &plane_barrier, &dead);
      __syncwarp();
      fast::tmem_fence_after();
      float2 v[32];
      tri::read_row(ta + 64 * b, v);
      column_bits(v);
      to_tmem(ta + 64 * b, v);
    }
  } else {
    const float* x = static_cast<const float*>(P.x) + e0;
    const LaneWord lw(t);
#pragma unroll 1
    for (int k = 0; k < C::BPW; ++k) {
      const int b = worker + C::WORKERS * k;
      const uint32_t d = tc::smem_u32(slot);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int q = t + 128 * i, o = tri::TILE * b + 4 * q;
        tri::cp_async16z(d + (q >> 4) * 256 + (((q & 15) ^ ((q >> 4) & 7)) << 4), x + (o < lv ? o : 0), o < lv);
      }
      fast::cp_async_commit();
      fast::cp_async_wait_all();
      tri::worker_sync(worker);
      {
        float2 a[16][2];
        read_chunks(slot, t, a);
        low_bits(a);
        write_chunks(slot, t, a);
      }
      tri::worker_sync(worker);
      float2 v[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = make_float2(slot[lw(2 * j)], slot[lw(2 * j + 1)]);
      if (k + 1 < C::BPW) tri::worker_sync(worker);  // the slot is free for the next block
      column_bits(v);
      to_tmem(ta + 64 * b, v);
    }
  }
  // block bits, gain, block bits: the rows 64 s + low .. of this lane, s = 0..NB-1
  const float* g = static_cast<const float*>(P.g) + t;
  auto load_gains = [&](float2 (&gg)[16], int low) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float* p = g + 128 * (64 * (k / WP) + low + 2 * (k % WP));
      gg[k] = make_float2(__ldg(p), __ldg(p + 128));
    }
  };
  auto pass_of = [&](const float2 (&gg)[16], int low) {
    float2 v[16];
#pragma unroll
    for (int s = 0; s < NB; ++s) tri::ld_pairs<WP>(ta + 64 * s + low, v + WP * s);
    fast::tmem_wait_ld();
    auto across = [&] {
#pragma unroll
      for (int h = WP; h < 16; h <<= 1)
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if ((k & h) == 0) bf2(v[k], v[k + h]);
    };
    across();
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = mul2(v[k], mul2(gg[k], sc));
    across();
#pragma unroll
    for (int s = 0; s < NB; ++s) tri::st_pairs<WP>(ta + 64 * s + low, v + WP * s);
  };
  {
    const int low0 = (64 / C::WORKERS) * worker;
    float2 ga[16], gb[16];
    load_gains(ga, low0);
    warps_sync();
#pragma unroll 1
    for (int pass = 0; pass < C::PASSES; pass += 2) {
      load_gains(gb, low0 + W * (pass + 1));
      pass_of(ga, low0 + W * pass);
      if (pass + 2 < C::PASSES) load_gains(ga, low0 + W * (pass + 2));
      pass_of(gb, low0 + W * (pass + 1));
    }
    warps_sync();
  }
  // bits 7..12, and out
  const LaneWord lw(t);
#pragma unroll 1
  for (int k = 0; k < C::BPW; ++k) {
    const int b = worker + C::WORKERS * k;
    {
      float2 v[32];
      tri::read_row(ta + 64 * b, v);
      column_bits(v);
      if (!C::MMA || k > 0) tri::worker_sync(worker);  // the slot's last reads (bf16, k = 0: X's products are done)
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        slot[lw(2 * j)] = v[j].x;
        slot[lw(2 * j + 1)] = v[j].y;
      }
    }
    tri::worker_sync(worker);
    float2 a[16][2];
    read_chunks(slot, t, a);
    low_bits(a);
    const int first = tri::TILE * b;
    if constexpr (D == DT_BF16) {
      tri::worker_sync(worker);
      // 64 elements (128 bytes) a thread, 16-byte chunk j of row t at j ^ (t mod 8)
      unsigned char* st = reinterpret_cast<unsigned char*>(slot);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(a[2 * j + (i >> 1)][i & 1].x, a[2 * j + (i >> 1)][i & 1].y);
          w[i] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(st + t * 128 + ((j ^ (t & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      tri::worker_sync(worker);
      unsigned short* y = static_cast<unsigned short*>(P.y) + e0 + first;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int q = t + 128 * i, R = q >> 3;
        const uint4 u = *reinterpret_cast<const uint4*>(st + R * 128 + (((q & 7) ^ (R & 7)) << 4));
        if (first + 8 * q < lv) __stcs(reinterpret_cast<uint4*>(y + 8 * q), u);
      }
    } else {
      write_chunks(slot, t, a);
      tri::worker_sync(worker);
      float* y = static_cast<float*>(P.y) + e0 + first;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int q = t + 128 * i;
        const float4 u = *chunk_of(slot, q >> 4, q & 15);
        if (first + 4 * q < lv) __stcs(reinterpret_cast<float4*>(y + 4 * q), u);
      }
    }
  }
  pdl_trigger();
  fast::tmem_fence_before();
  __syncthreads();
  fast::tmem_fence_after();
  if (threadIdx.x < 32) tc::tmem_dealloc(tmem_slot, C::COLS);
}

}  // namespace pln
}  // namespace whtmix

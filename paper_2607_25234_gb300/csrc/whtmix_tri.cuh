// whtmix_tri.cuh -- three-phase forward for fp32 / bf16 planes, every workspace and input access staged
// asynchronously through shared memory (Section III-B map; see whtmix_kernels.cuh for the flattening).
//
// A plane of 2^m elements is 2^Q rows of 2^13 contiguous elements (m = 13 + Q), transformed as
//   phase 1  every row: its 13 bits                                     X  -> workspace (fp32)
//   phase 2  every column: its Q bits, gain G/L, the Q bits again       workspace -> workspace
//   phase 3  every row: its 13 bits again                               workspace -> Y
// with the bounded device-wide barrier between phases.  The workspace is in natural order.
//
// One CTA of 16 warps per SM, 64 elements a thread (128 registers).  A worker of 128 threads holds a row; a ring of
// shared-memory slots keeps the next rows in flight, so that loads, butterflies and stores of different rows overlap.
//   rows of bf16 X  the 7 low bits on the tensor cores: D[i, n] = sum_k H_128[i, k] x[128 n + k] (M = 128,
//            N = 64, K = 128; bf16 times +-1 is exact, fp32 accumulation), then lane i of the worker reads its
//            64 values n from tensor memory and runs the other 6 bits in registers: no exchange at all;
//   other rows  two register rounds with one exchange inside the slot: A on bits {0, 1, 9..12} (16-byte
//            vectors), B on bits {3..8} and, by one shuffle stage, bit 2;
//   columns  a warp lane is a column (a warp reads and writes whole row segments): up to 64 rows in a thread's registers,
//            taller columns in that lane's tensor memory, which the warps of a lane quarter share.
// Slots are XOR-swizzled so that every access is conflict-free.
//
// What bounds it: the fp32 workspace crosses between SMs through L2 twice (32 MiB each way at 2^23 elements;
// measured without arithmetic: 4.4 us to write it, 5.9 to read and write it by columns, 1.8 to read it back,
// 1.4 per barrier), and within an SM the shared-memory data path (one 128-byte wavefront a cycle) more than the
// additions.  Measured against the previous kernel (8 warps, 128 elements a thread, columns read straight from
// L2): [32, 4096, 64] f32 40.6 -> 32.9 us, [1, 4096, 64] bf16 11.6 -> 8.9, [1, 65536, 128] bf16 41.9 -> 38.1, with
// log gains 39.2 -> 35.4, [1, 32768, 128] bf16 28.4 -> 26.6, [8, 4096, 256] f32 42.6 -> 36.7; of that the tensor-core
// rows took phase 1 of the 2^23-element plane from 13.5 to 8.7 us.
//
// What the tensor cores' additions cost in precision: their fp32 accumulator truncates where an addition rounds.  bf16 outputs hide
// it.  dG, the one fp32 result of bf16 inputs, against 64 bits, as a multiple of the error of the same values passed as fp32 (whose
// rows are additions): 0.97 to 1.02 (8e-8 to 1.4e-7) for N(0, 1) activations and gradients, planes of 2^14 to 2^23; 1.5 to 2.0
// (2.1e-7 to 3.1e-7) where a few values dominate their row, N(0, 1) e^(2 N(0, 1)).  Two accumulators of 64 k each make the latter
// 1.2 to 1.4, the backward of single small planes 3 to 6% slower; rows by additions 1.0, the training step 349 -> 376 us.
#pragma once

#include <type_traits>

#include "whtmix_fast.cuh"
#include "whtmix_tc.cuh"

namespace whtmix {
namespace tri {

using fast::add2;
using fast::bf2;
using fast::bf_in;
using fast::mul2;

constexpr int THREADS = 512;
constexpr int WORKERS = 4;
constexpr int WT = 128;              // threads per worker
constexpr int R = 13;                // row bits
constexpr int TILE = 1 << R;         // elements per row
constexpr int SLOTS = 6;             // ring of rows
constexpr int XSLOTS = 3;            // bf16 X rows (16 KiB) staged per worker
constexpr int H_BYTES = 128 * 128 * 2;  // H_128 in bf16, the tensor cores' A operand
constexpr int SLOT_BYTES = SLOTS * TILE * 4;
static_assert(WORKERS * XSLOTS * TILE * 2 <= SLOT_BYTES, "the X staging areas share the slots");
// more than half an SM: one CTA per SM (both for the barriers and for tensor memory)
template <int D>
constexpr size_t smem_bytes() { return SLOT_BYTES + (D == DT_BF16 ? H_BYTES : 0); }

// Mbarriers of the ring: two per slot, taken in turn, so that all uses of one barrier belong to one worker (12 is a
// multiple of four workers) and no wait can start two phases ahead.
constexpr int ROW_BARS = 2 * SLOTS;

__device__ __forceinline__ void worker_sync(int worker) {
  asm volatile("bar.sync %0, %1;" ::"r"(worker + 1), "r"(WT) : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// this thread arrives on `full` once its earlier cp.async copies have landed
__device__ __forceinline__ void cp_async_arrive(uint64_t* full) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(full)) : "memory");
}
// Bounded wait for phase `parity` of an mbarrier.  A wait that gives up sets the workspace's error word
// and `dead`, which ends every later wait at once; the kernel then runs to its end on whatever the buffers
// hold.
__device__ __forceinline__ void wait_bar(uint64_t* bar, uint32_t parity, GridBarrier* gb, volatile int* dead) {
  const uint32_t a = tc::smem_u32(bar);
  unsigned long long t0 = 0;
  for (unsigned polls = 0;; ++polls) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (done) return;
    if ((polls & 63u) == 63u) {
      if (*dead) return;
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > BARRIER_TIMEOUT_NS) {
        atomicOr(&gb->err, 1u);
        *dead = 1;
        return;
      }
    }
  }
}
// use `seq` of a ring of `bars` barriers
__device__ __forceinline__ void wait_full(uint64_t* full, unsigned seq, unsigned bars, GridBarrier* gb, volatile int* dead) {
  wait_bar(full + seq % bars, (seq / bars) & 1u, gb, dead);
}
// Share of CTA blockIdx.x of `units` units (units < 2^22: the product fits 32 bits)
__device__ __forceinline__ void share(unsigned units, int* begin, int* end) {
  *begin = static_cast<int>(units * blockIdx.x / gridDim.x);
  *end = static_cast<int>(units * (blockIdx.x + 1) / gridDim.x);
}

// Butterflies over bits [B0, 5) of the index of v[32] (packed pairs).
template <int B0>
__device__ __forceinline__ void bfly32(float2 (&v)[32]) {
#pragma unroll
  for (int b = B0 < 0 ? 0 : B0; b < 5; ++b)
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if ((i & (1 << b)) == 0) bf2(v[i], v[i + (1 << b)]);
}

// ---------------------------------------------------------------------------------------------
// Rows of bf16 X on the tensor cores.  Both operands are K-major in 128-byte-swizzled panels of 64 k
// (16-byte chunk j of row r at chunk j ^ (r mod 8)).
//
// H_128 (A: 128 rows, two panels of 16 KiB): entry (i, k) = (-1)^popcount(i & k).
template <int NT = THREADS>
__device__ __forceinline__ void build_h(unsigned char* sh) {
  for (int q = threadIdx.x; q < 128 * 16; q += NT) {
    const int i = q >> 4, c = q & 15;  // k = 8 c ..
    const uint32_t flip = (__popc(i & (8 * c)) & 1) ? 0x80008000u : 0u;
    uint32_t w[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t lo = (__popc(i & (2 * p)) & 1) ? 0xBF80u : 0x3F80u;
      const uint32_t hi = (__popc(i & (2 * p + 1)) & 1) ? 0xBF80u : 0x3F80u;
      w[p] = (lo | (hi << 16)) ^ flip;
    }
    *reinterpret_cast<uint4*>(sh + (c >> 3) * 16384 + i * 128 + (((c & 7) ^ (i & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
// X row (64 tile rows n of 128 contiguous elements, B: two panels of 8 KiB) by the worker's cp.async; elements
// at offsets >= lim are zero.
__device__ __forceinline__ void load_x_bf16(const unsigned short* src, int lim, uint32_t dst, int t) {
  const int n = t >> 4, c = t & 15;
  const uint32_t d = dst + (c >> 3) * 8192 + n * 128 + (((c & 7) ^ (n & 7)) << 4);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int o = 8 * t + 1024 * i;
    cp_async16z(d + 1024 * i, src + (o < lim ? o : 0), o < lim);
  }
}
// D (TMEM columns d .. d + 63) = H_128 x row, one thread
__device__ __forceinline__ void mma_row(uint32_t d, uint32_t h, uint32_t x) {
#pragma unroll
  for (int k = 0; k < 8; ++k)
    tc::mma_bf16(d, tc::sw128_desc(h + (k >> 2) * 16384 + (k & 3) * 32), tc::sw128_desc(x + (k >> 2) * 8192 + (k & 3) * 32),
                 tc::instr_desc(128, 64), k > 0);
}
// this thread's lane of D: element r = t + 128 n, pairs (n, n + 1)
__device__ __forceinline__ void read_row(uint32_t ta, float2 (&v)[32]) {
  float f[64];
#pragma unroll
  for (int c = 0; c < 64; c += 16) fast::tmem_ld16(ta + c, *reinterpret_cast<float(*)[16]>(f + c));
  fast::tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = make_float2(f[2 * i], f[2 * i + 1]);
}

// ---------------------------------------------------------------------------------------------
// Rows in registers.  Round A: thread t holds the quads (r0, r1) at 4 t + 512 v, v = 0..15 (r9..r12); round B:
// lane l holds r0, r1, r2 = l mod 8, r9, r10 = l / 8, warp r11, r12, registers r3..r8 as pairs (s, s + 32).  In
// the slot, word bits 3, 4 are XORed with r9, r10.
__device__ __forceinline__ int quad_word(int t, int v) { return ((4 * t) ^ ((v & 3) << 3)) + 512 * v; }
__device__ __forceinline__ void round_a(float2 (&a)[16][2]) {
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    bf_in(a[v][0]);
    bf_in(a[v][1]);
    bf2(a[v][0], a[v][1]);
  }
#pragma unroll
  for (int h = 1; h < 16; h <<= 1)
#pragma unroll
    for (int v = 0; v < 16; ++v)
      if ((v & h) == 0) {
        bf2(a[v][0], a[v + h][0]);
        bf2(a[v][1], a[v + h][1]);
      }
}
__device__ __forceinline__ void round_b(float2 (&b)[32]) {
#pragma unroll
  for (int s = 0; s < 32; ++s) bf_in(b[s]);
  bfly32<0>(b);
  // r2 across lanes l, l ^ 4
  const float2 sgn = (threadIdx.x & 4) ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
#pragma unroll
  for (int s = 0; s < 32; ++s) {
    const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, b[s].x, 4), __shfl_xor_sync(0xffffffffu, b[s].y, 4));
    b[s] = fast::fma2(b[s], sgn, p);
  }
}
// Slot word of round B's element s.
struct RowB {
  int q[4];
  __device__ __forceinline__ RowB(int t) {
    const int l = t & 31, h = l >> 3, w = t >> 5;
    const int base = (l & 7) + 512 * (h + 4 * w);
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = base + 8 * (k ^ h);
  }
  __device__ __forceinline__ int word(int s) const { return q[s & 3] + 32 * (s >> 2); }
};
// A row of fp32 (lim elements present, the rest zero) into a slot, by one worker.
__device__ __forceinline__ void load_row(const float* src, int lim, float* slot, int t, uint64_t* full) {
  const uint32_t d = tc::smem_u32(slot);
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const int o = 4 * t + 512 * v;
    cp_async16z(d + 4 * quad_word(t, v), src + (o < lim ? o : 0), o < lim);
  }
  cp_async_arrive(full);
}

// Phase 1, fp32: the row in `slot` -> workspace row.  `done` is called once the slot is free.
template <class Done>
__device__ __forceinline__ void row_in(float* slot, float* ws_row, int t, int worker, const Done& done) {
  {
    float2 a[16][2];
#pragma unroll
    for (int v = 0; v < 16; ++v) {
      const float4 q = *reinterpret_cast<const float4*>(slot + quad_word(t, v));
      a[v][0] = make_float2(q.x, q.y);
      a[v][1] = make_float2(q.z, q.w);
    }
    round_a(a);
#pragma unroll
    for (int v = 0; v < 16; ++v)
      *reinterpret_cast<float4*>(slot + quad_word(t, v)) = make_float4(a[v][0].x, a[v][0].y, a[v][1].x, a[v][1].y);
  }
  worker_sync(worker);
  const RowB rb(t);
  float2 b[32];
#pragma unroll
  for (int s = 0; s < 32; ++s) b[s] = make_float2(slot[rb.word(s)], slot[rb.word(s + 32)]);
  worker_sync(worker);
  done();
  round_b(b);
  float* dst = ws_row + (t & 7) + 512 * (t >> 3);
#pragma unroll
  for (int s = 0; s < 32; ++s) {
    __stcg(dst + 8 * s, b[s].x);
    __stcg(dst + 8 * (s + 32), b[s].y);
  }
}

// Phase 3: the row bits of the workspace row in `slot`, into the quads of round A.  `done` is called once the slot is
// free.
template <class Done>
__device__ __forceinline__ void row_transform(float* slot, float2 (&a)[16][2], int t, int worker, const Done& done) {
  {
    const RowB rb(t);
    float2 b[32];
#pragma unroll
    for (int s = 0; s < 32; ++s) b[s] = make_float2(slot[rb.word(s)], slot[rb.word(s + 32)]);
    round_b(b);
#pragma unroll
    for (int s = 0; s < 32; ++s) {
      slot[rb.word(s)] = b[s].x;
      slot[rb.word(s + 32)] = b[s].y;
    }
  }
  worker_sync(worker);
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const float4 q = *reinterpret_cast<const float4*>(slot + quad_word(t, v));
    a[v][0] = make_float2(q.x, q.y);
    a[v][1] = make_float2(q.z, q.w);
  }
  worker_sync(worker);
  done();
  round_a(a);
}
// ... and out: the first lim elements of Y's row at dst + e0.
template <int D, class Done>
__device__ __forceinline__ void row_out(float* slot, void* dst, long long e0, int lim, int t, int worker, const Done& done) {
  float2 a[16][2];
  row_transform(slot, a, t, worker, done);
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const int o = 4 * t + 512 * v;
    if (o < lim) {
      if constexpr (D == DT_BF16) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(a[v][0].x, a[v][0].y), h1 = __floats2bfloat162_rn(a[v][1].x, a[v][1].y);
        __stcs(reinterpret_cast<uint2*>(static_cast<unsigned short*>(dst) + e0 + o),
               make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1)));
      } else {
        __stcs(reinterpret_cast<float4*>(static_cast<float*>(dst) + e0 + o),
               make_float4(a[v][0].x, a[v][0].y, a[v][1].x, a[v][1].y));
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Columns.
// Gains of one column: rows2(j) = rows j and j + 1 (j even).
template <int Q>
struct LaneFull {
  const float* p;
  __device__ __forceinline__ LaneFull(const Params& P, const float*, int col) : p(static_cast<const float*>(P.g) + col) {}
  __device__ __forceinline__ float2 rows2(int j) const { return make_float2(__ldg(p + (j << R)), __ldg(p + ((j + 1) << R))); }
};
// Separable log gains: G[n, c] = et[n] ec[c] from two tables that phase 1 builds (tab); the token table is
// stored so that a column's rows are consecutive, et[(column >> cb) 2^Q + row].
template <int Q>
struct LaneSep {
  const float* p;
  float e;
  __device__ __forceinline__ LaneSep(const Params& P, const float* tab, int col)
      : p(tab + (static_cast<long long>(col >> P.cbits) << Q)), e(tab[(1ll << (P.m - P.cbits)) + (col & ((1 << P.cbits) - 1))]) {}
  __device__ __forceinline__ float2 rows2(int j) const { return mul2(*reinterpret_cast<const float2*>(p + j), make_float2(e, e)); }
};

// C = 2^14, two rows a token: rows j and j + 1 are one token's two halves of the channels, et[j / 2] (ec[col], ec[2^13 + col]), and
// the token table is in natural order.
template <int Q>
struct LaneSepWide {
  const float* p;
  float2 e;
  __device__ __forceinline__ LaneSepWide(const Params& P, const float* tab, int col)
      : p(tab), e(make_float2(tab[(1 << (Q - 1)) + col], tab[(1 << (Q - 1)) + TILE + col])) {}
  __device__ __forceinline__ float2 rows2(int j) const { return mul2(make_float2(p[j >> 1], p[j >> 1]), e); }
};
enum Gains { FULL, LOG, LOG_WIDE };
template <int Q, Gains G> struct LaneGain { using T = LaneFull<Q>; };
template <int Q> struct LaneGain<Q, LOG> { using T = LaneSep<Q>; };
template <int Q> struct LaneGain<Q, LOG_WIDE> { using T = LaneSepWide<Q>; };

// The token of entry i of the table.
template <int Q, Gains G>
__device__ __forceinline__ long long sep_token_of(long long i, int cb) {
  return G == LOG_WIDE ? i : ((i & ((1ll << Q) - 1)) << (R - cb)) | (i >> Q);
}

__device__ __forceinline__ void tmem_ld8(uint32_t ta, float (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
               : "r"(ta) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t ta, const float (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(ta), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]) : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t ta, float (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(ta) : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t ta, const float (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
               ::"r"(ta), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]) : "memory");
}

// Staging of a warp's column blocks: NR rows of 32 columns (128 bytes a row), by the warp's own cp.async.  No group is
// committed here: the caller commits and counts groups (col_regs), or waits for every copy (col_lanes: cp_async_wait_all).
template <int NR>
__device__ __forceinline__ void stage_block(const float* src32, float* stg, int lane) {  // src32: the block's first column
  const float* s = src32 + (static_cast<long long>(lane >> 3) << R) + 4 * (lane & 7);
  const uint32_t d = tc::smem_u32(stg) + 16 * lane;
#pragma unroll
  for (int j = 0; j < NR / 4; ++j) cp_async16(d + 512 * j, s + (static_cast<long long>(4 * j) << R));
}
constexpr int WARP_STAGE = SLOT_BYTES / 4 / (THREADS / 32);  // floats of the slots per warp (12 KiB)

// Columns of up to 64 rows, whole in a thread's registers; a warp's next blocks are staged behind it.
template <int Q, class GainT>
__device__ __forceinline__ void col_regs(float* ws, int cols, const Params& P, const float* tab, float* slots) {
  constexpr int NR = 1 << Q, NP = NR / 2, m = R + Q;
  constexpr int PER = 32 * (NR < 4 ? 4 : NR);
  constexpr int RING = WARP_STAGE / PER > 3 ? 3 : WARP_STAGE / PER;  // blocks in flight
  static_assert(RING >= 1, "a block fits the warp's staging area");
  const float2 sc = make_float2(P.scale, P.scale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int first = warp * gridDim.x + blockIdx.x, step = gridDim.x * (THREADS / 32), n = cols / 32;
  float* stg = slots + warp * WARP_STAGE;
  auto block = [&](int w) { return ws + (static_cast<long long>((32 * w) >> R) << m) + ((32 * w) & (TILE - 1)); };
  auto stage = [&](int w, int slot) {
    if (w < n) {
      if constexpr (NR >= 4) {
        stage_block<NR>(block(w), stg + slot * PER, lane);
      } else {  // two rows: half the warp
        if (lane < 8 * NR)
          cp_async16(tc::smem_u32(stg + slot * PER) + 16 * lane, block(w) + (static_cast<long long>(lane >> 3) << R) + 4 * (lane & 7));
      }
    }
    fast::cp_async_commit();
  };
#pragma unroll
  for (int k = 0; k < RING; ++k) stage(first + k * step, k);
  int slot = 0;
  for (int w = first; w < n; w += step) {
    float* base = block(w) + lane;
    const GainT gain(P, tab, ((32 * w) & (TILE - 1)) + lane);
    constexpr int NG = NP < 16 ? NP : 16;  // gains loaded at a time
    float2 v[NP], gg[NG];
#pragma unroll
    for (int j = 0; j < NG; ++j) gg[j] = gain.rows2(2 * j);
    asm volatile("cp.async.wait_group %0;" ::"n"(RING - 1) : "memory");
    __syncwarp();
    const float* b = stg + slot * PER + lane;
#pragma unroll
    for (int j = 0; j < NP; ++j) v[j] = make_float2(b[64 * j], b[64 * j + 32]);
    __syncwarp();
    stage(w + RING * step, slot);
    slot = slot + 1 == RING ? 0 : slot + 1;
#pragma unroll
    for (int j = 0; j < NP; ++j) bf_in(v[j]);
    fast::bfly_all<NP>(v);
#pragma unroll
    for (int h = 0; h < NP; h += NG) {
      if (h > 0) {
#pragma unroll
        for (int j = 0; j < NG; ++j) gg[j] = gain.rows2(2 * (h + j));
      }
#pragma unroll
      for (int j = 0; j < NG; ++j) v[h + j] = mul2(v[h + j], mul2(gg[j], sc));
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) bf_in(v[j]);
    fast::bfly_all<NP>(v);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      __stcg(base + ((2 * j) << R), v[j].x);
      __stcg(base + ((2 * j + 1) << R), v[j].y);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The column passes of 512 rows and up serve the backward in two more modes: SPECTRUM on the workspace of X (the
// column bits alone) and then ADJOINT on the workspace of dY, which is FWD and on the way replaces the spectrum of X,
// at the same positions of xws, by the dG term (W X)(W dY)/L (or stores the term to the same position of another plane,
// `terms`).  Both take the same columns in the same thread.
enum Mode { FWD, SPECTRUM, ADJOINT };

// Columns of 128 rows and up.  NW warps of a tensor-memory lane quarter hold a group of columns, 64 NB rows of each (up to
// 512, bits 0..8 of the row), two blocks of 64 rows per warp.  All four warps of a quarter run on one sub-partition of the
// SM, so columns are given to as few warps as tensor memory (512 words a lane) allows: the groups then drift apart and
// one group's loads overlap another's butterflies.
//   round A  blocks of 64 rows, bits 0..5: workspace -> registers -> tensor memory (the second block staged
//            in shared memory meanwhile);
//   round B  bits 6.. across the NB blocks, 32 values a pass, each pass's gains loaded a pass ahead;
//   round C  blocks of 64 rows, bits 0..5 again -> workspace.
// Taller columns (Q >= 10) are 16 to a group: the upper half of the lanes holds row bit 9, whose butterfly is a shuffle
// in round B.  For Q = 11 and 12 the NQ = 2 or 4 quarters of a set hold row bits 10 (and 11) of the same columns: in round
// B the warps at the same place of their quarters trade values through shared memory, each then holding all NQ of 16 / NQ
// row pairs, and trade them back after the gain.  Against units of 2^14 elements in shared memory (8 columns of 1024 or 2048
// rows, 4 of 4096: 32- and 16-byte row segments, each a whole wavefront of the SM's data path): 2^23 elements 39.6 -> 38.0 us
// (log gains 37.9 -> 35.5, backward included 148 -> 132), 2^24 116 -> 101, 2^25 526 -> 222 (generic engine:
// 967); with their groups strided over the CTAs 88 and 189.
template <int Q>
struct Lane {
  static constexpr bool TALL = Q >= 10;
  static constexpr int NB = TALL ? 8 : 1 << (Q - 6);  // blocks of 64 rows
  static constexpr int NW = NB / 2;                   // warps per group
  static constexpr int NQ = Q <= 10 ? 1 : 1 << (Q - 10);        // quarters per set
  static constexpr int GROUPS = THREADS / 32 / NW / NQ;         // groups a CTA works on at a time
  static constexpr int W = 32 / NB;                   // rows of each block per pass of round B: four passes
  static constexpr int COLS = TALL ? 16 : 32;         // columns per group
  static constexpr int LOG_GROUPS = TALL ? R - 4 : R - 5;       // log2 of the groups of a plane
};
template <int NW>
__device__ __forceinline__ void lane_sync(int group) {
  fast::tmem_wait_st();
  if constexpr (NW > 1) {
    fast::tmem_fence_before();
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(32 * NW) : "memory");
    fast::tmem_fence_after();
  }
}
// words ta .. ta + 2 N - 1 of this lane <-> N pairs
template <int N>
__device__ __forceinline__ void ld_pairs(uint32_t ta, float2* v) {
  float f[2 * N];
  if constexpr (N == 8) fast::tmem_ld16(ta, f);
  else if constexpr (N == 4) tmem_ld8(ta, f);
  else tmem_ld4(ta, f);
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = make_float2(f[2 * k], f[2 * k + 1]);
}
template <int N>
__device__ __forceinline__ void st_pairs(uint32_t ta, const float2* v) {
  float f[2 * N];
#pragma unroll
  for (int k = 0; k < N; ++k) f[2 * k] = v[k].x, f[2 * k + 1] = v[k].y;
  if constexpr (N == 8) fast::tmem_st16(ta, f);
  else if constexpr (N == 4) tmem_st8(ta, f);
  else tmem_st4(ta, f);
}
template <int Q, class GainT, Mode MODE = FWD>
__device__ __forceinline__ void col_lanes(float* ws, int begin, int end, int total, const Params& P, const float* tab, uint32_t tmem,
                                          float* slots, const float* xws = nullptr, float* terms = nullptr) {
  using C = Lane<Q>;
  constexpr int m = R + Q, NB = C::NB, NW = C::NW, W = C::W, WP = W / 2, NQ = C::NQ, COLS = C::COLS;
  static_assert(MODE == FWD || NQ == 1, "the backward modes: Q <= 10");
  const float2 sc = make_float2(P.scale, P.scale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = warp & 3;
  const int half = (warp >> 2) / NW, i = (warp >> 2) % NW;  // warps of a group share a quarter
  const int bar = quarter + 4 * half, group = bar / NQ, sub = quarter % NQ;  // this warp's quarter of the set
  const uint32_t ta = tmem + (static_cast<uint32_t>(32 * quarter) << 16) + half * (64 * NB);
  float* stg = slots + warp * WARP_STAGE;
  const int lcol = lane & (COLS - 1);
  const int row0 = (C::TALL ? 512 * (lane >> 4) : 0) + 1024 * sub;  // this lane's first row
  auto first_col = [&](int g) { return (COLS * g) & (TILE - 1); };
  auto plane = [&](int g) { return ws + (static_cast<long long>((COLS * g) >> R) << m) + first_col(g); };
  // this lane's column of group g, from its row 64 b on
  auto block = [&](int g, int b) { return plane(g) + lcol + (static_cast<long long>(row0 + 64 * b) << R); };
  auto stage = [&](int g) {
    if constexpr (C::TALL) {  // lanes 0..3 and 4..7 of a row copy the two halves
      const float* src = plane(g) + 4 * (lane & 3) + (static_cast<long long>(1024 * sub + 512 * ((lane >> 2) & 1) + 64 * (i + NW) + (lane >> 3)) << R);
      const uint32_t d = tc::smem_u32(stg) + 16 * lane;
#pragma unroll
      for (int j = 0; j < 16; ++j) cp_async16(d + 512 * j, src + (static_cast<long long>(4 * j) << R));
    } else {
      stage_block<64>(plane(g) + (static_cast<long long>(64 * (i + NW)) << R), stg, lane);
    }
  };
  // neighbouring CTAs take neighbouring groups where the plane lies in HBM (the rows' segments then fall into the same DRAM pages at
  // the same time), else each CTA a contiguous range
  const int first = NQ > 1 ? static_cast<int>(blockIdx.x) * C::GROUPS + group : begin + group;
  const int step = NQ > 1 ? static_cast<int>(gridDim.x) * C::GROUPS : C::GROUPS;
  if constexpr (NQ > 1) end = total;
  fast::tmem_fence_after();  // with the fence before the device-wide barrier: other warps read rows out of these words
  if (first < end) stage(first);
  for (int g = first; g < end; g += step) {
    const GainT gain(P, tab, first_col(g) + lcol);
    auto round_ac = [&](float2 (&v)[32]) {
#pragma unroll
      for (int j = 0; j < 32; ++j) bf_in(v[j]);
      bfly32<0>(v);
    };
    {
      float2 v[32];
      const float* src = block(g, i);
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = make_float2(__ldcg(src + ((2 * j) << R)), __ldcg(src + ((2 * j + 1) << R)));
      round_ac(v);
#pragma unroll
      for (int q = 0; q < 4; ++q) st_pairs<8>(ta + 64 * i + 16 * q, v + 8 * q);
      fast::cp_async_wait_all();
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = make_float2(stg[64 * j + lane], stg[64 * j + 32 + lane]);
      __syncwarp();
      if (g + step < end) stage(g + step);
      round_ac(v);
#pragma unroll
      for (int q = 0; q < 4; ++q) st_pairs<8>(ta + 64 * (i + NW) + 16 * q, v + 8 * q);
    }
    // round B: pair k of a pass is rows pair_row(k) and + 1 of this lane; after the trade between quarters, rows of quarter
    // k / (16 / NQ) at the place of pair (16 / NQ) sub + k mod (16 / NQ)
    const int low0 = (64 / NW) * i;
    constexpr int KQ = 16 / NQ;
    auto pair_row = [&](int k, int pass) { return 64 * (k / WP) + low0 + W * pass + 2 * (k % WP); };
    auto load_gains = [&](float2 (&gg)[16], int pass) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        if constexpr (NQ == 1) {
          gg[k] = gain.rows2(row0 + pair_row(k, pass));
        } else {
          const int kk = k % KQ, r = 64 * (sub * (KQ / WP) + kk / WP) + low0 + W * pass + 2 * (kk % WP);
          gg[k] = gain.rows2(row0 - 1024 * sub + 1024 * (k / KQ) + r);
        }
      }
    };
    auto trade_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(5 + i * (4 / NQ) + group % (4 / NQ)), "r"(32 * NQ) : "memory"); };
    auto round_b_pass = [&](const float2 (&gg)[16], int pass) {
      float2 v[16];
#pragma unroll
      for (int s = 0; s < NB; ++s) ld_pairs<WP>(ta + 64 * s + low0 + W * pass, v + WP * s);
      fast::tmem_wait_ld();
      auto across = [&] {
#pragma unroll
        for (int h = WP; h < 16; h <<= 1)
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if ((k & h) == 0) bf2(v[k], v[k + h]);
      };
      auto lane_bit = [&] {  // row bit 9: lanes l, l ^ 16
        if constexpr (C::TALL) {
          const float2 sgn = (lane & 16) ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, v[k].x, 16), __shfl_xor_sync(0xffffffffu, v[k].y, 16));
            v[k] = fast::fma2(v[k], sgn, p);
          }
        }
      };
      across();
      lane_bit();
      if constexpr (MODE == SPECTRUM) {
        float* o = block(g, 0);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          __stcg(o + (static_cast<long long>(pair_row(k, pass)) << R), v[k].x);
          __stcg(o + (static_cast<long long>(pair_row(k, pass) + 1) << R), v[k].y);
        }
      } else {
        if constexpr (MODE == ADJOINT) {
          const float* xp = xws + (block(g, 0) - ws);
          float* tp = terms + (block(g, 0) - ws);
          float2 xh[16];
#pragma unroll
          for (int k = 0; k < 16; ++k)
            xh[k] = make_float2(__ldcg(xp + (static_cast<long long>(pair_row(k, pass)) << R)),
                                __ldcg(xp + (static_cast<long long>(pair_row(k, pass) + 1) << R)));
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const float2 pr = mul2(mul2(xh[k], v[k]), sc);
            __stcg(tp + (static_cast<long long>(pair_row(k, pass)) << R), pr.x);
            __stcg(tp + (static_cast<long long>(pair_row(k, pass) + 1) << R), pr.y);
          }
        }
        // the trade areas lie behind the staged blocks
        auto area = [&](int s) { return reinterpret_cast<float2*>(slots + (warp - sub + s) * WARP_STAGE + 64 * 32) + lane; };
        auto quarters = [&] {
#pragma unroll
          for (int h = KQ; h < 16; h <<= 1)
#pragma unroll
            for (int k = 0; k < 16; ++k)
              if ((k & h) == 0) bf2(v[k], v[k + h]);
        };
        if constexpr (NQ > 1) {
#pragma unroll
          for (int k = 0; k < 16; ++k) area(sub)[32 * k] = v[k];
          trade_sync();
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = area(k / KQ)[32 * (KQ * sub + k % KQ)];
          quarters();
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = mul2(v[k], mul2(gg[k], sc));
        if constexpr (NQ > 1) {
          quarters();
#pragma unroll
          for (int k = 0; k < 16; ++k) area(k / KQ)[32 * (KQ * sub + k % KQ)] = v[k];
          trade_sync();
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = area(sub)[32 * k];
        }
        lane_bit();
        across();
#pragma unroll
        for (int s = 0; s < NB; ++s) st_pairs<WP>(ta + 64 * s + low0 + W * pass, v + WP * s);
      }
    };
    if constexpr (MODE == FWD) {
      float2 ga[16], gb[16];
      load_gains(ga, 0);
      lane_sync<NW>(bar);
#pragma unroll 1
      for (int pass = 0; pass < 4; pass += 2) {
        load_gains(gb, pass + 1);
        round_b_pass(ga, pass);
        if (pass == 0) load_gains(ga, 2);
        round_b_pass(gb, pass + 1);
      }
    } else {  // (the spectrum's registers leave no room to load gains a pass ahead)
      lane_sync<NW>(bar);
#pragma unroll 1
      for (int pass = 0; pass < 4; ++pass) {
        float2 gg[16];
        if constexpr (MODE == ADJOINT) load_gains(gg, pass);
        round_b_pass(gg, pass);
      }
    }
    lane_sync<NW>(bar);
#pragma unroll 1
    for (int it = 0; it < (MODE == SPECTRUM ? 0 : 2); ++it) {
      float2 v[32];
      float* dst = block(g, i + NW * it);
      read_row(ta + 64 * (i + NW * it), v);
      round_ac(v);
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        __stcg(dst + ((2 * j) << R), v[j].x);
        __stcg(dst + ((2 * j + 1) << R), v[j].y);
      }
    }
    // the next columns' round A writes only this warp's own blocks, which the others stopped reading at the
    // second lane_sync
  }
}

// Backward columns of up to 256 rows, X and dY of a column in one pass: the spectrum of X waits on chip (in
// registers up to 32 rows, else in tensor memory) while dY is transformed; dY goes through gain and column bits to its
// place in wsd.  Against a pass over X that stores its spectrum and a pass over dY that reads it back, the exchange is a
// third smaller.
// The dG terms (W X)(W dY)/L never reach the workspace: a team of pl warps (groups of warps above 64 rows) takes the same
// 32 columns of pl planes, its terms meet in shared memory, and each warp adds some rows up in ascending b.  What bounds
// these phases is the exchange through L2: storing the terms and reading them back after a barrier was 8 of a group's 62 us
// (four planes of 2^21), and the stores part of its 22 us of columns.  Forward and backward, back to back, with terms in
// the workspace and in shared memory: [16, 8192, 256] bf16 375 -> 353 us, [32, 4000 of 4096, 64] f32 log gains 110 -> 104,
// [256, 512, 64] bf16 94 -> 77, [512, 256, 64] 124 -> 92, [1, 256, 64] 15.3 -> 14.5, [8, 4096, 128] bf16 52.3 -> 52.0.
template <int Q>
__device__ __forceinline__ void col_regs_bwd(const float* wsx, float* wsd, int nb, bool first, const Params& P, uint32_t tmem,
                                             float* slots) {
  constexpr int NR = 1 << Q, NP = NR / 2, m = R + Q;
  constexpr int NG = NP < 16 ? NP : 16;  // pairs per batch of gains and of dG terms
  constexpr int PER = 32 * (NR < 4 ? 4 : NR), TERMS = 64 * NG;
  constexpr int RING = (WARP_STAGE - TERMS) / PER > 3 ? 3 : (WARP_STAGE - TERMS) / PER;  // blocks in flight: X, dY, X, ...
  static_assert(RING >= 1, "a block and a batch of dG terms");
  const float2 sc = make_float2(P.scale, P.scale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ta = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + 64 * (warp >> 2);
  float *stg = slots + warp * WARP_STAGE, *terms = stg + RING * PER;
  int pl = 1;  // planes a team of warps holds at a time
  constexpr int MAXPL = THREADS / 32;
  while (pl < nb && pl < MAXPL) pl <<= 1;
  // a team of pl >= NG warps owns at most two rows of a batch per warp and keeps their sums in registers over its sets of pl
  // planes; among these, the pl with the fewest rounds of the CTA's warps
  if constexpr (NG < MAXPL) {
    const int blocks = (TILE / 32 + gridDim.x - 1) / gridDim.x;
    auto rounds = [&](int p) { return (nb + p - 1) / p * ((blocks * p + MAXPL - 1) / MAXPL); };
    for (int p = pl / 2; p >= NG; p /= 2)
      if (rounds(p) < rounds(pl)) pl = p;
  }
  // 64 rows, 9 to 12 planes: two teams of eight, whose second set is small, on the CTA's two blocks at once, against one team with
  // idle warps on one after the other ([12, 8192, 64] bf16 45.0 -> 43.4 us, [9, 8192, 64] 35.4 -> 35.0)
  if constexpr (NG == MAXPL && NP > 16) {
    if (nb > MAXPL / 2 && nb <= 12) pl = MAXPL / 2;
  }
  const int team = warp / pl, member = warp % pl, teams = MAXPL / pl;
  auto team_sync = [&] {
    if (pl > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(32 * pl) : "memory");
    else __syncwarp();
  };
  const bool direct = first && nb == 1;  // the only terms: stored as they are
  int gb, ge;  // blocks of 32 columns
  share(TILE / 32, &gb, &ge);
  int sg = gb + team, sb = member, sd = 0, sslot = 0;  // the next block to stage
  auto stage = [&] {
    if (sg < ge && sb < nb) {
      const float* b = (sd ? wsd : wsx) + (sb << m) + 32 * sg;
      if constexpr (NR >= 4) {
        stage_block<NR>(b, stg + sslot * PER, lane);
      } else {
        if (lane < 8 * NR)
          cp_async16(tc::smem_u32(stg + sslot * PER) + 16 * lane, b + (static_cast<long long>(lane >> 3) << R) + 4 * (lane & 7));
      }
    }
    fast::cp_async_commit();
    sslot = sslot + 1 == RING ? 0 : sslot + 1;
    if (sd) {
      sb += pl;
      if (sb >= nb) sb = member, sg += teams;
    }
    sd ^= 1;
  };
  if constexpr (NP > 16) fast::tmem_fence_after();  // as in col_lanes
#pragma unroll
  for (int k = 0; k < RING; ++k) stage();
  int slot = 0;
  auto take = [&](float2 (&v)[NP]) {  // the next staged block, its column bits done
    asm volatile("cp.async.wait_group %0;" ::"n"(RING - 1) : "memory");
    __syncwarp();
    const float* b = stg + slot * PER + lane;
#pragma unroll
    for (int j = 0; j < NP; ++j) v[j] = make_float2(b[64 * j], b[64 * j + 32]);
    __syncwarp();
    stage();
    slot = slot + 1 == RING ? 0 : slot + 1;
#pragma unroll
    for (int j = 0; j < NP; ++j) bf_in(v[j]);
    fast::bfly_all<NP>(v);
  };
  // dG at rows h + member, h + member + pl, ... of the batch: the team's terms in ascending b
  auto add_terms = [&](float (&own)[2], int g, int b, int h) {
    const int np = min(pl, nb - b);
    if (NP <= 16 && pl >= NG) {
      auto keep = [&](auto full) {  // (with the full team's constants 6% faster on large batches)
        constexpr bool FULL = decltype(full)::value;
        const int ps = FULL ? MAXPL : pl;
        const float* t = slots + (FULL ? 0 : team * pl) * WARP_STAGE + RING * PER + lane + 32 * member;
        for (int p = 0; p < np; ++p) {
          if (member < 2 * NG) own[0] += t[p * WARP_STAGE];
          if (member + ps < 2 * NG) own[1] += t[p * WARP_STAGE + 32 * ps];
        }
        if (b + ps >= nb) {
          float* o = static_cast<float*>(P.dg) + 32 * g + lane + ((h + member) << R);
          if (member < 2 * NG) __stcg(o, own[0]);
          if (member + ps < 2 * NG) __stcg(o + (ps << R), own[1]);
        }
      };
      if (NG == MAXPL || pl == MAXPL) keep(std::true_type{});
      else keep(std::false_type{});
      return;
    }
    float* o = static_cast<float*>(P.dg) + 32 * g + lane + (h << R);
#pragma unroll 1
    for (int r = member; r < 2 * NG; r += 4 * pl) {
      float acc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[k] = (first && b == 0) || r + k * pl >= 2 * NG ? 0.f : __ldcg(o + ((r + k * pl) << R));
#pragma unroll 1
      for (int p = 0; p < np; ++p) {
        const float* t = slots + (team * pl + p) * WARP_STAGE + RING * PER + lane;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (r + k * pl < 2 * NG) acc[k] += t[32 * (r + k * pl)];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (r + k * pl < 2 * NG) __stcg(o + ((r + k * pl) << R), acc[k]);
    }
  };
  for (int g = gb + team; g < ge; g += teams) {
    float own[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int r = member + (NG == MAXPL ? MAXPL : pl) * k;
      own[k] = first || NP > 16 || pl < NG || r >= 2 * NG ? 0.f : __ldcg(static_cast<float*>(P.dg) + 32 * g + lane + (r << R));
    }
    for (int b0 = 0; b0 < nb; b0 += pl) {
      const int b = b0 + member;
      if (b >= nb) {  // no plane for this warp: only its share of the sums
#pragma unroll 1
        for (int h = 0; h < NP; h += NG) {
          team_sync();
          team_sync();
          add_terms(own, g, b0, 2 * h);
        }
        continue;
      }
      const LaneFull<Q> gain(P, nullptr, 32 * g + lane);
      float2 xh[NG];
      float2 v[NP];
      take(v);
      if constexpr (NP > 16) {
#pragma unroll
        for (int q = 0; q < NP / 8; ++q) st_pairs<8>(ta + 16 * q, v + 8 * q);
        fast::tmem_wait_st();
      } else {
#pragma unroll
        for (int j = 0; j < NP; ++j) xh[j] = v[j];
      }
      take(v);
#pragma unroll
      for (int h = 0; h < NP; h += NG) {
        if constexpr (NP > 16) {
#pragma unroll
          for (int q = 0; q < 2; ++q) ld_pairs<8>(ta + 2 * h + 16 * q, xh + 8 * q);
          fast::tmem_wait_ld();
        }
        float2 gg[NG];
#pragma unroll
        for (int j = 0; j < NG; ++j) gg[j] = gain.rows2(2 * (h + j));
        if (direct) {
          float* d = static_cast<float*>(P.dg) + 32 * g + lane;
#pragma unroll
          for (int j = 0; j < NG; ++j) {
            const float2 pr = mul2(mul2(xh[j], v[h + j]), sc);
            __stcg(d + ((2 * (h + j)) << R), pr.x);
            __stcg(d + ((2 * (h + j) + 1) << R), pr.y);
          }
        } else {
          team_sync();  // the batch before this one has been added up
#pragma unroll
          for (int j = 0; j < NG; ++j) {
            const float2 pr = mul2(mul2(xh[j], v[h + j]), sc);
            terms[64 * j + lane] = pr.x;
            terms[64 * j + 32 + lane] = pr.y;
          }
        }
#pragma unroll
        for (int j = 0; j < NG; ++j) v[h + j] = mul2(v[h + j], mul2(gg[j], sc));
        if (!direct) {
          team_sync();
          add_terms(own, g, b0, 2 * h);
        }
      }
      float* o = wsd + (b << m) + 32 * g + lane;
#pragma unroll
      for (int j = 0; j < NP; ++j) bf_in(v[j]);
      fast::bfly_all<NP>(v);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        __stcg(o + ((2 * j) << R), v[j].x);
        __stcg(o + ((2 * j + 1) << R), v[j].y);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// 128 and 256 rows: NB = 2, 4 warps (a group) hold 32 columns of a plane, one block of 64 rows of X and of dY each.  The
// groups of a team of pl take the same columns of consecutive planes and add their dG terms up as above, eight rows of dG
// loaded before the team meets (after: their latency cost half the gain; before a pass: its registers spill).
template <int Q>
__device__ __forceinline__ void col_lanes_bwd(const float* wsx, float* wsd, int nb, bool first, const Params& P,
                                              uint32_t tmem, float* slots) {
  constexpr int m = R + Q, NB = 1 << (Q - 6), W = 32 / NB, WP = W / 2, GROUPS = THREADS / 32 / NB;
  constexpr int STAGED = 64 * 32;  // floats: a block of dY, then the warp's 32 x 32 dG terms of a pass
  static_assert(STAGED + 32 * 32 <= WARP_STAGE, "a block and its dG terms");
  const float2 sc = make_float2(P.scale, P.scale);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = warp & 3;
  const int half = (warp >> 2) / NB, i = (warp >> 2) % NB, group = quarter + 4 * half;
  // words of the lane: the spectrum of X, then dY
  const uint32_t tx = tmem + (static_cast<uint32_t>(32 * quarter) << 16) + half * (128 * NB), td = tx + 64 * NB;
  float *stg = slots + warp * WARP_STAGE, *terms = stg + STAGED;
  int pl = 1;  // planes a team holds at a time
  while (pl < nb && pl < GROUPS) pl <<= 1;
  const int team = group / pl, member = group % pl, teams = GROUPS / pl;
  auto team_sync = [&] {
    fast::tmem_wait_st();
    fast::tmem_fence_before();
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(32 * NB * pl) : "memory");
    fast::tmem_fence_after();
  };
  int gb, ge;  // blocks of 32 columns
  share(TILE / 32, &gb, &ge);
  const int own = (64 * i) << R;
  auto stage = [&](int g, int b) {
    if (g < ge && b < nb) stage_block<64>(wsd + (b << m) + 32 * g + own, stg, lane);
  };
  auto rows64 = [&](float2 (&v)[32]) {
#pragma unroll
    for (int j = 0; j < 32; ++j) bf_in(v[j]);
    bfly32<0>(v);
  };
  auto across = [&](float2 (&v)[16]) {
#pragma unroll
    for (int h = WP; h < 16; h <<= 1)
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if ((k & h) == 0) bf2(v[k], v[k + h]);
  };
  const int low0 = (64 / NB) * i;
  // dG at this warp's share of the 32 rows of a pass, eight rows at a time (row r of the terms is row
  // low + 64 (r / W) + r % W of the column); the first eight are loaded before the team meets
  const int r0 = member * (32 / pl), r1 = r0 + 32 / pl;
  const bool direct = first && nb == 1;  // the only terms: stored as they are
  auto dg_row = [&](int g, int low, int r) { return static_cast<float*>(P.dg) + 32 * g + lane + ((low + 64 * (r / W) + r % W) << R); };
  auto load_dg = [&](float (&acc)[8], int g, int b, int low, int r) {
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = (first && b == 0) || r + k >= r1 ? 0.f : __ldcg(dg_row(g, low, r + (k & 4)) + ((k & 3) << R));
  };
  auto add_terms = [&](float (&acc)[8], int g, int b, int low) {
    const int np = min(pl, nb - b);
#pragma unroll 1
    for (int r = r0;;) {
      for (int p = 0; p < np; ++p) {
        const int gr = team * pl + p;
        const float* t = slots + ((gr & 3) + 4 * ((gr >> 2) * NB + i)) * WARP_STAGE + STAGED + 32 * r + lane;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (r + k < r1) acc[k] += t[32 * k];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (r + k < r1) __stcg(dg_row(g, low, r + (k & 4)) + ((k & 3) << R), acc[k]);
      r += 8;
      if (r >= r1) break;
      load_dg(acc, g, b, low, r);
    }
  };
  fast::tmem_fence_after();  // as in col_lanes
  stage(gb + team, member);
  for (int g = gb + team; g < ge; g += teams)
    for (int b0 = 0; b0 < nb; b0 += pl) {
      const int b = b0 + member;
      const bool active = b < nb;  // of the whole warp
      const int o = (b << m) + 32 * g + lane;  // (a group's workspace is below 2^31 elements)
      const LaneFull<Q> gain(P, nullptr, 32 * g + lane);
      float2 gg[16];
      if (active) {
        float2 v[32];
        const float* src = wsx + o + own;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = make_float2(__ldcg(src + ((2 * j) << R)), __ldcg(src + ((2 * j + 1) << R)));
        rows64(v);
#pragma unroll
        for (int q = 0; q < 4; ++q) st_pairs<8>(tx + 64 * i + 16 * q, v + 8 * q);
        fast::cp_async_wait_all();
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = make_float2(stg[64 * j + lane], stg[64 * j + 32 + lane]);
        __syncwarp();
        if (b + pl < nb) stage(g, b + pl);
        else stage(g + teams, member);
        rows64(v);
#pragma unroll
        for (int q = 0; q < 4; ++q) st_pairs<8>(td + 64 * i + 16 * q, v + 8 * q);
#pragma unroll
        for (int k = 0; k < 16; ++k) gg[k] = gain.rows2(64 * (k / WP) + low0 + 2 * (k % WP));
      }
      team_sync();
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        const int low = low0 + W * pass;
        if (active) {
          float2 xh[16], v[16];
#pragma unroll
          for (int s = 0; s < NB; ++s) ld_pairs<WP>(tx + 64 * s + low, xh + WP * s);
#pragma unroll
          for (int s = 0; s < NB; ++s) ld_pairs<WP>(td + 64 * s + low, v + WP * s);
          fast::tmem_wait_ld();
          across(xh);
          across(v);
#pragma unroll
          for (int k = 0; k < 16; ++k) xh[k] = mul2(mul2(xh[k], v[k]), sc);
          if (direct) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              float* d = static_cast<float*>(P.dg) + 32 * g + lane + ((low + 64 * (k / WP) + 2 * (k % WP)) << R);
              __stcg(d, xh[k].x);
              __stcg(d + TILE, xh[k].y);
            }
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              terms[64 * k + lane] = xh[k].x;
              terms[64 * k + 32 + lane] = xh[k].y;
            }
          }
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = mul2(v[k], mul2(gg[k], sc));
          if (pass == 0) {
#pragma unroll
            for (int k = 0; k < 16; ++k) gg[k] = gain.rows2(64 * (k / WP) + low0 + W + 2 * (k % WP));
          }
          across(v);
#pragma unroll
          for (int s = 0; s < NB; ++s) st_pairs<WP>(td + 64 * s + low, v + WP * s);
        }
        if (direct) continue;
        float acc[8];
        load_dg(acc, g, b0, low, r0);
        team_sync();
        add_terms(acc, g, b0, low);
        if (pass == 0) team_sync();  // (the next block's first team_sync is the other one)
      }
      if (direct) team_sync();
      if (active) {
        float2 v[32];
        float* dst = wsd + o + own;
        read_row(td + 64 * i, v);
        rows64(v);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          __stcg(dst + ((2 * j) << R), v[j].x);
          __stcg(dst + ((2 * j + 1) << R), v[j].y);
        }
      }
    }
}

// ---------------------------------------------------------------------------------------------
// What the phases of one CTA share.
struct Cta {
  float* slots;
  uint64_t* full_row;
  uint64_t (*mma_done)[2];
  volatile int* dead;
  GridBarrier* bar;
  uint32_t tmem;
  int worker, t;
  unsigned row_seq, mma_seq;  // rows taken from the ring, and multiplied, so far
};
struct __align__(8) CtaShared {
  uint64_t full_row[ROW_BARS], mma_done[WORKERS][2];
  int flag, dead;
  uint32_t tmem_slot;
};
__host__ __device__ constexpr bool uses_tmem(int dtype, int q) { return dtype == DT_BF16 || q >= 6; }

// Before the launch wait: tensor memory, H_128, the barriers.
template <int D, int Q>
__device__ __forceinline__ Cta cta_begin(unsigned char* smem, CtaShared& sh, const Params& P) {
  if constexpr (uses_tmem(D, Q)) {
    if (threadIdx.x < 32) fast::tmem_alloc_512(&sh.tmem_slot);
  }
  if constexpr (D == DT_BF16) {
    build_h(smem + SLOT_BYTES);
    fence_async();
  }
  if (threadIdx.x == 0) {
    sh.dead = 0;
    for (int i = 0; i < ROW_BARS; ++i) tc::mbar_init(&sh.full_row[i], WT);
    for (int i = 0; i < WORKERS; ++i)
      for (int k = 0; k < 2; ++k) tc::mbar_init(&sh.mma_done[i][k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fast::tmem_fence_before();
  __syncthreads();
  fast::tmem_fence_after();
  return {reinterpret_cast<float*>(smem), sh.full_row, sh.mma_done, &sh.dead, P.bar, uses_tmem(D, Q) ? sh.tmem_slot : 0u,
          static_cast<int>(threadIdx.x) / WT, static_cast<int>(threadIdx.x) % WT, 0, 0};
}
template <int D, int Q>
__device__ __forceinline__ void cta_end(CtaShared& sh) {
  if constexpr (uses_tmem(D, Q)) {
    fast::tmem_fence_before();
    __syncthreads();
    fast::tmem_fence_after();
    if (threadIdx.x < 32) fast::tmem_dealloc_512(sh.tmem_slot);
  }
}

// Row bits of the CTA's n rows.  src(k, &p, &lim): row k's first element and how many are present; dst(k): its
// workspace row; each(k): called by one thread per row.
template <int D, class Src, class Dst, class Each>
__device__ __forceinline__ void rows_in(Cta& c, int n, const Src& src, const Dst& dst, const Each& each) {
  const int worker = c.worker, t = c.t;
  if constexpr (D == DT_BF16) {
    // the worker's i-th row (row worker + 4 i of the CTA's) is staged in its area i mod 3 and multiplied into its
    // accumulator i mod 2
    const int nw = (n - worker + WORKERS - 1) / WORKERS;
    const uint32_t xs = tc::smem_u32(c.slots) + worker * (XSLOTS * TILE * 2);
    const uint32_t sh = tc::smem_u32(c.slots) + SLOT_BYTES;
    const uint32_t acc = c.tmem + 128u * worker;
    auto load = [&](int i) {
      if (i < nw) {
        const void* p;
        int lim;
        src(worker + WORKERS * i, &p, &lim);
        load_x_bf16(static_cast<const unsigned short*>(p), lim, xs + (i % XSLOTS) * (TILE * 2), t);
      }
      fast::cp_async_commit();
    };
    auto multiply = [&](int i) {  // a row that has been staged -> its accumulator
      fence_async();
      fast::tmem_fence_before();
      worker_sync(worker);
      if (t == 0) {
        fast::tmem_fence_after();
        mma_row(acc + 64u * (i & 1), sh, xs + (i % XSLOTS) * (TILE * 2));
        tc::mma_commit(&c.mma_done[worker][(c.mma_seq + i) & 1]);
      }
    };
    for (int i = 0; i < XSLOTS; ++i) load(i);
    if (nw > 0) {
      asm volatile("cp.async.wait_group %0;" ::"n"(XSLOTS - 1) : "memory");
      multiply(0);
    }
    for (int i = 0; i < nw; ++i) {
      if (t == 0) each(worker + WORKERS * i);
      if (i + 1 < nw) {
        asm volatile("cp.async.wait_group %0;" ::"n"(XSLOTS - 2) : "memory");
        multiply(i + 1);
      }
      wait_bar(&c.mma_done[worker][(c.mma_seq + i) & 1], ((c.mma_seq + i) >> 1) & 1u, c.bar, c.dead);
      __syncwarp();
      fast::tmem_fence_after();
      float2 v[32];
      read_row(acc + 64u * (i & 1) + (static_cast<uint32_t>(32 * ((threadIdx.x >> 5) & 3)) << 16), v);
      load(i + XSLOTS);
#pragma unroll
      for (int j = 0; j < 32; ++j) bf_in(v[j]);
      bfly32<0>(v);
      float* o = dst(worker + WORKERS * i) + t;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        __stcg(o + 256 * j, v[j].x);
        __stcg(o + 256 * j + 128, v[j].y);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    c.mma_seq += nw;
    fast::tmem_fence_before();
  } else {
    auto load = [&](int k) {
      const void* p;
      int lim;
      src(k, &p, &lim);
      load_row(static_cast<const float*>(p), lim, c.slots + (c.row_seq + k) % SLOTS * TILE, t, &c.full_row[(c.row_seq + k) % ROW_BARS]);
    };
    for (int k = worker; k < SLOTS && k < n; k += WORKERS) load(k);
    for (int k = worker; k < n; k += WORKERS) {
      if (t == 0) each(k);
      wait_full(c.full_row, c.row_seq + k, ROW_BARS, c.bar, c.dead);
      row_in(c.slots + (c.row_seq + k) % SLOTS * TILE, dst(k), t, worker, [&] {
        if (k + SLOTS < n) load(k + SLOTS);
      });
    }
    c.row_seq += n;
  }
}

// Row bits of the CTA's n workspace rows at wsr -> dst: loc(k, &e0, &lim) is row k's place in dst.
template <int D, class Loc>
__device__ __forceinline__ void rows_out(Cta& c, int n, const float* wsr, void* dst, const Loc& loc) {
  auto load = [&](int k) {
    load_row(wsr + (static_cast<long long>(k) << R), TILE, c.slots + (c.row_seq + k) % SLOTS * TILE, c.t,
             &c.full_row[(c.row_seq + k) % ROW_BARS]);
  };
  for (int k = c.worker; k < SLOTS && k < n; k += WORKERS) load(k);
  for (int k = c.worker; k < n; k += WORKERS) {
    long long e0;
    int lim;
    loc(k, &e0, &lim);
    wait_full(c.full_row, c.row_seq + k, ROW_BARS, c.bar, c.dead);
    row_out<D>(c.slots + (c.row_seq + k) % SLOTS * TILE, dst, e0, lim, c.t, c.worker, [&] {
      if (k + SLOTS < n) load(k + SLOTS);
    });
  }
  c.row_seq += n;
}

// Column bits of nb planes of a workspace, all CTAs together.
template <int Q, Gains G, Mode MODE>
__device__ __forceinline__ void columns(Cta& c, float* ws, int nb, const Params& P, const float* tab, const float* xws = nullptr,
                                        float* terms = nullptr) {
  using LaneT = typename LaneGain<Q, G>::T;
  if constexpr (Q <= 6) {
    col_regs<Q, LaneT>(ws, nb << R, P, tab, c.slots);
  } else {
    int gb, ge;
    share(static_cast<unsigned>(nb) << Lane<Q>::LOG_GROUPS, &gb, &ge);
    col_lanes<Q, LaneT, MODE>(ws, gb, ge, nb << Lane<Q>::LOG_GROUPS, P, tab, c.tmem, c.slots, xws, terms);
    fast::tmem_fence_before();
  }
}

// Backward columns of nb planes: dY through gain and back over wsd; dG's terms over wsx or, where sums_dg(Q) (a plane group of
// taller columns is one or two planes), added to P.dg
// (which holds the earlier groups' sum unless `first`).
__host__ __device__ constexpr bool sums_dg(int q) { return q <= 8; }
// Taller columns: a first and only plane's terms are dG itself ([1, 65536, 128] bf16, forward and backward: 132.9 -> 125.8 us
// against terms in the workspace and a pass that copies them).
__device__ __forceinline__ bool dg_is_terms(int nb, bool first) { return first && nb == 1; }
template <int Q>
__device__ __forceinline__ void columns_bwd(Cta& c, float* wsx, float* wsd, int nb, bool first, const Params& P) {
  if constexpr (Q <= 6) {
    col_regs_bwd<Q>(wsx, wsd, nb, first, P, c.tmem, c.slots);
    fast::tmem_fence_before();
  } else if constexpr (Q <= 8) {
    col_lanes_bwd<Q>(wsx, wsd, nb, first, P, c.tmem, c.slots);
    fast::tmem_fence_before();
  } else {
    columns<Q, FULL, SPECTRUM>(c, wsx, nb, P, nullptr);
    columns<Q, FULL, ADJOINT>(c, wsd, nb, P, nullptr, wsx, dg_is_terms(nb, first) ? static_cast<float*>(P.dg) : wsx);
  }
}

// This CTA's share of G, fetched into L2 over phase 1's rows.
struct GainPrefetch {
  const char* g;
  long long begin, end;  // 16-byte chunks
  __device__ __forceinline__ GainPrefetch(const void* p, int m) : g(static_cast<const char*>(p)) {
    const long long chunks = (4ll << m) >> 4;
    begin = chunks * blockIdx.x / gridDim.x;
    end = chunks * (blockIdx.x + 1) / gridDim.x;
  }
  __device__ __forceinline__ void operator()(int k, int n) const {  // piece k of n
    const long long step = (end - begin + n - 1) / n, c0 = begin + step * k, c1 = min(c0 + step, end);
    if (c1 > c0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(g + (c0 << 4)), "r"(static_cast<unsigned>((c1 - c0) << 4)) : "memory");
  }
};
// (planes that fill L2 by themselves read G from HBM in phase 2: a prefetch would push the workspace out)
__host__ __device__ constexpr bool prefetches_gains(int q) { return q <= 10; }

// ---------------------------------------------------------------------------------------------
// Forward kernel: persistent grid (one CTA per SM, all resident), plane groups of P.gp planes.
template <int D, int Q, Gains G>
__global__ void __launch_bounds__(THREADS, 1) k_forward_fast(Params P) {
  extern __shared__ __align__(1024) unsigned char tri_smem[];
  __shared__ CtaShared sh;
  constexpr int m = R + Q;
  constexpr int ES = D == DT_BF16 ? 2 : 4;
  float* ws = static_cast<float*>(P.ws);
  float* tab = ws + (static_cast<long long>(P.gp) << m);
  {
    int rb, re;
    share(static_cast<unsigned>(min(static_cast<long long>(P.gp), P.B)) << Q, &rb, &re);
    fast::l2_prefetch_first_rows<D, R, Q>(P.x, rb, re, P.lv);
  }
  Cta c = cta_begin<D, Q>(tri_smem, sh, P);
  // tensor memory is allocated before the wait: the previous kernel's CTA on this SM has left
  pdl_wait();
  GridSync gsync(P.bar, &sh.flag);
  const GainPrefetch prefetch(P.g, m);
  if constexpr (G != FULL) {  // the gain tables, part of the first phase 1
    const long long n_t = 1ll << (m - P.cbits), n_tab = n_t + (1ll << P.cbits);
    for (long long i = static_cast<long long>(blockIdx.x) * THREADS + threadIdx.x; i < n_tab;
         i += static_cast<long long>(gridDim.x) * THREADS)
      tab[i] = expf(i < n_t ? P.gt[sep_token_of<Q, G>(i, P.cbits)] : P.gc[i - n_t]);
  }
  for (long long b0 = 0; b0 < P.B; b0 += P.gp) {
    const int nb = static_cast<int>(min(static_cast<long long>(P.gp), P.B - b0));
    int rb, re;
    share(static_cast<unsigned>(nb) << Q, &rb, &re);
    const int n = re - rb;
    // phase 1: X -> workspace, row bits
    rows_in<D>(
        c, n,
        [&](int k, const void** p, int* lim) {
          long long e0;
          fast::row_loc<R, Q>(b0, rb + k, P.lv, &e0, lim);
          *p = static_cast<const char*>(P.x) + e0 * ES;
        },
        [&](int k) { return ws + (static_cast<long long>(rb + k) << R); },
        [&](int k) {
          if (G == FULL && prefetches_gains(Q) && b0 == 0) prefetch(k, n);
        });
    if (!gsync()) break;
    // phase 2: columns
    columns<Q, G, FWD>(c, ws, nb, P, tab);
    if (!gsync()) break;
    // phase 3: workspace -> Y, row bits
    rows_out<D>(c, n, ws + (static_cast<long long>(rb) << R), P.y,
                [&](int k, long long* e0, int* lim) { fast::row_loc<R, Q>(b0, rb + k, P.lv, e0, lim); });
    if (b0 + P.gp < P.B && !gsync()) break;
  }
  pdl_trigger();
  cta_end<D, Q>(sh);
}

// Backward kernel (planes of 2^14 .. 2^23 elements).  Against the previous one (8 warps, one column a thread or two passes
// through tensor memory, dG summed plane after plane), forward and backward together: [16, 8192, 256] bf16 465 -> 350 us,
// [8, 4096, 256] bf16 118 -> 90, [1, 65536, 128] bf16 186 -> 124, [4, 16384, 256] bf16 335 -> 219, [32, 1024, 64] bf16
// 36.3 -> 30.6.  A group's workspaces (64 MiB) and the streamed X, dY, dX do not fit L2 together (531 MB of HBM traffic a call at
// [16, 8192, 256], 218 MB of them X, dY, dX and the gains); smaller groups lose more to phases and barriers than they save
// (48 MiB 403 us, 32 MiB 400), and 128 MiB take as long (349).
// Per group of planes the same three phases over X and dY
// together,
//   phase 1  rows of X and dY                                            X, dY -> wsx, wsd
//   phase 2  columns: the spectrum of X, then dY through gain and back, the terms (W X)(W dY)/L added to dG (0 for
//            the first group) in ascending b, so that dG is summed over b = 0, 1, ..., B-1 in that order
//                                                                        wsx, wsd -> wsd, dG
//   phase 3  rows of wsd -> dX; for columns above 256 rows whose terms replaced the spectrum in wsx, then dG.
// dG at plane positions [lb, le) (multiples of 4), NPOS positions of NPL planes loaded at a time (four loads in flight a thread:
// eight made the phases around it spill registers).  A plane group of these columns is one or two planes ([4, 65536, 64] bf16
// backward 162 -> 152 us against four planes' loads at a position, two of them always off).
template <int NPOS, int NPL>
__device__ __forceinline__ void dg_sum(float* dg, const float* wsx, int m, int nb, bool first, long long lb, long long le) {
  for (long long l0 = lb + 4 * threadIdx.x; l0 < le; l0 += 4 * THREADS * NPOS) {
    float4 acc[NPOS], p[NPOS][NPL];
#pragma unroll
    for (int i = 0; i < NPOS; ++i) {
      const long long l = l0 + 4 * THREADS * i;
      acc[i] = first || l >= le ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldcg(reinterpret_cast<const float4*>(dg + l));
    }
    for (int b = 0; b < nb; b += NPL) {
#pragma unroll
      for (int i = 0; i < NPOS; ++i)
#pragma unroll
        for (int k = 0; k < NPL; ++k) {
          const long long l = l0 + 4 * THREADS * i;
          if (l < le && b + k < nb) p[i][k] = __ldcg(reinterpret_cast<const float4*>(wsx + (static_cast<long long>(b + k) << m) + l));
        }
#pragma unroll
      for (int i = 0; i < NPOS; ++i)
#pragma unroll
        for (int k = 0; k < NPL; ++k)
          if (b + k < nb) {
            acc[i].x += p[i][k].x;
            acc[i].y += p[i][k].y;
            acc[i].z += p[i][k].z;
            acc[i].w += p[i][k].w;
          }
    }
#pragma unroll
    for (int i = 0; i < NPOS; ++i) {
      const long long l = l0 + 4 * THREADS * i;
      if (l < le) __stcg(reinterpret_cast<float4*>(dg + l), acc[i]);
    }
  }
}
__device__ __forceinline__ void dg_reduce(float* dg, const float* wsx, int m, int nb, bool first, long long lb, long long le) {
  if (nb == 1) dg_sum<4, 1>(dg, wsx, m, nb, first, lb, le);
  else dg_sum<2, 2>(dg, wsx, m, nb, first, lb, le);
}
template <int D, int Q>
__global__ void __launch_bounds__(THREADS, 1) k_backward_fast(Params P) {
  extern __shared__ __align__(1024) unsigned char tri_smem[];
  __shared__ CtaShared sh;
  constexpr int m = R + Q;
  constexpr int ES = D == DT_BF16 ? 2 : 4;
  float* wsx = static_cast<float*>(P.ws);
  float* wsd = wsx + (static_cast<long long>(P.gp) << m);
  Cta c = cta_begin<D, Q>(tri_smem, sh, P);
  pdl_wait();
  GridSync gsync(P.bar, &sh.flag);
  const GainPrefetch prefetch(P.g, m);
  const long long L = 1ll << m;
  const long long lb = ((L >> 2) * blockIdx.x / gridDim.x) << 2, le = ((L >> 2) * (blockIdx.x + 1) / gridDim.x) << 2;
  for (long long b0 = 0; b0 < P.B; b0 += P.gp) {
    const int nb = static_cast<int>(min(static_cast<long long>(P.gp), P.B - b0));
    const int rows = nb << Q;
    {
      int ub, ue;
      share(2u * static_cast<unsigned>(rows), &ub, &ue);
      const int n = ue - ub;
      rows_in<D>(
          c, n,
          [&](int k, const void** p, int* lim) {
            const int u = ub + k;
            long long e0;
            fast::row_loc<R, Q>(b0, u < rows ? u : u - rows, P.lv, &e0, lim);
            *p = static_cast<const char*>(u < rows ? P.x : P.dy) + e0 * ES;
          },
          [&](int k) {
            const int u = ub + k;
            return u < rows ? wsx + (static_cast<long long>(u) << R) : wsd + (static_cast<long long>(u - rows) << R);
          },
          [&](int k) {
            if (b0 == 0) prefetch(k, n);
          });
    }
    if (!gsync()) break;
    columns_bwd<Q>(c, wsx, wsd, nb, b0 == 0, P);
    if (!gsync()) break;
    int rb, re;
    share(static_cast<unsigned>(rows), &rb, &re);
    rows_out<D>(c, re - rb, wsd + (static_cast<long long>(rb) << R), P.dx,
                [&](int k, long long* e0, int* lim) { fast::row_loc<R, Q>(b0, rb + k, P.lv, e0, lim); });
    if (!sums_dg(Q) && !dg_is_terms(nb, b0 == 0)) dg_reduce(static_cast<float*>(P.dg), wsx, m, nb, b0 == 0, lb, le);
    if (b0 + P.gp < P.B && !gsync()) break;
  }
  pdl_trigger();
  cta_end<D, Q>(sh);
}

}  // namespace tri
}  // namespace whtmix

// whtmix_block.cuh -- the whole mixer block of Section III-B, Eq. 1-4, as one persistent launch for bf16 planes of 64 or
// 128 channels:
//   Y_b = ( H_N (G o (H_N (X_b W_in^T) H_C)) H_C / (N C) ) W_out^T
// The three-phase forward (whtmix_tri.cuh) with the projections in its row phases, on the tensor cores:
//   phase 1  a row is 128 consecutive elements k (the channels, and for C = 64 two tokens) by 64 values n.  Two forms:
//            Z rounded to bf16 (the block's activation, what whtmix_block_backward recomputes): Z = W_in x row, rounded over
//            the row's own staging area, then H_128 x Z as the forward multiplies X;
//            Z not rounded (C = 128, 2^21 elements and up): the forward's H_128 replaced by A = H_128 W_in, so that the
//            input projection and the seven low transform bits are one contraction and Z is never formed.  A is computed
//            in fp32 and used as three bf16 terms (together its 24 significand bits);
//   phase 2  the forward's columns;
//   phase 3  the forward's rows, whose result M, rounded to bf16 (the block's activation), becomes the B operand of a
//            product with W_out: lane i of the worker holds output channel i of the row's 64 values.
// For C = 64 a projection is two products, one per token of the pair (k < 64 and k >= 64), with W_out's or W_in's rows stacked
// twice, so that no token meets another's values.  X and Y cross HBM once.
//
// Bound as the forward is, by the exchange of the workspace and the row transforms: full image [1, 65536, 128] 48.5 us against the
// mixer's 38.0 (before: 61.3, with a row's exchange and both projections in one worker of 128 elements a thread).  With Z
// rounded, two products a row and 64 two-byte stores a thread take less than the three terms' 24 products and their table:
// [8, 4096, 128] 25.1 -> 23.3 us, [32, 4096, 64] 37.9 -> 34.3, [1, 1024, 128] 13.3 -> 11.9.
#pragma once

#include "whtmix_tri.cuh"

namespace whtmix {
namespace tri {

// Whether Z is rounded to bf16 before the mixer.  Where the block runs in three launches it is, and a shape that moves from three
// launches to this kernel keeps its result; C = 128 from 2^21 elements has always run fused, without the rounding.
template <int Q, int C>
__host__ __device__ constexpr bool rounds_z() { return !(C == 128 && Q >= 8); }

constexpr int BLK_XSLOTS = 2;                 // X rows staged per worker
constexpr int BLK_A = WORKERS * BLK_XSLOTS * TILE * 2;  // 128 KiB: behind the X staging areas A's three terms, or H_128 and W_in
constexpr int BLK_W = SLOT_BYTES;             // W_out behind the slots (phase 3)
constexpr size_t BLK_SMEM = SLOT_BYTES + H_BYTES;
static_assert(BLK_A + 3 * H_BYTES == static_cast<int>(BLK_SMEM), "the terms fill shared memory");

// byte offset of element (row r, k) of a K-major operand of 128 k: two 128-byte-swizzled panels of `rows` rows
__device__ __forceinline__ int panel_off(int r, int k, int rows) {
  return (k >> 6) * (rows * 128) + r * 128 + ((((k & 63) >> 3) ^ (r & 7)) << 4) + (k & 7) * 2;
}

// A = H_128 W (C = 128) as three bf16 terms at sm + BLK_A; sm[BLK_A ..] also holds the transform's exchange buffer (64 KiB), and
// the whole CTA takes part.
__device__ __forceinline__ void build_hw(unsigned char* sm, const __nv_bfloat16* __restrict__ w) {
  float* buf = reinterpret_cast<float*>(sm + BLK_A);
  const int k = threadIdx.x & 127, part = threadIdx.x >> 7;
  float v[32];  // rows 32 part .. of column k
#pragma unroll
  for (int r = 0; r < 32; ++r) v[r] = __bfloat162float(w[(32 * part + r) * 128 + k]);
#pragma unroll
  for (int h = 1; h < 32; h <<= 1)
#pragma unroll
    for (int r = 0; r < 32; ++r)
      if ((r & h) == 0) {
        const float a = v[r], b = v[r + h];
        v[r] = a + b;
        v[r + h] = a - b;
      }
#pragma unroll
  for (int r = 0; r < 32; ++r) buf[(32 * part + r) * 128 + k] = v[r];
  __syncthreads();
  float u[8][4];  // rows r + 32 j, r = 8 part ..
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    float q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = buf[(32 * j + 8 * part + r) * 128 + k];
    const float s0 = q[0] + q[1], d0 = q[0] - q[1], s1 = q[2] + q[3], d1 = q[2] - q[3];
    u[r][0] = s0 + s1;
    u[r][1] = d0 + d1;
    u[r][2] = s0 - s1;
    u[r][3] = d0 - d1;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float rest = u[r][j];
      const int o = panel_off(32 * j + 8 * part + r, k, 128);
#pragma unroll
      for (int term = 0; term < 3; ++term) {
        const __nv_bfloat16 b = __float2bfloat16_rn(rest);
        *reinterpret_cast<__nv_bfloat16*>(sm + BLK_A + term * H_BYTES + o) = b;
        rest -= __bfloat162float(b);
      }
    }
}
// W as the A operand of project_row at `dst`; for C = 64 its 64 rows twice.
template <int C>
__device__ __forceinline__ void load_w(unsigned char* dst, const __nv_bfloat16* __restrict__ w) {
  constexpr int CHUNKS = C / 8;
  for (int q = threadIdx.x; q < 128 * CHUNKS; q += THREADS) {
    const int r = q / CHUNKS, k = (q % CHUNKS) * 8;
    *reinterpret_cast<uint4*>(dst + panel_off(r, k, 128)) = __ldg(reinterpret_cast<const uint4*>(w + (r & (C - 1)) * C + k));
  }
}
// D = W x row, one thread: lane o of the columns at d holds output channel o (C = 128); for C = 64 lanes 0..63 of the
// columns at d the even token's channels, lanes 64..127 of those at d + 64 the odd token's (proj_lane).
template <int C>
__device__ __forceinline__ void project_row(uint32_t d, uint32_t w, uint32_t x) {
  if constexpr (C == 128) {
    mma_row(d, w, x);
  } else {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        tc::mma_bf16(d + 64 * s, tc::sw128_desc(w + k * 32), tc::sw128_desc(x + s * 8192 + k * 32), tc::instr_desc(128, 64), k > 0);
  }
}
template <int C>
__device__ __forceinline__ uint32_t proj_lane(uint32_t d, int t) { return d + (C == 64 ? 64u * (t >> 6) : 0u); }

template <int Q, int C>
__global__ void __launch_bounds__(THREADS, 1) k_block_fast(Params P, const __nv_bfloat16* __restrict__ w_in,
                                                            const __nv_bfloat16* __restrict__ w_out) {
  extern __shared__ __align__(1024) unsigned char tri_smem[];
  __shared__ CtaShared sh;
  constexpr int m = R + Q;
  float* ws = static_cast<float*>(P.ws);
  {
    int rb, re;
    share(static_cast<unsigned>(min(static_cast<long long>(P.gp), P.B)) << Q, &rb, &re);
    fast::l2_prefetch_first_rows<DT_BF16, R, Q>(P.x, rb, re, P.lv);
  }
  Cta c = cta_begin<DT_F32, 9>(tri_smem, sh, P);  // tensor memory, no H_128
  pdl_wait();
  GridSync gsync(P.bar, &sh.flag);
  const GainPrefetch prefetch(P.g, m);
  const uint32_t smem = tc::smem_u32(tri_smem);
  const int worker = c.worker, t = c.t;
  const uint32_t acc = c.tmem + 128u * worker, lane_bits = static_cast<uint32_t>(32 * ((threadIdx.x >> 5) & 3)) << 16;
  for (long long b0 = 0; b0 < P.B; b0 += P.gp) {
    const int nb = static_cast<int>(min(static_cast<long long>(P.gp), P.B - b0));
    int rb, re;
    share(static_cast<unsigned>(nb) << Q, &rb, &re);
    const int n = re - rb, nw = (n - worker + WORKERS - 1) / WORKERS;
    const unsigned short* xr = static_cast<const unsigned short*>(P.x) + (b0 << m) + (static_cast<long long>(rb) << R);
    const uint32_t xs = smem + worker * (BLK_XSLOTS * TILE * 2);
    auto load = [&](int i) {
      if (i < nw) load_x_bf16(xr + (static_cast<long long>(worker + WORKERS * i) << R), TILE, xs + (i % BLK_XSLOTS) * (TILE * 2), t);
      fast::cp_async_commit();
    };
    auto prefetch_gains = [&](int i) {
      if (t == 0 && b0 == 0 && prefetches_gains(Q)) prefetch(worker + WORKERS * i, n);
    };
    auto row_bits_out = [&](int i, float2 (&v)[32]) {  // the other six bits, and to the workspace
#pragma unroll
      for (int j = 0; j < 32; ++j) bf_in(v[j]);
      bfly32<0>(v);
      float* o = ws + (static_cast<long long>(rb + worker + WORKERS * i) << R) + t;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        __stcg(o + 256 * j, v[j].x);
        __stcg(o + 256 * j + 128, v[j].y);
      }
    };
    for (int i = 0; i < BLK_XSLOTS; ++i) load(i);
    if constexpr (rounds_z<Q, C>()) {
      // phase 1, Z rounded (a worker has at most four rows of a plane group, and the four workers' chains overlap: the products
      // of one are not pipelined)
      constexpr int A_H = BLK_A, A_W = BLK_A + H_BYTES;
      build_h(tri_smem + A_H);
      load_w<C>(tri_smem + A_W, w_in);
      fence_async();
      __syncthreads();
      auto product = [&](auto issue) {  // this worker's next product, completed; the worker's shared-memory writes lie before it
        fence_async();
        fast::tmem_fence_before();
        worker_sync(worker);
        uint64_t* done = &c.mma_done[worker][c.mma_seq & 1];
        if (t == 0) {
          fast::tmem_fence_after();
          issue();
          tc::mma_commit(done);
        }
        wait_bar(done, (c.mma_seq >> 1) & 1u, c.bar, c.dead);
        ++c.mma_seq;
        __syncwarp();
        fast::tmem_fence_after();
      };
      for (int i = 0; i < nw; ++i) {
        prefetch_gains(i);
        const uint32_t x = xs + (i % BLK_XSLOTS) * (TILE * 2);
        asm volatile("cp.async.wait_group %0;" ::"n"(BLK_XSLOTS - 1) : "memory");
        product([&] { project_row<C>(acc, smem + A_W, x); });
        float2 v[32];
        read_row(proj_lane<C>(acc, t) + lane_bits, v);
        unsigned char* z = tri_smem + (x - smem);  // over the row of X
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          *reinterpret_cast<__nv_bfloat16*>(z + panel_off(2 * j, t, 64)) = __float2bfloat16_rn(v[j].x);
          *reinterpret_cast<__nv_bfloat16*>(z + panel_off(2 * j + 1, t, 64)) = __float2bfloat16_rn(v[j].y);
        }
        product([&] { mma_row(acc, smem + A_H, x); });
        load(i + BLK_XSLOTS);
        read_row(acc + lane_bits, v);
        row_bits_out(i, v);
      }
    } else {
      // phase 1 (as rows_in, with A's terms for H_128 and two rows staged ahead)
      auto multiply = [&](int i) {
        fence_async();
        fast::tmem_fence_before();
        worker_sync(worker);
        if (t == 0) {
          fast::tmem_fence_after();
          const uint32_t x = xs + (i % BLK_XSLOTS) * (TILE * 2), d = acc + 64u * (i & 1);
#pragma unroll
          for (int term = 2; term >= 0; --term)  // smallest first
#pragma unroll
            for (int k = 0; k < 8; ++k)
              tc::mma_bf16(d, tc::sw128_desc(smem + BLK_A + term * H_BYTES + (k >> 2) * 16384 + (k & 3) * 32),
                           tc::sw128_desc(x + (k >> 2) * 8192 + (k & 3) * 32), tc::instr_desc(128, 64), term < 2 || k > 0);
          tc::mma_commit(&c.mma_done[worker][(c.mma_seq + i) & 1]);
        }
      };
      build_hw(tri_smem, w_in);
      fence_async();
      __syncthreads();
      if (nw > 0) {
        asm volatile("cp.async.wait_group %0;" ::"n"(BLK_XSLOTS - 1) : "memory");
        multiply(0);
      }
      for (int i = 0; i < nw; ++i) {
        prefetch_gains(i);
        if (i + 1 < nw) {
          asm volatile("cp.async.wait_group %0;" ::"n"(BLK_XSLOTS - 2) : "memory");
          multiply(i + 1);
        }
        wait_bar(&c.mma_done[worker][(c.mma_seq + i) & 1], ((c.mma_seq + i) >> 1) & 1u, c.bar, c.dead);
        __syncwarp();
        fast::tmem_fence_after();
        float2 v[32];
        read_row(acc + 64u * (i & 1) + lane_bits, v);
        load(i + BLK_XSLOTS);
        row_bits_out(i, v);
      }
      c.mma_seq += nw;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    fast::tmem_fence_before();
    if (!gsync()) break;
    // phase 2
    columns<Q, FULL, FWD>(c, ws, nb, P, nullptr);
    fast::tmem_fence_before();
    if (!gsync()) break;
    // phase 3 (as rows_out up to the row in registers)
    load_w<C>(tri_smem + BLK_W, w_out);
    fence_async();
    const float* wsr = ws + (static_cast<long long>(rb) << R);
    auto load_m = [&](int k) {
      load_row(wsr + (static_cast<long long>(k) << R), TILE, c.slots + (c.row_seq + k) % SLOTS * TILE, t,
               &c.full_row[(c.row_seq + k) % ROW_BARS]);
    };
    for (int k = worker; k < SLOTS && k < n; k += WORKERS) load_m(k);
    __syncthreads();
    for (int k = worker, i = 0; k < n; k += WORKERS, ++i) {
      float* slot = c.slots + (c.row_seq + k) % SLOTS * TILE;
      const uint32_t d = acc + (C == 128 ? 64u * (i & 1) : 0u);
      wait_full(c.full_row, c.row_seq + k, ROW_BARS, c.bar, c.dead);
      float2 a[16][2];
      row_transform(slot, a, t, worker, [] {});
      // the row as the B operand, over its own slot
      unsigned char* mb = reinterpret_cast<unsigned char*>(slot);
#pragma unroll
      for (int v = 0; v < 16; ++v) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(a[v][0].x, a[v][0].y), h1 = __floats2bfloat162_rn(a[v][1].x, a[v][1].y);
        *reinterpret_cast<uint2*>(mb + panel_off((t >> 5) + 4 * v, 4 * (t & 31), 64)) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
      }
      fence_async();
      fast::tmem_fence_before();
      worker_sync(worker);
      if (t == 0) {
        fast::tmem_fence_after();
        project_row<C>(d, smem + BLK_W, tc::smem_u32(mb));
        tc::mma_commit(&c.mma_done[worker][(c.mma_seq + i) & 1]);
      }
      wait_bar(&c.mma_done[worker][(c.mma_seq + i) & 1], ((c.mma_seq + i) >> 1) & 1u, c.bar, c.dead);
      __syncwarp();
      fast::tmem_fence_after();
      if (k + SLOTS < n) load_m(k + SLOTS);
      float2 v[32];
      read_row(proj_lane<C>(d, t) + lane_bits, v);
      __nv_bfloat16* y = static_cast<__nv_bfloat16*>(P.y) + (b0 << m) + (static_cast<long long>(rb + k) << R) + t;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        y[256 * j] = __float2bfloat16_rn(v[j].x);
        y[256 * j + 128] = __float2bfloat16_rn(v[j].y);
      }
    }
    c.row_seq += n;
    c.mma_seq += nw;
    fast::tmem_fence_before();
    if (b0 + P.gp < P.B && !gsync()) break;
  }
  pdl_trigger();
  cta_end<DT_F32, 9>(sh);
}

}  // namespace tri
}  // namespace whtmix

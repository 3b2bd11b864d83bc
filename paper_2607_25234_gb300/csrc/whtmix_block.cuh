// whtmix_block.cuh -- the whole mixer block of Section III-B, Eq. 1-4, as one persistent launch for bf16 planes of 64 or
// 128 channels:
//   Y_b = ( H_N (G o (H_N (X_b W_in^T) H_C)) H_C / (N C) ) W_out^T
// The three-phase forward (whtmix_tri.cuh) with the projections in its row phases, on the tensor cores:
//   phase 1  a row is 128 consecutive elements k (the channels, and for C = 64 two tokens) by 64 values n.  The
//            forward multiplies it by H_128; here by A = H_128 W, W = W_in (C = 128) or diag(W_in, W_in) (C = 64), so
//            that the input projection and the seven low transform bits are one contraction: Z = X W_in^T is never
//            formed.  A is computed in fp32 and used as three bf16 terms (together its 24 significand bits), so the
//            products keep the precision of an unrounded Z;
//   phase 2  the forward's columns;
//   phase 3  the forward's rows, whose result M, rounded to bf16 (the block's activation), becomes the B operand of a
//            product with W_out: lane i of the worker holds output channel i of the row's 64 values.
// X and Y cross HBM once.
//
// Bound as the forward is, by the exchange of the workspace and the row transforms: full image [1, 65536, 128] 48.5 us against the
// mixer's 38.0 (before: 61.3, with a row's exchange and both projections in one worker of 128 elements a thread).
#pragma once

#include "whtmix_tri.cuh"

namespace whtmix {
namespace tri {

constexpr int BLK_XSLOTS = 2;                 // X rows staged per worker
constexpr int BLK_A = WORKERS * BLK_XSLOTS * TILE * 2;  // 128 KiB: A's three terms behind the X staging areas
constexpr int BLK_W = SLOT_BYTES;             // W_out behind the slots (phase 3)
constexpr size_t BLK_SMEM = SLOT_BYTES + H_BYTES;
static_assert(BLK_A + 3 * H_BYTES == static_cast<int>(BLK_SMEM), "the terms fill shared memory");

// byte offset of element (row r, k) of a K-major operand of 128 k: two 128-byte-swizzled panels of `rows` rows
__device__ __forceinline__ int panel_off(int r, int k, int rows) {
  return (k >> 6) * (rows * 128) + r * 128 + ((((k & 63) >> 3) ^ (r & 7)) << 4) + (k & 7) * 2;
}

// A = H_128 W as three bf16 terms at sm + BLK_A; sm[BLK_A ..] also holds the transform's exchange buffer (64 KiB), and the
// whole CTA takes part.
template <int C>
__device__ __forceinline__ void build_hw(unsigned char* sm, const __nv_bfloat16* __restrict__ w) {
  float* buf = reinterpret_cast<float*>(sm + BLK_A);
  const int k = threadIdx.x & 127, part = threadIdx.x >> 7;
  float v[32];  // rows 32 part .. of column k
#pragma unroll
  for (int r = 0; r < 32; ++r) {
    const int o = 32 * part + r;
    const bool in = C == 128 || (o >> 6) == (k >> 6);
    v[r] = in ? __bfloat162float(w[(o & (C - 1)) * C + (k & (C - 1))]) : 0.f;
  }
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
// W_out, or diag(W_out, W_out) for C = 64, as the A operand at sm + BLK_W.
template <int C>
__device__ __forceinline__ void load_w_out(unsigned char* sm, const __nv_bfloat16* __restrict__ w) {
  for (int q = threadIdx.x; q < 128 * 16; q += THREADS) {
    const int r = q >> 4, k = (q & 15) * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (C == 128 || (r >> 6) == (k >> 6)) v = __ldg(reinterpret_cast<const uint4*>(w + (r & (C - 1)) * C + (k & (C - 1))));
    *reinterpret_cast<uint4*>(sm + BLK_W + panel_off(r, k, 128)) = v;
  }
}

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
    // phase 1 (as rows_in, with A's terms for H_128 and two rows staged ahead)
    const uint32_t xs = smem + worker * (BLK_XSLOTS * TILE * 2);
    auto load = [&](int i) {
      if (i < nw) load_x_bf16(xr + (static_cast<long long>(worker + WORKERS * i) << R), TILE, xs + (i % BLK_XSLOTS) * (TILE * 2), t);
      fast::cp_async_commit();
    };
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
    for (int i = 0; i < BLK_XSLOTS; ++i) load(i);
    build_hw<C>(tri_smem, w_in);
    fence_async();
    __syncthreads();
    if (nw > 0) {
      asm volatile("cp.async.wait_group %0;" ::"n"(BLK_XSLOTS - 1) : "memory");
      multiply(0);
    }
    for (int i = 0; i < nw; ++i) {
      if (t == 0 && b0 == 0 && prefetches_gains(Q)) prefetch(worker + WORKERS * i, n);
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
#pragma unroll
      for (int j = 0; j < 32; ++j) bf_in(v[j]);
      bfly32<0>(v);
      float* o = ws + (static_cast<long long>(rb + worker + WORKERS * i) << R) + t;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        __stcg(o + 256 * j, v[j].x);
        __stcg(o + 256 * j + 128, v[j].y);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    c.mma_seq += nw;
    fast::tmem_fence_before();
    if (!gsync()) break;
    // phase 2
    columns<Q, false, FWD>(c, ws, nb, P, nullptr);
    fast::tmem_fence_before();
    if (!gsync()) break;
    // phase 3 (as rows_out up to the row in registers)
    load_w_out<C>(tri_smem, w_out);
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
        mma_row(acc + 64u * (i & 1), smem + BLK_W, tc::smem_u32(mb));
        tc::mma_commit(&c.mma_done[worker][(c.mma_seq + i) & 1]);
      }
      wait_bar(&c.mma_done[worker][(c.mma_seq + i) & 1], ((c.mma_seq + i) >> 1) & 1u, c.bar, c.dead);
      __syncwarp();
      fast::tmem_fence_after();
      if (k + SLOTS < n) load_m(k + SLOTS);
      float2 v[32];
      read_row(acc + 64u * (i & 1) + lane_bits, v);
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

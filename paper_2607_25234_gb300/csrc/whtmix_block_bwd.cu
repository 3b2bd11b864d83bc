// whtmix_block_bwd.cu -- the pieces of the mixer block's backward (Section III-B, Eq. 1-4) that the
// forward kernels do not already provide: the weight gradients
//     dW[o, i] = sum over tokens t of A[t, o] B[t, i]      (dW_out = dY^T M, dW_in = dZ^T X)
// on the 5th-generation tensor cores, and the weight transposes the projections need.
//
// A and B are [T, C] bf16 token rows; the contraction runs over the tokens.  k_wgrad splits the tokens into one chunk per
// CTA (one persistent CTA per SM, 128 threads): K tiles of 64 tokens of both operands are copied as they are by 16-byte
// cp.async into 128-byte-swizzled panels of 64 channels, up to five tiles ahead, and multiplied from there as
// M-major and N-major operands (the channels are contiguous, the contraction runs down the panel's rows), so nothing is
// transposed; one thread issues tcgen05.mma (kind::f16, M = 128, N = C, K = 16) into a TMEM accumulator per 128 input
// channels i.  A lane of the accumulator is an i, a column an o, so that a warp stores 32 consecutive floats of the chunk's
// fp32 partial [C, C] at a time (with the roles swapped, 32 rows at a stride: 16384 tokens of 256 channels 16.9 us, so 11.8);
// k_wgrad_reduce adds the partials in a fixed order, so dW is the same bit for bit on every run.
// A chunk is a few tiles (3.4 at 32768 tokens), so its time is the latency of its chain: with 8 x 8 transposes in registers
// and one tile ahead it took 13.2 us, now 9.0 (32768 tokens, C = 128; whole block_train step [8, 4096, 128] 140 -> 124).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "whtmix_kernels.cuh"
#include "whtmix_tc.cuh"

namespace whtmix {
namespace bbwd {

using namespace tc;

constexpr int KT = 64;             // tokens per K tile (one 128-byte row of bf16 per operand row)
constexpr int WG_THREADS = 128;    // one thread per TMEM lane
constexpr int TR_THREADS = 256;
constexpr size_t SMEM_MIN = 120 * 1024;  // more than half an SM: one CTA per SM, so TMEM allocation never waits

// out0 = in0^T and out1 = in1^T, bf16 [C, C], C a multiple of 64: both weights' transposes in one launch.
__global__ void __launch_bounds__(TR_THREADS) k_transpose2(const uint16_t* __restrict__ in0, uint16_t* __restrict__ out0,
                                                           const uint16_t* __restrict__ in1, uint16_t* __restrict__ out1, int C) {
  __shared__ uint16_t tile[64][66];
  pdl_wait();
  const int n = C / 64, blk = blockIdx.x % (n * n), tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
  const int r0 = 64 * (blk / n), c0 = 64 * (blk % n);
  const uint16_t* in = static_cast<int>(blockIdx.x) < n * n ? in0 : in1;
  uint16_t* out = static_cast<int>(blockIdx.x) < n * n ? out0 : out1;
#pragma unroll
  for (int r = ty; r < 64; r += TR_THREADS / 64) tile[r][tx] = in[(r0 + r) * C + c0 + tx];
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 64; r += TR_THREADS / 64) out[(c0 + r) * C + r0 + tx] = tile[tx][r];
  pdl_trigger();
}

// Shared-memory descriptor of an M- or N-major operand in 128-byte-swizzled panels of 64 channels (rows of 128 bytes, one
// token each; 16-byte chunk j of token t at chunk j ^ (t mod 8)): `panel` bytes to the next 64 channels, 1024 to the next 8
// tokens.
__device__ __forceinline__ uint64_t mn_desc(uint32_t addr, uint32_t panel) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(panel >> 4) << 16) |
         (static_cast<uint64_t>(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// instr_desc with A and B M- and N-major
constexpr uint32_t MN_MAJOR = (1u << 15) | (1u << 16);

template <int C>
struct Wg {
  static constexpr int MT = C > 128 ? C / 128 : 1;             // MMA tiles of 128 input channels
  static constexpr uint32_t PANEL = KT * 128, OPERAND = C / 64 * PANEL, STAGE = 2 * OPERAND;
  static constexpr int STAGES = C == 256 ? 3 : 6;
  static constexpr size_t SMEM = STAGES * STAGE + 1024 > SMEM_MIN ? STAGES * STAGE + 1024 : SMEM_MIN;  // 1024: alignment slack
  static constexpr uint32_t TCOLS = MT * C;                    // 64, 128 or 512 TMEM columns
};

// Partial weight gradient of token chunk blockIdx.x: part[chunk][o][i] = sum over the chunk's tokens t of A[t][o] B[t][i], with A
// and B the [T, C] token rows as given.  C in {64, 128, 256}.
template <int C>
__global__ void __launch_bounds__(WG_THREADS, 1) k_wgrad(const uint16_t* __restrict__ A, const uint16_t* __restrict__ B,
                                                         float* __restrict__ part, long long T, int nchunk,
                                                         unsigned int* err) {
  using G = Wg<C>;
  constexpr int MT = G::MT, S = G::STAGES;
  constexpr uint32_t TCOLS = G::TCOLS;
  static_assert(C == 64 || C == 128 || C == 256, "channels");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint64_t mbar[S];
  __shared__ uint32_t tmem_slot;
  // the swizzle pattern is a function of the address: stage buffers start on 1024-byte boundaries
  const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid < 32) tmem_alloc(&tmem_slot, TCOLS);
  if (tid == 0) {
    for (int i = 0; i < S; ++i) mbar_init(&mbar[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  pdl_wait();
  const uint32_t tmem = tmem_slot;
  const long long ntiles = (T + KT - 1) / KT;
  const long long k0 = ntiles * blockIdx.x / nchunk, k1 = ntiles * (blockIdx.x + 1) / nchunk;
  const int n = static_cast<int>(k1 - k0);

  auto load = [&](int i) {  // tile i of the chunk into stage i mod S; tokens past T are zero
    if (i < n) {
      const uint32_t st = smem + (i % S) * G::STAGE;
#pragma unroll
      for (int j = 0; j < C * KT / 8 / WG_THREADS; ++j) {
        const int q = tid + WG_THREADS * j, tok = q / (C / 8), c = q % (C / 8);
        const long long t = (k0 + i) * KT + tok;
        const bool in = t < T;
        const long long off = (in ? t : 0) * C + 8 * c;
        const uint32_t d = st + (c >> 3) * G::PANEL + tok * 128 + (((c & 7) ^ (tok & 7)) << 4);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(A + off), "r"(in ? 16 : 0) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + G::OPERAND), "l"(B + off), "r"(in ? 16 : 0) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // the products of tile i have completed (all threads; false if the wait gave up)
  auto done = [&](int i) { return __syncthreads_and(mbar_wait(&mbar[i % S], (i / S) & 1) ? 1 : 0) != 0; };

  const uint32_t idesc = instr_desc(128, C) | MN_MAJOR;
  bool ok = true;
  for (int i = 0; i < S - 1; ++i) load(i);
  for (int i = 0; i < n; ++i) {
    asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = smem + (i % S) * G::STAGE, sb = sa + G::OPERAND;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int ks = 0; ks < KT / 16; ++ks)  // K steps of 16 tokens: 2048 bytes down the panels
          // (C = 64: rows 64 .. 127 of the product read the only panel again and are not used)
          mma_bf16(tmem + mt * C, mn_desc(sb + 2 * mt * G::PANEL + ks * 2048, C > 64 ? G::PANEL : 0),
                   mn_desc(sa + ks * 2048, C > 64 ? G::PANEL : 0), idesc, (i > 0 || ks > 0) ? 1u : 0u);
      mma_commit(&mbar[i % S]);
    }
    if (i + S - 1 < n && i > 0) {  // the stage of tile i - 1 is next
      ok = done(i - 1);
      if (!ok) break;
    }
    load(i + S - 1);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (ok && n > 0) ok = done(n - 1);  // the last commit covers every product issued before it
  if (!ok && tid == 0) atomicOr(err, 1u << 13);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // lane i = mt * 128 + tid, column o of the accumulator -> this chunk's partial (zeros for an empty chunk)
  float* pc = part + static_cast<long long>(blockIdx.x) * C * C;
  const bool live = ok && n > 0;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const int i = mt * 128 + tid;
#pragma unroll 4
    for (int c0 = 0; c0 < C; c0 += 16) {
      float v[16];
      tmem_ld16(tmem + (static_cast<uint32_t>(32 * warp) << 16) + mt * C + c0, v);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (i < C) {
#pragma unroll
        for (int q = 0; q < 16; ++q) pc[(c0 + q) * C + i] = live ? v[q] : 0.f;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  pdl_trigger();
  if (tid < 32) tmem_dealloc(tmem, TCOLS);
}

// dW = the sum of the chunks' partials (float32) in a fixed order: RG runs of consecutive chunks,
// each summed in ascending order by one thread, then the RG run sums in ascending order.  A CTA
// covers 32 float4 outputs x RG runs.
constexpr int RG = TR_THREADS / 32;
__global__ void __launch_bounds__(TR_THREADS) k_wgrad_reduce(const float4* __restrict__ part, float4* __restrict__ out,
                                                             int cc4, int nchunk) {
  __shared__ float4 sums[RG][32];
  pdl_wait();
  const int o = blockIdx.x * 32 + (threadIdx.x & 31), g = threadIdx.x >> 5;
  const int c0 = nchunk * g / RG, c1 = nchunk * (g + 1) / RG;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (o < cc4) {
    int c = c0;
    for (; c + 4 <= c1; c += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldcs(part + static_cast<long long>(c + u) * cc4 + o);
#pragma unroll
      for (int u = 0; u < 4; ++u) acc = make_float4(acc.x + v[u].x, acc.y + v[u].y, acc.z + v[u].z, acc.w + v[u].w);
    }
    for (; c < c1; ++c) {
      const float4 v = __ldcs(part + static_cast<long long>(c) * cc4 + o);
      acc = make_float4(acc.x + v.x, acc.y + v.y, acc.z + v.z, acc.w + v.w);
    }
  }
  sums[g][threadIdx.x & 31] = acc;
  __syncthreads();
  if (g == 0 && o < cc4) {
    float4 s = sums[0][threadIdx.x];
#pragma unroll
    for (int r = 1; r < RG; ++r) {
      const float4 v = sums[r][threadIdx.x];
      s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w);
    }
    out[o] = s;
  }
  pdl_trigger();
}

// ---- host ----

// Token chunks of one weight gradient over T tokens: one per SM, and at least C / 64 K tiles a chunk: a partial is C / 64 times a
// tile's size or more, and is written and read again (C = 256, 16384 tokens: k_wgrad 18.8
// us and its reduction 9.6 with 152 chunks, 16.9 and 5.9 with 64).
int wgrad_chunks(long long T, int C, int sms) {
  const long long nt = (T + KT - 1) / KT, most = (nt + C / 64 - 1) / (C / 64);
  return static_cast<int>(most < sms ? (most < 1 ? 1 : most) : sms);
}

cudaError_t transpose2(const void* in0, void* out0, const void* in1, void* out1, int C, cudaStream_t stream) {
  const uint16_t *i0 = static_cast<const uint16_t*>(in0), *i1 = static_cast<const uint16_t*>(in1);
  uint16_t *o0 = static_cast<uint16_t*>(out0), *o1 = static_cast<uint16_t*>(out1);
  void* args[] = {&i0, &o0, &i1, &o1, &C};
  return launch_pdl(reinterpret_cast<const void*>(k_transpose2), static_cast<unsigned>(2 * (C / 64) * (C / 64)), TR_THREADS, 0, stream, args);
}

template <int C>
cudaError_t wgrad_c(const void* a_tok, const void* b_tok, float* part, float* out, long long T, int sms, unsigned int* err,
                    cudaStream_t stream) {
  constexpr size_t smem = Wg<C>::SMEM;
  const void* k = reinterpret_cast<const void*>(k_wgrad<C>);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  int nchunk = wgrad_chunks(T, C, sms);
  const uint16_t* a = static_cast<const uint16_t*>(a_tok);
  const uint16_t* b = static_cast<const uint16_t*>(b_tok);
  void* args[] = {&a, &b, &part, &T, &nchunk, &err};
  e = launch_pdl(k, static_cast<unsigned>(nchunk), WG_THREADS, smem, stream, args);
  if (e != cudaSuccess) return e;
  int cc4 = C * C / 4;
  const float4* pc = reinterpret_cast<const float4*>(part);
  float4* o4 = reinterpret_cast<float4*>(out);
  void* rargs[] = {&pc, &o4, &cc4, &nchunk};
  return launch_pdl(reinterpret_cast<const void*>(k_wgrad_reduce), static_cast<unsigned>((cc4 + 31) / 32), TR_THREADS, 0,
                    stream, rargs);
}

// dW = A^T B over the T tokens of the [T, C] bf16 operands a_tok, b_tok; part holds
// wgrad_chunks(T, C, sms) partial [C, C] fp32 planes; out is 16-byte aligned.
cudaError_t wgrad(const void* a_tok, const void* b_tok, float* part, float* out, long long T, int C, int sms,
                  unsigned int* err, cudaStream_t stream) {
  switch (C) {
    case 64: return wgrad_c<64>(a_tok, b_tok, part, out, T, sms, err, stream);
    case 128: return wgrad_c<128>(a_tok, b_tok, part, out, T, sms, err, stream);
    case 256: return wgrad_c<256>(a_tok, b_tok, part, out, T, sms, err, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace bbwd
}  // namespace whtmix

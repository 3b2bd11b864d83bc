// whtmix_fast_launch.cuh -- host-side launcher of the fast forward and backward kernels for one I/O dtype.
// Included by whtmix_fast_f32.cu and whtmix_fast_bf16.cu (one translation unit each, compiled in
// parallel).  Returns a cudaError_t; the C ABI maps it to a status.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>

#include "whtmix_tri.cuh"
#include "whtmix_x16.cuh"

namespace whtmix {
namespace fast {

// Resident CTAs per SM for one kernel and smem size, per device (first query also raises the
// kernel's dynamic shared memory limit).
inline cudaError_t occupancy_cached(const void* kernel, int threads, size_t smem, int* occ) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> cache;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  auto it = cache.find({dev, kernel});
  if (it != cache.end()) {
    *occ = it->second;
    return cudaSuccess;
  }
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (*occ < 1) return cudaErrorInvalidConfiguration;
  cache[{dev, kernel}] = *occ;
  return cudaSuccess;
}

// Every variant requests more than half an SM's shared memory, so exactly one CTA runs per SM:
// two CTAs on one SM would both ask for all 512 TMEM columns, and the second would wait in
// tcgen05.alloc while the first waits for it at the device-wide barrier.  The grid is one CTA per
// SM, all resident at once; it is launched with programmatic stream serialisation (launch_pdl),
// which lets its launch and tensor-memory allocation overlap the previous kernel's tail.
inline cudaError_t launch_persistent(const void* k, const Params& P, int grid, cudaStream_t stream, int threads, size_t smem) {
  int occ = 0;
  cudaError_t e = occupancy_cached(k, threads, smem, &occ);
  if (e != cudaSuccess) return e;
  if (occ != 1) return cudaErrorInvalidConfiguration;
  Params p = P;
  void* args[] = {&p};
  return launch_pdl(k, static_cast<unsigned>(grid), threads, smem, stream, args);
}
// CTAs of a three-phase launch: one per SM, or one per row of a small batch (at least 64, for the columns): the
// device-wide barriers wait for fewer arrivals ([1, 4096, 64] bf16, 32 rows: 152 CTAs 9.8 us, 64 8.9, 32 9.4;
// [1, 2048, 64] 9.4, 8.4, 8.6; [1, 16384, 64], 128 rows: 14.4 with 152, 14.2 with 128).  The backward's rows are X's
// and dY's.
inline int tri_grid(long long rows, int sms) {
  const long long want = rows < 64 ? 64 : rows;
  return want < sms ? static_cast<int>(want) : sms;
}

// The three-phase kernels (whtmix_tri.cuh) of a 2^m-element plane: 2^(m-13) rows of 2^13.  LOG: log gains (P.gt, P.gc) instead of G,
// whose channels lie within a row, 1 <= P.cbits <= 13; at 2^21 elements also C = 2^14, whose tokens are two rows each
// (WIDE_M, WIDE_CBITS; measured at use_fast_separable).
constexpr int WIDE_M = 21, WIDE_CBITS = 14;
template <int D, tri::Gains G, int M = 14>
cudaError_t launch_forward_tri(const Params& P, int sms, cudaStream_t stream) {
  if constexpr (M <= 25) {
    if (P.m != M) return launch_forward_tri<D, G, M + 1>(P, sms, stream);
    const void* k = reinterpret_cast<const void*>(tri::k_forward_fast<D, M - tri::R, G>);
    if constexpr (G == tri::LOG && M == WIDE_M) {
      if (P.cbits == WIDE_CBITS) k = reinterpret_cast<const void*>(tri::k_forward_fast<D, M - tri::R, tri::LOG_WIDE>);
    }
    return launch_persistent(k, P, tri_grid(P.B << (M - tri::R), sms), stream, tri::THREADS, tri::smem_bytes<D>());
  }
  return cudaErrorInvalidValue;
}
template <int D, int M = 14>
cudaError_t launch_backward(const Params& P, int sms, cudaStream_t stream) {
  if constexpr (M <= 23) {
    if (P.m != M) return launch_backward<D, M + 1>(P, sms, stream);
    return launch_persistent(reinterpret_cast<const void*>(tri::k_backward_fast<D, M - tri::R>), P, tri_grid(2 * P.B << (M - tri::R), sms), stream,
                             tri::THREADS, tri::smem_bytes<D>());
  }
  return cudaErrorInvalidValue;
}

// The bf16-exchange forward (whtmix_forward_x16; whtmix_x16.cuh).  Rows of 2^13 elements at every size but 2^21;
// 2^23-element planes take 1024-row columns (two lanes per column).  With 152 SMs, 1024 rows of 2^13 spread as 7 or 6
// per CTA, where 512 rows of 2^14 give 56 CTAs four rows against three; 2^21-element planes take rows of 2^14 and
// 128-row columns, one column per thread in registers, instead of 256-row columns in tensor memory.
template <int D, int R, int Q>
cudaError_t launch_x16_one(const Params& P, int sms, cudaStream_t stream) {
  return launch_persistent(reinterpret_cast<const void*>(x16::k_forward_x16<D, R, Q>), P, sms, stream, x16::THREADS, x16::SMEM_BYTES);
}
template <int D>
cudaError_t launch_forward_x16(const Params& P, int sms, cudaStream_t stream) {
  switch (P.m) {
    case 14: return launch_x16_one<D, 13, 1>(P, sms, stream);
    case 15: return launch_x16_one<D, 13, 2>(P, sms, stream);
    case 16: return launch_x16_one<D, 13, 3>(P, sms, stream);
    case 17: return launch_x16_one<D, 13, 4>(P, sms, stream);
    case 18: return launch_x16_one<D, 13, 5>(P, sms, stream);
    case 19: return launch_x16_one<D, 13, 6>(P, sms, stream);
    case 20: return launch_x16_one<D, 13, 7>(P, sms, stream);
    case 21: return launch_x16_one<D, 14, 7>(P, sms, stream);
    case 22: return launch_x16_one<D, 13, 9>(P, sms, stream);
    case 23: return launch_x16_one<D, 13, 10>(P, sms, stream);
    default: return cudaErrorInvalidValue;
  }
}

// Entry points defined in whtmix_fast_f32.cu / whtmix_fast_bf16.cu.
cudaError_t forward_f32(const Params& P, int sms, cudaStream_t stream);
cudaError_t forward_bf16(const Params& P, int sms, cudaStream_t stream);
cudaError_t backward_f32(const Params& P, int sms, cudaStream_t stream);
cudaError_t backward_bf16(const Params& P, int sms, cudaStream_t stream);
// whtmix_fast_x16.cu: the forward with a bf16 exchange workspace
cudaError_t forward_x16_f32(const Params& P, int sms, cudaStream_t stream);
cudaError_t forward_x16_bf16(const Params& P, int sms, cudaStream_t stream);
// whtmix_fast_sep_f32.cu / whtmix_fast_sep_bf16.cu
cudaError_t forward_sep_f32(const Params& P, int sms, cudaStream_t stream);
cudaError_t forward_sep_bf16(const Params& P, int sms, cudaStream_t stream);

}  // namespace fast
}  // namespace whtmix

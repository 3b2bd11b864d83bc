// One-plane-per-CTA forward (planes of 2^14 .. 2^16 elements in tensor memory): host-side launcher,
// fp32 and bf16 I/O.
#include <cuda_runtime.h>

#include <map>
#include <mutex>

#include "whtmix_plane.cuh"

namespace whtmix {
namespace pln {

// Per device and kernel: raise the dynamic shared memory limit once.  `dev_out`: the current device.
static std::mutex g_mu;
static std::map<std::pair<int, const void*>, cudaError_t> g_prepared;

static cudaError_t prepare(const void* k, size_t smem) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_prepared.find({dev, k});
  if (it != g_prepared.end()) return it->second;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  g_prepared[{dev, k}] = e;
  return e;
}

// The kernels' error header on device `dev` (the current one), or null if none of them was launched there.
void* error_header(int dev) {
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_prepared.lower_bound({dev, nullptr});
    if (it == g_prepared.end() || it->first.first != dev) return nullptr;
  }
  void* p = nullptr;
  return cudaGetSymbolAddress(&p, plane_barrier) == cudaSuccess ? p : nullptr;
}

template <int D, int M>
cudaError_t launch_m(const Params& P, cudaStream_t stream) {
  using C = Plane<D, M>;
  const void* k = reinterpret_cast<const void*>(k_forward_plane<D, M>);
  cudaError_t e = prepare(k, C::SMEM);
  if (e != cudaSuccess) return e;
  Params p = P;
  void* args[] = {&p};
  return launch_pdl(k, static_cast<unsigned>(P.B), C::THREADS, C::SMEM, stream, args);
}

template <int D>
cudaError_t launch(const Params& P, cudaStream_t stream) {
  switch (P.m) {
    case 14: return launch_m<D, 14>(P, stream);
    case 15: return launch_m<D, 15>(P, stream);
    case 16: return launch_m<D, 16>(P, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t forward_f32(const Params& P, cudaStream_t stream) { return launch<DT_F32>(P, stream); }
cudaError_t forward_bf16(const Params& P, cudaStream_t stream) { return launch<DT_BF16>(P, stream); }

}  // namespace pln
}  // namespace whtmix

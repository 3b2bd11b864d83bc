// fp32 / bf16 planes of 2^10 .. 2^13 elements: host-side launchers (whtmix_small.cuh).
#include <cuda_runtime.h>

#include "whtmix_small.cuh"

namespace whtmix {
namespace sml {

template <int D, int M>
cudaError_t forward_m(const Params& P, cudaStream_t stream) {
  const long long tiles = (P.B + (1ll << (13 - M)) - 1) >> (13 - M);
  if (tiles > 0x7fffffff) return cudaErrorInvalidConfiguration;
  Params p = P;
  void* args[] = {&p};
  return launch_pdl(reinterpret_cast<const void*>(k_forward_small<D, M>), static_cast<unsigned>(tiles), WT, 0, stream, args);
}

// Groups of P.gp planes (what the workspace holds): the dG terms of a group, then their sum.
template <int D, int M>
cudaError_t backward_m(const Params& P, cudaStream_t stream) {
  constexpr size_t ES = D == DT_BF16 ? 2 : 4;
  for (long long b0 = 0; b0 < P.B; b0 += P.gp) {
    Params p = P;
    const size_t skip = static_cast<size_t>(b0) * static_cast<size_t>(P.lv) * ES;
    p.x = static_cast<const char*>(P.x) + skip;
    p.dy = static_cast<const char*>(P.dy) + skip;
    p.dx = static_cast<char*>(P.dx) + skip;
    long long nb = P.B - b0 < P.gp ? P.B - b0 : P.gp;
    p.B = nb;
    void* args[] = {&p};
    const long long tiles = (nb + (1ll << (13 - M)) - 1) >> (13 - M);
    cudaError_t e = launch_pdl(reinterpret_cast<const void*>(k_backward_small<D, M>), static_cast<unsigned>(tiles), WT, 0, stream, args);
    if (e != cudaSuccess) return e;
    float* dg = static_cast<float*>(P.dg);
    const float* part = static_cast<const float*>(P.ws);
    int m = M, first = b0 == 0;
    void* rargs[] = {&dg, &part, &m, &nb, &first};
    e = launch_pdl(reinterpret_cast<const void*>(k_small_dg), 1u << (M - 5), DG_THREADS, 0, stream, rargs);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int D>
cudaError_t run(bool backward, const Params& P, cudaStream_t stream) {
  switch (P.m) {
    case 10: return backward ? backward_m<D, 10>(P, stream) : forward_m<D, 10>(P, stream);
    case 11: return backward ? backward_m<D, 11>(P, stream) : forward_m<D, 11>(P, stream);
    case 12: return backward ? backward_m<D, 12>(P, stream) : forward_m<D, 12>(P, stream);
    case 13: return backward ? backward_m<D, 13>(P, stream) : forward_m<D, 13>(P, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t run_f32(bool backward, const Params& P, cudaStream_t stream) { return run<DT_F32>(backward, P, stream); }
cudaError_t run_bf16(bool backward, const Params& P, cudaStream_t stream) { return run<DT_BF16>(backward, P, stream); }

}  // namespace sml
}  // namespace whtmix

// Fused mixer block (Section III-B, Eq. 1-4) for bf16 planes of 64 or 128 channels and 2^17..2^23 elements: one persistent
// launch (one CTA per SM, all resident; programmatic stream serialisation).
#include "whtmix_block.cuh"
#include "whtmix_fast_launch.cuh"

namespace whtmix {
namespace blk {

template <int Q, int C>
cudaError_t launch(const Params& P, const void* w_in, const void* w_out, int sms, cudaStream_t stream) {
  const void* k = reinterpret_cast<const void*>(tri::k_block_fast<Q, C>);
  int occ = 0;
  cudaError_t e = fast::occupancy_cached(k, tri::THREADS, tri::BLK_SMEM, &occ);
  if (e != cudaSuccess) return e;
  if (occ != 1) return cudaErrorInvalidConfiguration;  // all 512 TMEM columns per CTA: one CTA per SM
  Params p = P;
  const __nv_bfloat16* wi = static_cast<const __nv_bfloat16*>(w_in);
  const __nv_bfloat16* wo = static_cast<const __nv_bfloat16*>(w_out);
  void* args[] = {&p, &wi, &wo};
  return launch_pdl(k, static_cast<unsigned>(fast::tri_grid(P.B << (P.m - tri::R), sms)), tri::THREADS, tri::BLK_SMEM, stream, args);
}

template <int C>
cudaError_t launch_c(const Params& P, const void* w_in, const void* w_out, int sms, cudaStream_t stream) {
  switch (P.m) {
    case 17: return launch<4, C>(P, w_in, w_out, sms, stream);
    case 18: return launch<5, C>(P, w_in, w_out, sms, stream);
    case 19: return launch<6, C>(P, w_in, w_out, sms, stream);
    case 20: return launch<7, C>(P, w_in, w_out, sms, stream);
    case 21: return launch<8, C>(P, w_in, w_out, sms, stream);
    case 22: return launch<9, C>(P, w_in, w_out, sms, stream);
    case 23: return launch<10, C>(P, w_in, w_out, sms, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t forward_bf16(const Params& P, const void* w_in, const void* w_out, int sms, cudaStream_t stream) {
  return P.cbits == 7 ? launch_c<128>(P, w_in, w_out, sms, stream) : launch_c<64>(P, w_in, w_out, sms, stream);
}

}  // namespace blk
}  // namespace whtmix

// Fused decode kernel instantiations: f32 caches, Hamming scores, deferred selection (steps that append a key to units whose
// blocks have few keys).
#include "decode_launch.cuh"
cudaError_t bpc_launch_decode_f32_short(bpc_ctx* ctx, const DecodeParams& p, cudaStream_t stream) {
  return bpcdev::launch_dtype<float, 0, 4>(ctx, p, stream);
}

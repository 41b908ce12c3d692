// Fused decode kernel instantiations: bf16 caches, Hamming scores, deferred selection (steps that append a key to units whose
// blocks have few keys).
#include "decode_launch.cuh"
cudaError_t bpc_launch_decode_bf16_short(bpc_ctx* ctx, const DecodeParams& p, cudaStream_t stream) {
  return bpcdev::launch_dtype<__nv_bfloat16, 0, 4>(ctx, p, stream);
}

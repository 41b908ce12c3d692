// Fused decode kernel instantiations: bf16 caches, Hamming scores, two blocks per SM (batches of unequal lengths).
#include "decode_launch.cuh"
cudaError_t bpc_launch_decode_bf16_duo(bpc_ctx* ctx, const DecodeParams& p, cudaStream_t stream) {
  return bpcdev::launch_dtype<__nv_bfloat16, 0, 5>(ctx, p, stream);
}
cudaError_t bpc_decode_limits_bf16_duo(const bpc_ctx* ctx, int nbins, int* max_cluster, int* chunk_cap, size_t* smem) {
  return bpcdev::limits_dtype<__nv_bfloat16, 0, 5>(ctx, nbins, max_cluster, chunk_cap, smem);
}

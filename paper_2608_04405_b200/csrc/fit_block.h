// Blocked fit (fit_block.cu): workspace layout and launcher.
#pragma once
#include "common.cuh"

// The blocked fit serves every configuration without power iterations (those change the directions from bit to bit), up to
// the length at which the byte sums of a block of keys in a cluster of eight stay below 2^32.
inline bool bpc_fit_blocked_covers(const bpc_config* c) { return c->fit_power_iters == 0 && c->n_max <= (1 << 27); }
// workspace behind the fitted codes (which stay at offset 0)
size_t bpc_fit_blocked_bytes(const bpc_config* c);
cudaError_t bpc_launch_fit_blocked(bpc_ctx* ctx, const void* k_cache, const float* v_star, uint32_t* hfit, unsigned char* ws,
                                   cudaStream_t stream, int* launches);

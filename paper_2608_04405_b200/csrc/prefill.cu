// Prefill-side and cache-write kernels: projection finalisation, Algorithm 1 (fit), Algorithm 2 on CUDA
// cores (fp32 caches and shapes the tensor-core encode does not cover), and the per-step append.
#include "fit_block.h"

namespace {

// --------------------------------------------------------------------------- projection finalisation
// P (float) -> P_h in the cache dtype (the hash function is defined on these rounded values),
// the same values as float, and the Gram matrix G = P_h P_h^T used by the Gram form of Algorithm 2:
// t_i = k.P_i - sum_{j<i} u_j G_ji is the decision value r.P_i of the residual form.
template <typename KV>
__global__ void round_projection_kernel(const float* __restrict__ P, KV* __restrict__ Ph, float* __restrict__ Phf, size_t n) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    KV v = (KV)P[i];
    Ph[i] = v;
    Phf[i] = to_float(v);
  }
}
template <> __global__ void round_projection_kernel<__nv_bfloat16>(const float* __restrict__ P, __nv_bfloat16* __restrict__ Ph,
                                                                   float* __restrict__ Phf, size_t n) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    __nv_bfloat16 v = __float2bfloat16_rn(P[i]);
    Ph[i] = v;
    Phf[i] = __bfloat162float(v);
  }
}

// C[i][j] = A_i . B_j for 16 x 32 tiles of row pairs, fp64 products summed in channel order; grid (tiles of A, tiles of B,
// sets).  Rows are converted to fp64 once on their way to shared memory and a thread keeps 2 x 2 sums.  fp64 issue bounds
// it: small tiles spread few sets over more SMs, and a Gram matrix (A = B, `symmetric`) leaves the tiles left of the
// diagonal to their mirror images.  (One thread per sum with a conversion per operand of each product: 266 us for the Gram
// matrices of 32 sets of 128 bits.)
constexpr int kDotThreads = 128;
constexpr int kDotChannels = 64;
__global__ void __launch_bounds__(kDotThreads)
dots_kernel(const float* A, size_t a_set, const float* B, size_t b_set, float* __restrict__ C, size_t c_set, int ldc,
            int symmetric) {
  pdl_wait();
  pdl_release();
  __shared__ double as[16][kDotChannels + 1], bs[32][kDotChannels + 1];
  const int i0 = 16 * blockIdx.x, j0 = 32 * blockIdx.y;
  if (symmetric && j0 + 31 < i0) return;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const float* a = A + blockIdx.z * a_set + (size_t)i0 * BPC_D;
  const float* b = B + blockIdx.z * b_set + (size_t)j0 * BPC_D;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int c0 = 0; c0 < BPC_D; c0 += kDotChannels) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16 * kDotChannels / kDotThreads; ++k) {
      const int e = tid + k * kDotThreads;
      as[e / kDotChannels][e % kDotChannels] = (double)a[(size_t)(e / kDotChannels) * BPC_D + c0 + e % kDotChannels];
    }
#pragma unroll
    for (int k = 0; k < 32 * kDotChannels / kDotThreads; ++k) {
      const int e = tid + k * kDotThreads;
      bs[e / kDotChannels][e % kDotChannels] = (double)b[(size_t)(e / kDotChannels) * BPC_D + c0 + e % kDotChannels];
    }
    __syncthreads();
#pragma unroll 16
    for (int c = 0; c < kDotChannels; ++c) {
      const double b0 = bs[tx][c], b1 = bs[tx + 16][c], a0 = as[ty][c], a1 = as[ty + 8][c];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
  }
  float* out = C + blockIdx.z * c_set;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + ty + 8 * (q >> 1), j = j0 + tx + 16 * (q & 1);
    out[(size_t)i * ldc + j] = (float)acc[q >> 1][q & 1];
    if (symmetric && j > i) out[(size_t)j * ldc + i] = (float)acc[q >> 1][q & 1];
  }
}

// --------------------------------------------------------------------------- Algorithm 2 on CUDA cores
// Blocks of 32 keys.  Decision values t = k P_h^T: a register-tiled product in fp64 (a thread owns 2 keys x 4 bits at a
// time, four running sums per value), kept as fp32 in shared memory.  The greedy sweep u_i = sign(t_i), t_j -= u_i G_ij
// (j > i) runs with one lane per column of a 32-bit block and four keys per warp: a decision is a shuffle, its corrections
// one FMA per 32 columns, and a block's word is one ballot at its end, because a decided column keeps its decision value.  The
// chunks of the projection are requested one ahead and the Gram matrix arrives by asynchronous copies, so that no global latency but
// the first is waited for.  Bound by the product's fp64 issue and shared-memory reads (two channels a read) and by the chain of
// decisions, with eight warps per SM to hide it.  4096 keys x 64 bits: 18.4 -> 12.3 us with those, 12.1 with the keys requested
// before anything is waited for (160 with one thread per key, its own conversions and a column-by-column sweep, which filled 32 SMs).
constexpr int kEncThreads = 256;
constexpr int kEncKeys = 32;
constexpr int kEncBits = 64;                                         // bits of a projection pass
constexpr int kEncChannels = 32;                                     // channels of P staged at a time
constexpr int kEncGramBits = 128;                                    // up to this code length the Gram matrix is kept in shared memory

template <int NB>
struct EncSmem {
  double k[kEncKeys][BPC_D + 2];                                     // (even strides: read two channels at a time)
  double p[kEncBits][kEncChannels + 2];
  float t[kEncKeys][32 * NB + 1];
};

template <typename KV, int NB>                                       // NB = code words per key
__global__ void __launch_bounds__(kEncThreads)
encode_simple_kernel(const KV* k_cache, const float* Phf, const float* gram,
                     const int32_t* unit_lens, uint64_t* __restrict__ codes, int n_kv_heads, int n_max,
                     int row_stride, int shared_sets, int residual_correction, float* __restrict__ key_err) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int b = 32 * NB;
  EncSmem<NB>& sm = *reinterpret_cast<EncSmem<NB>*>(smem);
  float* g_s = reinterpret_cast<float*>(smem + sizeof(EncSmem<NB>));     // [b][b] where it fits
  const int unit = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  pdl_release();
  const int n = min(unit_lens[unit], n_max);
  if (blockIdx.x * kEncKeys >= n) return;                            // uniform over the block
  const int set = shared_sets ? unit % n_kv_heads : unit;
  const float* Pset = Phf + (size_t)set * b * BPC_D;
  const float* Gset = gram + (size_t)set * b * b;
  // the rows of the projection one chunk ahead, in registers: chunk s holds channels 32 (s % 4) .. of bits 64 (s / 4) ..
  constexpr int JN = (b < kEncBits ? b : kEncBits) / 16;             // bits of a thread: tx, tx + 16, ...
  constexpr int kChunks = BPC_D / kEncChannels, kSteps = (b + kEncBits - 1) / kEncBits * kChunks;
  constexpr int kAhead = 16 * JN * kEncChannels / kEncThreads;
  float ahead[kAhead];
  auto fetch = [&](int s) {
#pragma unroll
    for (int m = 0; m < kAhead; ++m) {
      const int e = tid + m * kEncThreads;
      ahead[m] = Pset[(size_t)(kEncBits * (s / kChunks) + e / kEncChannels) * BPC_D + kEncChannels * (s % kChunks) + e % kEncChannels];
    }
  };
  fetch(0);
  // the keys as well, in 16-byte pieces (cache rows start on 16 bytes), but with 32 bits, where the registers cost more than the latency
  // (8 x 4K keys 35.2 us against 37.2; 4K keys of 64 bits 12.4 with, 12.7 without, 4K of 256 55.2 and 56.6)
  constexpr bool kKeysAhead = NB > 1;
  constexpr int kVec = 16 / (int)sizeof(KV), kKeysEach = kEncKeys * BPC_D / kVec / kEncThreads;
  uint4 keys[kKeysEach];
  auto fetch_keys = [&](int key0) {
#pragma unroll
    for (int m = 0; m < kKeysEach; ++m) {
      const int e = (tid + m * kEncThreads) * kVec, r = e / BPC_D, c = e % BPC_D;
      keys[m] = key0 + r < n ? *reinterpret_cast<const uint4*>(k_cache + ((size_t)unit * n_max + key0 + r) * row_stride + c) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if constexpr (kKeysAhead) fetch_keys(blockIdx.x * kEncKeys);
  if (b <= kEncGramBits && residual_correction)
    for (int i = tid; i < b * b / 4; i += kEncThreads)               // (lands during the product)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(g_s + 4 * i)), "l"(Gset + 4 * i) : "memory");
  for (int key0 = blockIdx.x * kEncKeys; key0 < n; key0 += gridDim.x * kEncKeys) {
    if (kKeysAhead && key0 != blockIdx.x * kEncKeys) fetch_keys(key0);
    __syncthreads();
    if constexpr (kKeysAhead) {
#pragma unroll
      for (int m = 0; m < kKeysEach; ++m) {
        const int e = (tid + m * kEncThreads) * kVec;
        const KV* x = reinterpret_cast<const KV*>(&keys[m]);
        double* row = &sm.k[e / BPC_D][e % BPC_D];
#pragma unroll
        for (int i = 0; i < kVec; i += 2) *reinterpret_cast<double2*>(row + i) = make_double2((double)to_float(x[i]), (double)to_float(x[i + 1]));
      }
    } else {
      for (int e = tid; e < kEncKeys * BPC_D; e += kEncThreads) {
        const int r = e / BPC_D, c = e % BPC_D;
        sm.k[r][c] = key0 + r < n ? (double)to_float(k_cache[((size_t)unit * n_max + key0 + r) * row_stride + c]) : 0.0;
      }
    }
    const int tx = tid & 15, ty = tid >> 4;
    for (int j0 = 0; j0 < b; j0 += kEncBits) {
      double acc[2][JN][4];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < JN; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[r][j][q] = 0.0;
      for (int c0 = 0; c0 < BPC_D; c0 += kEncChannels) {
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kAhead; ++m) {
          const int e = tid + m * kEncThreads;
          sm.p[e / kEncChannels][e % kEncChannels] = (double)ahead[m];
        }
        fetch((j0 / kEncBits * kChunks + c0 / kEncChannels + 1) % kSteps);   // (behind the last chunk: the next keys' first)
        __syncthreads();
#pragma unroll 2
        for (int c = 0; c < kEncChannels; c += 4) {
#pragma unroll
          for (int q = 0; q < 4; q += 2) {
            const double2 k0 = *reinterpret_cast<const double2*>(&sm.k[ty][c0 + c + q]), k1 = *reinterpret_cast<const double2*>(&sm.k[ty + 16][c0 + c + q]);
#pragma unroll
            for (int j = 0; j < JN; ++j) {
              const double2 pv = *reinterpret_cast<const double2*>(&sm.p[tx + 16 * j][c + q]);
              acc[0][j][q] = fma(k0.x, pv.x, acc[0][j][q]);
              acc[1][j][q] = fma(k1.x, pv.x, acc[1][j][q]);
              acc[0][j][q + 1] = fma(k0.y, pv.y, acc[0][j][q + 1]);
              acc[1][j][q + 1] = fma(k1.y, pv.y, acc[1][j][q + 1]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < JN; ++j) {
        sm.t[ty][j0 + tx + 16 * j] = (float)((acc[0][j][0] + acc[0][j][1]) + (acc[0][j][2] + acc[0][j][3]));
        sm.t[ty + 16][j0 + tx + 16 * j] = (float)((acc[1][j][0] + acc[1][j][1]) + (acc[1][j][2] + acc[1][j][3]));
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");                 // (the Gram matrix)
    __syncthreads();
    // sweep: keys 4 warp .. 4 warp + 3; lane = column of each 32-bit block
    float t[4][NB];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int w = 0; w < NB; ++w) t[r][w] = sm.t[4 * warp + r][32 * w + lane];
    double abs_sum[4] = {0.0, 0.0, 0.0, 0.0};                        // this lane's part of the sums of |t_i| at decision time
#pragma unroll
    for (int cb = 0; cb < NB; ++cb) {
      // (a column takes no more corrections once it is decided: after the block lane i still holds decision value i)
      if (residual_correction) {
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
          float g[NB];
#pragma unroll
          for (int w = cb; w < NB; ++w) {
            const size_t at = (size_t)(32 * cb + i) * b + 32 * w + lane;
            g[w] = b <= kEncGramBits ? g_s[at] : Gset[at];
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float nu = __shfl_sync(0xffffffffu, t[r][cb], i) >= 0.f ? -1.f : 1.f;
            if (lane > i) t[r][cb] = fmaf(nu, g[cb], t[r][cb]);
#pragma unroll
            for (int w = cb + 1; w < NB; ++w) t[r][w] = fmaf(nu, g[w], t[r][w]);
          }
        }
      }
      uint32_t word[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        word[r] = __ballot_sync(0xffffffffu, t[r][cb] >= 0.f);
        if (key_err != nullptr) abs_sum[r] += (double)fabsf(t[r][cb]);       // (this lane's columns)
      }
      if (lane < 4 && key0 + 4 * warp + lane < n) {
        const uint32_t v = lane == 0 ? word[0] : lane == 1 ? word[1] : lane == 2 ? word[2] : word[3];
        (reinterpret_cast<uint32_t*>(codes) + ((size_t)unit * n_max + key0 + 4 * warp + lane) * NB)[cb] = v;
      }
    }
    if (key_err != nullptr) {
      // squared reconstruction error (Eq. 8) from the sweep: ||k - hP||^2 = ||k||^2 - 2 sum|t_i| + trace(G)
      double trg = 0.0;
      for (int i = lane; i < b; i += 32) trg += (double)Gset[(size_t)i * b + i];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        double v = trg - 2.0 * abs_sum[r];
        for (int c = lane; c < BPC_D; c += 32) v = fma(sm.k[4 * warp + r][c], sm.k[4 * warp + r][c], v);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && key0 + 4 * warp + r < n)
          key_err[(size_t)unit * n_max + key0 + 4 * warp + r] = (float)fmax(0.0, v);
      }
    }
  }
}

// --------------------------------------------------------------------------- append (cache write + Algorithm 2 on one key)
// One block per unit.  The decision values come from a warp-cooperative fp32 mat-vec; the greedy sweep is
// split in 32-bit column blocks: warp B owns columns 32B..32B+31, sweeps its diagonal block with register
// shuffles, publishes its 32 signs, and the later warps apply that rank-32 update.
constexpr int kAppThreads = 256;

template <typename KV>
__global__ void __launch_bounds__(kAppThreads)
append_kernel(const KV* k_new, const KV* v_new, KV* __restrict__ k_cache, KV* __restrict__ v_cache,
              uint64_t* __restrict__ codes, const KV* Ph, const float* gram,
              int32_t* __restrict__ unit_lens, int32_t* __restrict__ err, int n_kv_heads, int n_max, int row_stride,
              int b, int shared_sets, int residual_correction) {
  pdl_wait();
  pdl_release();
  extern __shared__ __align__(16) unsigned char smem[];
  // the 32 x 32 blocks of the Gram matrix on and to the right of the diagonal (the only ones the sweep reads), block
  // (r, c) at slot r * nb - r (r - 1) / 2 + (c - r): 144 KB at 256 bits
  float* gs = reinterpret_cast<float*>(smem);
  __shared__ float t_s[256];
  __shared__ float k_s[BPC_D];
  __shared__ uint32_t ubits_s[8];
  const int unit = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = unit_lens[unit];
  if (n >= n_max || n < 0) {
    if (tid == 0) atomicOr(err, BPC_DEVERR_APPEND_CAP);
    return;
  }
  const int set = shared_sets ? unit % n_kv_heads : unit;
  const float* Gset = gram + (size_t)set * b * b;
  const int nb = b / 32;
  if (residual_correction) {
    float4* dst = reinterpret_cast<float4*>(gs);
    int slot = 0;
    for (int r = 0; r < nb; ++r) {
      for (int c = r; c < nb; ++c, ++slot) {                         // one block per pass of the 256 threads: row tid / 8, four columns
        const int i = tid >> 3, l4 = tid & 7;
        dst[slot * 256 + tid] = *reinterpret_cast<const float4*>(Gset + (size_t)(32 * r + i) * b + 32 * c + 4 * l4);
      }
    }
  }
  const KV* kn = k_new + (size_t)unit * BPC_D;
  const KV* vn = v_new + (size_t)unit * BPC_D;
  if (tid < BPC_D) {
    const KV kv = kn[tid];
    k_s[tid] = to_float(kv);
    k_cache[((size_t)unit * n_max + n) * row_stride + tid] = kv;
  } else if (tid < 2 * BPC_D) {
    v_cache[((size_t)unit * n_max + n) * row_stride + (tid - BPC_D)] = vn[tid - BPC_D];
  }
  __syncthreads();
  // t_j = P_h[j] . k
  {
    const KV* Pset = Ph + (size_t)set * b * BPC_D;
    const float k0 = k_s[4 * lane], k1 = k_s[4 * lane + 1], k2 = k_s[4 * lane + 2], k3 = k_s[4 * lane + 3];
#pragma unroll 4
    for (int j = warp; j < b; j += kAppThreads / 32) {
      const KV* row = Pset + (size_t)j * BPC_D + 4 * lane;
      float s = to_float(row[0]) * k0;
      s = fmaf(to_float(row[1]), k1, s);
      s = fmaf(to_float(row[2]), k2, s);
      s = fmaf(to_float(row[3]), k3, s);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) t_s[j] = s;
    }
  }
  __syncthreads();
  auto gblock = [&](int r, int c) { return gs + (size_t)(r * nb - r * (r - 1) / 2 + (c - r)) * 1024; };
  float t = warp < nb ? t_s[32 * warp + lane] : 0.f;
  float gd[32];                                                      // diagonal block column of this lane
  if (warp < nb && residual_correction) {
    const float* gb = gblock(warp, warp);
#pragma unroll
    for (int i = 0; i < 32; ++i) gd[i] = gb[32 * i + lane];
  }
  for (int blk = 0; blk < nb; ++blk) {
    if (warp == blk) {
      uint32_t bits = 0;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float ti = __shfl_sync(0xffffffffu, t, i);
        const bool pos = ti >= 0.f;
        bits |= (pos ? 1u : 0u) << i;
        if (residual_correction && lane > i) t -= pos ? gd[i] : -gd[i];
      }
      if (lane == 0) {
        ubits_s[blk] = bits;
        (reinterpret_cast<uint32_t*>(codes) + ((size_t)unit * n_max + n) * (b / 32))[blk] = bits;
      }
    }
    __syncthreads();
    if (residual_correction && warp > blk && warp < nb) {
      const uint32_t bits = ubits_s[blk];
      const float* gcol = gblock(blk, warp) + lane;
      float a = 0.f;
#pragma unroll 8
      for (int i = 0; i < 32; ++i) {
        const float g = gcol[32 * i];
        a += ((bits >> i) & 1u) ? g : -g;
      }
      t -= a;
    }
  }
  if (tid == 0) unit_lens[unit] = n + 1;
}

// --------------------------------------------------------------------------- Algorithm 1 (fit)
// The residual is never stored.  With the signs u_j of the earlier bits kept as packed code words (the codes H that
// Algorithm 1 itself produces) and P_j = v_j, a row's residual is R_row = K_row - sum_j u_j v_j, hence
//   t = R_row . d        = K_row . d - sum_{j<i} u_j (v_j . d)          (d = the direction of bit i)
//   u_i R = u_i K - sum_{j<i} (u_i . u_j) v_j                            (u_i . u_j = 2 * agreements - N, an integer)
// Iteration i therefore reads the key row and its code words (272 bytes per row instead of 1 KB of fp32 residual read and
// written back), writes one bit, and leaves per block a partial sum of +-K rows and the per-bit agreement counts; a
// small kernel before the pass prepares d and the b inner products v_j . d, a small one after it forms v_i.
constexpr int kFitThreads = 256;
constexpr int kFitRowsPerBlock = 1024;

// before the pass of bit `it`: dir[unit] = direction (the caller's draw, unless the power-iteration kernel already
// wrote one), dots[unit][j] = v_j . dir for j < it and 0 for the other bits
__global__ void __launch_bounds__(BPC_D)
fit_prep_kernel(const float* __restrict__ P, const float* __restrict__ v_star, float* __restrict__ dir, float* __restrict__ dots,
                int b, int it, int have_dir) {
  const int unit = blockIdx.x, tid = threadIdx.x;
  __shared__ float d_s[BPC_D];
  float dv = have_dir ? dir[(size_t)unit * BPC_D + tid] : v_star[((size_t)unit * b + it) * BPC_D + tid];
  d_s[tid] = dv;
  if (!have_dir) dir[(size_t)unit * BPC_D + tid] = dv;
  __syncthreads();
  for (int j = tid; j < b; j += BPC_D) {
    double acc = 0.0;
    if (j < it) {
      const float* pj = P + ((size_t)unit * b + j) * BPC_D;
      for (int c = 0; c < BPC_D; ++c) acc += (double)pj[c] * (double)d_s[c];
    }
    dots[(size_t)unit * b + j] = (float)acc;
  }
}

// Eight lanes share a row (16 channels and b/8 earlier bits each), so a warp works on four rows at once.
template <typename KV, int JPL>          // JPL = b / 8 bits per lane
__global__ void __launch_bounds__(kFitThreads, 4)   // latency-bound: four blocks (32 warps) per SM
fit_pass_kernel(const KV* __restrict__ k_cache, uint32_t* __restrict__ hfit, const float* __restrict__ dir,
                const float* __restrict__ dots, float* __restrict__ partials, int32_t* __restrict__ agree,
                const int32_t* __restrict__ unit_lens, int n_max, int row_stride, int it, int blocks_per_unit) {
  constexpr int b = JPL * 8, WORDS = b / 32;
  constexpr int CPLN = 16;                                    // channels per lane
  const int unit = blockIdx.y;
  const int n = min(unit_lens[unit], n_max);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane & 7, grp = lane >> 3;                  // lane within the row's group, row within the warp's four
  const int row0 = blockIdx.x * kFitRowsPerBlock;
  float dv[CPLN];
#pragma unroll
  for (int c = 0; c < CPLN; ++c) dv[c] = dir[(size_t)unit * BPC_D + sub * CPLN + c];
  // sum_j u_j (v_j . d) over a lane's bits is looked up four bits at a time: lut[sub][nibble][pattern] = sum over the
  // nibble's bits of +-(v_j . d) (the inner products of bits >= it are zero, so later bits add nothing)
  constexpr int NIB = JPL / 4;
  __shared__ float lut[8][NIB][16];
  for (int e = tid; e < 8 * NIB * 16; e += kFitThreads) {
    const int m = e & 15, nb = (e >> 4) % NIB, sb = e / (16 * NIB);
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float d = dots[(size_t)unit * b + sb * JPL + 4 * nb + q];
      v += ((m >> q) & 1) ? d : -d;
    }
    lut[sb][nb][m] = v;
  }
  __syncthreads();
  const int my_word = (sub * JPL) >> 5, my_shift = (sub * JPL) & 31;
  float acc[CPLN];
#pragma unroll
  for (int c = 0; c < CPLN; ++c) acc[c] = 0.f;
  // agreements with the earlier bits are counted in six bit-sliced counter planes (at most 32 rows per lane group)
  uint32_t pl[6] = {0u, 0u, 0u, 0u, 0u, 0u};
  const int row_end = min(n, row0 + kFitRowsPerBlock);
  constexpr int ROWS_PER_ITER = (kFitThreads / 32) * 4;
  // Rows reach the lanes through a small ring in shared memory filled by asynchronous copies, NSTG - 1 row sets ahead
  // (the pass is bound by memory latency).  Every lane copies and later reads only its own 16-byte pieces, so the ring
  // needs no barrier.
  constexpr int NV = CPLN * (int)sizeof(KV) / 16;            // 16-byte vectors per lane and row
  constexpr int NSTG = sizeof(KV) == 2 ? 4 : 2;
  __shared__ uint4 ring[NSTG][kFitThreads][NV];
  __shared__ uint32_t ringw[NSTG][kFitThreads];
  auto issue = [&](int slot, int rb) {
    const int r = rb + warp * 4 + grp;
    if (r < row_end) {
      const uint4* kr = reinterpret_cast<const uint4*>(k_cache + ((size_t)unit * n_max + r) * row_stride + sub * CPLN);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(&ring[slot][tid][v]);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(kr + v) : "memory");
      }
      if (it > 0) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(&ringw[slot][tid]);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(hfit + ((size_t)unit * n_max + r) * WORDS + my_word) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s0 = 0; s0 < NSTG - 1; ++s0) issue(s0, row0 + s0 * ROWS_PER_ITER);
  int slot = 0;
  for (int rb = row0; rb < row_end; rb += ROWS_PER_ITER) {   // uniform trip count: the shuffles below need whole warps
    issue(slot == 0 ? NSTG - 1 : slot - 1, rb + (NSTG - 1) * ROWS_PER_ITER);
    asm volatile("cp.async.wait_group %0;" ::"n"(NSTG - 1) : "memory");
    const int r = rb + warp * 4 + grp;
    const bool live = r < row_end;
    float x[CPLN];
    if (sizeof(KV) == 2) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint4 q = ring[slot][tid][v];
        const uint32_t ww[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) { x[8 * v + 2 * c] = __uint_as_float(ww[c] << 16); x[8 * v + 2 * c + 1] = __uint_as_float(ww[c] & 0xffff0000u); }
      }
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint4 q = ring[slot][tid][v];
        x[4 * v] = __uint_as_float(q.x); x[4 * v + 1] = __uint_as_float(q.y); x[4 * v + 2] = __uint_as_float(q.z); x[4 * v + 3] = __uint_as_float(q.w);
      }
    }
    if (!live) {                                             // nothing was copied for this lane: keep the arithmetic finite
#pragma unroll
      for (int c = 0; c < CPLN; ++c) x[c] = 0.f;
    }
    const uint32_t mine = (it > 0 && live) ? (ringw[slot][tid] >> my_shift) : 0u;       // this lane's JPL earlier bits
    slot = slot + 1 == NSTG ? 0 : slot + 1;
    float tk = 0.f;
#pragma unroll
    for (int c = 0; c < CPLN; ++c) tk = fmaf(x[c], dv[c], tk);
    float tc = 0.f;
#pragma unroll
    for (int nb = 0; nb < NIB; ++nb) tc += lut[sub][nb][(mine >> (4 * nb)) & 15u];
    double t = (double)tk - (double)tc;
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    const bool pos = t >= 0.0;
    if (live) {
      if (sub == 0) {
        uint32_t* w = hfit + ((size_t)unit * n_max + r) * WORDS + (it >> 5);
        const uint32_t prev = (it & 31) ? *w : 0u;
        *w = prev | ((pos ? 1u : 0u) << (it & 31));
      }
      const float sg = pos ? 1.f : -1.f;
#pragma unroll
      for (int c = 0; c < CPLN; ++c) acc[c] = fmaf(sg, x[c], acc[c]);
      uint32_t carry = pos ? mine : ~mine;                                              // bit e: u_j agrees with u_i
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const uint32_t nc = pl[k] & carry;
        pl[k] ^= carry;
        carry = nc;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();                                           // the ring is free: it now holds the block's partial sums
  float (*red)[BPC_D] = reinterpret_cast<float (*)[BPC_D]>(&ring[0][0][0]);
  int32_t (*redc)[b] = reinterpret_cast<int32_t (*)[b]>(reinterpret_cast<unsigned char*>(&ring[0][0][0]) + (kFitThreads / 32) * BPC_D * 4);
  // the four row groups of a warp hold partial sums for the same channels and bits
#pragma unroll
  for (int c = 0; c < CPLN; ++c) {
    acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 8);
    acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 16);
  }
  int cnt[JPL];
#pragma unroll
  for (int e = 0; e < JPL; ++e) {
    int c = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) c += (int)((pl[k] >> e) & 1u) << k;
    c += __shfl_xor_sync(0xffffffffu, c, 8);
    c += __shfl_xor_sync(0xffffffffu, c, 16);
    cnt[e] = c;
  }
  if (grp == 0) {
#pragma unroll
    for (int c = 0; c < CPLN; ++c) red[warp][sub * CPLN + c] = acc[c];
#pragma unroll
    for (int e = 0; e < JPL; ++e) redc[warp][sub * JPL + e] = cnt[e];
  }
  __syncthreads();
  if (tid < BPC_D) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kFitThreads / 32; ++w) s += red[w][tid];
    partials[((size_t)unit * blocks_per_unit + blockIdx.x) * BPC_D + tid] = s;
  }
  for (int j = tid; j < b; j += kFitThreads) {
    int c = 0;
#pragma unroll
    for (int w = 0; w < kFitThreads / 32; ++w) c += redc[w][j];
    agree[((size_t)unit * blocks_per_unit + blockIdx.x) * b + j] = c;
  }
}

// v_i = (sum of the blocks' +-K partial sums - sum_{j<i} (2 * agreements_j - N) v_j) / N.  Four thread groups split
// the blocks and the earlier bits; every sum is formed in a fixed order (group partials added 0..3).
constexpr int kRedGroups = 4;
__global__ void __launch_bounds__(BPC_D * kRedGroups)
fit_reduce_kernel(const float* __restrict__ partials, const int32_t* __restrict__ agree, float* __restrict__ P,
                  const int32_t* __restrict__ unit_lens, int n_max, int b, int it, int blocks_per_unit, int rows_per_block) {
  const int unit = blockIdx.x, c = threadIdx.x & (BPC_D - 1), q = threadIdx.x / BPC_D;
  const int n = min(unit_lens[unit], n_max);
  const int nblk = (n + rows_per_block - 1) / rows_per_block;
  __shared__ double corr[256];                               // u_i . u_j for j < it
  __shared__ double part[kRedGroups][BPC_D];
  __shared__ int agp[kRedGroups][256];
  // agreement counts: group q adds the blocks k = q, q + 4, ... (eight loads in flight per thread), then the groups are added
  for (int j = c; j < it; j += BPC_D) {
    int a8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int k = q;
    for (; k + 7 * kRedGroups < nblk; k += 8 * kRedGroups) {
#pragma unroll
      for (int e = 0; e < 8; ++e) a8[e] += agree[((size_t)unit * blocks_per_unit + k + e * kRedGroups) * b + j];
    }
    for (; k < nblk; k += kRedGroups) a8[0] += agree[((size_t)unit * blocks_per_unit + k) * b + j];
    agp[q][j] = ((a8[0] + a8[1]) + (a8[2] + a8[3])) + ((a8[4] + a8[5]) + (a8[6] + a8[7]));
  }
  __syncthreads();
  for (int j = threadIdx.x; j < it; j += BPC_D * kRedGroups) {
    const long long a = (long long)agp[0][j] + agp[1][j] + agp[2][j] + agp[3][j];
    corr[j] = (double)(2 * a - (long long)n);
  }
  __syncthreads();
  double s = 0.0;
  {
    double s8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int k = q;
    for (; k + 7 * kRedGroups < nblk; k += 8 * kRedGroups) {
#pragma unroll
      for (int e = 0; e < 8; ++e) s8[e] += (double)partials[((size_t)unit * blocks_per_unit + k + e * kRedGroups) * BPC_D + c];
    }
    for (; k < nblk; k += kRedGroups) s8[0] += (double)partials[((size_t)unit * blocks_per_unit + k) * BPC_D + c];
    s = ((s8[0] + s8[1]) + (s8[2] + s8[3])) + ((s8[4] + s8[5]) + (s8[6] + s8[7]));
  }
  {
    double t8[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int j = q;
    for (; j + 7 * kRedGroups < it; j += 8 * kRedGroups) {
#pragma unroll
      for (int e = 0; e < 8; ++e) t8[e] += corr[j + e * kRedGroups] * (double)P[((size_t)unit * b + j + e * kRedGroups) * BPC_D + c];
    }
    for (; j < it; j += kRedGroups) t8[0] += corr[j] * (double)P[((size_t)unit * b + j) * BPC_D + c];
    s -= ((t8[0] + t8[1]) + (t8[2] + t8[3])) + ((t8[4] + t8[5]) + (t8[6] + t8[7]));
  }
  part[q][c] = s;
  __syncthreads();
  if (q == 0) {
    double t = 0.0;
#pragma unroll
    for (int g = 0; g < kRedGroups; ++g) t += part[g][c];
    P[((size_t)unit * b + it) * BPC_D + c] = n > 0 ? (float)(t / (double)n) : 0.f;
  }
}

// --------------------------------------------------------------------------- power-iteration fit
// u = sign((R R^T)^n R v*^T) = sign(R z) with z = (R^T R)^n v*^T.  C = R^T R (D x D, fp64) is formed once from the keys
// and then follows the residual through C <- C - N v^T v (u R = N v and u u^T = N make the cross terms collapse), so
// a power-iteration fit costs one extra pass over the keys and a D x D product per bit.
constexpr int kGramRows = 8192;          // key rows per block of the initial Gram pass

// One block per (row slab, unit): its 256 threads own 8 x 8 tiles of the D x D partial sum.  Rows are staged 32 at a
// time in shared memory; a tile of 32 rows is summed in fp32 and added to fp64 accumulators.
template <typename KV>
__global__ void __launch_bounds__(256, 1)
fit_gram0_kernel(const KV* __restrict__ k_cache, double* __restrict__ cpart, const int32_t* __restrict__ unit_lens,
                 int n_max, int row_stride, int slabs_per_unit) {
  const int unit = blockIdx.y, tid = threadIdx.x;
  const int n = min(unit_lens[unit], n_max);
  const int row0 = blockIdx.x * kGramRows, row_end = min(n, row0 + kGramRows);
  __shared__ float tile[32][BPC_D + 4];
  const int i0 = (tid >> 4) * 8, j0 = (tid & 15) * 8;
  double acc[8][8];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[a][c] = 0.0;
  for (int r0 = row0; r0 < row_end; r0 += 32) {
    __syncthreads();
    for (int e = tid; e < 32 * BPC_D; e += 256) {
      const int r = e >> 7, c = e & 127;
      tile[r][c] = (r0 + r < row_end) ? to_float(k_cache[((size_t)unit * n_max + r0 + r) * row_stride + c]) : 0.f;
    }
    __syncthreads();
    float part[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int c = 0; c < 8; ++c) part[a][c] = 0.f;
#pragma unroll 4
    for (int r = 0; r < 32; ++r) {
      float xa[8], xb[8];
#pragma unroll
      for (int a = 0; a < 8; ++a) { xa[a] = tile[r][i0 + a]; xb[a] = tile[r][j0 + a]; }
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 8; ++c) part[a][c] = fmaf(xa[a], xb[c], part[a][c]);
    }
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[a][c] += (double)part[a][c];
  }
  double* dst = cpart + ((size_t)unit * slabs_per_unit + blockIdx.x) * BPC_D * BPC_D;
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < 8; ++c) dst[(size_t)(i0 + a) * BPC_D + j0 + c] = acc[a][c];
}

// C[unit] = sum of the slabs' partial sums, in slab order
__global__ void fit_gram0_reduce_kernel(const double* __restrict__ cpart, double* __restrict__ C,
                                        const int32_t* __restrict__ unit_lens, int n_max, int slabs_per_unit) {
  const int unit = blockIdx.y, e = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = min(unit_lens[unit], n_max);
  const int nslab = (n + kGramRows - 1) / kGramRows;
  double s = 0.0;
  for (int k = 0; k < nslab; ++k) s += cpart[((size_t)unit * slabs_per_unit + k) * BPC_D * BPC_D + e];
  C[(size_t)unit * BPC_D * BPC_D + e] = s;
}

// One block of D threads per unit, before the pass of bit `it`: apply the previous bit's downdate C -= N v v^T (v = row
// it-1 of P), then z = C^n v*_it with a rescale between the products, written as the pass's direction (fp32).
__global__ void __launch_bounds__(BPC_D)
fit_direction_kernel(double* __restrict__ C, const float* __restrict__ P, const float* __restrict__ v_star,
                     float* __restrict__ dir, const int32_t* __restrict__ unit_lens, int n_max, int b, int it, int power_iters) {
  const int unit = blockIdx.x, j = threadIdx.x;
  const int n = min(unit_lens[unit], n_max);
  double* Cu = C + (size_t)unit * BPC_D * BPC_D;
  __shared__ double z[BPC_D];
  __shared__ double red[BPC_D / 32];
  __shared__ float vprev[BPC_D];
  if (it > 0) {
    vprev[j] = P[((size_t)unit * b + (it - 1)) * BPC_D + j];
    __syncthreads();
    const double nv = (double)n * (double)vprev[j];
    for (int c = 0; c < BPC_D; ++c) Cu[(size_t)c * BPC_D + j] -= nv * (double)vprev[c];   // column j (C is symmetric)
  }
  z[j] = (double)v_star[((size_t)unit * b + it) * BPC_D + j];
  __syncthreads();
  for (int k = 0; k < power_iters; ++k) {
    double s = 0.0;
    for (int c = 0; c < BPC_D; ++c) s += Cu[(size_t)c * BPC_D + j] * z[c];                // (C z)_j, reading column j
    double q = s * s;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    __syncthreads();                                        // everyone has read z
    if ((j & 31) == 0) red[j >> 5] = q;
    __syncthreads();
    double nrm = 0.0;
#pragma unroll
    for (int w = 0; w < BPC_D / 32; ++w) nrm += red[w];
    nrm = sqrt(nrm);
    z[j] = nrm > 0.0 ? s / nrm : s;
    __syncthreads();
  }
  dir[(size_t)unit * BPC_D + j] = (float)z[j];
}

// --------------------------------------------------------------------------- error-aware safeguard set
// One block per unit: the m keys with the largest squared reconstruction error, ties to the lowest index, written
// in ascending index order.  The errors are non-negative floats, so their bit patterns order like unsigned
// integers: a 4-pass radix select (8 bits per pass) finds the m-th largest pattern, then one ordered pass compacts.
constexpr int kEasThreads = 1024;

__global__ void __launch_bounds__(kEasThreads)
build_eas_kernel(const float* __restrict__ key_err, const int32_t* __restrict__ unit_lens, int32_t* __restrict__ eas_idx,
                 int32_t* __restrict__ eas_cnt, int n_max, int eas_ppm, int eas_cap) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t wsum[kEasThreads / 32];
  __shared__ uint32_t s_prefix, s_need, s_run_gt, s_run_eq;
  const int unit = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = min(unit_lens[unit], n_max);
  int m = (int)(((long long)n * eas_ppm + 999999) / 1000000);
  m = min(min(m, n), eas_cap);
  const uint32_t* e = reinterpret_cast<const uint32_t*>(key_err + (size_t)unit * n_max);
  if (m <= 0) { if (tid == 0) eas_cnt[unit] = 0; return; }
  if (tid == 0) { s_prefix = 0u; s_need = (uint32_t)m; }
  __syncthreads();
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0u;
    __syncthreads();
    const uint32_t prefix = s_prefix, himask = shift == 24 ? 0u : ~((1u << (shift + 8)) - 1u);
    for (int i = tid; i < n; i += kEasThreads) {
      const uint32_t v = e[i];
      if ((v & himask) == prefix) atomicAdd(&hist[(v >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid == 0) {                                          // 256 bins: a serial walk from the top is cheap enough
      uint32_t need = s_need, acc = 0;
      int d = 255;
      for (; d > 0; --d) { if (acc + hist[d] >= need) break; acc += hist[d]; }
      s_need = need - acc;                                   // still to take among values with this digit
      s_prefix = prefix | ((uint32_t)d << shift);
    }
    __syncthreads();
  }
  const uint32_t thr = s_prefix, need_eq = s_need;           // take every v > thr and the first need_eq with v == thr
  if (tid == 0) { s_run_gt = 0u; s_run_eq = 0u; }
  __syncthreads();
  int32_t* out = eas_idx + (size_t)unit * eas_cap;
  for (int i0 = 0; i0 < n; i0 += kEasThreads) {
    const int i = i0 + tid;
    const uint32_t v = i < n ? e[i] : 0u;
    const bool gt = i < n && v > thr, eq = i < n && v == thr;
    const uint32_t bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
    if (lane == 0) wsum[warp] = (uint32_t)__popc(bg) | ((uint32_t)__popc(be) << 16);
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int w = 0; w < kEasThreads / 32; ++w) { if (w < warp) before += wsum[w]; total += wsum[w]; }
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t gt_before = s_run_gt + (before & 0xffffu) + (uint32_t)__popc(bg & lt);
    const uint32_t eq_before = s_run_eq + (before >> 16) + (uint32_t)__popc(be & lt);
    if (gt || (eq && eq_before < need_eq)) out[gt_before + min(eq_before, need_eq)] = i;
    __syncthreads();
    if (tid == 0) { s_run_gt += total & 0xffffu; s_run_eq += total >> 16; }
    __syncthreads();
  }
  if (tid == 0) eas_cnt[unit] = m;
}

}  // namespace

// =========================================================================== host launchers
cudaError_t bpc_launch_dots(const float* A, size_t a_set, const float* B, size_t b_set, float* C, size_t c_set, int ldc, int tiles_a, int tiles_b,
                            int sets, bool early, cudaStream_t stream) {
  return launch_pdl(early, dots_kernel, dim3(2 * tiles_a, tiles_b, sets), kDotThreads, 0, stream, A, a_set, B, b_set, C, c_set, ldc, A == B);
}

cudaError_t bpc_launch_finalize_projection(bpc_ctx* ctx, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  const size_t n = (size_t)c.hash_sets * c.code_bits * BPC_D;
  const int th = 256;
  const unsigned blocks = (unsigned)((n + th - 1) / th);
  const cudaError_t e = c.kv_dtype == BPC_BF16
      ? launch_pdl(false, round_projection_kernel<__nv_bfloat16>, blocks, th, 0, stream, ctx->P, (__nv_bfloat16*)ctx->P_h, ctx->P_hf, n)
      : launch_pdl(false, round_projection_kernel<float>, blocks, th, 0, stream, ctx->P, (float*)ctx->P_h, ctx->P_hf, n);
  if (e != cudaSuccess) return e;
  ctx->launches += 2;
  const size_t set = (size_t)c.code_bits * BPC_D;
  return bpc_launch_dots(ctx->P_hf, set, ctx->P_hf, set, ctx->gram, (size_t)c.code_bits * c.code_bits, c.code_bits, c.code_bits / 32,
                         c.code_bits / 32, c.hash_sets, ctx->use_pdl, stream);
}

template <typename KV, int NB>
static cudaError_t launch_encode_simple(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  constexpr int b = 32 * NB;
  const size_t smem = sizeof(EncSmem<NB>) + (b <= kEncGramBits ? (size_t)b * b * 4 : 0);
  cudaError_t e = cudaFuncSetAttribute(encode_simple_kernel<KV, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // a block per 32 keys up to about eight per SM over all units; longer units loop (the Gram matrix is staged once per block)
  int blocks = (c.n_max + kEncKeys - 1) / kEncKeys;
  const int most = (8 * ctx->sm_count + ctx->units - 1) / ctx->units;
  if (blocks > most) blocks = most;
  e = launch_pdl(ctx->use_pdl, encode_simple_kernel<KV, NB>, dim3(blocks, ctx->units), kEncThreads, smem, stream,
      (const KV*)k_cache, ctx->P_hf, ctx->gram, ctx->unit_lens, codes, c.n_kv_heads, c.n_max, ctx->row_stride, c.hash_sets != ctx->units,
      c.residual_correction, ctx->key_err);
  ctx->launches += 1;
  return e;
}

template <typename KV>
static cudaError_t launch_encode_simple_bits(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  switch (ctx->cfg.code_bits) {
    case 32: return launch_encode_simple<KV, 1>(ctx, k_cache, codes, stream);
    case 64: return launch_encode_simple<KV, 2>(ctx, k_cache, codes, stream);
    case 128: return launch_encode_simple<KV, 4>(ctx, k_cache, codes, stream);
    default: return launch_encode_simple<KV, 8>(ctx, k_cache, codes, stream);
  }
}

cudaError_t bpc_launch_encode_simple(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  return ctx->cfg.kv_dtype == BPC_BF16 ? launch_encode_simple_bits<__nv_bfloat16>(ctx, k_cache, codes, stream)
                                       : launch_encode_simple_bits<float>(ctx, k_cache, codes, stream);
}

cudaError_t bpc_launch_append(bpc_ctx* ctx, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                              uint64_t* codes, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  const int b = c.code_bits;
  const size_t smem = (size_t)(b / 32) * (b / 32 + 1) / 2 * 4096;   // Gram blocks on and right of the diagonal
  const int smem_limit = 8 * 9 / 2 * 4096;                 // (for every code length: the limit is shared by all threads' contexts)
  const int shared_sets = c.hash_sets != ctx->units;
  cudaError_t e;
  if (c.kv_dtype == BPC_BF16) {
    e = cudaFuncSetAttribute(append_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    if (e != cudaSuccess) return e;
    e = launch_pdl(ctx->use_pdl, append_kernel<__nv_bfloat16>, ctx->units, kAppThreads, smem, stream,
        (const __nv_bfloat16*)k_new, (const __nv_bfloat16*)v_new, (__nv_bfloat16*)k_cache, (__nv_bfloat16*)v_cache, codes,
        (const __nv_bfloat16*)ctx->P_h, ctx->gram, ctx->unit_lens, ctx->dev_err, c.n_kv_heads, c.n_max, ctx->row_stride, b, shared_sets,
        c.residual_correction);
  } else {
    e = cudaFuncSetAttribute(append_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    if (e != cudaSuccess) return e;
    e = launch_pdl(ctx->use_pdl, append_kernel<float>, ctx->units, kAppThreads, smem, stream,
        (const float*)k_new, (const float*)v_new, (float*)k_cache, (float*)v_cache, codes, (const float*)ctx->P_h,
        ctx->gram, ctx->unit_lens, ctx->dev_err, c.n_kv_heads, c.n_max, ctx->row_stride, b, shared_sets,
        c.residual_correction);
  }
  ctx->launches += 1;
  return e;
}

static inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// extra workspace of the power-iteration fit, placed after the fitted codes: C, the slabs' partial sums, the directions
static size_t fit_power_bytes(const bpc_config* c) {
  if (c->fit_power_iters <= 0) return 0;
  const size_t units = (size_t)c->batch * c->n_kv_heads;
  const size_t slabs = ((size_t)c->n_max + kGramRows - 1) / kGramRows;
  return align256(units * BPC_D * BPC_D * 8) + align256(units * slabs * BPC_D * BPC_D * 8) + align256(units * BPC_D * 4);
}

// workspace layout: fitted codes H | per-block partial sums | per-block agreement counts | direction | inner products
// | (power-iteration fit) C, its slab partial sums
static size_t fit_off_partials(const bpc_config* c) {
  const size_t units = (size_t)c->batch * c->n_kv_heads;
  return align256(units * c->n_max * (c->code_bits / 8));
}
static size_t fit_off_agree(const bpc_config* c) {
  const size_t units = (size_t)c->batch * c->n_kv_heads;
  const size_t bpu = ((size_t)c->n_max + kFitRowsPerBlock - 1) / kFitRowsPerBlock;
  return fit_off_partials(c) + align256(units * bpu * BPC_D * 4);
}
static size_t fit_off_dir(const bpc_config* c) {
  const size_t units = (size_t)c->batch * c->n_kv_heads;
  const size_t bpu = ((size_t)c->n_max + kFitRowsPerBlock - 1) / kFitRowsPerBlock;
  return fit_off_agree(c) + align256(units * bpu * c->code_bits * 4);
}
static size_t fit_off_power(const bpc_config* c) {
  const size_t units = (size_t)c->batch * c->n_kv_heads;
  return fit_off_dir(c) + align256(units * BPC_D * 4) + align256(units * c->code_bits * 4);
}

size_t bpc_fit_workspace_min_bytes_impl(const bpc_config* c) { return fit_off_power(c) + fit_power_bytes(c); }

size_t bpc_fit_workspace_bytes_impl(const bpc_config* c) {
  const size_t passes = bpc_fit_workspace_min_bytes_impl(c);
  if (!bpc_fit_blocked_covers(c)) return passes;
  const size_t blocked = fit_off_partials(c) + bpc_fit_blocked_bytes(c);   // (either path: the diagnostic switch changes it per call)
  return blocked > passes ? blocked : passes;
}

size_t bpc_fit_codes_offset_impl(const bpc_config* c) { (void)c; return 0; }

cudaError_t bpc_launch_fit(bpc_ctx* ctx, const void* k_cache, const float* v_star, void* workspace, size_t workspace_bytes,
                           cudaStream_t stream, int* launches) {
  const bpc_config& c = ctx->cfg;
  // without power iterations the fit runs in blocks of 32 bits where the workspace has room for their columns (132 B per key:
  // 0.55 of 0.64 GB at 32 x 128K keys); one pass over the keys per bit otherwise
  if (bpc_fit_blocked_covers(&c) && !ctx->no_tc_encode && workspace_bytes >= bpc_fit_workspace_bytes_impl(&c)) {
    const cudaError_t e =
        bpc_launch_fit_blocked(ctx, k_cache, v_star, (uint32_t*)workspace, (unsigned char*)workspace + fit_off_partials(&c), stream, launches);
    if (e != cudaErrorNotSupported) return e;
  }
  const size_t units = (size_t)ctx->units;
  int bpu = (c.n_max + kFitRowsPerBlock - 1) / kFitRowsPerBlock;
  int rows_per_block = kFitRowsPerBlock;
  // bf16 caches: the pass runs on the tensor cores, with longer row ranges per block (never
  // more blocks than the workspace was sized for)
  const bool tc_pass = bpc_fit_tc_covers(ctx);
  if (tc_pass) bpc_fit_tc_geometry(ctx, &bpu, &rows_per_block);
  unsigned char* ws = (unsigned char*)workspace;
  uint32_t* hfit = (uint32_t*)ws;
  float* partials = (float*)(ws + fit_off_partials(&c));
  int32_t* agree = (int32_t*)(ws + fit_off_agree(&c));
  float* dir = (float*)(ws + fit_off_dir(&c));
  float* dots = (float*)(ws + fit_off_dir(&c) + align256(units * BPC_D * 4));
  const dim3 grid(bpu, ctx->units);
  if (tc_pass) {
    // the tensor-core pass ORs each new bit into its code word and reads the earlier bits back: the words must not
    // carry anything an earlier fit left in the workspace (masking them in the pass instead was measured: 15 % slower)
    cudaError_t e = cudaMemsetAsync(hfit, 0, units * (size_t)c.n_max * (size_t)(c.code_bits / 8), stream);
    if (e != cudaSuccess) return e;
  }
  const int npow = c.fit_power_iters;
  double* Cm = nullptr;
  if (npow > 0) {
    const int slabs = (c.n_max + kGramRows - 1) / kGramRows;
    unsigned char* pw = ws + fit_off_power(&c);
    Cm = (double*)pw;
    double* cpart = (double*)(pw + align256(units * BPC_D * BPC_D * 8));
    const dim3 g0(slabs, ctx->units);
    if (c.kv_dtype == BPC_BF16)
      fit_gram0_kernel<__nv_bfloat16><<<g0, 256, 0, stream>>>((const __nv_bfloat16*)k_cache, cpart, ctx->unit_lens, c.n_max, ctx->row_stride, slabs);
    else
      fit_gram0_kernel<float><<<g0, 256, 0, stream>>>((const float*)k_cache, cpart, ctx->unit_lens, c.n_max, ctx->row_stride, slabs);
    fit_gram0_reduce_kernel<<<dim3(BPC_D * BPC_D / 256, ctx->units), 256, 0, stream>>>(cpart, Cm, ctx->unit_lens, c.n_max, slabs);
    *launches += 2;
  }
  for (int it = 0; it < c.code_bits; ++it) {
    if (npow > 0) {
      fit_direction_kernel<<<ctx->units, BPC_D, 0, stream>>>(Cm, ctx->P, v_star, dir, ctx->unit_lens, c.n_max, c.code_bits, it, npow);
      *launches += 1;
    }
    fit_prep_kernel<<<ctx->units, BPC_D, 0, stream>>>(ctx->P, v_star, dir, dots, c.code_bits, it, npow > 0 ? 1 : 0);
#define BPC_FIT_PASS(KV, JPL)                                                                                          \
    fit_pass_kernel<KV, JPL><<<grid, kFitThreads, 0, stream>>>((const KV*)k_cache, hfit, dir, dots, partials, agree,   \
                                                                ctx->unit_lens, c.n_max, ctx->row_stride, it, bpu)
    if (tc_pass) {
      cudaError_t e = bpc_launch_fit_pass_tc(ctx, k_cache, hfit, dir, dots, partials, agree, it, stream);
      if (e != cudaSuccess) return e;
    } else if (c.kv_dtype == BPC_BF16) {
      if (c.code_bits == 32) BPC_FIT_PASS(__nv_bfloat16, 4); else if (c.code_bits == 64) BPC_FIT_PASS(__nv_bfloat16, 8); else if (c.code_bits == 128) BPC_FIT_PASS(__nv_bfloat16, 16); else BPC_FIT_PASS(__nv_bfloat16, 32);
    } else {
      if (c.code_bits == 32) BPC_FIT_PASS(float, 4); else if (c.code_bits == 64) BPC_FIT_PASS(float, 8); else if (c.code_bits == 128) BPC_FIT_PASS(float, 16); else BPC_FIT_PASS(float, 32);
    }
#undef BPC_FIT_PASS
    fit_reduce_kernel<<<ctx->units, BPC_D * kRedGroups, 0, stream>>>(partials, agree, ctx->P, ctx->unit_lens, c.n_max, c.code_bits, it, bpu, rows_per_block);
    *launches += 3;
  }
  return cudaGetLastError();
}

cudaError_t bpc_launch_build_eas(bpc_ctx* ctx, cudaStream_t stream) {
  build_eas_kernel<<<ctx->units, kEasThreads, 0, stream>>>(ctx->key_err, ctx->unit_lens, ctx->eas_idx, ctx->eas_cnt,
                                                           ctx->cfg.n_max, ctx->cfg.eas_ppm, ctx->eas_cap);
  ctx->launches += 1;
  return cudaGetLastError();
}

// Algorithm 1 (fit) in blocks of 32 bits: four kernels per block instead of one pass over the keys per bit.
//
// Algorithm 1 decides bit i of every key by t = R_i d_i (R_i = K - sum_{j<i} u_j v_j, d_i the caller's direction) and forms
// v_i = u_i^T R_i / n.  With the plain rule (no power iterations) all directions are known from the start, so what a bit
// needs from its predecessors is not the residual rows but only the scalars c_{j,i} = v_j . d_i:
//     t_i = (K D^T)_i - sum_{j<i} u_j c_{j,i}.
// Per block of 32 bits:
//   * project: T = K D_blk^T - U_prev C_prev for the block's 32 columns, one key per row; both terms are contractions and
//     run on the tensor cores (directions and scalars as three bf16 terms each: 24 mantissa bits, products exact).
//   * sweep: the 32 sequential bits on T alone.  A key costs 4 bytes of new data per bit (its entry of the next column)
//     where the row pass costs 272.  Pass j decides bit j from column j and already sums u_i T[:, j+1] for all i <= j;
//     those sums and the agreement counts u_j . u_i give c_{i,j+1} in fp64, because
//     n c_{i,l} = u_i^T T_l - sum_{m<i} (u_i . u_m) c_{m,l}: a triangular system, whose inverse grows by one row per bit.  One
//     thread block cluster per unit: the exchange per bit is a few hundred bytes per block, stored asynchronously into the
//     peers' shared memory (added there) and counted on their mbarriers.
//   * gather: W = U_blk^T K and the agreement counts of the block's bits with all bits so far (tensor cores again, the key
//     tile read channel-major).
//   * rows: v_i = (W_i - sum_{j<i} (u_i . u_j) v_j) / n in fp64, then the next block's scalars C = V D_next^T in fp64.
// The keys are read twice per 32 bits instead of 32 times.  fp32 caches take CUDA-core versions of project and gather.
#include <mutex>
#include "tma.cuh"
#include "fit_block.h"

namespace {
using namespace umma;

constexpr int kTileKeys = 128;
constexpr int kGroupThreads = 128;
constexpr int kTileBytes = kTileKeys * 256;
constexpr int kBits = 32;                                  // bits of a block = one code word

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kGroupThreads) : "memory"); }

// 32 consecutive accumulator columns of this thread's TMEM lane (no wait: several can be in flight)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
               "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                 "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
                 "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                 "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                 "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 x 32 bit transposes across the lanes of a warp, N words at once: lane i returns bit i of every lane.  Halves and bytes
// move with one byte permute, smaller fields with a rotation and a merge.
template <int N>
__device__ __forceinline__ void warp_transpose(uint32_t (&x)[N], int lane) {
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const int o = 16 >> st;
    const bool up = lane & o;
    const uint32_t low = o == 16 ? 0u : o == 8 ? 0u : o == 4 ? 0x0F0F0F0Fu : o == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t keep = up ? ~low : low, sel = o == 16 ? (up ? 0x3276u : 0x5410u) : (up ? 0x3715u : 0x6240u);
    const int rot = up ? 32 - o : o;
    uint32_t y[N];
#pragma unroll
    for (int k = 0; k < N; ++k) y[k] = __shfl_xor_sync(0xffffffffu, x[k], o);
#pragma unroll
    for (int k = 0; k < N; ++k)
      x[k] = o >= 8 ? __byte_perm(x[k], y[k], sel) : ((x[k] & keep) | (__funnelshift_l(y[k], y[k], rot) & ~keep));
  }
}
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
  uint32_t v[1] = {x};
  warp_transpose<1>(v, lane);
  return v[0];
}

// Largest |T| per column, in the upper halves of the words (sign off, exponent, seven bits of the mantissa; infinities and NaN are
// above every number): two columns to a register, the larger of each.
__device__ __forceinline__ uint32_t max_abs2(uint32_t a, float even, float odd) {
  const uint32_t v = __byte_perm(__float_as_uint(even), __float_as_uint(odd), 0x7632) & 0x7fff7fffu;
  asm("max.u16x2 %0, %0, %1;" : "+r"(a) : "r"(v));
  return a;
}
// such maxima of a warp's lanes (register q: columns 2q, 2q + 1): lane l returns column l's
__device__ __forceinline__ uint32_t warp_column_max(uint32_t (&v)[kBits / 2], int lane) {
#pragma unroll
  for (int o = 16; o >= 2; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o / 2; ++i) {
      const uint32_t keep = up ? v[i + o / 2] : v[i], give = up ? v[i] : v[i + o / 2];
      v[i] = __vmaxu2(keep, __shfl_xor_sync(0xffffffffu, give, o));
    }
  }
  const uint32_t m = __vmaxu2(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1));
  return lane & 1 ? m >> 16 : m & 0xffffu;
}
// where project leaves them, by unit and block of project: in the unit's partial sums, which the gather writes later
__host__ __device__ inline size_t column_max_at(int unit, int part, int parts) { return ((size_t)unit * parts * BPC_D * 2 + part) * kBits; }

// rows of a unit that block `blk` of `blocks` takes: equal shares of whole tiles
__host__ __device__ inline int block_rows(int n, int blocks) { return ((n + blocks - 1) / blocks + kTileKeys - 1) / kTileKeys * kTileKeys; }

// ---- sweep geometry (the projection fills the columns up to a whole group of keys)
constexpr int kSweepThreads = 512;
constexpr int kSweepWarps = kSweepThreads / 32;
constexpr int kSweepKeys = 8;                              // keys of a thread per round: two runs of four, 128 apart
constexpr int kSweepGroup = 32 * kSweepKeys;               // keys of a warp per round
// keys of a sweep block: equal shares in whole groups (columns are zero up to a whole group past the last key)
__host__ __device__ inline int sweep_share(int n, int blocks) { return ((n + blocks - 1) / blocks + kSweepGroup - 1) / kSweepGroup * kSweepGroup; }

// --------------------------------------------------------------------------- project (tensor cores, bf16 caches)
// T[l][key] for the 32 columns of block `blk`.  Per tile of 128 keys: eight MMAs K_tile x D (N = 96: three bf16 terms of
// the 32 directions), then two MMAs per earlier code word, U x (-C), into the same accumulator.  GROUPS warpgroups with
// their own tile, sign operand and accumulator.  The signs are laid out while the tile is on its way; the tile's buffer is
// refilled as soon as the MMAs are done, so the next load runs under the 32 column stores.
constexpr int kSignCols = 96;                              // signs expanded at a time (three words)
constexpr int kProjN = 3 * kBits;

template <int GROUPS>
__global__ void __launch_bounds__(kGroupThreads * GROUPS, 1)
fit_project_tc_kernel(const __grid_constant__ CUtensorMap kmap, const uint32_t* hfit, const float* __restrict__ v_star,
                      const float* cross, float* __restrict__ T, uint32_t* __restrict__ t_max,
                      const int32_t* __restrict__ unit_lens, int32_t* __restrict__ err, int n_max, int b, int blk, int t_stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  constexpr int kThreads = kGroupThreads * GROUPS;
  constexpr int U_BYTES = kTileKeys * kSignCols * 2;
  constexpr unsigned U_LBO = (kTileKeys / 8) * 128, C_LBO = (kProjN / 8) * 128;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int grp = tid / kGroupThreads, gtid = tid % kGroupThreads;
  unsigned char* a_t = smem + (size_t)grp * kTileBytes;
  unsigned char* b_s = smem + (size_t)GROUPS * kTileBytes;             // directions, three terms: [96 x 128], 128-byte swizzle
  unsigned char* u_s = b_s + kProjN * 256 + (size_t)grp * U_BYTES;     // this warpgroup's signs: [128 x 96], no swizzle
  unsigned char* c_s = b_s + kProjN * 256 + (size_t)GROUPS * U_BYTES;  // -C, three terms: [96 x 32 blk], no swizzle
  __shared__ __align__(128) uint2 sign_table[16];
  __shared__ unsigned long long bar_s[GROUPS], tile_bar_s[GROUPS];
  __shared__ uint32_t tmem_base_s, max_s[kBits];
  __shared__ int timed_out_g[GROUPS];
  const unsigned st_a = smem_u32(sign_table);
  // The keys that the gather before read last come first: some of them are still in L2 (32 x 128K keys 273 -> 262 us a launch).
  const int unit = gridDim.y - 1 - blockIdx.y, part = gridDim.x - 1 - blockIdx.x;
  const int n = min(unit_lens[unit], n_max);
  const int rows = block_rows(n, gridDim.x);
  const int row0 = part * rows;
  if (row0 >= n) { pdl_wait(); return; }                               // uniform over the block, nothing set up yet
  const int row_end = min(n, row0 + rows);
  const int ntile = (row_end - row0 + kTileKeys - 1) / kTileKeys;
  const int words = b / 32;

  if (tid == 0) {
    for (int g = 0; g < GROUPS; ++g) { mbar_init(&bar_s[g], 1); mbar_init(&tile_bar_s[g], 1); timed_out_g[g] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // (the warpgroups' first tiles: no kernel of the fit writes keys)
    for (int g = 0; g < min(GROUPS, ntile); ++g)
      tma::load_key_tile(smem + (size_t)g * kTileBytes, &kmap, unit * n_max + row0 + (ntile - 1 - g) * kTileKeys, &tile_bar_s[g]);
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  unsigned long long* tile_bar = &tile_bar_s[grp];
  auto load_tile = [&](int tile) { tma::load_key_tile(a_t, &kmap, unit * n_max + row0 + (ntile - 1 - tile) * kTileKeys, tile_bar); };   // (one thread)
  fill_sign_table(sign_table, tid);
  if (tid < kBits) max_s[tid] = 0u;
  for (int c = tid; c < kBits * BPC_D / 8; c += kThreads) {             // eight elements at a time: a 16-byte store per term
    const int l = c >> 4, ch = c & 15;
    const float4* src = reinterpret_cast<const float4*>(v_star + ((size_t)unit * b + kBits * blk + l) * BPC_D + 8 * ch);
    const float4 x = src[0], y = src[1];
    const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    uint4 t3[3];
    split3x8(v, t3);
#pragma unroll
    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(b_s + sw128_offset(kProjN, p * kBits + l, ch)) = t3[p];
  }
  pdl_wait();                                                          // (launched early by the kernel that forms the scalars)
  for (int c = tid; c < kBits * blk * kBits / 8; c += kThreads) {
    const int j = 8 * (c >> 5), l = c & 31;                            // eight earlier bits, column
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = -cross[((size_t)unit * b + j + e) * kBits + l];
    uint4 t3[3];
    split3x8(v, t3);
#pragma unroll
    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(c_s + nosw_offset(kProjN, p * kBits + l, j)) = t3[p];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pdl_release();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_all = tmem_base_s;
  const uint32_t tm_d = tmem_all + (uint32_t)(grp * kProjN);
  const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
  unsigned long long* bar = &bar_s[grp];
  const uint32_t idesc = umma_idesc_bf16(kTileKeys, kProjN);

  unsigned ph = 0, tph = 0;
  uint32_t first[kSignCols / 32];                                      // the next tile's first code words of this thread's key
  auto load_words = [&](int tile) {
    const int r = row0 + (ntile - 1 - tile) * kTileKeys + gtid;
    const uint32_t* h = hfit + ((size_t)unit * n_max + r) * words;
#pragma unroll
    for (int w = 0; w < kSignCols / 32; ++w) first[w] = (w < blk && r < row_end) ? h[w] : 0u;
  };
  auto put_signs = [&](int w, uint32_t x) {                            // word w of the operand's row `gtid`
    unsigned char* d = u_s + (size_t)(4 * w) * U_LBO + (size_t)(gtid >> 3) * 128 + (size_t)(gtid & 7) * 16;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint2 lo = signs4(st_a, x, 2 * c), hi = signs4(st_a, x, 2 * c + 1);
      *reinterpret_cast<uint4*>(d + (size_t)c * U_LBO) = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
  };
  auto issue_signs = [&](int w0, int wn) {
    for (int ks = 0; ks < 2 * wn; ++ks)
      umma_bf16(tm_d, umma_desc_nosw(u_s + (size_t)ks * 2 * U_LBO, U_LBO, 128),
                umma_desc_nosw(c_s + (size_t)(4 * w0 + 2 * ks) * C_LBO, C_LBO, 128), idesc, 1u);
  };
  if (grp < ntile) load_words(grp);
  uint32_t t_abs[kBits / 2] = {};                                      // largest |T| of this thread's keys
  for (int tl = grp; tl < ntile; tl += GROUPS) {
    const int row = row0 + (ntile - 1 - tl) * kTileKeys + gtid;
    const bool live = row < row_end;
    const int w1 = min(blk, kSignCols / 32);
#pragma unroll
    for (int w = 0; w < kSignCols / 32; ++w)                           // (while the tile is on its way)
      if (w < w1) put_signs(w, first[w]);
    if (tl + GROUPS < ntile) load_words(tl + GROUPS);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    group_sync(grp);                                                   // the signs are there
    if (timed_out_g[grp]) {                                            // (set before a barrier, so all 128 threads agree)
      if (gtid == 0) (void)mbar_wait(tile_bar, tph);                   // the copy in flight
      break;
    }
    if (gtid == 0) {
      if (!mbar_wait(tile_bar, tph)) timed_out_g[grp] = 1;             // and the tile
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        const size_t aoff = (size_t)(ks >> 2) * (kTileKeys * 128) + (size_t)(ks & 3) * 32;
        const size_t boff = (size_t)(ks >> 2) * (kProjN * 128) + (size_t)(ks & 3) * 32;
        umma_bf16(tm_d, umma_desc_sw128(a_t + aoff), umma_desc_sw128(b_s + boff), idesc, ks > 0 ? 1u : 0u);
      }
      issue_signs(0, w1);
      umma_commit(bar);
    }
    if (!mbar_wait(bar, ph)) timed_out_g[grp] = 1;
    ph ^= 1u;
    tph ^= 1u;
    if (tl + GROUPS < ntile && gtid == 0) load_tile(tl + GROUPS);
    for (int w0 = kSignCols / 32; w0 < blk; w0 += kSignCols / 32) {    // 256-bit codes: the words beyond the third
      const int wn = min(blk - w0, kSignCols / 32);
      const uint32_t* h = hfit + ((size_t)unit * n_max + (live ? row : row0)) * words + w0;
      for (int w = 0; w < wn; ++w) put_signs(w, h[w]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      group_sync(grp);
      if (gtid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue_signs(w0, wn);
        umma_commit(bar);
      }
      if (!mbar_wait(bar, ph)) timed_out_g[grp] = 1;
      ph ^= 1u;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    uint32_t r0[32], r1[32], r2[32];
    tmem_ld32(tm_d + lane_off, r0);
    tmem_ld32(tm_d + lane_off + 32, r1);
    tmem_ld32(tm_d + lane_off + 64, r2);
    tmem_wait_ld();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    float* dst = T + (size_t)unit * kBits * t_stride + row;            // (rows of the last tile past the end: zeros)
#pragma unroll
    for (int l = 0; l < kBits; l += 2) {
      const float v = (__uint_as_float(r0[l]) + __uint_as_float(r1[l])) + __uint_as_float(r2[l]);
      const float w = (__uint_as_float(r0[l + 1]) + __uint_as_float(r1[l + 1])) + __uint_as_float(r2[l + 1]);
      const float tv = live ? v + 0.f : 0.f, tw = live ? w + 0.f : 0.f;   // (never -0)
      dst[(size_t)l * t_stride] = tv;
      dst[(size_t)(l + 1) * t_stride] = tw;
      t_abs[l / 2] = max_abs2(t_abs[l / 2], tv, tw);
    }
  }
  atomicMax(&max_s[tid & 31], warp_column_max(t_abs, tid & 31));
  // the sweep reads whole groups of keys: zeros behind the unit's last tile where that ends half a group
  for (int i = row0 + ntile * kTileKeys + tid; row_end == n && i < (n + kSweepGroup - 1) / kSweepGroup * kSweepGroup; i += kThreads)
    for (int l = 0; l < kBits; ++l) T[((size_t)unit * kBits + l) * t_stride + i] = 0.f;
  if (timed_out_g[grp] && gtid == 0) atomicOr(err, BPC_DEVERR_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid < kBits) t_max[column_max_at(unit, part, gridDim.x) + tid] = max_s[tid];
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_all), "r"(512) : "memory");
}

// --------------------------------------------------------------------------- project (CUDA cores, fp32 caches)
// One thread per key.  Both sums run in fp64 and are rounded once, on their way to the column (sums of 16 channels and of 32
// earlier bits in fp32 left the decisions less precise than one pass per bit has them).
__global__ void __launch_bounds__(kTileKeys)
fit_project_f32_kernel(const float* __restrict__ k_cache, const uint32_t* __restrict__ hfit, const float* __restrict__ v_star,
                       const float* __restrict__ cross, float* __restrict__ T, uint32_t* __restrict__ t_max,
                       const int32_t* __restrict__ unit_lens, int n_max, int row_stride, int b, int blk, int t_stride, int parts) {
  const int unit = blockIdx.y, tid = threadIdx.x;
  const int n = min(unit_lens[unit], n_max);
  const int row = blockIdx.x * kTileKeys + tid;
  if (blockIdx.x * kTileKeys >= (n + kSweepGroup - 1) / kSweepGroup * kSweepGroup) return;   // (zeros up to a whole sweep group)
  const bool live = row < n;
  __shared__ __align__(16) double d_s[BPC_D][kBits];                   // directions, channel-major; then the scalars of 32 bits
  double acc[kBits];
#pragma unroll
  for (int l = 0; l < kBits; ++l) acc[l] = 0.0;
  for (int c = tid; c < kBits * BPC_D; c += kTileKeys) d_s[c & 127][c >> 7] = (double)v_star[((size_t)unit * b + kBits * blk + (c >> 7)) * BPC_D + (c & 127)];
  __syncthreads();
  const float4* kr = reinterpret_cast<const float4*>(k_cache + ((size_t)unit * n_max + (live ? row : 0)) * row_stride);
  for (int c0 = 0; c0 < BPC_D; c0 += 4) {
    const float4 q = kr[c0 / 4];
    const double x[4] = {(double)q.x, (double)q.y, (double)q.z, (double)q.w};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int l = 0; l < kBits; ++l) acc[l] = fma(x[c], d_s[c0 + c][l], acc[l]);
  }
  for (int w = 0; w < blk; ++w) {
    __syncthreads();
    for (int c = tid; c < kBits * kBits; c += kTileKeys) d_s[c >> 5][c & 31] = (double)cross[((size_t)unit * b + 32 * w + (c >> 5)) * kBits + (c & 31)];
    __syncthreads();
    const uint32_t x = hfit[((size_t)unit * n_max + (live ? row : 0)) * (b / 32) + w];
    for (int j = 0; j < 32; ++j) {
      const double u = ((x >> j) & 1u) ? 1.0 : -1.0;
#pragma unroll
      for (int l = 0; l < kBits; ++l) acc[l] = fma(-u, d_s[j][l], acc[l]);
    }
  }
  float* dst = T + (size_t)unit * kBits * t_stride + row;
  uint32_t t_abs[kBits / 2] = {};
#pragma unroll
  for (int l = 0; l < kBits; l += 2) {
    const float tv = live ? (float)acc[l] + 0.f : 0.f, tw = live ? (float)acc[l + 1] + 0.f : 0.f;   // (never -0)
    dst[(size_t)l * t_stride] = tv;
    dst[(size_t)(l + 1) * t_stride] = tw;
    t_abs[l / 2] = max_abs2(t_abs[l / 2], tv, tw);
  }
  atomicMax(&t_max[column_max_at(unit, 0, parts) + (tid & 31)], warp_column_max(t_abs, tid & 31));
}

// --------------------------------------------------------------------------- gather (tensor cores, bf16 caches)
// W[i][c] = sum over keys of u_i K[c] for the block's 32 bits, and the inner products u_i . u_j with all bits j so far.
// Per tile of 128 keys the signs of all R = 32 (blk + 1) bits so far are laid out bit-major, U [R x 128 keys] (each warp
// transposes its 32 keys' code words across lanes, one lane then writes one bit's 32 keys); then eight MMAs K_tile^T
// (channel-major view of the tile, M = 128 channels) x U_blk (N = 32) and eight per 128 bits U x U_blk.  An A operand of 128
// rows reaches past the R rows of U into whatever follows; those accumulator rows are not read.  Channel sums move to fp64
// registers every kFlushTiles tiles (the tensor cores' fp32 sums lose with their length: 5.0e-8 of a row over 1024 keys, 3.0e-8
// over 512; the pass per bit sums at least 384); the inner products are integers below 2^24 and stay exact in fp32.
// A tile occupies its buffer from the start of its load to the end of its MMAs and the load is most of that, so as many
// warpgroups with one buffer each as shared memory holds beat fewer with two (two groups of two buffers: 261 to 372 us at
// 32 x 128K keys).
constexpr int kFlushTiles = 3;

template <int GROUPS>
__global__ void __launch_bounds__(kGroupThreads * GROUPS, 1)
fit_gather_tc_kernel(const __grid_constant__ CUtensorMap kmap, const uint32_t* hfit, double* __restrict__ wpart,
                     int32_t* __restrict__ apart, const int32_t* __restrict__ unit_lens, int32_t* __restrict__ err, int n_max,
                     int b, int blk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  constexpr int kThreads = kGroupThreads * GROUPS;
  constexpr int kMaxWords = 8;
  const int R = kBits * (blk + 1);                         // operand rows (bits)
  const unsigned LBO = (unsigned)(R / 8) * 128;            // bytes between core matrices along K (keys)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = tid / kGroupThreads, gtid = tid % kGroupThreads;
  unsigned char* a_t = smem + (size_t)grp * kTileBytes;
  unsigned char* u_s = smem + (size_t)GROUPS * kTileBytes + (size_t)grp * R * kTileKeys * 2;
  __shared__ __align__(128) uint2 sign_table[16];
  __shared__ unsigned long long bar_s[GROUPS], tile_bar_s[GROUPS];
  __shared__ uint32_t tmem_base_s;
  __shared__ int timed_out_g[GROUPS];
  const unsigned st_a = smem_u32(sign_table);
  const int unit = blockIdx.y, words = b / 32;
  const int n = min(unit_lens[unit], n_max);
  const int rows = block_rows(n, gridDim.x);
  const int row0 = blockIdx.x * rows;
  if (row0 >= n) { pdl_wait(); return; }                   // (the reduction skips blocks without rows)
  const int row_end = min(n, row0 + rows);
  const int ntile = (row_end - row0 + kTileKeys - 1) / kTileKeys;
  if (tid == 0) {
    for (int g = 0; g < GROUPS; ++g) { mbar_init(&bar_s[g], 1); mbar_init(&tile_bar_s[g], 1); timed_out_g[g] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int g = 0; g < min(GROUPS, ntile); ++g)           // (the warpgroups' first tiles: no kernel of the fit writes keys)
      tma::load_key_tile(smem + (size_t)g * kTileBytes, &kmap, unit * n_max + row0 + g * kTileKeys, &tile_bar_s[g]);
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  unsigned long long* tile_bar = &tile_bar_s[grp];
  auto load_tile = [&](int tile) { tma::load_key_tile(a_t, &kmap, unit * n_max + row0 + tile * kTileKeys, tile_bar); };   // (one thread)
  uint32_t nxt[kMaxWords];                                 // code words of this thread's key of the next tile
  auto load_words = [&](int tile) {
    const int r = row0 + tile * kTileKeys + gtid;
    const uint32_t* h = hfit + ((size_t)unit * n_max + r) * words;
#pragma unroll
    for (int w = 0; w < kMaxWords; ++w) nxt[w] = (w <= blk && r < row_end) ? h[w] : 0u;
  };
  fill_sign_table(sign_table, tid);
  pdl_wait();                                              // (launched early: the code words are there)
  if (grp < ntile) load_words(grp);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pdl_release();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_all = tmem_base_s;
  const uint32_t tm_w = tmem_all + (uint32_t)(grp * 96), tm_a = tm_w + 32;   // channel sums; inner products, 128 bits per 32 columns
  const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
  unsigned long long* bar = &bar_s[grp];
  const uint32_t idesc = umma_idesc_bf16(128, kBits);
  double acc[kBits];                                       // channel gtid
#pragma unroll
  for (int i = 0; i < kBits; ++i) acc[i] = 0.0;
  unsigned ph = 0, tph = 0;
  int since_flush = 0;
  bool first = true;
  for (int tl = grp; tl < ntile; tl += GROUPS) {
    // this warp's 32 keys, one bit per lane; keys past the end become 0 instead of +-1 (while the tile is on its way)
    const int live = min(max(row_end - (row0 + tl * kTileKeys + 32 * (warp & 3)), 0), 32);
#pragma unroll
    for (int w = 0; w < kMaxWords; ++w) {
      if (w > blk) break;
      const uint32_t m = warp_transpose(nxt[w], lane);
      unsigned char* dst = u_s + (size_t)(4 * (warp & 3)) * LBO + (size_t)(32 * w + lane) * 16;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint2 lo = signs4(st_a, m, 2 * c), hi = signs4(st_a, m, 2 * c + 1);
        uint32_t h[4] = {lo.x, lo.y, hi.x, hi.y};
        if (live < 32) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int k0 = 8 * c + 2 * e;
            h[e] &= (k0 < live ? 0xFFFFu : 0u) | (k0 + 1 < live ? 0xFFFF0000u : 0u);
          }
        }
        *reinterpret_cast<uint4*>(dst + (size_t)c * LBO) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
    if (tl + GROUPS < ntile) load_words(tl + GROUPS);
    const int tile_rows = min(row_end - (row0 + tl * kTileKeys), kTileKeys);
    if (tile_rows < kTileKeys) {                           // the unit's last tile: what the cache holds past the end becomes zero
      if (!mbar_wait(tile_bar, tph)) timed_out_g[grp] = 1;
      if (gtid >= tile_rows) {
#pragma unroll
        for (int ch = 0; ch < 16; ++ch) *reinterpret_cast<uint4*>(a_t + sw128_offset(kTileKeys, gtid, ch)) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // (a flush's accumulator reads are done)
    group_sync(grp);
    if (timed_out_g[grp]) {                                // (set before a barrier, so all 128 threads agree)
      if (gtid == 0) (void)mbar_wait(tile_bar, tph);       // the copy in flight
      break;
    }
    if (gtid == 0) {
      if (!mbar_wait(tile_bar, tph)) timed_out_g[grp] = 1;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned char* ub = u_s + (size_t)(4 * blk) * 128;          // rows of this block's 32 bits
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        umma_bf16(tm_w, umma_desc_sw128_mn(a_t + (size_t)ks * 2048, 16384, 1024), umma_desc_nosw(ub + (size_t)ks * 2 * LBO, LBO, 128),
                  idesc | kIdescAMnMajor, (since_flush > 0 || ks > 0) ? 1u : 0u);
      for (int hf = 0; 4 * hf <= blk; ++hf) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
          umma_bf16(tm_a + (uint32_t)(32 * hf), umma_desc_nosw(u_s + (size_t)hf * 2048 + (size_t)ks * 2 * LBO, LBO, 128),
                    umma_desc_nosw(ub + (size_t)ks * 2 * LBO, LBO, 128), idesc, (!first || ks > 0) ? 1u : 0u);
      }
      umma_commit(bar);
    }
    first = false;
    if (!mbar_wait(bar, ph)) timed_out_g[grp] = 1;
    ph ^= 1u;
    tph ^= 1u;
    if (tl + GROUPS < ntile && gtid == 0) load_tile(tl + GROUPS);
    ++since_flush;
    if (since_flush == kFlushTiles || tl + GROUPS >= ntile) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t r[16];
        tmem_ld16(tm_w + lane_off + 16 * h, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[16 * h + i] += (double)__uint_as_float(r[i]);
      }
      since_flush = 0;
    }
  }
  if (timed_out_g[grp] && gtid == 0) atomicOr(err, BPC_DEVERR_TIMEOUT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncthreads();                                         // the tile buffers are free in all warpgroups
  double* red = reinterpret_cast<double*>(smem);           // [groups][32][128]
#pragma unroll
  for (int i = 0; i < kBits; ++i) red[((size_t)grp * kBits + i) * BPC_D + gtid] = acc[i];
  int32_t* redc = reinterpret_cast<int32_t*>(smem + (size_t)GROUPS * kBits * BPC_D * 8);   // [groups][R][33]
  for (int hf = 0; 4 * hf <= blk; ++hf) {
    const int j = 128 * hf + gtid;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t r[16];
      tmem_ld16(tm_a + (uint32_t)(32 * hf + 16 * h) + lane_off, r);
      tmem_wait_ld();
      if (j < R) {
#pragma unroll
        for (int i = 0; i < 16; ++i) redc[((size_t)grp * R + j) * 33 + 16 * h + i] = grp < ntile ? (int)__uint_as_float(r[i]) : 0;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  double* wo = wpart + ((size_t)unit * gridDim.x + blockIdx.x) * kBits * BPC_D;
  for (int e = tid; e < kBits * BPC_D; e += kThreads) {
    double v = 0.0;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) v += red[(size_t)g * kBits * BPC_D + e];
    wo[e] = v;
  }
  int32_t* ao = apart + ((size_t)unit * gridDim.x + blockIdx.x) * kBits * b;
  for (int e = tid; e < kBits * R; e += kThreads) {
    const int i = e / R, j = e % R;
    int v = 0;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) v += redc[((size_t)g * R + j) * 33 + i];
    ao[(size_t)i * b + j] = v;
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_all), "r"(512) : "memory");
}

// --------------------------------------------------------------------------- gather (CUDA cores, fp32 caches)
// Thread (half, channel) adds +-K over kGatherRows rows in fp32 and the sums in fp64; the inner products come from ballots: lane i holds bit i of
// the block over a warp's 32 keys, every earlier bit's 32 keys are one broadcast word.
constexpr int kGatherRows = 32;

__global__ void __launch_bounds__(256)
fit_gather_f32_kernel(const float* __restrict__ k_cache, const uint32_t* __restrict__ hfit, double* __restrict__ wpart,
                      int32_t* __restrict__ apart, const int32_t* __restrict__ unit_lens, int n_max, int row_stride, int b, int blk) {
  const int unit = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, words = b / 32;
  const int n = min(unit_lens[unit], n_max);
  const int rows = block_rows(n, gridDim.x);
  const int row0 = blockIdx.x * rows;
  if (row0 >= n) return;
  const int row_end = min(n, row0 + rows);
  __shared__ int cnt_s[kBits][256 + 1];
  for (int e = tid; e < kBits * 257; e += 256) (&cnt_s[0][0])[e] = 0;
  const int half = tid >> 7, c = tid & 127;
  double acc64[kBits];
#pragma unroll
  for (int i = 0; i < kBits; ++i) acc64[i] = 0.0;
  const uint32_t* h = hfit + (size_t)unit * n_max * words;
  for (int r0 = row0; r0 < row_end; r0 += 2 * kGatherRows) {
    float acc[kBits];
#pragma unroll
    for (int i = 0; i < kBits; ++i) acc[i] = 0.f;
    for (int r = r0 + half; r < min(row_end, r0 + 2 * kGatherRows); r += 2) {
      const float x = k_cache[((size_t)unit * n_max + r) * row_stride + c];
      const uint32_t w = h[(size_t)r * words + blk];
#pragma unroll
      for (int i = 0; i < kBits; ++i) acc[i] += ((w >> i) & 1u) ? x : -x;
    }
#pragma unroll
    for (int i = 0; i < kBits; ++i) acc64[i] += (double)acc[i];
  }
  __syncthreads();
  for (int r0 = row0 + 32 * warp; r0 < row_end; r0 += 256) {
    const int r = r0 + lane;
    const uint32_t live = __ballot_sync(0xffffffffu, r < row_end);
    const uint32_t mine = warp_transpose(r < row_end ? h[(size_t)r * words + blk] : 0u, lane);   // bit `lane` of the block
    for (int w = 0; w <= blk; ++w) {
      const uint32_t other = warp_transpose(r < row_end ? h[(size_t)r * words + w] : 0u, lane);
      for (int j = 0; j < 32; ++j) {
        const uint32_t x = __shfl_sync(0xffffffffu, other, j);
        const int d = __popc(live) - 2 * __popc((mine ^ x) & live);
        atomicAdd(&cnt_s[lane][32 * w + j], d);
      }
    }
  }
  double* wo = wpart + ((size_t)unit * gridDim.x + blockIdx.x) * kBits * BPC_D;
  if (half == 0)
    for (int i = 0; i < kBits; ++i) wo[(size_t)i * BPC_D + c] = acc64[i];
  __syncthreads();
  if (half == 1)
    for (int i = 0; i < kBits; ++i) wo[(size_t)i * BPC_D + c] += acc64[i];
  int32_t* ao = apart + ((size_t)unit * gridDim.x + blockIdx.x) * kBits * b;
  const int nj = kBits * (blk + 1);
  for (int e = tid; e < kBits * nj; e += 256) ao[(size_t)(e / nj) * b + e % nj] = cnt_s[e / nj][e % nj];
}

// --------------------------------------------------------------------------- sweep
// The 32 sequential bits of a block on the columns T.  Block r of the unit's cluster owns an equal share of the keys; a
// thread takes eight keys at a time, two runs of four.  Per key and bit: compare with sum_i u_i c_i (one table look-up per five
// bits) and decide; then the next column's sums over the keys whose bit i is set (u_i^T T = 2 sum - total).
// Those sums and the agreements with the earlier bits are one contraction over the keys and run on the warp-level integer
// tensor path (mma.sync m16n8k32, u8 x u8 -> s32, exact): rows = the block's bits, columns = the four bytes of T in 32-bit
// fixed point, a column of ones (keys set) and the new bit itself (keys set in both).  A warp keeps its keys' bits a second
// time for that, bit-major: lane (g, t) holds bits g, g + 8, g + 16, g + 24 of the keys of lanes 8t .. 8t + 7, bit 8b + s of
// word h being key (lane 8t + s, entry 4h + b), so that (word & 0x01010101 << s) is an operand register of four keys and a new
// bit costs six byte permutes of its ballots.  The bytes of T are transposed by byte permutes and pass through rows of
// shared memory of the warp's own.  One logic operation per 128 (bit, key) pairs, where predicated adds took two
// instructions per 32.  Per 32 bits, against sums in fp32 with the agreements counted bit-sliced, byte tables for sum_i u_i c_i, 16-way
// exchange slots and a copy ring: 8 x 32K keys 102 -> 77 us, 32 x 128K 372 -> 342.  With one group per warp a bit takes 2.4 us, half of
// it the exchange (send 0.2, transit 0.2, scalars 0.4, tables 0.2) and the rest a chain of latencies; with several, the integer pipe
// and the shared-memory pipe (shuffles and operand staging) share the bound at 2.1 us per group of keys and 32 bits.
// The bit-major words stay in registers where a warp has one group of keys, in tensor memory (a scratchpad here: the kernel
// issues no tcgen05.mma) beside key-major words in shared memory, and over column 0 of T, which is dead after bit 0, where a block
// has more keys than fit on chip.
// Precision: T enters the sums as a 32-bit integer with a power-of-two scale, rounded by at most 2^-30 of the largest |T| of
// its column in the unit; everything after that is exact up to the fp64 scalars.  Each column has its own scale, so that a long
// direction, or a channel far larger than the others, takes no bits from the other columns.  A key's own T stays the fp32 value.

constexpr int kOneGroup = 0, kWordsOnChip = 1, kWordsGlobal = 2;

// one round of a warp: this lane's entries of a column, keys 4 lane .. + 3 and 128 + 4 lane .. + 3 of a group
__device__ __forceinline__ void load_entries(float4 (&v)[2], const float* src) {
  v[0] = __ldcg(reinterpret_cast<const float4*>(src));
  v[1] = __ldcg(reinterpret_cast<const float4*>(src + 128));
}

__device__ __forceinline__ void mma_u8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Operand B of a round, per warp: five rows (the bytes of T, least significant first, and the new bit), each 32 lanes x 2 words;
// 80 bytes per eight lanes and 320 per row keep the 16-byte reads of a quarter warp (two rows, all four parts) on different banks.
constexpr int kStagePart = 80, kStageRow = 320, kStageWarp = 5 * kStageRow;
// sums of a block: six columns (bytes 0 .. 3, keys set, keys set in both) of 32 bits; a stride of 36 spreads the lanes' banks
constexpr int kSumStride = 36;
constexpr int kLeastExp = 29;                              // biased exponent of a column's largest |T| from which one factor scales it
constexpr int kTabBits = 5, kTabs = 7;                     // sum_i u_i c_i: five bits per look-up

// What a warp carries from pass to pass.
struct SweepWarp {
  float tab[kTabs];                                        // entry `lane` of the look-up tables
  float4 t[2], nx[2];                                      // this lane's entries of columns j and j + 1, requested a round ahead
  uint32_t aw[4][2];                                       // bit-major words (of the warp's only group, or of the one at hand)
  uint32_t w[kSweepKeys];                                  // the same key-major
};

// One pass over this block's keys: decides bit j; unless it is the block's last bit, also the sums for column j + 1.
// TILES = tiles of 16 bits in play.  The last row of the last tile is all ones (the totals) until its own bit is
// decided, so bit 15 already takes two tiles.  Keys past the end (up to 255, all in the last group of the unit's last
// block, entries zero) take part like any others and are subtracted by the sender: they all carry the same code word.
// sum_i u_i c_i comes from tables of 32 sums held by the lanes of the warp, one shuffle per five bits: no address arithmetic and
// no bank conflicts (byte tables in shared memory: 3.4 wavefronts a look-up, which bounded the pass).  An entry is rounded once
// and the look-ups are added as a tree: four roundings deep (added in a row, with entries summed from rounded scalars, nine).
template <int TILES, bool LAST, int WORDS>
__device__ __forceinline__ void sweep_pass(SweepWarp& st, uint32_t* __restrict__ ws, const float* __restrict__ Tw, int t_stride,
                                           uint32_t aw_tmem, uint32_t* __restrict__ aw_g, int j, int nk, int e_next, int warp, int lane,
                                           unsigned stage, unsigned ones, unsigned* __restrict__ sums) {
  const uint32_t bit = 1u << j;
  // 2^(156 - e_next) for the next column's entries, in two factors where that is more than 2^127
  const float scale = e_next == 255 ? 0.f : __uint_as_float((uint32_t)(283 - max(e_next, kLeastExp)) << 23);
  [[maybe_unused]] const float boost = __uint_as_float((uint32_t)(127 + kLeastExp - e_next) << 23);
  const int ng = nk / kSweepGroup, g = lane >> 2, t = lane & 3;
  const int nl = (j + kTabBits - 1) / kTabBits;            // tables in play
  uint32_t (&aw)[4][2] = st.aw;
  int acc[TILES][4][4];                                    // [tile][s & 3]: counts times 2^(s & 3)
#pragma unroll
  for (int r = 0; r < TILES; ++r)
#pragma unroll
    for (int s = 0; s < 4; ++s) acc[r][s][0] = acc[r][s][1] = acc[r][s][2] = acc[r][s][3] = 0;
  const unsigned sel = (unsigned)t | ((unsigned)(t + 4) << 4);
  // operand B: lane g reads row g of the bytes, the column of ones, the new bit (columns 6 and 7 are not used)
  const unsigned b_src = (g < 4 || g == 5 ? stage + (unsigned)((g == 5 ? 4 : g) * kStageRow) : ones) + (unsigned)(t * kStagePart);
  const unsigned st_dst = stage + (unsigned)((lane >> 3) * kStagePart + (lane & 7) * 8);
  const float* col = Tw + (size_t)j * t_stride + 4 * lane;
#pragma unroll 1
  for (int gr = warp; gr < ng; gr += kSweepWarps) {
    uint32_t* pw = ws + gr * kSweepGroup + 4 * lane;
    if constexpr (!LAST && WORDS == kWordsOnChip) {
      const uint32_t a = aw_tmem + (uint32_t)(gr / kSweepWarps) * 8u;
      if (TILES == 1 || j == 15) {
        if (j > 0) asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                : "=r"(aw[0][0]), "=r"(aw[0][1]), "=r"(aw[1][0]), "=r"(aw[1][1]) : "r"(a));
      } else {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(aw[0][0]), "=r"(aw[0][1]), "=r"(aw[1][0]), "=r"(aw[1][1]), "=r"(aw[2][0]), "=r"(aw[2][1]), "=r"(aw[3][0]), "=r"(aw[3][1]) : "r"(a));
      }
    }
    uint32_t (&w)[kSweepKeys] = st.w;
    if (WORDS != kOneGroup) {
      const uint4 wl = *reinterpret_cast<const uint4*>(pw), wh = *reinterpret_cast<const uint4*>(pw + 128);
      w[0] = wl.x; w[1] = wl.y; w[2] = wl.z; w[3] = wl.w; w[4] = wh.x; w[5] = wh.y; w[6] = wh.z; w[7] = wh.w;
    }
    float c[kSweepKeys];
#pragma unroll
    for (int e = 0; e < kSweepKeys; ++e) c[e] = __shfl_sync(0xffffffffu, st.tab[0], w[e]);
    // ((0 + 1) + (2 + 3)) + ((4 + 5) + 6), as far as there are tables
    auto look = [&](int q, int e) { return __shfl_sync(0xffffffffu, st.tab[q], w[e] >> (kTabBits * q)); };
    if (nl > 1) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += look(1, e);
    }
    if (nl > 3) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += look(2, e) + look(3, e);
    } else if (nl > 2) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += look(2, e);
    }
    if (nl > 6) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += (look(4, e) + look(5, e)) + look(6, e);
    } else if (nl > 5) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += look(4, e) + look(5, e);
    } else if (nl > 4) {
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) c[e] += look(4, e);
    }
    uint32_t f[2] = {0u, 0u};                              // the new bit, a byte per key
    [[maybe_unused]] uint32_t x[kSweepKeys];
    {
      const float tv[kSweepKeys] = {st.t[0].x, st.t[0].y, st.t[0].z, st.t[0].w, st.t[1].x, st.t[1].y, st.t[1].z, st.t[1].w};
#pragma unroll
      for (int e = 0; e < kSweepKeys; ++e) {
        const bool set = !(tv[e] < c[e]);
        if (set) w[e] |= bit;
        if (!LAST) {
          if (set) f[e >> 2] |= 1u << (8 * (e & 3));
          x[e] = __ballot_sync(0xffffffffu, set);
        }
      }
    }
    if (WORDS != kOneGroup || LAST) {
      *reinterpret_cast<uint4*>(pw) = make_uint4(w[0], w[1], w[2], w[3]);
      *reinterpret_cast<uint4*>(pw + 128) = make_uint4(w[4], w[5], w[6], w[7]);
    } else if (lane == 31) {
      pw[131] = w[7];                                      // (the last key's: the sender may need it)
    }
    // The registers just used take the next round's entries, or the next pass's first.
    const bool more = WORDS != kOneGroup && gr + kSweepWarps < ng;
    const float* next = more ? col + (gr + kSweepWarps) * kSweepGroup : col + t_stride + warp * kSweepGroup;
    if (WORDS != kOneGroup && (!LAST || more)) load_entries(st.t, next);
    if constexpr (!LAST) {
      // the next column in fixed point, its bytes and the new bit to the warp's staging rows
      uint32_t v[kSweepKeys], z[5][2];
      {
        float nv[kSweepKeys] = {st.nx[0].x, st.nx[0].y, st.nx[0].z, st.nx[0].w, st.nx[1].x, st.nx[1].y, st.nx[1].z, st.nx[1].w};
        if (e_next < kLeastExp) {
#pragma unroll
          for (int e = 0; e < kSweepKeys; ++e) nv[e] *= boost;
        }
#pragma unroll
        for (int e = 0; e < kSweepKeys; ++e) v[e] = (uint32_t)__float2int_rn(nv[e] * scale);
      }
      if (WORDS == kOneGroup) { st.t[0] = st.nx[0]; st.t[1] = st.nx[1]; }
      if (more || j + 2 < kBits) load_entries(st.nx, next + t_stride);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t p0 = __byte_perm(v[4 * h], v[4 * h + 1], 0x5140), p1 = __byte_perm(v[4 * h + 2], v[4 * h + 3], 0x5140);
        const uint32_t q0 = __byte_perm(v[4 * h], v[4 * h + 1], 0x7362), q1 = __byte_perm(v[4 * h + 2], v[4 * h + 3], 0x7362);
        z[0][h] = __byte_perm(p0, p1, 0x5410);
        z[1][h] = __byte_perm(p0, p1, 0x7632);
        z[2][h] = __byte_perm(q0, q1, 0x5410);
        z[3][h] = __byte_perm(q0, q1, 0x7632) ^ 0x80808080u;         // (the integer plus 2^31)
        z[4][h] = f[h];
      }
      __syncwarp();                                        // every lane has read the rows of the round before
#pragma unroll
      for (int d = 0; d < 5; ++d)
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(st_dst + (unsigned)(d * kStageRow)), "r"(z[d][0]), "r"(z[d][1]) : "memory");
      // the new bit joins the bit-major words
      if constexpr (WORDS == kWordsOnChip) {
        if (TILES == 1)
          asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(aw[0][0]), "+r"(aw[0][1]), "+r"(aw[1][0]), "+r"(aw[1][1]) :: "memory");
        else
          asm volatile("tcgen05.wait::ld.sync.aligned;"
                       : "+r"(aw[0][0]), "+r"(aw[0][1]), "+r"(aw[1][0]), "+r"(aw[1][1]), "+r"(aw[2][0]), "+r"(aw[2][1]), "+r"(aw[3][0]), "+r"(aw[3][1]) :: "memory");
      }
      [[maybe_unused]] uint4* ag = reinterpret_cast<uint4*>(aw_g + gr * kSweepGroup + 8 * lane);
      if constexpr (WORDS == kWordsGlobal) {
        if (j > 0) {
          const uint4 lo = ag[0];
          aw[0][0] = lo.x; aw[0][1] = lo.y; aw[1][0] = lo.z; aw[1][1] = lo.w;
          if (TILES == 2 && j > 15) {
            const uint4 hi = ag[1];
            aw[2][0] = hi.x; aw[2][1] = hi.y; aw[3][0] = hi.z; aw[3][1] = hi.w;
          }
        }
      }
      if (TILES == 1 && j == 0) {
        aw[0][0] = aw[0][1] = 0u;
        aw[1][0] = aw[1][1] = g == 7 ? ~0u : 0u;
      }
      if (TILES == 2 && j == 15) {
        aw[2][0] = aw[2][1] = 0u;
        aw[3][0] = aw[3][1] = g == 7 ? ~0u : 0u;
      }
      {
        uint32_t nw[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          nw[h] = __byte_perm(__byte_perm(x[4 * h], x[4 * h + 1], sel), __byte_perm(x[4 * h + 2], x[4 * h + 3], sel), 0x5410);
#pragma unroll
        for (int q = 0; q < 2 * TILES; ++q)
          if (lane >> 2 == j - 8 * q) { aw[q][0] = nw[0]; aw[q][1] = nw[1]; }
      }
      if constexpr (WORDS == kWordsOnChip) {
        const uint32_t a = aw_tmem + (uint32_t)(gr / kSweepWarps) * 8u;
        if (TILES == 1)
          asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(aw[0][0]), "r"(aw[0][1]), "r"(aw[1][0]), "r"(aw[1][1]) : "memory");
        else
          asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                       ::"r"(a), "r"(aw[0][0]), "r"(aw[0][1]), "r"(aw[1][0]), "r"(aw[1][1]), "r"(aw[2][0]), "r"(aw[2][1]), "r"(aw[3][0]), "r"(aw[3][1]) : "memory");
      }
      __syncwarp();                                        // the bytes are there
      if constexpr (WORDS == kWordsGlobal) {               // (over column 0, whose entries every lane has used)
        ag[0] = make_uint4(aw[0][0], aw[0][1], aw[1][0], aw[1][1]);
        if (TILES == 2) ag[1] = make_uint4(aw[2][0], aw[2][1], aw[3][0], aw[3][1]);
      }
      uint32_t lo[TILES][4], hi[TILES][4];                 // (operand A's registers of bits g, g + 8, word 0, 1; low and high half bytes)
#pragma unroll
      for (int r = 0; r < TILES; ++r) {
        lo[r][0] = aw[2 * r][0]; lo[r][1] = aw[2 * r + 1][0]; lo[r][2] = aw[2 * r][1]; lo[r][3] = aw[2 * r + 1][1];
#pragma unroll
        for (int q = 0; q < 4; ++q) hi[r][q] = lo[r][q] >> 4;
      }
#pragma unroll
      for (int s2 = 0; s2 < 4; ++s2) {                     // keys of lanes 8t + 2 s2, 8t + 2 s2 + 1
        uint32_t b[4];
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(b_src + 16u * s2) : "memory");
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int s = (2 * s2 + e) & 3;
          const uint32_t m = 0x01010101u << s;
#pragma unroll
          for (int r = 0; r < TILES; ++r) {
            const uint32_t* a = s2 < 2 ? lo[r] : hi[r];
            mma_u8(acc[r][s], a[0] & m, a[1] & m, a[2] & m, a[3] & m, b[2 * e], b[2 * e + 1]);
          }
        }
      }
    }
    if (WORDS == kOneGroup) break;
  }
  if constexpr (!LAST) {
    if (WORDS == kWordsOnChip) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    if (warp < ng && t < 3) {                              // lane (g, t): columns 2t, 2t + 1 of bits g, g + 8 of a tile
#pragma unroll
      for (int r = 0; r < TILES; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const unsigned v = (8u * (unsigned)acc[r][0][q] + 4u * (unsigned)acc[r][1][q] + 2u * (unsigned)acc[r][2][q] + (unsigned)acc[r][3][q]) >> 3;
          atomicAdd(&sums[(2 * t + (q & 1)) * kSumStride + 16 * r + g + 8 * (q >> 1)], v);
        }
    }
  }
}

// arrival of this thread plus `bytes` still to come on the barrier's current phase
__device__ __forceinline__ void mbar_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bounded wait for a phase whose data other blocks of the cluster sent; false when the iteration budget runs out
__device__ __forceinline__ bool mbar_wait_cluster(unsigned long long* bar, unsigned parity, int tries) {
  for (int it = 0; it < tries; ++it) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
// asynchronous addition to rank r's copy of `dst`, counted on rank r's copy of `bar`
__device__ __forceinline__ void add_b64(const void* dst, const void* bar, int r, unsigned long long v) {
  asm volatile("{\n\t.reg .b32 d, b;\n\tmapa.shared::cluster.u32 d, %0, %2;\n\tmapa.shared::cluster.u32 b, %1, %2;\n\t"
               "red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.add.u64 [d], %3, [b];\n\t}\n"
               ::"r"(smem_u32(dst)), "r"(smem_u32(bar)), "r"(r), "l"(v) : "memory");
}
__device__ __forceinline__ void add_b32(const void* dst, const void* bar, int r, uint32_t v) {
  asm volatile("{\n\t.reg .b32 d, b;\n\tmapa.shared::cluster.u32 d, %0, %2;\n\tmapa.shared::cluster.u32 b, %1, %2;\n\t"
               "red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.add.u32 [d], %3, [b];\n\t}\n"
               ::"r"(smem_u32(dst)), "r"(smem_u32(bar)), "r"(r), "r"(v) : "memory");
}

template <int WORDS>
__global__ void __launch_bounds__(kSweepThreads, 1)
fit_sweep_kernel(float* __restrict__ T, uint32_t* __restrict__ hfit, uint32_t* __restrict__ words_g, const uint32_t* t_max,
                 const int32_t* __restrict__ unit_lens, int32_t* __restrict__ err, int n_max, int b, int blk, int t_stride, int parts,
                 int t_parts, int cluster_size, int wait_tries) {
  extern __shared__ __align__(16) unsigned char sweep_smem[];   // this block's code words (unless global)
  __shared__ __align__(16) unsigned char stage_s[kSweepWarps * kStageWarp];
  __shared__ __align__(16) uint32_t ones_s[kStageRow / 4]; // operand B's column of ones
  __shared__ unsigned sum_s[2][6 * kSumStride];            // this block's sums; two passes alternate
  // the cluster's u_i^T T (fixed point) and keys whose new bit agrees with bit i; of four passes, so that a buffer is cleared two
  // exchanges before anyone adds to it again
  __shared__ unsigned long long slot_s[4][32];
  __shared__ int slot_c[4][32];
  __shared__ unsigned long long bar_s[2];                  // the cluster's sums of this parity have arrived
  __shared__ double tot_s[32];
  __shared__ double inv_s[32][33];                         // c = inv_s * sums: the inverse of the triangle n I + (u_i . u_m), m < i
  __shared__ double agree_s[32];                           // u_j . u_m of the newest bit
  __shared__ double c_s[kTabs * kTabBits];                 // the scalars of the next column
  __shared__ float tab_s[kTabs][32];                       // and their look-up tables
  __shared__ int timed_out;
  __shared__ uint32_t tmem_base_s, max_s[kSweepWarps][kBits];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % cluster_size, unit = blockIdx.x / cluster_size;
  const int n = min(unit_lens[unit], n_max);
  if (n <= 0) { pdl_wait(); return; }                      // (the whole cluster)
  const int share = sweep_share(n, cluster_size);
  const int row0 = rank * share;
  const int nkeys = max(0, min(n - row0, share));          // keys of this block; nk = the same in whole groups
  const int nk = (nkeys + kSweepGroup - 1) / kSweepGroup * kSweepGroup;
  uint32_t* ws = WORDS != kWordsGlobal ? reinterpret_cast<uint32_t*>(sweep_smem) : words_g + (size_t)unit * t_stride + row0;
  float* Tu = T + (size_t)unit * kBits * t_stride + row0;
  SweepWarp st;
#pragma unroll
  for (int q = 0; q < kTabs; ++q) st.tab[q] = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) st.aw[q][0] = st.aw[q][1] = st.w[2 * q] = st.w[2 * q + 1] = 0u;
  if (WORDS == kWordsGlobal) pdl_wait();                   // (the words below are not this block's own memory)
  for (int i = tid; i < nk / 4; i += kSweepThreads) reinterpret_cast<uint4*>(ws)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid < kTabs * kTabBits) c_s[tid] = 0.0;
  if (tid < kStageRow / 4) ones_s[tid] = 0x01010101u;
  for (int i = tid; i < 2 * 6 * kSumStride; i += kSweepThreads) (&sum_s[0][0])[i] = 0u;
  for (int i = tid; i < 32 * 33; i += kSweepThreads) (&inv_s[0][0])[i] = 0.0;
  if (tid < 4 * 32) { (&slot_s[0][0])[tid] = 0ull; (&slot_c[0][0])[tid] = 0; }
  pdl_wait();                                              // (launched early: the columns are there)
  if (warp * kSweepGroup < nk) {
    load_entries(st.t, Tu + warp * kSweepGroup + 4 * lane);
    load_entries(st.nx, Tu + t_stride + warp * kSweepGroup + 4 * lane);
  }
  {                                                        // largest |T| of the unit's columns (lane: column), by block of the projection
    const int used = t_parts > 1 ? (n + block_rows(n, parts) - 1) / block_rows(n, parts) : 1;
    uint32_t m = 0u;
    for (int i = warp; i < used; i += kSweepWarps) m = max(m, t_max[column_max_at(unit, i, parts) + lane]);
    max_s[warp][lane] = m;
  }
  if (WORDS == kWordsOnChip && warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    timed_out = 0;
    for (int q = 0; q < 2; ++q) {
      mbar_init(&bar_s[q], 1);
      mbar_expect(&bar_s[q], (unsigned)cluster_size * 32u * 12u);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (WORDS == kWordsOnChip) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // every rank's barriers are armed
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  pdl_release();
  if (WORDS == kWordsOnChip) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  double new_row = 0.0;
  const uint32_t aw_tmem = WORDS == kWordsOnChip ? tmem_base_s + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(warp >> 2) * 128u : 0u;
  uint32_t* aw_g = reinterpret_cast<uint32_t*>(Tu);        // (column 0)
  // Fixed point: 2^(156 - e) for a column whose largest |T| is below 2^(e - 126), so that every entry is below 2^30.  Infinities and
  // NaN among the entries make the column's scalars NaN.
  int e_col = 0;                                           // e of column `lane`
#pragma unroll
  for (int w = 0; w < kSweepWarps; ++w) e_col = max(e_col, (int)(max_s[w][lane] >> 7));
  const double inv_n = 1.0 / (double)n;
  const unsigned ones_a = smem_u32(ones_s), stage_a = smem_u32(stage_s) + (unsigned)(warp * kStageWarp);
  for (int j = 0; j < kBits; ++j) {
    const int buf = j & 1, e_next = __shfl_sync(0xffffffffu, e_col, (j + 1) & 31);
#define BPC_SWEEP(TILES, LAST) sweep_pass<TILES, LAST, WORDS>(st, ws, Tu, t_stride, aw_tmem, aw_g, j, nk, e_next, warp, lane, stage_a, ones_a, sum_s[buf])
    if (j == kBits - 1) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // (this block sends no more: see the end)
      BPC_SWEEP(1, true);
      break;
    }
    if (j < 15) BPC_SWEEP(1, false);
    else BPC_SWEEP(2, false);
#undef BPC_SWEEP
    int stop = timed_out;                                  // (last set between the previous bit's barriers)
    __syncthreads();
    const unsigned phase = (unsigned)(j >> 1) & 1u;
    // Exchange within the cluster: warp r sends the block's sums to rank r; the sends complete on the receiver's barrier of this
    // parity (a rank sends bit j + 2 only after it has everybody's bit j + 1).  A block that gave up a wait sends no more (its
    // peers then miss its sums and give up in turn: every wait is bounded) and runs to the end on what it has.
    if (!stop && warp < cluster_size) {
      const unsigned* s = sum_s[buf];
      const int all = j < 15 ? 15 : 31;                    // the row of ones
      auto fixed = [&](int i) {
        return (long long)(s[i] + ((unsigned long long)s[kSumStride + i] << 8) + ((unsigned long long)s[2 * kSumStride + i] << 16) +
                           ((unsigned long long)s[3 * kSumStride + i] << 24)) - ((long long)s[4 * kSumStride + i] << 31);
      };
      int agree = nk - (int)s[4 * kSumStride + j] - (int)s[4 * kSumStride + lane] + 2 * (int)s[5 * kSumStride + lane];
      if (nkeys < nk) {                                    // take off the keys past the end
        const uint32_t wp = ws[nk - 1], same = ((wp >> j) & 1u) ? wp : ~wp;
        agree -= (nk - nkeys) * (int)((same >> lane) & 1u);
      }
      add_b64(&slot_s[j & 3][lane], &bar_s[buf], warp, (unsigned long long)(2 * fixed(lane) - fixed(all)));
      add_b32(&slot_c[j & 3][lane], &bar_s[buf], warp, (uint32_t)agree);
    }
    if (warp == 15) {                                      // (what was read before the last barrier, or two passes ago)
      for (int i = lane; i < 6 * kSumStride; i += 32) sum_s[buf ^ 1][i] = 0u;
      slot_s[(j + 2) & 3][lane] = 0ull;
      slot_c[(j + 2) & 3][lane] = 0;
    }
    // n c_{i,j+1} = u_i^T T - sum_{m<i} (u_i . u_m) c_{m,j+1}: c_i for i < j are rows of the triangle's inverse times the
    // sums, c_j follows from them (warp 0); the new bit's row of the inverse (warp 8) is needed one bit later.
    if (warp == 0 || warp == 8) {
      if (!stop && !mbar_wait_cluster(&bar_s[buf], phase, wait_tries)) stop = timed_out = 1;
      const int c = slot_c[j & 3][lane];
      const double agree = lane < j ? (double)(2 * c - n) : 0.0;         // u_j . u_lane
      if (warp == 0) {
        const double unscale = __longlong_as_double(e_next == 255 ? 0x7ff8000000000000ll : (long long)(1023 - 156 + e_next) << 52);
        const double sum = (double)(long long)slot_s[j & 3][lane] * unscale;
        tot_s[lane] = sum;
        __syncwarp();
        double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
        for (int m = 0; m < j; m += 4)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] += inv_s[lane][m + q] * tot_s[m + q];   // (zero beyond the row's own bit)
        double ci = (a[0] + a[1]) + (a[2] + a[3]);
        double x = lane < j ? agree * ci : 0.0;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == j) ci = (sum - x) * inv_n;
        c_s[lane] = lane <= j ? ci : 0.0;
      } else {
        agree_s[lane] = agree;
        __syncwarp();
        double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
        for (int k = 0; k < j; k += 4)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] += agree_s[k + q] * inv_s[k + q][lane];    // (rows from j on are zero)
        new_row = lane == j ? inv_n : -((a[0] + a[1]) + (a[2] + a[3])) * inv_n;
      }
    }
    if (tid == 0 && !stop) mbar_expect(&bar_s[buf], (unsigned)cluster_size * 32u * 12u);   // arms the barrier for bit j + 2
    // The tables in play, one to a warp: entries are sums of the fp64 scalars, rounded once.
    if (warp < kTabs) {
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kTabs) : "memory");
      if (kTabBits * warp <= j) {
        const double* cv = c_s + kTabBits * warp;
        double v[kTabBits];
#pragma unroll
        for (int k = 0; k < kTabBits; ++k) v[k] = ((lane >> k) & 1) ? cv[k] : -cv[k];
        tab_s[warp][lane] = (float)(((v[0] + v[1]) + (v[2] + v[3])) + v[4]);
      }
    }
    __syncthreads();
    if (warp == 8) inv_s[j][lane] = new_row;               // (read again behind the next pass's barrier)
#pragma unroll
    for (int q = 0; q < kTabs; ++q)
      if (kTabBits * q <= j) st.tab[q] = tab_s[q][lane];
  }
  if (WORDS == kWordsOnChip) asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (WORDS == kWordsOnChip && warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base_s), "r"(512) : "memory");
  }
  uint32_t* h = hfit + ((size_t)unit * n_max + row0) * (b / 32) + blk;
  for (int i = tid; i < nkeys; i += kSweepThreads) h[(size_t)i * (b / 32)] = ws[i];
  // No block leaves while a peer may still send to it.  With all sums received nothing is under way; a block that gave up a wait
  // leaves what was sent to it before this barrier the time to land (microseconds).
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (timed_out) {
    if (tid == 0) atomicOr(err, BPC_DEVERR_TIMEOUT);
    for (int i = 0; i < 100; ++i) __nanosleep(1000);
  }
}

// --------------------------------------------------------------------------- rows and scalars
// The blocks' partial sums of a unit, added in block order into the first block's place; grid (16 + 4 (blk + 1), units), one
// sum per thread (the loads are independent: a latency or two in all).
__global__ void __launch_bounds__(256)
fit_sum_parts_kernel(double* __restrict__ wpart, int32_t* __restrict__ apart, const int32_t* __restrict__ unit_lens, int n_max, int b,
                     int blk, int parts) {
  pdl_wait();
  pdl_release();
  const int unit = blockIdx.y;
  const int n = min(unit_lens[unit], n_max);
  if (n <= 0) return;
  const int rows = block_rows(n, parts), used = (n + rows - 1) / rows;
  if (blockIdx.x < 16) {
    double* w = wpart + (size_t)unit * parts * kBits * BPC_D + blockIdx.x * 256 + threadIdx.x;
    double s = w[0];
#pragma unroll 16
    for (int p = 1; p < used; ++p) s += w[(size_t)p * kBits * BPC_D];
    w[0] = s;
  } else {
    const int e = (blockIdx.x - 16) * 256 + threadIdx.x, nj = kBits * (blk + 1);
    int32_t* a = apart + (size_t)unit * parts * kBits * b + (size_t)(e / nj) * b + e % nj;
    int s = a[0];
#pragma unroll 16
    for (int p = 1; p < used; ++p) s += a[(size_t)p * kBits * b];
    a[0] = s;
  }
}

// v_i = (W_i - sum_{j<i} (u_i . u_j) v_j) / n for the block's 32 bits; grid (4, units), a block has 32 channels.  Thread
// (row pair, channel) takes off the earlier blocks' rows, then one warp runs the block's own triangle in registers.
__global__ void __launch_bounds__(512)
fit_rows_kernel(const double* wpart, const int32_t* apart, float* __restrict__ P,
                const int32_t* __restrict__ unit_lens, int n_max, int b, int blk, int parts) {
  pdl_wait();
  pdl_release();
  extern __shared__ __align__(16) double rows_smem[];
  const int nj = kBits * (blk + 1), np = kBits * blk;
  double* corr = rows_smem;                                // [32][nj] u_i . u_j
  double* v_s = corr + kBits * nj;                         // [np][32] earlier rows, this block's channels
  double* w_s = v_s + (size_t)np * 32;                     // [32][32]
  const int unit = blockIdx.y, tid = threadIdx.x, lane = tid & 31, r = tid >> 5, c = 32 * blockIdx.x + lane;
  const int n = min(unit_lens[unit], n_max);
  float* Pu = P + (size_t)unit * b * BPC_D;
  if (n <= 0) {
    for (int i = r; i < kBits; i += 16) Pu[(size_t)(np + i) * BPC_D + c] = 0.f;
    return;
  }
  const double* w = wpart + (size_t)unit * parts * kBits * BPC_D;
  const int32_t* a = apart + (size_t)unit * parts * kBits * b;
  double acc[2][2] = {{w[(size_t)r * BPC_D + c], 0.0}, {w[(size_t)(r + 16) * BPC_D + c], 0.0}};
  for (int e = tid; e < kBits * nj; e += 512) corr[e] = (double)a[(size_t)(e / nj) * b + e % nj];
  for (int j = r; j < np; j += 16) v_s[j * 32 + lane] = (double)Pu[(size_t)j * BPC_D + c];
  __syncthreads();
#pragma unroll 4
  for (int j = 0; j < np; j += 2) {
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const double v = v_s[(j + o) * 32 + lane];
      acc[0][o] -= corr[r * nj + j + o] * v;
      acc[1][o] -= corr[(r + 16) * nj + j + o] * v;
    }
  }
  w_s[r * 32 + lane] = acc[0][0] + acc[0][1];
  w_s[(r + 16) * 32 + lane] = acc[1][0] + acc[1][1];
  __syncthreads();
  if (r != 0) return;
  double x[kBits];
#pragma unroll
  for (int i = 0; i < kBits; ++i) x[i] = w_s[i * 32 + lane];
  const double inv_n = 1.0 / (double)n;
#pragma unroll
  for (int i = 0; i < kBits; ++i) {
    const float v = (float)(x[i] * inv_n);
    Pu[(size_t)(np + i) * BPC_D + c] = v;
#pragma unroll
    for (int k = i + 1; k < kBits; ++k) x[k] -= corr[k * nj + np + i] * (double)v;
  }
}

// The same in one launch, for a few units (see bpc_launch_fit_blocked): a cluster per unit adds the partial sums, forms the rows and then
// the next block's scalars C = V D_next^T.  Block r of the cluster owns 16 channels of the rows, 1 / 8 of the inner products (sums sent to
// every block) and 1 / 8 of the scalars.  Nothing here is limited by a rate of the chip but by a launch, a round of loads, two cluster
// barriers and a chain of 32 FMAs, so every load is requested at the start, and both contractions take four rows per thread
// and split their sums over the warps (with one output per thread they were bound by shared-memory reads, two per FMA).  Three kernels
// take 21 to 27 us per 32 bits of 8 x 32K keys, this one 12 to 15.
// The rows of the block enter each other's corrections in fp64, before they are rounded.
constexpr int kFinishBlocks = 8;
constexpr int kFinishThreads = 512;
constexpr int kFinishChannels = BPC_D / kFinishBlocks;
constexpr int kFinishRows = kBits / kFinishBlocks;         // rows of inner products, and per 32 bits so far of scalars, of a block
constexpr int kFinishSlices = 4;                           // of the sum over the earlier rows
constexpr int kDirStride = BPC_D + 1, kRowStride = kFinishChannels + 1;
static_assert(kBits * kFinishChannels == kFinishThreads && kFinishChannels == kFinishThreads / 32, "a thread per row and channel; a warp per channel");
static_assert(kFinishRows == 4 && kFinishThreads / 32 == 16, "four rows per thread, sums split over the warps");

struct FinishSmem {                                        // (doubles)
  int corr, v, w, d, p, part, total;                       // u_i . u_j over n; earlier rows, own channels; sums; next directions; rows of the own scalars; partial sums
  __host__ __device__ explicit FinishSmem(int blk) {
    corr = 0;                                              // [32][32 (blk + 1) + 2]
    v = corr + kBits * (kBits * (blk + 1) + 2);            // [32 blk][16]
    w = v + kBits * blk * kFinishChannels;                 // [4][32][17]
    d = w + kFinishSlices * kBits * kRowStride;            // [32][129]
    p = d + kBits * kDirStride;                            // [4 (blk + 1)][128]
    part = p + kFinishRows * (blk + 1) * BPC_D;            // [16 warps][4][32]
    total = part + 16 * kFinishRows * kBits;
  }
};

__device__ __forceinline__ void store_peer(const double* dst, int r, double v) {
  asm volatile("{\n\t.reg .b32 d;\n\tmapa.shared::cluster.u32 d, %0, %1;\n\tst.shared::cluster.f64 [d], %2;\n\t}\n" ::"r"(smem_u32(dst)), "r"(r), "d"(v) : "memory");
}

__global__ void __cluster_dims__(kFinishBlocks, 1, 1) __launch_bounds__(kFinishThreads, 1)
fit_finish_kernel(const double* wpart, const int32_t* apart, const float* __restrict__ v_star, float* __restrict__ P,
                  float* __restrict__ cross, const int32_t* __restrict__ unit_lens, int n_max, int b, int blk, int parts) {
  extern __shared__ __align__(16) double finish_smem[];
  const FinishSmem at(blk);
  const int nj = kBits * (blk + 1), np = kBits * blk, cstride = nj + 2;
  double *corr = finish_smem + at.corr, *v_s = finish_smem + at.v, *w_s = finish_smem + at.w, *d_s = finish_smem + at.d, *p_s = finish_smem + at.p,
         *part_s = finish_smem + at.part;
  const int rank = blockIdx.x % kFinishBlocks, unit = blockIdx.x / kFinishBlocks, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i = tid / kFinishChannels, c = tid % kFinishChannels;        // this thread's row and channel
  const int n = min(unit_lens[unit], n_max);
  float* Pu = P + (size_t)unit * b * BPC_D;
  if (n <= 0) {                                            // (the whole cluster)
    pdl_wait();
    Pu[(size_t)(np + i) * BPC_D + kFinishChannels * rank + c] = 0.f;
    return;
  }
  const bool last = nj == b;                               // no further block
  const int rows = block_rows(n, parts), used = (n + rows - 1) / rows;
  const double inv_n = 1.0 / (double)n;
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  constexpr int kDirs = kBits * BPC_D / kFinishThreads;
  float dir[kDirs];
  if (!last) {
#pragma unroll
    for (int k = 0; k < kDirs; ++k) dir[k] = v_star[((size_t)unit * b + nj) * BPC_D + tid + k * kFinishThreads];
  }
  pdl_wait();                                              // (the lengths and directions are older than the kernel before)
  pdl_release();
  const double* w = wpart + (size_t)unit * parts * kBits * BPC_D + (size_t)i * BPC_D + kFinishChannels * rank + c;
  double ws = w[0];
#pragma unroll 16
  for (int p = 1; p < used; ++p) ws += w[(size_t)p * kBits * BPC_D];
  const int32_t* a = apart + ((size_t)unit * parts * kBits + kFinishRows * rank) * b;   // inner products of rows 4 rank .. 4 rank + 3
  auto product = [&](int e) {
    int s = 0;
#pragma unroll 16
    for (int p = 0; p < used; ++p) s += a[(size_t)p * kBits * b + (size_t)(e / nj) * b + e % nj];
    return s;
  };
  const int first = tid < kFinishRows * nj ? product(tid) : 0;
  for (int j = i; j < np; j += kBits) v_s[j * kFinishChannels + c] = (double)Pu[(size_t)j * BPC_D + kFinishChannels * rank + c];
  if (!last) {
#pragma unroll
    for (int k = 0; k < kDirs; ++k) {
      const int e = tid + k * kFinishThreads;
      d_s[(e >> 7) * kDirStride + (e & 127)] = (double)dir[k];
    }
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");    // (every block of the cluster runs: its shared memory may be written)
  for (int e = tid; e < kFinishRows * nj; e += kFinishThreads) {
    const double v = (double)(e == tid ? first : product(e)) * inv_n;
#pragma unroll
    for (int q = 0; q < kFinishBlocks; ++q) store_peer(corr + (size_t)(kFinishRows * rank + e / nj) * cstride + e % nj, q, v);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  {                                                        // earlier rows: four rows and a quarter of the sum per thread
    const int slice = tid >> 7, r0 = 4 * ((tid >> 4) & 7);
    double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (int j = slice * (np / kFinishSlices); j < (slice + 1) * (np / kFinishSlices); j += 2) {
      const double v0 = v_s[j * kFinishChannels + c], v1 = v_s[(j + 1) * kFinishChannels + c];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double2 k = *reinterpret_cast<const double2*>(corr + (r0 + q) * cstride + j);
        x[q] = fma(k.x, v0, x[q]);
        x[q] = fma(k.y, v1, x[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) w_s[(slice * kBits + r0 + q) * kRowStride + c] = x[q];
    __syncthreads();
    const double* y = w_s + i * kRowStride + c;
    const double sum = (y[0] + y[kBits * kRowStride]) + (y[2 * kBits * kRowStride] + y[3 * kBits * kRowStride]);
    w_s[i * kRowStride + c] = fma(ws, inv_n, -sum);        // (its own place; the other slices are not read again)
  }
  __syncthreads();
  {                                                        // the block's own triangle: a warp per channel, a row per lane
    double x = w_s[lane * kRowStride + warp];
    const double* col = corr + (size_t)lane * cstride + np;
#pragma unroll 4
    for (int k = 0; k < kBits; ++k) {
      const double v = __shfl_sync(0xffffffffu, x, k);
      if (lane > k) x = fma(-col[k], v, x);
    }
    Pu[(size_t)(np + lane) * BPC_D + kFinishChannels * rank + warp] = (float)x;
  }
  if (last) return;                                        // (nobody writes to another block any more)
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");    // the unit's new rows are in memory
  const int groups = blk + 1;                              // of four rows: this block's scalars
  for (int e = tid; e < kFinishRows * groups * BPC_D; e += kFinishThreads) p_s[e] = (double)__ldcg(Pu + (size_t)kFinishRows * groups * rank * BPC_D + e);
  __syncthreads();
  const int slices = 16 / groups, slice = warp / groups, grp = warp % groups;   // (warps beyond groups x slices: none)
  if (slice < slices) {
    const int k0 = BPC_D * slice / slices & ~1, k1 = BPC_D * (slice + 1) / slices & ~1;
    double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (int k = k0; k < k1; k += 2) {
      const double d0 = d_s[lane * kDirStride + k], d1 = d_s[lane * kDirStride + k + 1];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double2 v = *reinterpret_cast<const double2*>(p_s + (4 * grp + q) * BPC_D + k);
        x[q] = fma(v.x, d0, x[q]);
        x[q] = fma(v.y, d1, x[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) part_s[(warp * 4 + q) * kBits + lane] = x[q];
  }
  __syncthreads();
  for (int e = tid; e < kFinishRows * groups * kBits; e += kFinishThreads) {   // row e / 32 of the block's, column e % 32
    const int q = e >> 5;
    double s = 0.0;
    for (int sl = 0; sl < slices; ++sl) s += part_s[((sl * groups + (q >> 2)) * 4 + (q & 3)) * kBits + (e & 31)];
    cross[((size_t)unit * b + kFinishRows * groups * rank) * kBits + e] = (float)s;
  }
}

// --------------------------------------------------------------------------- host side
constexpr int kSms = 148;
constexpr int kSweepMaxKeys = 1 << 24;                     // keys of a sweep block
constexpr size_t kSweepMaxSmem = 186 * 1024;               // dynamic shared memory of a sweep block: its code words

constexpr size_t kMaxSmem = 226 * 1024;                    // dynamic shared memory a block may ask for next to its static part
// The limit of a kernel belongs to the process: one value for every launch, whatever it needs, so that a thread's launch does
// not fall between another's lower limit and that one's launch.
template <typename K>
cudaError_t allow_smem(K* kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem); }
// tiles, signs of 32 (blk + 1) bits, room for the last A operand (128 rows a half) to reach past its signs, and alignment
inline size_t gather_smem(int groups, int blk) {
  return (size_t)groups * (kTileBytes + (size_t)kBits * (blk + 1) * kTileKeys * 2) + (size_t)(2048 * (blk / 4 + 1) - 512 * (blk + 1)) + 1024;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
inline int t_stride_of(const bpc_config* c) { return sweep_share(c->n_max, 1); }

// Blocks per unit of project and gather (one block per SM): the first count from one wave up whose last wave is at least
// 90 % full (32 units: 9, 8 units: 18, 128 units: 8), not below 384 keys per block.
int parts_of(const bpc_config* c) {
  const int units = c->batch * c->n_kv_heads;
  int p = kSms / units > 0 ? kSms / units : 1;
  for (int tries = 0; tries < 16; ++tries) {
    const int rem = (int)(((long long)units * p) % kSms);
    if (rem == 0 || rem * 10 >= kSms * 9) break;
    ++p;
  }
  const int most = (c->n_max + 383) / 384;
  return p < most ? p : most;
}

struct Layout {
  size_t t, words, wpart, apart, cross, total;
  explicit Layout(const bpc_config* c) {
    const size_t units = (size_t)c->batch * c->n_kv_heads, ts = t_stride_of(c), parts = parts_of(c);
    t = 0;
    words = align256(units * kBits * ts * 4);
    wpart = words + align256(units * ts * 4);
    apart = wpart + align256(units * parts * kBits * BPC_D * 8);
    cross = apart + align256(units * parts * kBits * c->code_bits * 4);
    total = cross + align256(units * c->code_bits * kBits * 4);
  }
};

// Resident sweep clusters by size on a device (the kernel takes a whole SM per block, so this depends on nothing else);
// asked for until it succeeds, then kept.  The kernel after the gather is such a kernel too.
struct SweepLimits {
  std::mutex lock;
  bool known;
  int active[BPC_MAX_CLUSTER + 1];
};
SweepLimits g_sweep_limits[64];

cudaLaunchConfig_t sweep_config(cudaLaunchAttribute* attr, int units, int cs, size_t smem, cudaStream_t stream, bool early = false) {   // (two attributes)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * cs));
  cfg.blockDim = dim3(kSweepThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cs;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (early) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  return cfg;
}

cudaError_t sweep_limits(int device, const SweepLimits** out) {
  if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
  SweepLimits* l = &g_sweep_limits[device];
  *out = l;
  std::lock_guard<std::mutex> hold(l->lock);
  if (l->known) return cudaSuccess;
  const void* kernels[3] = {(const void*)fit_sweep_kernel<kOneGroup>, (const void*)fit_sweep_kernel<kWordsOnChip>, (const void*)fit_sweep_kernel<kWordsGlobal>};
  for (const void* k : kernels) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSweepMaxSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  for (int cs = 1; cs <= BPC_MAX_CLUSTER; ++cs) {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg = sweep_config(&attr, 1, cs, kSweepMaxSmem, nullptr);
    if (cudaOccupancyMaxActiveClusters(&l->active[cs], fit_sweep_kernel<kWordsOnChip>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      l->active[cs] = 0;
    }
    l->known = l->known || l->active[cs] > 0;
  }
  return l->known ? cudaSuccess : cudaErrorInvalidConfiguration;
}

// Cluster size of the sweep: the smallest estimate, in microseconds per 32 bits, of waves x (groups of keys per block + the exchanges,
// which grow with the ranks).  With at most one group per warp the first groups hide behind each other's latencies (1.3 each to two
// per scheduler, 3.1 from there); several groups per warp are issue-bound at 2.13 each, half as much again with the words in global
// memory.  Measured against every size from 1 to 16 on fifteen shapes of 1 to 128 units and 4K to 256K keys: the estimate picks the
// fastest or one within 3 %.
// No block takes more than 2^24 keys: the sums of their bytes are 32 bits wide.
int sweep_cluster(const bpc_config* c, const int* active) {
  const int units = c->batch * c->n_kv_heads;
  double best_cost = 0.0;
  int best = 0;
  for (int cs = 1; cs <= BPC_MAX_CLUSTER; ++cs) {
    const int nk = sweep_share(c->n_max, cs), groups = nk / kSweepGroup;
    if (active[cs] < 1 || nk > kSweepMaxKeys) continue;
    const int waves = (units + active[cs] - 1) / active[cs];
    const double words = (size_t)nk * 4 > kSweepMaxSmem ? 1.5 : 1.0;
    const double keys = groups > kSweepWarps ? 2.13 * words * groups + 56.0
                                             : 1.3 * (groups < 4 ? 4 : groups) + 1.8 * (groups < 8 ? 0 : groups - 8) + 50.0;
    const double cost = waves * (keys + 0.7 * cs);
    if (best_cost == 0.0 || cost < best_cost) { best_cost = cost; best = cs; }
  }
  return best;
}

template <int GROUPS>
cudaError_t launch_project_tc(const bpc_ctx* ctx, const CUtensorMap& kmap, const uint32_t* hfit, const float* v_star, const float* cross, float* T,
                              uint32_t* t_max, int blk, int parts, int ts, bool early, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  const size_t smem = (size_t)GROUPS * (kTileBytes + kTileKeys * kSignCols * 2) + (size_t)kProjN * 256 + (size_t)blk * kProjN * 64 + 1024;
  cudaError_t e = allow_smem(fit_project_tc_kernel<GROUPS>);
  if (e != cudaSuccess) return e;
  return launch_pdl(early, fit_project_tc_kernel<GROUPS>, dim3(parts, ctx->units), kGroupThreads * GROUPS, smem, stream, kmap, hfit, v_star, cross, T, t_max,
                      (const int32_t*)ctx->unit_lens, ctx->dev_err, (int)c.n_max, (int)c.code_bits, blk, ts);
}

template <int GROUPS>
cudaError_t launch_gather_tc(const bpc_ctx* ctx, const CUtensorMap& kmap, const uint32_t* hfit, double* wpart, int32_t* apart, int blk, int parts,
                             bool early, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  const size_t smem = gather_smem(GROUPS, blk);
  cudaError_t e = allow_smem(fit_gather_tc_kernel<GROUPS>);
  if (e != cudaSuccess) return e;
  return launch_pdl(early, fit_gather_tc_kernel<GROUPS>, dim3(parts, ctx->units), kGroupThreads * GROUPS, smem, stream, kmap, hfit, wpart, apart,
                      (const int32_t*)ctx->unit_lens, ctx->dev_err, (int)c.n_max, (int)c.code_bits, blk);
}

}  // namespace

size_t bpc_fit_blocked_bytes(const bpc_config* c) { return Layout(c).total; }

int bpc_fit_sweep_cluster(const bpc_config* c, const int* active) { return sweep_cluster(c, active); }

cudaError_t bpc_launch_fit_blocked(bpc_ctx* ctx, const void* k_cache, const float* v_star, uint32_t* hfit, unsigned char* ws,
                                   cudaStream_t stream, int* launches) {
  const bpc_config& c = ctx->cfg;
  const Layout lay(&c);
  float* T = (float*)(ws + lay.t);
  uint32_t* words_g = (uint32_t*)(ws + lay.words);
  double* wpart = (double*)(ws + lay.wpart);
  int32_t* apart = (int32_t*)(ws + lay.apart);
  float* cross = (float*)(ws + lay.cross);
  uint32_t* t_max = (uint32_t*)wpart;                      // (see column_max_at)
  const int ts = t_stride_of(&c), parts = parts_of(&c), b = c.code_bits;
  const SweepLimits* lim = nullptr;
  cudaError_t e = sweep_limits(ctx->device, &lim);
  if (e != cudaSuccess) return e;
  const int cs = sweep_cluster(&c, lim->active);
  if (cs == 0) return cudaErrorNotSupported;
  const size_t sweep_smem = (size_t)sweep_share(c.n_max, cs) * 4;
  const bool tc = c.kv_dtype == BPC_BF16;
  // One kernel after the gather while all its clusters are resident at once: like the sweep it takes an SM per block, so the sweep's limit is
  // its own (15 clusters of eight on a B200).  Three kernels -> one, 128 bits, early launches: 32K keys 8 units 537 -> 511 us, 12 605 -> 595,
  // 15 658 -> 644, but 16 785 -> 812 and 20 847 -> 871; 2K keys 8 units 329 -> 312, 15 329 -> 317, but 16 331 -> 355.  32 and 256 bits: the
  // same line (15 units of 32K keys 158 -> 157 and 1546 -> 1518, 16 189 -> 195 and 1806 -> 1880).
  const bool one_finish = ctx->units <= lim->active[kFinishBlocks];
  // Each kernel is launched to start while the one before it drains: what it can set up, and request, lies before its wait.  (fp32 caches: their
  // project and gather do not wait.)  Fits of 32K keys and 128 bits: 4 units 502 -> 461 us, 8 units 575 -> 535, 16 units 849 -> 809,
  // 32 units 1183 -> 1171.
  const bool early = tc && ctx->use_pdl;
  const dim3 grid(parts, ctx->units);
  CUtensorMap kmap;
  if (tc) e = tma::make_key_map(&kmap, k_cache, (unsigned long long)ctx->units * c.n_max, ctx->row_stride);
  for (int blk = 0; blk < b / kBits && e == cudaSuccess; ++blk) {
    if (blk > 0 && !one_finish) {                          // cross[j][l] = v_j . d_l for the bits so far and this block's columns
      const size_t set = (size_t)b * BPC_D;
      e = bpc_launch_dots(ctx->P, set, v_star + (size_t)kBits * blk * BPC_D, set, cross, (size_t)b * kBits, kBits, blk, 1, ctx->units, early, stream);
      if (e != cudaSuccess) return e;
    }
    if (tc) {
      // three warpgroups while the scalars of the earlier bits leave room for them (up to five earlier words)
      e = blk <= 5 ? launch_project_tc<3>(ctx, kmap, hfit, v_star, cross, T, t_max, blk, parts, ts, early && blk > 0, stream)
                   : launch_project_tc<2>(ctx, kmap, hfit, v_star, cross, T, t_max, blk, parts, ts, early && blk > 0, stream);
    } else {
      e = cudaMemset2DAsync(t_max, column_max_at(1, 0, parts) * 4, 0, kBits * 4, ctx->units, stream);
      if (e != cudaSuccess) return e;
      e = launch_pdl(false, fit_project_f32_kernel, dim3(ts / kTileKeys, ctx->units), kTileKeys, 0, stream, (const float*)k_cache, hfit, v_star, cross, T,
                     t_max, ctx->unit_lens, c.n_max, ctx->row_stride, b, blk, ts, parts);
    }
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2];
    const bool words_fit = sweep_smem <= kSweepMaxSmem, one = sweep_share(c.n_max, cs) <= kSweepWarps * kSweepGroup;
    cudaLaunchConfig_t cfg = sweep_config(attr, ctx->units, cs, words_fit ? sweep_smem : 0, stream, early);
    auto sweep = !words_fit ? fit_sweep_kernel<kWordsGlobal> : one ? fit_sweep_kernel<kOneGroup> : fit_sweep_kernel<kWordsOnChip>;
    e = cudaLaunchKernelEx(&cfg, sweep, T, hfit, words_g, (const uint32_t*)t_max, (const int32_t*)ctx->unit_lens, ctx->dev_err, (int)c.n_max, b, blk,
                           ts, parts, tc ? parts : 1, cs, ctx->wait_tries);
    if (e != cudaSuccess) return e;
    if (tc) {
      // as many warpgroups as their tile and sign buffers leave room for (four up to the third word, two from the sixth)
      if (gather_smem(4, blk) <= kMaxSmem) e = launch_gather_tc<4>(ctx, kmap, hfit, wpart, apart, blk, parts, early, stream);
      else if (gather_smem(3, blk) <= kMaxSmem) e = launch_gather_tc<3>(ctx, kmap, hfit, wpart, apart, blk, parts, early, stream);
      else e = launch_gather_tc<2>(ctx, kmap, hfit, wpart, apart, blk, parts, early, stream);
    } else {
      e = launch_pdl(false, fit_gather_f32_kernel, grid, 256, 0, stream, (const float*)k_cache, hfit, wpart, apart, ctx->unit_lens, c.n_max, ctx->row_stride,
                     b, blk);
    }
    if (e != cudaSuccess) return e;
    if (one_finish) {
      e = allow_smem(fit_finish_kernel);
      if (e != cudaSuccess) return e;
      e = launch_pdl(early, fit_finish_kernel, dim3(kFinishBlocks * ctx->units), kFinishThreads, FinishSmem(blk).total * sizeof(double), stream,
                       (const double*)wpart, (const int32_t*)apart, v_star, ctx->P, cross, (const int32_t*)ctx->unit_lens, (int)c.n_max, b, blk, parts);
      *launches += 4;
      continue;
    }
    e = launch_pdl(early, fit_sum_parts_kernel, dim3(16 + 4 * (blk + 1), ctx->units), 256, 0, stream, wpart, apart, ctx->unit_lens, c.n_max, b, blk, parts);
    if (e != cudaSuccess) return e;
    const size_t rows_smem = (size_t)(kBits * kBits * (blk + 1) + kBits * blk * 32 + kBits * 32) * 8;
    e = allow_smem(fit_rows_kernel);
    if (e != cudaSuccess) return e;
    e = launch_pdl(early, fit_rows_kernel, dim3(4, ctx->units), 512, rows_smem, stream, wpart, apart, ctx->P, ctx->unit_lens, c.n_max, b, blk, parts);
    *launches += blk > 0 ? 6 : 5;
  }
  return e;
}

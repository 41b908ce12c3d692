// Tensor-core encode: Algorithm 2 for all cached keys of bf16 caches.
//
// The decision values before any correction are a dense contraction T = K P_h^T (keys x channels times
// channels x bits).  It runs on the 5th-generation tensor cores: per warpgroup, tiles of 128 keys (M = 128) against
// the unit's b projection rows (N = b: 32, 64 or 128) over the 128 channels (eight tcgen05.mma steps of K = 16), bf16
// operands in shared memory in the 128-byte-swizzled K-major layout, fp32 accumulator in tensor memory with one
// key per TMEM lane.  Algorithm 2's greedy sweep in its Gram form,
//     u_i = sign(t_i);  t_j -= u_i * G_ij  (j > i),   G = P_h P_h^T,
// (equal to updating the residual r <- r - u_i P_i and testing r . P_{i+1}) is blocked by 16 bits.  Inside a block the
// 16 sign decisions are sequential: each thread pulls its key's 16 decision values out of tensor memory (tcgen05.ld)
// and sweeps them in registers (120 FMAs).  The corrections of all LATER columns by those 16 signs are again a dense
// contraction, T[:, later] -= U (128 keys x 16 signs) G[block, later], and go to the tensor cores too: the signs are
// written over the block's own accumulator columns as a bf16 operand in tensor memory (+-1 is exact), the Gram rows are
// kept as three bf16 terms whose sum carries 24 mantissa bits (so the products are exact and the fp32 accumulation in
// tensor memory sees what an fp32 FMA chain would see up to rounding), and three small MMAs (one per term, K = 16)
// accumulate straight into the accumulator columns that still wait for their decisions.  That leaves 960 of the 8 128
// sign-dependent FMAs per key (128 bits) on the CUDA cores.  The small operands use the K-major layout without swizzle
// (8-row x 16-byte core matrices; leading-dimension offset = distance between core matrices along K, stride offset = 128
// bytes along M/N).
// A block holds four warpgroups of one tile each (tensor memory holds four accumulators of 128 columns), which share the
// projection rows and the Gram operands in shared memory and otherwise run independent pipelines (own key tile, own
// accumulator columns, own mbarrier, own hardware barrier), so that one warpgroup's sweep covers the others' MMA round
// trips; the next key tile of a warpgroup is copied in while it sweeps.  Measured at 32 x 128K keys, 128 bits: blocks of 32
// bits and three warpgroups with the signs in shared memory 1114 us, two warpgroups of two tiles with paired FMAs 874 us
// (a paired FMA with three different operands issues every four cycles, no faster than two single ones), this form 669 us.
//
// Waits on the MMA-completion mbarrier are bounded: on expiry the block raises the device error word, still
// releases its tensor memory and returns.
#include <stdlib.h>
#include "tma.cuh"

namespace {
using namespace umma;

constexpr int kTileKeys = 128;
constexpr int kGroupThreads = 128;   // a warpgroup: one TMEM lane per thread
constexpr int kGroups = 4;           // warpgroups per block, each with its own tile, accumulator columns and barrier
constexpr int kSub = 16;             // bits of a sweep block
// 256-bit codes run as two launches over 128 bits each.  HALF = 0: the code is NBITS long.  HALF = 1: bits 0..127 of a
// 256-bit code (projection rows 0..127, Gram block G[0:128, 0:128], code words 0..3 of 8).  HALF = 2: bits 128..255; their
// decision values start from P_h[128 + j] . k - sum_{i < 128} u_i G[i][128 + j], and that sum over the first half's signs
// (read back from the code words the first launch wrote) is one more contraction on the tensor cores, U1 (128 keys x
// 128 signs) times -G[0:128, 128:256] as three bf16 terms (96 KB of shared memory: one warpgroup per block then).
constexpr int kCrossBytes = 3 * 128 * 128 * 2;

// Gram terms of the corrections: three bf16 operands [columns after block p x 16] for every block p but the last
__host__ __device__ constexpr size_t gram_off(int bits, int p) { return (size_t)3 * 2 * kSub * (size_t)(p * bits - kSub * p * (p + 1) / 2); }
__host__ __device__ constexpr size_t gram_bytes(int bits) { return gram_off(bits, bits / kSub - 1); }

// Further warpgroups of a block that only take part in its set-up: the second launch of 256-bit codes has 128 x 128 cross terms
// to split in three, which one warpgroup needed some 70 us for.
__host__ __device__ constexpr int setup_groups(int half) { return half == 2 ? 2 : 0; }

// barrier among the 128 threads of one warpgroup (hardware barriers 1 .. kGroups; 0 is __syncthreads)
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kGroupThreads) : "memory"); }

// 16 consecutive accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&t)[kSub]) {
  uint32_t r[kSub];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < kSub; ++i) t[i] = __uint_as_float(r[i]) + 0.f;   // (-0 becomes 0)
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n\ttcgen05.wait::st.sync.aligned;"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

// Greedy sweep of one 16-bit column block held in registers (every index a compile-time constant).  On entry t already
// carries the corrections of all earlier blocks (no value is -0); on exit bit I of `word` is 1 where decision I came out
// positive or zero.  A NaN is not >= 0: the addition carries the canonical NaN, and nothing else, over into the sign bit
// (comparisons instead cost 1 % of the encode, NaN replaced on the way out of tensor memory 7 %).
template <int I, bool ERR>
__device__ __forceinline__ void diag_sweep(float (&t)[kSub], uint32_t& word, float& abs_sum, const float* g_diag) {
  if constexpr (I < kSub) {
    const uint32_t v = __float_as_uint(t[I]) + 0x007FFFFFu;
    word = __funnelshift_l(v, word, 1);                        // collects the sign bits, first decision on top
    if (ERR) abs_sum += fabsf(t[I]);
    const float nu = __uint_as_float((v & 0x80000000u) ^ 0xBF800000u);       // -u
    // row I of the diagonal block, columns after I: 16-byte broadcast reads
    const float4* gi = reinterpret_cast<const float4*>(g_diag + I * kSub);
#pragma unroll
    for (int j4 = (I + 1) / 4; j4 < kSub / 4; ++j4) {
      const float4 g = gi[j4];
      const float ge[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (4 * j4 + e > I) t[4 * j4 + e] = fmaf(nu, ge[e], t[4 * j4 + e]);
    }
    diag_sweep<I + 1, ERR>(t, word, abs_sum, g_diag);
  } else {
    word = (~__brev(word)) >> (32 - kSub);
  }
}

template <int NBITS, int GROUPS, int HALF, bool ERR>
__global__ void __launch_bounds__(kGroupThreads * (GROUPS + setup_groups(HALF)), 1)
encode_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __nv_bfloat16* Ph, const float* gram,
                 const int32_t* unit_lens, uint64_t* __restrict__ codes, int32_t* __restrict__ err,
                 int n_kv_heads, int n_max, int shared_sets, int residual_correction, int blocks_per_unit,
                 float* __restrict__ key_err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the swizzled operand tiles need 1024-byte alignment in the shared address space
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  constexpr int kGroups = GROUPS;                          // (shadows the default of the single-launch code lengths)
  constexpr int kThreads = kGroupThreads * (GROUPS + setup_groups(HALF));   // (the last ones only help with the set-up)
  static_assert(HALF == 0 || NBITS == 128, "the two-launch form is for 256-bit codes");
  constexpr int TOTAL = HALF == 0 ? NBITS : 256;           // bits of a whole code
  constexpr int ROW0 = HALF == 2 ? 128 : 0;                // first projection row (= first bit) of this launch
  constexpr int NB = NBITS / 32;                           // code words of this launch
  constexpr int NS = NBITS / kSub;                         // column blocks
  constexpr int NWK = TOTAL / 32;                          // code words per key
  constexpr int A_BYTES = kTileKeys * 256;                 // one key tile (128 rows x 128 bf16)
  constexpr int B_BYTES = NBITS * 256;                     // the projection rows
  constexpr int GD_BYTES = NS * kSub * kSub * 4;           // diagonal blocks of the Gram matrix, fp32
  // one bf16 term of -G[rows of block pb][columns after block pb] is an operand [NBITS - 16 (pb + 1) x 16]; the three
  // terms of block pb start at gb_off(pb)
  constexpr unsigned U_LBO = (kTileKeys / 8) * 128;        // bytes between core matrices along K of a [128 x K] operand
  const int tid = threadIdx.x, warp = tid >> 5;
  const int grp = tid / kGroupThreads, gtid = tid % kGroupThreads;   // warpgroup and thread within it
  unsigned char* a_t = smem + (size_t)grp * A_BYTES;       // this warpgroup's key tile (one buffer: see the loop)
  unsigned char* b_s = smem + kGroups * A_BYTES;
  float* gd_s = reinterpret_cast<float*>(b_s + B_BYTES);   // [NS][16][16]
  unsigned char* gb_s = reinterpret_cast<unsigned char*>(gd_s) + GD_BYTES;
  constexpr size_t GB_BYTES = gram_bytes(NBITS);
  unsigned char* x_s = gb_s + GB_BYTES;                    // HALF == 2: the three bf16 terms of -G[0:128, 128:256], operands [128 x 128]
  auto gb_cols = [](int pb) { return NBITS - kSub * (pb + 1); };                   // columns after block pb
  auto gb_off = [](int pb) { return gram_off(NBITS, pb); };
  __shared__ __align__(128) uint2 sign_table[16];
  __shared__ unsigned long long mma_bar_s[kGroups], tile_bar_s[kGroups];
  __shared__ uint32_t tmem_base_s;
  __shared__ int timed_out_g[kGroups];
  unsigned long long* mma_bar = &mma_bar_s[grp < kGroups ? grp : 0];
  unsigned long long* tile_bar = &tile_bar_s[grp < kGroups ? grp : 0];
  constexpr int kAccCols = kGroups * NBITS;                // fp32 accumulator columns of the tiles in flight
  constexpr int kTmemCols = kAccCols <= 32 ? 32 : kAccCols <= 64 ? 64 : kAccCols <= 128 ? 128 : kAccCols <= 256 ? 256 : 512;   // a power of two >= 32
  static_assert(kAccCols <= 512, "accumulators exceed tensor memory");

  const int unit = blockIdx.y;
  const int set = shared_sets ? unit % n_kv_heads : unit;

  // ---- one-time set-up: barrier, tensor memory, projection and Gram operands in shared memory
  fill_sign_table(sign_table, tid);
  const unsigned st_a = smem_u32(sign_table);
  if (tid == 0) {
    for (int g = 0; g < kGroups; ++g) { mbar_init(&mma_bar_s[g], 1); mbar_init(&tile_bar_s[g], 1); timed_out_g[g] = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // launched while the kernel before drains: nothing that one may be writing is read above
  pdl_wait();
  const int n = min(unit_lens[unit], n_max);
  const int ntiles = (n + kTileKeys - 1) / kTileKeys;
  if (tid == 0) {                                            // the warpgroups' first key tiles come in under the set-up
    for (int g = 0; g < kGroups; ++g)
      if (kGroups * (int)blockIdx.x + g < ntiles)
        tma::load_key_tile(smem + (size_t)g * A_BYTES, &kmap, unit * n_max + (kGroups * (int)blockIdx.x + g) * kTileKeys, &tile_bar_s[g]);
  }
  {
    // Projection rows, diagonal blocks (fp32, for the in-register sweep) and the Gram terms: everything is requested before anything is
    // stored, one latency in all.
    // -G[16 pb + i][j], j after block pb, as three bf16 terms (g = t1 + t2 + t3 up to 2^-24 |g|); operand rows j, K index i.  Eight
    // consecutive i at a time are one 16-byte store per term.  (One element at a time, in stores of 2 bytes, and one loop after
    // the other: 22.6 us for 8 x 4K keys, 15.4 now.)
    const uint4* psrc = reinterpret_cast<const uint4*>(Ph + ((size_t)set * TOTAL + ROW0) * BPC_D);
    const float* gfull = gram + (size_t)set * TOTAL * TOTAL;
    const float* gsrc = gfull + (size_t)ROW0 * TOTAL + ROW0;  // this launch's diagonal block of the Gram matrix, row stride TOTAL
    constexpr int kRows = NBITS * 16, kDiag = NS * kSub * kSub, kTerms = (NS - 1) * 2 * NBITS;
    constexpr int kRowsEach = (kRows + kThreads - 1) / kThreads, kDiagEach = (kDiag + kThreads - 1) / kThreads, kTermsEach = (kTerms + kThreads - 1) / kThreads;
    uint4 row[kRowsEach];
    float diag[kDiagEach], term[kTermsEach][8];
    auto put_terms = [&](unsigned char* base, int term_bytes, int rows, int r, int i0, const float (&v)[8]) {   // K elements i0 .. i0 + 7 of operand row r
      uint4 t3[3];
      split3x8(v, t3);
#pragma unroll
      for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(base + (size_t)p * term_bytes + nosw_offset(rows, r, i0)) = t3[p];
    };
#pragma unroll
    for (int k = 0; k < kRowsEach; ++k)
      if (tid + k * kThreads < kRows) row[k] = psrc[tid + k * kThreads];
#pragma unroll
    for (int k = 0; k < kDiagEach; ++k) {
      const int c = tid + k * kThreads, d = c / (kSub * kSub), i = c / kSub % kSub, j = c % kSub;
      if (c < kDiag) diag[k] = gsrc[(size_t)(kSub * d + i) * TOTAL + kSub * d + j];
    }
#pragma unroll
    for (int k = 0; k < kTermsEach; ++k) {
      const int c = tid + k * kThreads, pb = c / (2 * NBITS), i0 = 8 * (c / NBITS % 2), j = c % NBITS;
      if (c < kTerms && j >= kSub * (pb + 1)) {
#pragma unroll
        for (int e = 0; e < 8; ++e) term[k][e] = -gsrc[(size_t)(kSub * pb + i0 + e) * TOTAL + j];
      }
    }
#pragma unroll
    for (int k = 0; k < kRowsEach; ++k) {
      const int c = tid + k * kThreads;
      if (c < kRows) *reinterpret_cast<uint4*>(b_s + sw128_offset(NBITS, c >> 4, c & 15)) = row[k];
    }
#pragma unroll
    for (int k = 0; k < kDiagEach; ++k)
      if (tid + k * kThreads < kDiag) gd_s[tid + k * kThreads] = diag[k];
#pragma unroll
    for (int k = 0; k < kTermsEach; ++k) {
      const int c = tid + k * kThreads, pb = c / (2 * NBITS), i0 = 8 * (c / NBITS % 2), j = c % NBITS, j0 = kSub * (pb + 1);
      if (c < kTerms && j >= j0) put_terms(gb_s + gb_off(pb), gb_cols(pb) * kSub * 2, gb_cols(pb), j - j0, i0, term[k]);
    }
    if constexpr (HALF == 2) {
      // -G[i][128 + j] for the first half's bits i, as three bf16 terms; operand rows j, K index i, [128 x 128] each
#pragma unroll 2
      for (int c = tid; c < 16 * 128; c += kThreads) {
        const int i0 = 8 * (c >> 7), j = c & 127;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = -gfull[(size_t)(i0 + e) * TOTAL + 128 + j];
        put_terms(x_s, 32768, 128, j, i0, v);
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the tensor core
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  pdl_release();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_all = tmem_base_s;
  const uint32_t tmem_base = tmem_all + (uint32_t)(grp * NBITS);   // this warpgroup's accumulator columns
  float trace_g = 0.f;                                       // trace of the whole Gram matrix (added by the launch that finishes the code)
  if (ERR && HALF != 1) {
    if constexpr (HALF == 2)
      for (int i = 0; i < 128; ++i) trace_g += gram[(size_t)set * TOTAL * TOTAL + (size_t)i * TOTAL + i];
    for (int i = 0; i < NBITS; ++i) trace_g += gd_s[(i / kSub) * kSub * kSub + (i % kSub) * (kSub + 1)];
  }

  // (one thread) rows past n are never stored, whatever they hold
  auto load_tile = [&](int tile) { tma::load_key_tile(a_t, &kmap, unit * n_max + tile * kTileKeys, tile_bar); };
  const uint32_t idesc = umma_idesc_bf16(kTileKeys, NBITS);
  unsigned tph = 0;                                          // phase of the tile barrier the next wait refers to
  auto issue_gemm = [&]() {                                 // one thread, once the tile is there: 8 steps of K = 16 over the 128 channels
    if (!mbar_wait(tile_bar, tph)) timed_out_g[grp] = 1;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      const size_t aoff = (size_t)(ks >> 2) * (kTileKeys * 128) + (size_t)(ks & 3) * 32;
      const size_t boff = (size_t)(ks >> 2) * (NBITS * 128) + (size_t)(ks & 3) * 32;
      umma_bf16(tmem_base, umma_desc_sw128(a_t + aoff), umma_desc_sw128(b_s + boff), idesc, ks > 0 ? 1u : 0u);
    }
    umma_commit(mma_bar);                                    // arrives when all MMAs issued so far have completed
  };
  // corrections of the columns after block pb by the block's 16 signs (in the block's own columns of tensor memory):
  // T[:, j0..] += U x (-G[block rows, j0..]), three bf16 terms, accumulated into the columns that still wait for their
  // decisions
  auto issue_corrections = [&](int pb) {
    const int j0 = kSub * (pb + 1);
    const uint32_t idc = umma_idesc_bf16(kTileKeys, NBITS - j0);
    const unsigned lbo = (unsigned)(gb_cols(pb) >> 3) * 128;
#pragma unroll
    for (int part = 0; part < 3; ++part)
      umma_bf16_ta(tmem_base + (uint32_t)j0, tmem_base + (uint32_t)(kSub * pb),
                   umma_desc_nosw(gb_s + gb_off(pb) + (size_t)part * gb_cols(pb) * kSub * 2, lbo, 128), idc, 1u);
    umma_commit(mma_bar);
  };

  // HALF == 2: T[:, 0..127] += U1 x (-G[0:128, 128:256]); U1 sits in the key-tile buffer (the projection has completed),
  // three bf16 terms x eight K steps
  auto issue_cross = [&]() {
#pragma unroll
    for (int part = 0; part < 3; ++part) {
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        const unsigned char* ap = a_t + (size_t)ks * 2 * U_LBO;
        const unsigned char* bp = x_s + (size_t)part * 32768 + (size_t)ks * 2 * U_LBO;
        umma_bf16(tmem_base, umma_desc_nosw(ap, U_LBO, 128), umma_desc_nosw(bp, U_LBO, 128), idesc, 1u);
      }
    }
    umma_commit(mma_bar);
  };

  // Tiles of this warpgroup: kGroups * blockIdx.x + grp, then every kGroups * blocks_per_unit-th.  The warpgroups
  // run independent pipelines (own tile, own accumulator columns, own MMA barrier, own hardware barrier); all threads
  // of a warpgroup take the same branches, so its barrier is always reached by all 128 of them.
  const int tile_step = kGroups * blocks_per_unit;
  int tl = grp < kGroups ? kGroups * blockIdx.x + grp : ntiles;
  unsigned ph = 0;                                           // phase of the MMA barrier the next wait refers to
  if (tl < ntiles && gtid == 0) issue_gemm();
  for (; tl < ntiles; tl += tile_step) {
    const int next = tl + tile_step;
    // decision values of this tile: wait for the MMAs, then one TMEM lane (one key) per thread
    if (!mbar_wait(mma_bar, ph)) timed_out_g[grp] = 1;
    ph ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // The MMAs are the only readers of the key tile (besides the key norms below), and they have completed: the
    // buffer is refilled with the warpgroup's next tile right away, under the sweep.
    const int key = tl * kTileKeys + gtid;
    float k2 = 0.f;
    if (ERR && HALF != 2) {                                  // squared norm of this thread's key, from the operand tile
      if (!mbar_wait(tile_bar, tph)) timed_out_g[grp] = 1;   // (the copy's bytes, for this thread too)
#pragma unroll
      for (int ch = 0; ch < 16; ++ch) {
        const uint4 w = *reinterpret_cast<const uint4*>(a_t + sw128_offset(kTileKeys, gtid, ch));
        const float f0 = bf16_lo(w.x), f1 = bf16_hi(w.x), f2 = bf16_lo(w.y), f3 = bf16_hi(w.y);
        const float f4 = bf16_lo(w.z), f5 = bf16_hi(w.z), f6 = bf16_lo(w.w), f7 = bf16_hi(w.w);
        k2 += (f0 * f0 + f1 * f1) + (f2 * f2 + f3 * f3) + (f4 * f4 + f5 * f5) + (f6 * f6 + f7 * f7);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (reads before the refill's writes)
      group_sync(grp);                                       // every thread has read its row before the refill starts
    }
    if (HALF == 2 && residual_correction) {
      // the first half's 128 signs of this thread's key as row gtid of the bf16 operand U1, written over the key tile
      // (no reader of the tile is left: the MMAs have completed and this launch computes no key norms)
      const uint4 cw = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint32_t*>(codes) +
                                                       ((size_t)unit * n_max + (key < n ? key : 0)) * NWK);
      const uint32_t w4[4] = {cw.x, cw.y, cw.z, cw.w};
#pragma unroll
      for (int c = 0; c < 16; ++c) {                         // chunk c: signs 8c .. 8c+7
        const uint2 lo = signs4(st_a, w4[c >> 2], 2 * (c & 3)), hi = signs4(st_a, w4[c >> 2], 2 * (c & 3) + 1);
        *reinterpret_cast<uint4*>(a_t + (size_t)c * U_LBO + (size_t)(gtid >> 3) * 128 + (size_t)(gtid & 7) * 16) =
            make_uint4(lo.x, lo.y, hi.x, hi.y);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      group_sync(grp);
      if (gtid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue_cross();
      }
      if (!mbar_wait(mma_bar, ph)) timed_out_g[grp] = 1;     // the decision values now carry the first half's corrections
      ph ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    tph ^= 1u;
    if (next < ntiles && gtid == 0) load_tile(next);
    const uint32_t taddr = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16);   // a warp reaches the lanes of its quarter
    uint32_t words[NB];
    float abs_sum = 0.f;                                     // sum of |t_i| at decision time (for Eq. 8)
#pragma unroll
    for (int cb = 0; cb < NS; ++cb) {
      if (cb > 0 && residual_correction) {                   // the corrections by block cb - 1 (and all before it) have landed
        if (!mbar_wait(mma_bar, ph)) timed_out_g[grp] = 1;
        ph ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
      float t[kSub];
      tmem_ld16(taddr + (uint32_t)(kSub * cb), t);
      uint32_t word = 0u;
      if (residual_correction) {
        diag_sweep<0, ERR>(t, word, abs_sum, gd_s + (size_t)cb * kSub * kSub);
      } else {
#pragma unroll
        for (int i = 0; i < kSub; ++i) word |= (((__float_as_uint(t[i]) + 0x007FFFFFu) >> 31) ^ 1u) << i;
      }
      if (cb & 1) words[cb / 2] |= word << 16;
      else words[cb / 2] = word;
      if (cb + 1 < NS && residual_correction) {
        // this key's 16 signs as a row of the bf16 operand in tensor memory, over the columns just read
        uint32_t u[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) { const uint2 v = signs4(st_a, word, e); u[2 * e] = v.x; u[2 * e + 1] = v.y; }
        tmem_st8(taddr + (uint32_t)(kSub * cb), u);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        group_sync(grp);                                     // all rows of U are written (and the block's TMEM reads are done)
        if (gtid == 0) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          issue_corrections(cb);
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    group_sync(grp);                                         // the accumulators have been read by the whole warpgroup
    if (timed_out_g[grp]) {                                  // (written only by this warpgroup, before the barrier)
      if (next < ntiles && gtid == 0) (void)mbar_wait(tile_bar, tph);   // the copy in flight
      break;
    }
    if (next < ntiles && gtid == 0) issue_gemm();
    if (key < n) {
      // squared reconstruction error (Eq. 8) from the sweep: ||k - hP||^2 = ||k||^2 - 2 sum|t_i| + trace(G)
      // (256-bit codes: the first launch leaves ||k||^2 - 2 sum|t_i| of its bits, the second adds its own sum and the trace)
      if (ERR) {
        float* ke = key_err + (size_t)unit * n_max + key;
        if (HALF == 0) *ke = fmaxf(0.f, k2 - 2.f * abs_sum + trace_g);
        else if (HALF == 1) *ke = k2 - 2.f * abs_sum;
        else *ke = fmaxf(0.f, *ke - 2.f * abs_sum + trace_g);
      }
      uint32_t* dst = reinterpret_cast<uint32_t*>(codes) + ((size_t)unit * n_max + key) * NWK + (HALF == 2 ? 4 : 0);
      if (NB == 1) {
        dst[0] = words[0];
      } else if (NB == 2) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[1]);
      } else {
#pragma unroll
        for (int w = 0; w + 3 < NB; w += 4) *reinterpret_cast<uint4*>(dst + w) = make_uint4(words[w], words[w + 1], words[w + 2], words[w + 3]);
      }
    }
  }
  if (grp < kGroups && timed_out_g[grp] && gtid == 0) atomicOr(err, BPC_DEVERR_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();                                           // all warpgroups are done with tensor memory
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_all), "r"(kTmemCols) : "memory");
  }
}

template <int NBITS, int GROUPS, int HALF, bool ERR>
cudaError_t launch(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  const bpc_config& c = ctx->cfg;
  const size_t smem = (size_t)GROUPS * kTileKeys * 256 + (size_t)NBITS * 256 + (size_t)NBITS * kSub * 4 + gram_bytes(NBITS) +
                      (HALF == 2 ? (size_t)kCrossBytes : 0) + 1024;
  auto kern = encode_tc_kernel<NBITS, GROUPS, HALF, ERR>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int steps_max = ((c.n_max + kTileKeys - 1) / kTileKeys + GROUPS - 1) / GROUPS;   // a block takes GROUPS tiles at a time
  // Blocks per unit.  One block fits an SM (shared memory), so the grid runs in waves of sm_count blocks and a last,
  // partly filled wave costs as much as a full one: from one wave up, the first count whose last wave is at least 90 % full
  // (32 units on 148 SMs: 9 blocks per unit = 1.95 waves).  Every block lays out the Gram operands anew, so few waves: from
  // four waves up 32 x 128K keys take 621 us instead of 583, and 8 x 32K keys at 256 bits 296 instead of 273.
  int bpu = (ctx->sm_count + ctx->units - 1) / ctx->units;
  if (bpu < 1) bpu = 1;
  for (int tries = 0; tries < 16; ++tries) {
    const int rem = (int)(((long long)ctx->units * bpu) % ctx->sm_count);
    if (rem == 0 || rem * 10 >= ctx->sm_count * 9) break;
    ++bpu;
  }
  if (bpu > steps_max) bpu = steps_max;
  const dim3 grid(bpu, ctx->units);
  CUtensorMap kmap;
  e = tma::make_key_map(&kmap, k_cache, (unsigned long long)ctx->units * c.n_max, ctx->row_stride);
  if (e != cudaSuccess) return e;
  return launch_pdl(ctx->use_pdl, kern, grid, kGroupThreads * (GROUPS + setup_groups(HALF)), smem, stream,
                    kmap, (const __nv_bfloat16*)ctx->P_h, ctx->gram, ctx->unit_lens, codes, ctx->dev_err,
                    c.n_kv_heads, c.n_max, c.hash_sets != ctx->units, c.residual_correction, bpu, ctx->key_err);
}

template <bool ERR>
cudaError_t launch_bits(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  switch (ctx->cfg.code_bits) {
    case 32: return launch<32, kGroups, 0, ERR>(ctx, k_cache, codes, stream);
    case 64: return launch<64, kGroups, 0, ERR>(ctx, k_cache, codes, stream);
    case 128: return launch<128, kGroups, 0, ERR>(ctx, k_cache, codes, stream);
    case 256: {
      const cudaError_t e = launch<128, kGroups, 1, ERR>(ctx, k_cache, codes, stream);
      if (e != cudaSuccess) return e;
      ctx->launches += 1;
      return launch<128, 1, 2, ERR>(ctx, k_cache, codes, stream);
    }
    default: return cudaErrorNotSupported;
  }
}

}  // namespace

// bf16 caches run on the tensor cores: 32-, 64- and 128-bit codes in one launch, 256-bit codes in two (the bf16 terms of
// a 256 x 256 Gram matrix do not fit shared memory next to the operands, those of its 128 x 128 blocks do).  fp32 caches
// report "not supported" and the caller falls back to the CUDA-core kernel (they have no bf16 operands).  The kernel is
// compiled with and without the reconstruction errors that only the safeguard needs.
cudaError_t bpc_launch_encode_tc(bpc_ctx* ctx, const void* k_cache, uint64_t* codes, cudaStream_t stream) {
  if (ctx->cfg.kv_dtype != BPC_BF16) return cudaErrorNotSupported;
  if (ctx->no_tc_encode) return cudaErrorNotSupported;     // diagnostic switch: the CUDA-core kernel is asked for
  const cudaError_t e = ctx->key_err != nullptr ? launch_bits<true>(ctx, k_cache, codes, stream) : launch_bits<false>(ctx, k_cache, codes, stream);
  if (e == cudaSuccess) ctx->launches += 1;
  return e;
}

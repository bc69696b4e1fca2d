// Intra-chunk part of the causal linear branch.  When the query chunk is the most recently
// appended chunk, query i may only see the chunk's own keys up to its position; the state of
// everything before the chunk is applied by the forward kernel, and this kernel supplies
//   num[i,h,:] = sum_{q_pos0 <= j <= q_pos0+i} (phi(q_i).phi(k_j)) v_j,   den[i,h] = sum of weights
// K and V from the pool pages.
//
// phi(K) of the chunk is made first, by a kernel of its own, as bf16 tiles in the workspace (made in the kernel
// of the products it would be made again for every query tile behind a key; left there by the append, every
// append would pay for it): 5 us for a chunk of 1560 tokens, 12 heads of 128.
//
// In chunks of enough query tiles (sums_pay; head_dim 128) a tile does not walk through all of the chunk's pages in front of it:
// chunk_sums_kernel leaves T = sum_j phi(k_j) v_j^T and z = sum_j phi(k_j) over every group of four pages (two tiles)
// in the workspace, and a tile takes phi(Q) times the sum of T over the groups before its own, then the pages from
// its group's first on, at most five.  At head_dim 64 a tile always walks through all of them.
//
// One CTA per (128-row query tile, head), 576 threads:
//   warp 0       TMA producer: Q tile, then, page by page up to the tile's diagonal, phi(K) and V (64 keys per
//                step) into rings of two
//   warp 1       tcgen05.mma issuer
//   warps 2..17  sum of T, phi(Q), once; weights of a step: mask, row sum, split; running sum of num
// The map, the weights and the sums are fp32 quantities, so each operand is carried as three bf16 terms,
// hi + mid + lo (24 bits), with the products of down to 2^-16 of the largest:
//   A     = phi(Q) phi(K)^T  as  hi hi  +  (lo hi + hi lo + mid mid + mid hi + hi mid)    (fp32, TMEM)
//   num_j = A_lo V + A_mid V + A_hi V  of one step's 64 keys, with A masked and split     (fp32, TMEM)
// The tensor cores truncate what they add to.  The hi of phi(Q) and phi(K) are therefore multiples of 2^-6 of the
// largest value's power of two (per row and 32 dims): the sum of hi hi over 128 dims needs 22 bits and
// is exact, the other products have an accumulator of their own, and A is rounded once, when the two are added.
// In num small terms go first and the accumulator lives for one step: num and den are running sums in
// registers, rounded.
// The sum of T is split the same way (hi on a grid per dim of v and 32 dims of k), hi hi once more apart from the rest.
// Error of num and den against 64 bits (2-norm; 12 heads of 128, chunks of 256 / 1560, 4 heads, 3120 tokens): fp32
// SIMT kernel num 1.1e-7 / 2.2e-7 / 3.0e-7, den 0.6e-7 / 0.8e-7 / 1.0e-7; all pages in steps 0.7e-7 / 1.0e-7 / 1.3e-7 and
// 0.4e-7 / 0.5e-7 / 0.6e-7; with sums over groups 0.7e-7 / 0.6e-7 / 0.6e-7 and 0.4e-7 / 0.4e-7 / 0.4e-7.  (Two terms
// each and sums over the whole chunk in TMEM: num 2.7e-6 and more, den 6.0e-7.)
// An Inf or NaN meets zeros in the products (masked weights, terms of the split), also in rows before it: a row
// whose result is not finite is taken again key by key (cl_plain_row).
//
// What bounds it: latencies of a tile's chain.  The terms of phi(K) lie side by side, so that one product of phi(Q) hi
// with all three, one of mid with the first two and one of lo with the first form all sums: 8 x (96 + 64 + 32)
// cycles per step at head_dim 128, and 768 for num.  Time stamps, 12 heads of 128, 1560 tokens: sum of T there at 2
// to 5 us, phi(Q) 3 us later, its products with the sum read back after another 2.4, then 1.3 us per step and 2 at the
// end: 15 to 18 us per tile, where the longest took 36 step by step.  One CTA per query and head in fp32 on the CUDA
// cores took 1678 us for the chunk.
// The work of a tile grows with its position, so the last tiles are launched first and the forward kernel
// behind this one may start on the SMs that are through (see hsa_forward_kernel).
// TMEM: num (128 columns) | two step buffers of 192: hi hi | hi mid + mid hi | hi lo + mid mid + lo hi, 64 columns
// each.  The split weights overwrite them: 16 columns of hi hi become 8 of packed hi and 8 of packed mid, 16 of
// the next sum 8 of packed lo.
#include <cuda_bf16.h>

#include <cfloat>

#include "hsa_internal.h"
#include "ptx.cuh"

namespace hsa {

namespace {

constexpr int kClWorkers = 512;
constexpr int kClThreads = 64 + kClWorkers;
constexpr int kClTerms = kPhiTerms;
constexpr int kClStages = 2;
constexpr int kClGroup = 4;       // pages of a group: two query tiles
// Whether the sums over groups are made.  Their kernel is 5 us in front of the tiles, and the steps that they save, 1.3 us each,
// count along the longest tile: six query tiles at least.  Step by step the tiles also end one after another, and the
// forward's tiles start on the SMs that are left; with sums they all end together.  So on more than half of the
// SMs, and again where the tiles take a second wave, the work has to be larger: tiles * (heads + 15), the overheads of
// both ways being about 15 heads' worth.  A causal forward, lists of 32 blocks, all pages step by step -> with sums, heads x
// tiles (the rule's choice last): 2 x 6 38.9 -> 37.8 us (sums), 12 x 7 45.3 -> 51.6 (steps), 12 x 8 51.4 -> 54.8 (steps), 12 x 9
// 56.3 -> 54.5 (sums), 16 x 6 48.0 -> 53.1 (steps), 16 x 8 59.4 -> 56.9 (sums), 20 x 8 72.4 -> 80.2 (steps), 20 x 10 87.8 -> 86.1
// (sums), 24 x 7 74.4 -> 81.1 (steps), 24 x 9 89.3 -> 85.5 (sums), 40 x 16 314 -> 243 (sums).  It errs at 4 x 7 (40.7 -> 44.7) and,
// with lists of 8 blocks, at 12 x 8 (46.5 -> 44.4).
constexpr int kClMinTiles = 6, kClHalfWork = 220, kClWaveWork = 340;
bool sums_pay(int tiles, int heads, int nsm, bool alone) {
  const int64_t items = static_cast<int64_t>(tiles) * heads, work = items + 15 * static_cast<int64_t>(tiles);
  if (tiles < kClMinTiles) return false;
  if (items <= (alone ? nsm : nsm / 2)) return true;
  return work >= (items <= nsm ? kClHalfWork : kClWaveWork);
}
constexpr int kClSums = 128 * 128 + 128;  // floats of a group's sums
constexpr int kCsStages = 3, kCsThreads = 192;
constexpr int kCsSmem = kCsStages * (kClTerms + 1) * kBlock * 128 * 2 + 2048 + 256 + 1024;
constexpr uint32_t kClColNum = 0, kClColBuf = 128, kClBuf = kClTerms * kBlock;
constexpr uint32_t kClColPre = kClColBuf + kClBuf;  // sums over earlier groups, smaller products (before the steps)

template <int D>
struct ClSmem {
  static constexpr int kSlab = kBlock * 128;       // bytes of one [64 rows x 128 B] slab
  static constexpr int kPage = kBlock * D * 2;     // 64 keys
  static constexpr int kQHalf = kTileM * 128;      // bytes of one [128 rows x 128 B] slab of Q
  static constexpr int kQTile = kTileM * D * 2;
  static constexpr int kK = 0;                     // phi(K): stage, then slab, then term
  static constexpr int kV = kK + kClStages * kClTerms * kPage;
  static constexpr int kQ = kV + kClStages * kPage;  // terms of phi(Q); Q arrives in the last one's place
  static constexpr int kBars = kQ + kClTerms * kQTile;
  static constexpr int kTotal = kBars + 256 + D * 4 + 1024;
};

// (ring stage and step buffer of step j are both j % 2)
struct ClBars {
  uint64_t q_full, q_read;
  uint64_t s_ready;    // terms of the sums over earlier groups written (in the phi(K) ring's place)
  uint64_t pre_low;    // products of mid and lo of the sums formed, the ring's first stage free
  uint64_t pre_full;   // all their products with phi(Q) formed, the ring free
  uint64_t pre_read;   // and read back
  uint64_t k_full[2], v_full[2];
  uint64_t a_full[2];    // A of the step is formed, its phi(K) stage free
  uint64_t num_full[2];  // num of the step is formed, its V stage free
  uint64_t p_ready;      // weights of step j written, num of step j - 1 added up
  uint32_t tmem_base;
  volatile int abort_flag;
};
static_assert(kClStages == 2, "one barrier stands for a step buffer and a ring stage");
static_assert(sizeof(ClBars) <= 256 && sizeof(ClBars) % 16 == 0, "barrier block must fit its slot, z follows");

__device__ __forceinline__ bool cl_wait(uint64_t* bar, uint32_t parity, ClBars* bars, int32_t* status) {
  if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t i = 1; i < (1u << 24); ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 1023u) == 0u && bars->abort_flag) return false;
  }
  bars->abort_flag = 1;
  atomicCAS(status, 0, kDevTimeout);
  return false;
}

__device__ __forceinline__ float cl_phi(float x, int relu) { return relu ? fmaxf(x, 0.f) : (x > 0.f ? x + 1.f : expf(x)); }
// Adding and subtracting this rounds to multiples of 2^-6 of the power of two at or below `largest`.
__device__ __forceinline__ float cl_grid(float largest) {
  const uint32_t e = min(max(__float_as_uint(largest) >> 23, 27u), 227u);
  return __uint_as_float(((e + 17u) << 23) | 0x400000u);
}
// two fp32 values as packed bf16 terms, hi + mid + lo = value to 24 bits; grid: see cl_grid (0: hi is the rounded value)
__device__ __forceinline__ void cl_split(float a, float b, float grid, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = pack_bf16(__fsub_rn(__fadd_rn(a, grid), grid), __fsub_rn(__fadd_rn(b, grid), grid));
  a -= __uint_as_float(hi << 16);
  b -= __uint_as_float(hi & 0xffff0000u);
  mid = pack_bf16(a, b);
  lo = pack_bf16(a - __uint_as_float(mid << 16), b - __uint_as_float(mid & 0xffff0000u));
}

// element e of 8 that three bf16 terms make up
__device__ __forceinline__ float cl_join(const uint4 (&t)[kClTerms], int e) {
  float f[kClTerms];
#pragma unroll
  for (int m = 0; m < kClTerms; ++m) {
    const uint32_t w = (e >> 1) == 0 ? t[m].x : (e >> 1) == 1 ? t[m].y : (e >> 1) == 2 ? t[m].z : t[m].w;
    f[m] = __uint_as_float(e & 1 ? w & 0xffff0000u : w << 16);
  }
  return fabsf(f[0]) <= FLT_MAX ? f[0] + f[1] + f[2] : f[0];  // (the remainders of Inf are NaN)
}

// num of one row (D / 4 columns) and den, key by key in fp32.  q: terms of phi(Q) in shared memory, row r; phik: the
// head's hi tiles, mid and lo `term` elements further on each; keys `first` and the n_keys - 1 behind it, counted
// from the first of `pages`.
template <int D>
__device__ __noinline__ void cl_plain_row(const uint8_t* q, int r, const __nv_bfloat16* phik, size_t term,
                                          const __nv_bfloat16* v_pool, const int32_t* pages, int H, int h, int first, int n_keys,
                                          int col, float* num, float* den) {
  using L = ClSmem<D>;
  constexpr int NC = D / 4;
  float acc[NC], sum = 0.f;
#pragma unroll
  for (int i = 0; i < NC; ++i) acc[i] = 0.f;
#pragma unroll 1
  for (int t = first; t < first + n_keys; ++t) {
    float w = 0.f;
#pragma unroll 1
    for (int c = 0; c < D / 8; ++c) {
      uint4 qt[kClTerms], kt[kClTerms];
#pragma unroll
      for (int m = 0; m < kClTerms; ++m) {
        qt[m] = *reinterpret_cast<const uint4*>(q + m * L::kQTile + r * 128 + (c >> 3) * L::kQHalf + (((c & 7) ^ (r & 7)) << 4));
        kt[m] = *reinterpret_cast<const uint4*>(phik + m * term + static_cast<size_t>(t) * D + c * 8);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) w = fmaf(cl_join(qt, e), cl_join(kt, e), w);
    }
    sum += w;
    const __nv_bfloat16* v = v_pool + ((static_cast<size_t>(pages[t / kBlock]) * H + h) * kBlock + t % kBlock) * D + col;
#pragma unroll
    for (int i = 0; i < NC; ++i) acc[i] = fmaf(w, __bfloat162float(v[i]), acc[i]);
  }
#pragma unroll
  for (int i = 0; i < NC; ++i) num[i] = acc[i];
  if (den) *den = sum;
}

}  // namespace

// phi(K) of one page of one head: what bounds it is the bytes, 16 KB in and 48 KB out per page at head_dim 128.
template <int D>
__global__ void __launch_bounds__(256) phi_terms_kernel(CausalLinArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int h = blockIdx.y;
  const int64_t b = a.q_pos0 / kBlock + blockIdx.x;
  const uint4* src = reinterpret_cast<const uint4*>(a.k_pool + (static_cast<size_t>(a.page_table[b]) * a.H + h) * kBlock * D);
  uint4* dst = reinterpret_cast<uint4*>(a.phik + (static_cast<size_t>(h) * kClTerms * a.phik_blocks + blockIdx.x) * kBlock * D);
  const size_t term = static_cast<size_t>(a.phik_blocks) * kBlock * D / 8;  // from one term's tile to the next
#pragma unroll
  for (int i = 0; i < kBlock * D / 8 / 256; ++i) {
    const int c = threadIdx.x + 256 * i;
    const uint4 raw = src[c];
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
    float f[8], largest = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      f[e] = cl_phi(__uint_as_float(e & 1 ? w[e >> 1] & 0xffff0000u : w[e >> 1] << 16), a.relu);
      largest = fmaxf(largest, f[e]);
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) largest = fmaxf(largest, __shfl_xor_sync(0xffffffffu, largest, o));  // of 32 dims
    const float grid = cl_grid(largest);
    uint32_t t[kClTerms][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) cl_split(f[2 * e], f[2 * e + 1], grid, t[0][e], t[1][e], t[2][e]);
    if (b * kBlock + c / (D / 8) < a.q_pos0) {  // rows before the chunk add nothing to the sums over groups
#pragma unroll
      for (int m = 0; m < kClTerms; ++m)
#pragma unroll
        for (int e = 0; e < 4; ++e) t[m][e] = 0u;
    }
#pragma unroll
    for (int m = 0; m < kClTerms; ++m) dst[c + m * term] = make_uint4(t[m][0], t[m][1], t[m][2], t[m][3]);
  }
}

// Sums over a group of kClGroup pages of the chunk, head_dim 128: T = sum_j phi(k_j) v_j^T (stored [dim of k / 4][dim of v]
// [4]) and z = sum_j phi(k_j).  One CTA per (group, head), 192 threads: warp 0 TMA, warp 1 products, warps 2..5
// write-out.  phi(K) in its three terms, lo and mid into one accumulator, hi of every two pages into one of its own
// (the tensor cores truncate what they add to), added in rounded fp32.  V is the operand of 128 lanes, so that a
// thread of the write-out, and later of causal_linear_kernel, holds 32 dims of k beside each other.
struct CsBars {
  uint64_t full[kCsStages], empty[kCsStages], done;
  uint32_t tmem_base;
  volatile int abort_flag;
};
__global__ void __launch_bounds__(kCsThreads, 1)
chunk_sums_kernel(CausalLinArgs a, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v) {
  constexpr int D = 128, kSlab = kBlock * 128, kPage = kBlock * D * 2, kStage = (kClTerms + 1) * kPage;
  extern __shared__ uint8_t cl_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(cl_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* ones = smem + kCsStages * kStage;
  CsBars* bars = reinterpret_cast<CsBars*>(ones + 2048);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u = blockIdx.x, h = blockIdx.y;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kCsStages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    mbar_init(&bars->done, 1);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  for (int i = threadIdx.x; i < 2048 / 4; i += kCsThreads) reinterpret_cast<uint32_t*>(ones)[i] = 0x3F803F80u;
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    for (uint32_t i = 0; i < (1u << 24); ++i) {
      if (mbar_try_wait(bar, parity)) return true;
      if ((i & 1023u) == 1023u && bars->abort_flag) return false;
    }
    bars->abort_flag = 1;
    atomicCAS(a.status, 0, kDevTimeout);
    return false;
  };
  constexpr uint32_t kColHi = 128, kColZ = 384;
  int armed = 0;  // pages asked for (producer's lane)
  if (warp == 0) {
    if (elect_one_sync()) {
      const int64_t b0 = a.q_pos0 / kBlock + u * kClGroup;
      bool ok = true;
      for (int i = 0; i < kClGroup && ok; ++i) {
        const int s = i % kCsStages;
        uint8_t* st = smem + s * kStage;
        const int32_t y = (a.page_table[b0 + i] * a.H + h) * kBlock;
        ok = i < kCsStages || wait(&bars->empty[s], ((i / kCsStages) - 1) & 1);
        if (!ok) break;
        mbar_expect_tx(&bars->full[s], kStage);
        for (int dh = 0; dh < 2; ++dh) tma_load_2d(st + kClTerms * kPage + dh * kSlab, &tm_v, &bars->full[s], dh * 64, y);
        for (int t = kClTerms - 1; t >= 0; --t)
          for (int dh = 0; dh < 2; ++dh)
            tma_load_2d(st + t * kPage + dh * kSlab, &tm_k, &bars->full[s], dh * 64,
                        ((h * kClTerms + t) * a.phik_blocks + u * kClGroup + i) * kBlock);
        ++armed;
      }
    }
  } else if (warp == 1) {
    if (elect_one_sync()) {
      constexpr uint32_t kHiSw = desc_hi_sw128(1024), idesc = idesc_bf16_f32(128, D, 1, 1), idesc_1 = idesc_bf16_f32(128, 16, 1, 0);
      const uint32_t b_ones = desc_lo_sw128(smem_u32(ones), 16);
      bool ok = a.give_up == 0;
      if (!ok) {
        bars->abort_flag = 1;
        atomicCAS(a.status, 0, kDevTimeout);
      }
      for (int i = 0; i < kClGroup && ok; ++i) {
        const int s = i % kCsStages;
        ok = wait(&bars->full[s], (i / kCsStages) & 1);
        if (!ok) break;
        tc_fence_after();
        const uint32_t st = smem_u32(smem + s * kStage);
        const uint32_t v = desc_lo_sw128(st + kClTerms * kPage, kSlab);
#pragma unroll
        for (int t = kClTerms - 1; t >= 0; --t) {
          const uint32_t k = desc_lo_sw128(st + t * kPage, kSlab);
          const uint32_t acc = tmem + (t > 0 ? 0 : kColHi + 128 * (i >> 1)), acc_z = tmem + kColZ + 16 * (t > 0 ? 0 : 1 + (i >> 1));
          const bool more = t == kClTerms - 1 ? i > 0 : t > 0 || (i & 1) != 0;
#pragma unroll
          for (int kk = 0; kk < kBlock / 16; ++kk) tc_mma_ss_lo(acc, v + kk * 128, k + kk * 128, kHiSw, idesc, more || kk > 0 ? 1u : 0u);
#pragma unroll
          for (int kk = 0; kk < kBlock / 16; ++kk) tc_mma_ss_lo(acc_z, k + kk * 128, b_ones, kHiSw, idesc_1, more || kk > 0 ? 1u : 0u);
        }
        tc_commit(&bars->empty[s]);
      }
      tc_commit(&bars->done);
    }
  } else {
    const int quad = warp & 3, r = quad * 32 + lane;
    const uint32_t row = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    // (done alone does not say that every page is in)
    if (__all_sync(0xffffffffu, wait(&bars->done, 0) && bars->abort_flag == 0)) {
      tc_fence_after();
      float* dst = a.sums + (static_cast<size_t>(h) * a.sum_groups + u) * kClSums;
#pragma unroll 1
      for (int c = 0; c < D; c += 16) {
        uint32_t lo[16], h0[16], h1[16];
        tmem_ld16(row + c, lo);
        tmem_ld16(row + kColHi + c, h0);
        tmem_ld16(row + kColHi + 128 + c, h1);
        tc_wait_ld();
        auto sum = [&](int i) { return (__uint_as_float(h0[i]) + __uint_as_float(h1[i])) + __uint_as_float(lo[i]); };
#pragma unroll
        for (int i = 0; i < 16; i += 4)
          reinterpret_cast<float4*>(dst)[(c + i) / 4 * D + r] = make_float4(sum(i), sum(i + 1), sum(i + 2), sum(i + 3));
      }
      uint32_t z[3][16];
#pragma unroll
      for (int m = 0; m < 3; ++m) tmem_ld16(row + kColZ + 16 * m, z[m]);
      tc_wait_ld();
      dst[D * D + r] = (__uint_as_float(z[1][0]) + __uint_as_float(z[2][0])) + __uint_as_float(z[0][0]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (bars->abort_flag) {
    // whoever has given up: the copies issued land before the CTA's shared memory goes away, and the products end before TMEM
    // goes
    for (int s = 0; s < kCsStages; ++s)
      if (armed > s) mbar_wait(&bars->full[s], ((armed - 1 - s) / kCsStages) & 1, 1u << 16);
    if (warp == 1) mbar_wait(&bars->done, 0, 1u << 16);
  }
  __syncwarp();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// SUMS: compiled with the sums over earlier groups; an instance of its own, since a step without them takes 4 % longer in one
// that carries them (linear branch alone, 4 heads, 5 tiles: 43.9 us a call against 42.9)
template <int D, bool SUMS>
__global__ void __launch_bounds__(kClThreads, 1)
causal_linear_kernel(CausalLinArgs a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v) {  // tm_k: the phi(K) tiles
  using L = ClSmem<D>;
  constexpr int DH = D / 64;
  extern __shared__ uint8_t cl_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(cl_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  ClBars* bars = reinterpret_cast<ClBars*>(smem + L::kBars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tiles = (a.n_q + kTileM - 1) / kTileM;
  const int h = static_cast<int>(blockIdx.x) % a.H;
  const int row0 = (n_tiles - 1 - static_cast<int>(blockIdx.x) / a.H) * kTileM;  // longest tiles first

  if (threadIdx.x == 0) {
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->q_read, kClWorkers / 32);
    mbar_init(&bars->s_ready, kClWorkers / 32);
    mbar_init(&bars->pre_low, 1);
    mbar_init(&bars->pre_full, 1);
    mbar_init(&bars->pre_read, kClWorkers / 32);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->a_full[s], 1);
      mbar_init(&bars->num_full[s], 1);
    }
    mbar_init(&bars->p_ready, kClWorkers / 32);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  // everything before this kernel is complete from here on, for this grid and -- since the trigger
  // comes after the wait -- for the kernel launched behind it as a programmatic dependent
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // Pages of the chunk up to the last token this tile sees, one per step; with sums over groups from the tile's own
  // group on (the pages of a group start where its two tiles do, less the first page's older rows).
  const int b_first = static_cast<int>(a.q_pos0 / kBlock);
  const int64_t last = a.q_pos0 + min(row0 + kTileM, a.n_q) - 1;
  const int groups = SUMS ? row0 / kTileM * 2 / kClGroup : 0;  // groups before the tile's own
  const int p0 = groups * kClGroup;                            // first page of the steps
  const int nsteps = static_cast<int>(last / kBlock) - b_first + 1 - p0;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one lane)
    if (elect_one_sync()) {
      mbar_expect_tx(&bars->q_full, L::kQTile);
      for (int dh = 0; dh < DH; ++dh) tma_load_3d(smem + L::kQ + 2 * L::kQTile + dh * L::kQHalf, &tm_q, &bars->q_full, dh * 64, h, row0);
      int armed_k = 0, armed_v = 0;  // loads issued per ring, for the drain on abort
      auto load_k = [&](int j) -> bool {
        const int s = j % kClStages;
        if (j >= kClStages && !cl_wait(&bars->a_full[s], ((j / kClStages) - 1) & 1, bars, a.status)) return false;
        mbar_expect_tx(&bars->k_full[s], kClTerms * L::kPage);
        for (int t = 0; t < kClTerms; ++t)
          for (int dh = 0; dh < DH; ++dh)
            tma_load_2d(smem + L::kK + s * kClTerms * L::kPage + (dh * kClTerms + t) * L::kSlab, &tm_k, &bars->k_full[s], dh * 64,
                        ((h * kClTerms + t) * a.phik_blocks + p0 + j) * kBlock);
        ++armed_k;
        return true;
      };
      auto load_v = [&](int j) -> bool {
        const int s = j % kClStages;
        const int32_t y = (a.page_table[b_first + p0 + j] * a.H + h) * kBlock;  // (looked up ahead of the wait)
        if (j >= kClStages && !cl_wait(&bars->num_full[s], ((j / kClStages) - 1) & 1, bars, a.status)) return false;
        mbar_expect_tx(&bars->v_full[s], L::kPage);
        for (int dh = 0; dh < DH; ++dh)
          tma_load_2d(smem + L::kV + s * L::kPage + dh * L::kSlab, &tm_v, &bars->v_full[s], dh * 64, y);
        ++armed_v;
        return true;
      };
      // phi(K) one step further than V: its stage is free as soon as the sums of step j - 2 are formed, before
      // the weights of that step have met the V whose stage the next V takes (in one order 3500 cycles per step)
      bool ok = !SUMS || groups == 0 || cl_wait(&bars->pre_low, 0, bars, a.status);
      ok = ok && load_k(0) && (!SUMS || groups == 0 || cl_wait(&bars->pre_full, 0, bars, a.status));
      for (int j = 0; j < nsteps && ok; ++j) ok = (j + 1 >= nsteps || load_k(j + 1)) && load_v(j);
      if (!ok) {  // let every copy already issued land before the CTA's shared memory goes away
        mbar_wait(&bars->q_full, 0, 1u << 16);
        for (int s = 0; s < kClStages; ++s) {
          if (armed_k > s) mbar_wait(&bars->k_full[s], ((armed_k - 1 - s) / kClStages) & 1, 1u << 16);
          if (armed_v > s) mbar_wait(&bars->v_full[s], ((armed_v - 1 - s) / kClStages) & 1, 1u << 16);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one lane)
    if (elect_one_sync()) {
      constexpr uint32_t kHiSw = desc_hi_sw128(1024);
      const uint32_t q_lo = desc_lo_sw128(smem_u32(smem + L::kQ), 16);
      // What is waited for next is asked about while the products just issued still keep the pipe busy: a barrier
      // costs some 100 cycles to ask even if it is complete, and few products queue up.
      bool k_landed = false, ready = false;
      auto issue_qk = [&](int j, int next) -> bool {
        const uint32_t d = tmem + kClColBuf + kClBuf * (j & 1);
        const int s = j % kClStages;
        if (!k_landed && !cl_wait(&bars->k_full[s], (j / kClStages) & 1, bars, a.status)) return false;
        tc_fence_after();
        const uint32_t k_lo = desc_lo_sw128(smem_u32(smem + L::kK + s * kClTerms * L::kPage), 16);
        // term t of phi(Q) with the first 3 - t of phi(K), onto the sums from the t-th on
        auto product = [&](int t, int kk) {
          tc_mma_ss_lo(d + kBlock * t, q_lo + ((t * L::kQTile + (kk / 4) * L::kQHalf + (kk % 4) * 32) >> 4),
                       k_lo + (((kk / 4) * kClTerms * L::kSlab + (kk % 4) * 32) >> 4), kHiSw,
                       idesc_bf16_f32(128, kBlock * (kClTerms - t), 0, 0), (t > 0 || kk > 0) ? 1u : 0u);
        };
        // (the largest products last: the most work in the queue while the lane turns to the next step)
        product(0, 0);
#pragma unroll
        for (int t = kClTerms - 1; t > 0; --t)
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) product(t, kk);
        ready = next < nsteps && mbar_test_wait(&bars->v_full[next % kClStages], (next / kClStages) & 1) &&
                mbar_test_wait(&bars->p_ready, next & 1);
#pragma unroll
        for (int kk = 1; kk < D / 16; ++kk) product(0, kk);
        tc_commit(&bars->a_full[j & 1]);
        return true;
      };
      bool ok = cl_wait(&bars->q_read, 0, bars, a.status);  // phi(Q) is in shared memory
      if (SUMS && groups > 0 && ok) {
        // the sums over earlier groups: hi hi into the place of num, the smaller products into the second buffer's
        ok = cl_wait(&bars->s_ready, 0, bars, a.status);
        if (ok) {
          tc_fence_after();
          constexpr uint32_t idesc = idesc_bf16_f32(128, D, 0, 0);
          const uint32_t s_lo = desc_lo_sw128(smem_u32(smem + L::kK), 16);
          auto product = [&](int tq, int ts, uint32_t d, uint32_t more) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t off = ((kk / 4) * L::kQHalf + (kk % 4) * 32) >> 4;
              tc_mma_ss_lo(tmem + d, q_lo + ((tq * L::kQTile) >> 4) + off, s_lo + (((kClTerms - 1 - ts) * L::kQTile) >> 4) + off, kHiSw, idesc,
                           more || kk > 0 ? 1u : 0u);
            }
          };
          product(0, 2, kClColPre, 0u);
          product(1, 1, kClColPre, 1u);
          product(0, 1, kClColPre, 1u);
          tc_commit(&bars->pre_low);  // (phi(K) of the first step may come where lo and mid were)
          product(2, 0, kClColPre, 1u);
          product(1, 0, kClColPre, 1u);
          product(0, 0, kClColNum, 0u);
          tc_commit(&bars->pre_full);
          ok = cl_wait(&bars->pre_read, 0, bars, a.status);
          tc_fence_after();
        }
      }
      for (int j = 0; j < min(2, nsteps) && ok; ++j) {
        k_landed = false;
        ok = issue_qk(j, nsteps);
      }
#pragma unroll 1
      for (int j = 0; j < nsteps && ok; ++j) {
        const int s = j % kClStages;
        if (!ready)
          ok = cl_wait(&bars->v_full[s], (j / kClStages) & 1, bars, a.status) && cl_wait(&bars->p_ready, j & 1, bars, a.status);
        if (!ok) break;
        tc_fence_after();
        constexpr uint32_t idesc = idesc_bf16_f32(128, D, 0, 1);
        const uint32_t v_lo = desc_lo_sw128(smem_u32(smem + L::kV + s * L::kPage), L::kSlab);
        const uint32_t p_op = tmem + kClColBuf + kClBuf * (j & 1);
#pragma unroll
        for (int t = kClTerms - 1; t >= 0; --t) {
#pragma unroll
          for (int kk = 0; kk < kBlock / 16; ++kk)
            tc_mma_ts_lo(tmem + kClColNum, p_op + (t == 2 ? kBlock + 16 * kk : 16 * kk + 8 * t), v_lo + kk * 128, kHiSw, idesc,
                         (t < kClTerms - 1 || kk > 0) ? 1u : 0u);
          if (t == 1) k_landed = j + 2 < nsteps && mbar_test_wait(&bars->k_full[s], ((j + 2) / kClStages) & 1);
        }
        tc_commit(&bars->num_full[s]);
        // the weights of step j + 2 overwrite the ones just consumed: the tensor pipe runs in order
        ready = false;
        if (j + 2 < nsteps) ok = issue_qk(j + 2, j + 1);
      }
    }
  } else {
    // ------------------------------------------------------------------ weights, sums
    const int set = (warp - 2) >> 2;  // 16 of the 64 columns of a step, D / 4 of the dims
    const int quad = warp & 3;        // TMEM lane quadrant this warp may access
    const int r = quad * 32 + lane;   // row inside the tile
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    constexpr int NC = D / 4;
    float den = 0.f, num[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) num[i] = 0.f;
    const float* sums = a.sums + static_cast<size_t>(h) * a.sum_groups * kClSums;
    float* zs = reinterpret_cast<float*>(bars + 1);  // z over the groups before the tile's own
    if (SUMS && groups > 0) {
      if (set == 0) {
        float z = 0.f;
        for (int u = 0; u < groups; ++u) z += __ldcg(sums + static_cast<size_t>(u) * kClSums + D * D + r);
        zs[r] = z;
      }
      // Sums over the groups before the tile's own, in fp32 and in order: dim r of v, 32 dims of k; as three terms
      // where phi(K) comes later.
      float sv[32], largest = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) sv[i] = 0.f;
#pragma unroll 2
      for (int u = 0; u < groups; ++u) {
        const float4* src = reinterpret_cast<const float4*>(sums + static_cast<size_t>(u) * kClSums) + set * 8 * D + r;
        float4 x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = __ldcg(src + i * D);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          sv[4 * i] += x[i].x;
          sv[4 * i + 1] += x[i].y;
          sv[4 * i + 2] += x[i].z;
          sv[4 * i + 3] += x[i].w;
        }
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) largest = fmaxf(largest, fabsf(sv[i]));
      const float grid = cl_grid(largest);
      uint32_t t[kClTerms][16];
#pragma unroll
      for (int i = 0; i < 16; ++i) cl_split(sv[2 * i], sv[2 * i + 1], grid, t[0][i], t[1][i], t[2][i]);
#pragma unroll
      for (int m = 0; m < kClTerms; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cc = set * 4 + c;
          *reinterpret_cast<uint4*>(smem + L::kK + (kClTerms - 1 - m) * L::kQTile + r * 128 + (cc >> 3) * L::kQHalf + (((cc & 7) ^ (r & 7)) << 4)) =
              make_uint4(t[m][4 * c], t[m][4 * c + 1], t[m][4 * c + 2], t[m][4 * c + 3]);
        }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->s_ready);
      asm volatile("bar.sync 1, %0;" ::"n"(kClWorkers) : "memory");
    }
    bool ok = __all_sync(0xffffffffu, cl_wait(&bars->q_full, 0, bars, a.status));
    if (ok) {
      if (set * 32 < D) {
        // phi(q) of this thread's row, 32 dims, as the three bf16 A operands
        uint8_t* cell[4];  // 16-byte chunks of the row
        float f[32], largest = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cc = set * 4 + c;
          cell[c] = smem + L::kQ + r * 128 + (cc >> 3) * L::kQHalf + (((cc & 7) ^ (r & 7)) << 4);
          const uint4 raw = *reinterpret_cast<const uint4*>(cell[c] + 2 * L::kQTile);
          const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            f[c * 8 + e] = cl_phi(__uint_as_float(e & 1 ? w[e >> 1] & 0xffff0000u : w[e >> 1] << 16), a.relu);
            largest = fmaxf(largest, f[c * 8 + e]);
          }
        }
        if (SUMS && groups > 0) {
          float d8[8];
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            const float4 z = *reinterpret_cast<const float4*>(zs + set * 32 + i);
            d8[i / 4] = (f[i] * z.x + f[i + 1] * z.y) + (f[i + 2] * z.z + f[i + 3] * z.w);
          }
          den = ((d8[0] + d8[1]) + (d8[2] + d8[3])) + ((d8[4] + d8[5]) + (d8[6] + d8[7]));
        }
        const float grid = cl_grid(largest);
        uint32_t t[kClTerms][16];
#pragma unroll
        for (int i = 0; i < 16; ++i) cl_split(f[2 * i], f[2 * i + 1], grid, t[0][i], t[1][i], t[2][i]);
#pragma unroll
        for (int m = 0; m < kClTerms; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(cell[c] + m * L::kQTile) = make_uint4(t[m][4 * c], t[m][4 * c + 1], t[m][4 * c + 2], t[m][4 * c + 3]);
        fence_proxy_async_smem();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->q_read);
      if (SUMS && groups > 0) {
        ok = __all_sync(0xffffffffu, cl_wait(&bars->pre_full, 0, bars, a.status));
        if (ok) {
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < NC; c += 16) {
            uint32_t v[16], w[16];
            tmem_ld16(tmem + lane_off + kClColNum + NC * set + c, v);
            tmem_ld16(tmem + lane_off + kClColPre + NC * set + c, w);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) num[c + i] = __uint_as_float(v[i]) + __uint_as_float(w[i]);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->pre_read);
        }
      }
    }
    // adds the products of step j to the running sums
    auto add_step = [&](int j) -> bool {
      if (!__all_sync(0xffffffffu, cl_wait(&bars->num_full[j & 1], (j >> 1) & 1, bars, a.status))) return false;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < NC; c += 16) {
        uint32_t v[16];
        tmem_ld16(tmem + lane_off + kClColNum + NC * set + c, v);
        tc_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) num[c + i] += __uint_as_float(v[i]);
      }
      return true;
    };
#pragma unroll 1
    for (int j = 0; j < nsteps && ok; ++j) {
      ok = __all_sync(0xffffffffu, cl_wait(&bars->a_full[j & 1], (j >> 1) & 1, bars, a.status));
      if (!ok) break;
      tc_fence_after();
      const uint32_t buf = tmem + lane_off + kClColBuf + kClBuf * (j & 1);
      uint32_t v[16], u1[16], u2[16];
      tmem_ld16(buf + 16 * set, v);
      tmem_ld16(buf + kBlock + 16 * set, u1);
      tmem_ld16(buf + 2 * kBlock + 16 * set, u2);
      const int64_t base = static_cast<int64_t>(b_first + p0 + j) * kBlock;  // token of column 0
      const int lo_col = static_cast<int>(a.q_pos0 - base);             // first visible column (<= 0: all)
      const int hi_col = static_cast<int>(a.q_pos0 + row0 - base);      // last visible column of row 0
      tc_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) + (__uint_as_float(u1[i]) + __uint_as_float(u2[i])));
      if (lo_col > 0 || hi_col < kBlock - 1) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int c = 16 * set + i;
          if (c < lo_col || c > hi_col + r) v[i] = 0u;
        }
      }
      float s4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t t[kClTerms][8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x0 = __uint_as_float(v[2 * i]), x1 = __uint_as_float(v[2 * i + 1]);
        s4[(2 * i) & 3] += x0;
        s4[(2 * i + 1) & 3] += x1;
        cl_split(x0, x1, 0.f, t[0][i], t[1][i], t[2][i]);
      }
      // (over the thread's own columns, which it has read)
      tmem_st8(buf + 16 * set, t[0]);
      tmem_st8(buf + 16 * set + 8, t[1]);
      tmem_st8(buf + kBlock + 16 * set, t[2]);
      den += (s4[0] + s4[1]) + (s4[2] + s4[3]);
      tc_wait_st();
      if (j > 0) ok = add_step(j - 1);
      tc_fence_before();
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&bars->p_ready);
    }
    if (ok) ok = add_step(nsteps - 1);
    float* dsum = reinterpret_cast<float*>(smem + L::kK);  // [4][128], dead by now
    if (ok) dsum[set * 128 + r] = den;
    // (an aborted wait leaves the loop as well: the barrier takes every worker)
    asm volatile("bar.sync 1, %0;" ::"n"(kClWorkers) : "memory");
    const int row = row0 + r;
    if (ok && row < a.n_q) {
      float* dst = a.lin_num + (static_cast<size_t>(row) * a.H + h) * D + NC * set;
      float* dst_den = set == 0 ? a.lin_den + static_cast<size_t>(row) * a.H + h : nullptr;
      den = (dsum[r] + dsum[128 + r]) + (dsum[256 + r] + dsum[384 + r]);
      bool finite = fabsf(den) <= FLT_MAX;
#pragma unroll
      for (int i = 0; i < NC; ++i) finite = finite && fabsf(num[i]) <= FLT_MAX;
      if (finite) {
#pragma unroll
        for (int i = 0; i < NC / 4; ++i)
          reinterpret_cast<float4*>(dst)[i] = make_float4(num[4 * i], num[4 * i + 1], num[4 * i + 2], num[4 * i + 3]);
        if (dst_den) *dst_den = den;
      } else {
        const size_t term = static_cast<size_t>(a.phik_blocks) * kBlock * D;
        cl_plain_row<D>(smem + L::kQ, r, a.phik + h * kClTerms * term, term, a.v_pool, a.page_table + b_first, a.H, h,
                        static_cast<int>(a.q_pos0 - static_cast<int64_t>(b_first) * kBlock), row + 1, NC * set, dst, dst_den);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

namespace {
using ClKernel = void (*)(CausalLinArgs, CUtensorMap, CUtensorMap, CUtensorMap);
ClKernel cl_kernel(int D, bool sums) {
  return D == 64 ? causal_linear_kernel<64, false> : sums ? causal_linear_kernel<128, true> : causal_linear_kernel<128, false>;
}
int cl_smem(int D) { return D == 128 ? ClSmem<128>::kTotal : ClSmem<64>::kTotal; }
}  // namespace

cudaError_t causal_linear_init() {
  cudaError_t e = cudaFuncSetAttribute(chunk_sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCsSmem);
  for (int i = 0; i < 3 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(cl_kernel(i == 2 ? 64 : 128, i == 1), cudaFuncAttributeMaxDynamicSharedMemorySize, cl_smem(i == 2 ? 64 : 128));
  return e;
}

int causal_sum_groups(int tokens) { return (tokens + kTileM - 1) / kTileM * 2 / kClGroup; }
size_t causal_sums_bytes(int heads, int tokens) { return static_cast<size_t>(heads) * causal_sum_groups(tokens) * kClSums * 4; }

cudaError_t launch_causal_linear(const CausalLinArgs& a_in, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                                 const CUtensorMap& tm_v, cudaStream_t st) {
  CausalLinArgs a = a_in;
  const int n_tiles = (a.n_q + kTileM - 1) / kTileM;
  const int64_t pages = (a.q_pos0 + a.n_q - 1) / kBlock - a.q_pos0 / kBlock + 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(pages), a.H);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, a.D == 128 ? phi_terms_kernel<128> : phi_terms_kernel<64>, a);
  if (e != cudaSuccess) return e;
  if (a.D != 128 || !sums_pay(n_tiles, a.H, a.nsm, a.alone)) a.sums = nullptr;
  if (a.sums) {
    cfg.gridDim = dim3(static_cast<unsigned>((n_tiles - 1) * 2 / kClGroup), a.H);  // (nothing reads the last tiles' own group)
    cfg.blockDim = dim3(kCsThreads);
    cfg.dynamicSmemBytes = kCsSmem;
    const cudaError_t es = cudaLaunchKernelEx(&cfg, chunk_sums_kernel, a, tm_k, tm_v);
    if (es != cudaSuccess) return es;
  }
  cfg.gridDim = dim3(static_cast<unsigned>(n_tiles) * a.H);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = cl_smem(a.D);
  return cudaLaunchKernelEx(&cfg, cl_kernel(a.D, a.sums != nullptr), a, tm_q, tm_k, tm_v);
}

}  // namespace hsa

// hsa_append_kv kernels: pool write + per-block key sums, and the linear-branch state update
//   S[h] += sum_j phi(k_j)^T v_j,   z[h] += sum_j phi(k_j),   phi(x) = elu(x) + 1
// as a deterministic two-stage reduction (no floating-point atomics).
#include <cuda_bf16.h>

#include <cfloat>

#include "hsa_internal.h"
#include "ptx.cuh"

namespace hsa {

// ---------------------------------------------------------------------------------------
// Without a linear state: one CTA per (touched block, head).  Copies the new rows of K and V into the block's
// page and adds their column sums to the block's key sum.  A CTA owns its (head, block)
// exclusively, so the sum order is fixed.
// ---------------------------------------------------------------------------------------
template <int D, bool ALL_ROWS>  // ALL_ROWS: a thread asks for all of its rows before the first of them is consumed
__global__ void __launch_bounds__(256, ALL_ROWS && D == 128 ? 4 : kPageCtasPerSm) append_pool_ksum_kernel(AppendArgs a) {
  constexpr int CH = D / 8;     // 16-byte chunks per row
  constexpr int RP = 256 / CH;  // rows handled per pass
  __shared__ float red[RP][D];

  const int h = blockIdx.y;
  const int64_t b = a.n0 / kBlock + blockIdx.x;
  const int64_t t_lo = max(a.n0, b * kBlock);
  const int64_t t_hi = min(a.n0 + a.n_new, b * kBlock + kBlock);
  const int c8 = threadIdx.x % CH;
  const int rg = threadIdx.x / CH;
  const int page = a.page_table[b];
  const size_t row_base = (static_cast<size_t>(page) * a.H + h) * kBlock;

  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  auto add_row = [&acc](const uint4& kk) {
    const __nv_bfloat162* k2 = reinterpret_cast<const __nv_bfloat162*>(&kk);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __bfloat1622float2(k2[i]);
      acc[2 * i] += f.x;
      acc[2 * i + 1] += f.y;
    }
  };

  if constexpr (ALL_ROWS) {
    constexpr int NR = kBlock / RP;
    uint4 kk[NR], vv[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const int64_t t = t_lo + rg + i * RP;
      if (t < t_hi) {
        const size_t src = static_cast<size_t>(t - a.n0) * a.tok_stride + static_cast<size_t>(h) * a.head_stride + c8 * 8;
        kk[i] = *reinterpret_cast<const uint4*>(a.k + src);
        vv[i] = *reinterpret_cast<const uint4*>(a.v + src);
      }
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const int64_t t = t_lo + rg + i * RP;
      if (t < t_hi) {
        const size_t dst = (row_base + (t - b * kBlock)) * D + c8 * 8;
        *reinterpret_cast<uint4*>(a.k_pool + dst) = kk[i];
        *reinterpret_cast<uint4*>(a.v_pool + dst) = vv[i];
        add_row(kk[i]);
      }
    }
  } else {
    for (int64_t t = t_lo + rg; t < t_hi; t += RP) {
      const size_t src = static_cast<size_t>(t - a.n0) * a.tok_stride + static_cast<size_t>(h) * a.head_stride + c8 * 8;
      const uint4 kk = *reinterpret_cast<const uint4*>(a.k + src);
      const uint4 vv = *reinterpret_cast<const uint4*>(a.v + src);
      const size_t dst = (row_base + (t - b * kBlock)) * D + c8 * 8;
      *reinterpret_cast<uint4*>(a.k_pool + dst) = kk;
      *reinterpret_cast<uint4*>(a.v_pool + dst) = vv;
      add_row(kk);
    }
  }
  // Rows of a partial tail page past the last token are zero-filled: the forward kernel masks
  // their scores, but 0 * (uninitialised V) must not be able to produce a NaN.
  for (int64_t t = t_hi + rg; t < b * kBlock + kBlock; t += RP) {
    const size_t dst = (row_base + (t - b * kBlock)) * D + c8 * 8;
    *reinterpret_cast<uint4*>(a.k_pool + dst) = make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(a.v_pool + dst) = make_uint4(0, 0, 0, 0);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) red[rg][c8 * 8 + i] = acc[i];
  __syncthreads();
  if (threadIdx.x < D) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < RP; ++r) s += red[r][threadIdx.x];
    float* dst = a.ksum + (static_cast<size_t>(h) * a.max_pages + b) * D + threadIdx.x;
    float old = 0.f;
    if (t_lo > b * kBlock) {  // block already partly filled: its sum before this append
      float* saved = a.ksum_saved + static_cast<size_t>(h) * D + threadIdx.x;
      old = a.tail_from_saved ? *saved : *dst;
      if (!a.tail_from_saved) *saved = old;
    }
    *dst = old + s;
  }
  // Launched as a programmatic dependent (Linformer form: behind the compression kernel, whose
  // outputs it does not touch) this grid runs beside that kernel and waits for it only here, so
  // that its own end implies that kernel's.  Launched normally this is a no-op.
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// sum of phi(k) v (v null: of phi(k)) over n tokens, one after another in fp32.  (Plain arguments: the whole
// AppendArgs by reference would be copied to the stack by every thread of the caller.)
__device__ __noinline__ float chunk_sum(const __nv_bfloat16* k, const __nv_bfloat16* v, int64_t tok_stride, int n, int relu) {
  float sum = 0.f;
  for (int t = 0; t < n; ++t) {
    const float x = __bfloat162float(k[t * tok_stride]);
    const float f = relu ? fmaxf(x, 0.f) : (x > 0.f ? x + 1.f : expf(x));
    sum = v ? fmaf(f, __bfloat162float(v[t * tok_stride]), sum) : sum + f;
  }
  return sum;
}

// ---------------------------------------------------------------------------------------
// Reduction: S[dst] <- S[src] + sum of partials (fixed order), with its bf16 hi/lo split (the forward
// kernels feed hi and lo to the tensor cores as two bf16 operands), the same for z and its operand image.
// ---------------------------------------------------------------------------------------
template <int D>
__global__ void state_reduce_kernel(AppendArgs a) {
  constexpr int DD = D * D;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int h = blockIdx.y;
  if (idx >= DD + D) return;
  // results of the kernel before this one are needed from here on
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float* part = a.spart + static_cast<size_t>(h) * a.nsplit * (DD + D) + idx;
  // all partials are fetched at once (independent loads in flight); the sum order stays fixed
  float v[kStateSplitMax];
#pragma unroll
  for (int i = 0; i < kStateSplitMax; ++i)
    v[i] = (i < a.nsplit) ? __ldcg(&part[static_cast<size_t>(i) * (DD + D)]) : 0.f;
  float add = 0.f;
#pragma unroll
  for (int i = 0; i < kStateSplitMax; ++i) add += v[i];
  // head_dim 64: an Inf that meets the zeros of the split products (zero terms, Inf - Inf in the split itself)
  // gives NaN where the sum of phi(k) v is Inf, so a sum that is not finite is taken again term by term
  if (D == 64 && !(fabsf(add) <= FLT_MAX)) {
    const __nv_bfloat16* kh = a.k + static_cast<size_t>(h) * a.head_stride;
    const __nv_bfloat16* vh = a.v + static_cast<size_t>(h) * a.head_stride;
    add = idx < DD ? chunk_sum(kh + idx / D, vh + idx % D, a.tok_stride, a.n_new, a.relu)
                   : chunk_sum(kh + idx - DD, nullptr, a.tok_stride, a.n_new, a.relu);
  }
  const int dst = a.src_slot ^ 1;
  if (idx < DD) {
    const size_t o = static_cast<size_t>(h) * DD + idx;
    const float s_new = a.S[a.src_slot][o] + add;
    a.S[dst][o] = s_new;
    __nv_bfloat16* hl = a.hilo + (static_cast<size_t>(h) * 2 + dst) * 2 * DD + idx;
    const __nv_bfloat16 nh = __float2bfloat16_rn(s_new);
    hl[0] = nh;
    hl[DD] = __float2bfloat16_rn(s_new - __bfloat162float(nh));
  } else {
    const int k = idx - DD;
    const size_t o = static_cast<size_t>(h) * D + k;
    const float z_new = a.z[a.src_slot][o] + add;
    a.z[dst][o] = z_new;
    if (D == 128) {
      // operand image of z: element (row n, dim k) of a K-major tile with the 128-byte swizzle sits
      // at slab (k / 64), row n, 16-byte chunk ((k % 64) / 8) ^ (n % 8)
      const int slab = k >> 6, kk = k & 63, c = kk >> 3;
      uint8_t* img = a.zop + static_cast<size_t>(h * 2 + dst) * kZopBytes + slab * (kZopBytes / 2) + (kk & 7) * 2;
      const __nv_bfloat16 hi = __float2bfloat16_rn(z_new);
      *reinterpret_cast<__nv_bfloat16*>(img + 0 * 128 + ((c ^ 0) << 4)) = hi;
      *reinterpret_cast<__nv_bfloat16*>(img + 1 * 128 + ((c ^ 1) << 4)) = __float2bfloat16_rn(z_new - __bfloat162float(hi));
    }
  }
}

// ---------------------------------------------------------------------------------------
// Fused append with the linear state (the measured path): one pass over the chunk's K and V in which
// no thread touches global memory for the bulk data.
// grid (nsplit, H); a CTA owns a run of consecutive history blocks of one head.  Per block
//   * the producer lane brings the block's rows of K and V into a 4-deep ring by TMA (rows
//     outside the chunk arrive as zeros) and sends the same tiles on to the block's page by
//     TMA store (a block that already held tokens before this call is written row by row by
//     the workers instead, so that its old rows stay),
//   * sixteen worker warps (two groups on alternate blocks) read K from the ring and build phi(K) as
//     bf16 terms in the 128-byte-swizzled MN-major layout,
//   * the MMA lane lets the tensor cores accumulate, over the block's tokens (tcgen05, K = tokens)
//       S_part (d x d, fp32 in TMEM)   += phi(K)^T V      (V straight from the ring)
//       z_part (d x 16)                += phi(K)^T 1
//       ksum_b (d x 16)                 = K^T 1           (K straight from the ring)
//     and four more warps read ksum_b back as soon as it is final,
// and finally the CTA writes its partial S and z for the fixed-order reduction below.
// head_dim 128: phi(K) = hi + lo (~16 bits), two products into one accumulator of 128 lanes.
// head_dim 64: phi(K) = hi + mid + lo (~24 bits: this size was summed in fp32 before it came here).  A
// product has 128 lanes, so that hi and mid go through it together, as the two 64-lane halves of one
// operand (their tiles lie one behind the other), and lo with a tile of zeros (beside hi, on mid's lanes).
// Every product truncates what it adds to, so the products take turns at four accumulators, and those and
// the two halves are added in rounded fp32 when the partial state is written.  The key sums are taken by the
// workers and the key-sum warps, in rounded fp32 and, for a block that is new as a whole, in the order of the
// page kernel above.
// Error against 64 bits, the fp32 SIMT kernels this replaced -> now (2-norm, N(0, 1) inputs): 16 heads, 1000
// tokens, S 1.6e-7 -> 7.8e-8, z 7.4e-8 -> 5.1e-8; 40 heads, 4680 tokens, S 5.8e-7 -> 2.9e-7, z 4.9e-7 ->
// 3.4e-8; with one accumulator per two blocks S was 8.4e-8 and 6.3e-7.
// Measured, the whole append replayed from a graph: 16 heads, 1000 tokens 13.6 -> 7.6 us (the 8.3 MB take 1.3 us at
// the copy bandwidth: what is left is latency, of launch, first data and two kernels), 8 heads, 4680 tokens
// 26.2 -> 11.5 us.
// Every wait is bounded; on expiry the CTA records a timeout and leaves.
// ---------------------------------------------------------------------------------------

namespace {

constexpr int kAfDepth = 4;                      // ring stages
constexpr int kAfWorkers = 512;                  // worker threads (warps 2..17)
constexpr int kAfThreads = 64 + kAfWorkers + 128;  // + producer warp + MMA warp + 4 key-sum warps
constexpr int kAfOnes = 2048;                    // [16 x 64] bf16 ones (K-major operand)
constexpr uint32_t kAfColZ = 128, kAfColKs = 144;  // TMEM columns: S from 0, z, ksum[2]
constexpr uint32_t kAfColZ64 = 256;                 // head_dim 64: S[4] from 0, z[4]

template <int D>
struct AfSmem {
  static constexpr int kTile = 64 * D * 2;     // [64 tokens x D dims] bf16 = D / 64 swizzled slabs
  static constexpr int kSlab = 64 * 128;       // bytes of one slab
  static constexpr int kStage = 2 * kTile;     // K | V
  static constexpr int kTerms = D == 128 ? 2 : 3;
  static constexpr int kPhi = kTerms * kTile;  // phi(K) of a block: hi | lo or hi | mid | lo
  static constexpr int kZeros = D == 128 ? 0 : kTile;  // (a tile of zeros in front of the two phi buffers)
  static constexpr int kKsum = D == 128 ? 0 : 2 * 32 * D * 4;  // column sums of every 32nd row, two buffers
  static constexpr int kTotal = kAfDepth * kStage + 2 * kPhi + kZeros + kAfOnes + 256 + kKsum + 1024;
  static constexpr int kPitch = D + 4;  // floats per row of the staged partial state
  static constexpr uint32_t kTmemCols = D == 128 ? 256 : 512;
  static_assert(128 * kPitch * 4 <= 2 * kPhi + kZeros + kAfOnes, "partial state is staged in the phi + ones area");
};

struct AfBars {
  uint64_t full[kAfDepth];      // ring stage landed
  uint64_t consumed[kAfDepth];  // tensor cores are done with the stage
  uint64_t phi_ready[2];        // hi/lo buffer written
  uint64_t mma_done[2];         // tensor cores are done with the hi/lo buffer (and ksum is final)
  uint64_t ks_read[2];          // key-sum buffer read back
  uint32_t tmem_base;
  volatile int abort_flag;
};

__device__ __forceinline__ bool af_wait(uint64_t* bar, uint32_t parity, AfBars* bars, int32_t* status) {
  if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t i = 1; i < (1u << 24); ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 1023u) == 0u && bars->abort_flag) return false;
  }
  bars->abort_flag = 1;
  atomicCAS(status, 0, kDevTimeout);
  return false;
}

// Either feature map.  elu(x) + 1 = max(x, 0) + exp(min(x, 0)), branch-free; head_dim 128 takes the fast
// exponential (relative error ~1e-6, far inside what two bf16 terms carry), head_dim 64 expf.
template <int D, bool RELU>
__device__ __forceinline__ float af_phi(float x) {
  if (RELU) return fmaxf(x, 0.f);
  float e;
  if (D == 128)
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fminf(x, 0.f) * 1.4426950408889634f));
  else
    return x > 0.f ? x + 1.f : expf(x);
  return fmaxf(x, 0.f) + e;
}

__device__ __forceinline__ void tma_store_2d(const void* tmap, const void* smem_src, int32_t x, int32_t y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}

}  // namespace

// RELU: the feature map is max(x, 0) instead of elu(x) + 1 (an instance of its own: the map sits in
// the innermost loop of the worker warps)
template <int D, bool RELU>
__global__ void __launch_bounds__(kAfThreads, 1)
append_fused_kernel(AppendArgs a, int blocks_per_cta, const __grid_constant__ CUtensorMap tm_kin,
                    const __grid_constant__ CUtensorMap tm_vin, const __grid_constant__ CUtensorMap tm_kpool,
                    const __grid_constant__ CUtensorMap tm_vpool) {
  using L = AfSmem<D>;
  extern __shared__ uint8_t af_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(af_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* ring = smem;
  uint8_t* zeros = smem + kAfDepth * L::kStage;
  uint8_t* phi = zeros + L::kZeros;
  uint8_t* ones = phi + 2 * L::kPhi;
  AfBars* bars = reinterpret_cast<AfBars*>(ones + kAfOnes);

  // the reduction kernel behind this one may be scheduled early; it waits for this grid itself
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // This grid is itself launched as a programmatic dependent: it may be scheduled while the kernel
  // before it in the stream (the forward kernel of the layer before) is still finishing.  The
  // set-up below touches nothing of that kernel's; every thread waits for its end (wait_prior)
  // before the first load of the inputs is issued and before the CTA-wide barrier.
  auto wait_prior = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };

  const int h = blockIdx.y, split = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t b_first = a.n0 / kBlock, b_last = (a.n0 + a.n_new - 1) / kBlock;
  const int64_t bs = b_first + static_cast<int64_t>(split) * blocks_per_cta;
  const int64_t be = min64(b_last + 1, bs + blocks_per_cta);
  const int nblk = static_cast<int>(max64(0, be - bs));
  const int64_t n_end = a.n0 + a.n_new;

  auto issue_loads = [&](int bi) {
    const int s = bi % kAfDepth;
    uint8_t* st = ring + s * L::kStage;
    const int32_t row0 = static_cast<int32_t>((bs + bi) * kBlock - a.n0);  // may be negative: zero fill
    mbar_expect_tx(&bars->full[s], L::kStage);
#pragma unroll
    for (int dh = 0; dh < D / 64; ++dh) tma_load_3d(st + dh * L::kSlab, &tm_kin, &bars->full[s], dh * 64, h, row0);
#pragma unroll
    for (int dh = 0; dh < D / 64; ++dh)
      tma_load_3d(st + L::kTile + dh * L::kSlab, &tm_vin, &bars->full[s], dh * 64, h, row0);
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < kAfDepth; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->consumed[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->phi_ready[s], kAfWorkers / 2);  // one worker group per buffer
      mbar_init(&bars->mma_done[s], 1);
      mbar_init(&bars->ks_read[s], 4);
    }
    bars->abort_flag = 0;
    fence_mbar_init();
    wait_prior();
    // the first ring fill starts before the rest of the CTA is set up
    for (int bi = 0; bi < nblk && bi < kAfDepth; ++bi) issue_loads(bi);
    tma_prefetch_desc(&tm_kpool);
    tma_prefetch_desc(&tm_vpool);
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, L::kTmemCols);
    tmem_relinquish();
  }
  // bf16 1.0 everywhere: under any swizzle the tile reads as all ones
  for (int i = threadIdx.x; i < kAfOnes / 4; i += kAfThreads) reinterpret_cast<uint32_t*>(ones)[i] = 0x3F803F80u;
  for (int i = threadIdx.x; i < L::kZeros / 16; i += kAfThreads)
    reinterpret_cast<uint4*>(zeros)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  wait_prior();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (one lane)
    if (elect_one_sync()) {
      bool ok = true;
      for (int bi = 0; bi < nblk && ok; ++bi) {
        const int s = bi % kAfDepth;
        ok = af_wait(&bars->full[s], (bi / kAfDepth) & 1, bars, a.status);
        if (!ok) break;
        const int64_t b = bs + bi;
        if (b * kBlock >= a.n0) {  // the block holds nothing older: whole tiles go to its page
          uint8_t* st = ring + s * L::kStage;
          const int32_t prow = (a.page_table[b] * a.H + h) * kBlock;
#pragma unroll
          for (int dh = 0; dh < D / 64; ++dh) tma_store_2d(&tm_kpool, st + dh * L::kSlab, dh * 64, prow);
#pragma unroll
          for (int dh = 0; dh < D / 64; ++dh) tma_store_2d(&tm_vpool, st + L::kTile + dh * L::kSlab, dh * 64, prow);
        }
        tma_store_commit();
        if (bi >= 1 && bi - 1 + kAfDepth < nblk) {
          // refill the stage of block bi - 1: its stores have read it, the tensor cores are done
          asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
          ok = af_wait(&bars->consumed[(bi - 1) % kAfDepth], ((bi - 1) / kAfDepth) & 1, bars, a.status);
          if (ok) issue_loads(bi - 1 + kAfDepth);
        }
      }
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // every page write has landed
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one lane)
    if (elect_one_sync()) {
      constexpr uint32_t idesc_s = idesc_bf16_f32(128, D, 1, 1);
      constexpr uint32_t idesc_1 = idesc_bf16_f32(128, 16, 1, 0);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      const uint32_t b_ones = desc_lo_sw128(smem_u32(ones), 16);
      for (int bi = 0; bi < nblk; ++bi) {
        const int s = bi % kAfDepth, hb = bi & 1;
        if (!af_wait(&bars->phi_ready[hb], (bi >> 1) & 1, bars, a.status)) break;
        tc_fence_after();
        uint8_t* st = ring + s * L::kStage;
        uint8_t* ph = phi + hb * L::kPhi;
        // lanes 0..63 and 64..127 of the A operands: the two slabs of a tile (head_dim 128), two tiles
        // one behind the other or the zeros and lo (head_dim 64)
        const uint32_t a_k = desc_lo_sw128(smem_u32(st), L::kSlab);
        const uint32_t b_v = desc_lo_sw128(smem_u32(st + L::kTile), L::kSlab);
        const uint32_t a_1 = desc_lo_sw128(smem_u32(ph), L::kSlab);
        const uint32_t a_2 = D == 128 ? desc_lo_sw128(smem_u32(ph + L::kTile), L::kSlab)
                                      : desc_lo_sw128(smem_u32(zeros), L::kZeros + hb * L::kPhi + 2 * L::kTile);
        // accumulators of product kk and whether they hold earlier ones
        auto acc_s = [&](int kk) { return tmem + (D == 64 ? 64 * (2 * hb + (kk & 1)) : 0); };
        auto acc_z = [&](int kk) { return tmem + (D == 64 ? kAfColZ64 + 16 * (2 * hb + (kk & 1)) : kAfColZ); };
        auto more = [&](int kk) { return (D == 64 ? bi >= 2 || kk >= 2 : bi > 0 || kk > 0) ? 1u : 0u; };
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma_ss_lo(acc_s(kk), a_1 + kk * 128, b_v + kk * 128, hi, idesc_s, more(kk));
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc_mma_ss_lo(acc_s(kk), a_2 + kk * 128, b_v + kk * 128, hi, idesc_s, 1u);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma_ss_lo(acc_z(kk), a_1 + kk * 128, b_ones, hi, idesc_1, more(kk));
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) tc_mma_ss_lo(acc_z(kk), a_2 + kk * 128, b_ones, hi, idesc_1, 1u);
        if constexpr (D == 128) {
          if (bi >= 2 && !af_wait(&bars->ks_read[hb], ((bi >> 1) - 1) & 1, bars, a.status)) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc_mma_ss_lo(tmem + kAfColKs + hb * 16, a_k + kk * 128, b_ones, hi, idesc_1, kk > 0 ? 1u : 0u);
        }
        tc_commit(&bars->consumed[s]);
        tc_commit(&bars->mma_done[hb]);
      }
    }
  } else if (warp >= 2 + kAfWorkers / 32) {
    // ------------------------------------------------------------------ key-sum warps
    // key sum of each block: one warp per TMEM lane quadrant, as soon as the block's MMAs are done
    // (head_dim 64: two warps that add up the workers' sums)
    const int quad = warp & 3;
    for (int bj = 0; bj < nblk; ++bj) {
      if (!af_wait(D == 128 ? &bars->mma_done[bj & 1] : &bars->phi_ready[bj & 1], (bj >> 1) & 1, bars, a.status)) break;
      float sum = 0.f;
      if constexpr (D == 128) {
        tc_fence_after();
        uint32_t v[16];
        tmem_ld16(tmem + (static_cast<uint32_t>(quad * 32) << 16) + kAfColKs + (bj & 1) * 16, v);
        tc_wait_ld();
        sum = __uint_as_float(v[0]);
        tc_fence_before();
      } else if (quad * 32 < D) {
        const float* col = reinterpret_cast<const float*>(ones + kAfOnes + 256) + (bj & 1) * (L::kKsum / 8) + quad * 32 + lane;
#pragma unroll
        for (int r = 0; r < L::kKsum / (2 * D * 4); ++r) sum += col[r * D];
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(&bars->ks_read[bj & 1]);
      if (quad * 32 >= D) continue;
      const int64_t b = bs + bj;
      float* dst = a.ksum + (static_cast<size_t>(h) * a.max_pages + b) * D + quad * 32 + lane;
      float old = 0.f;
      if (a.n0 > b * kBlock) {  // block partly filled before: its sum before this append
        float* saved = a.ksum_saved + static_cast<size_t>(h) * D + quad * 32 + lane;
        old = a.tail_from_saved ? *saved : *dst;
        if (!a.tail_from_saved) *saved = old;
      }
      *dst = old + sum;
    }
  } else {
    // ------------------------------------------------------------------ workers
    // two groups of eight warps take alternate blocks, so that one group's waits hide under the
    // other's arithmetic
    const int w = threadIdx.x - 64;
    const int grp = w >> 8, wg = w & 255;
    constexpr int CH = D / 8;              // 16-byte chunks of a row (8 dims)
    constexpr int RS = kAfWorkers / 2 / CH;  // rows one pass of a group covers
    constexpr int NI = kBlock / RS;
    const int ch = wg % CH;
    const int rg = wg / CH;  // rows rg, rg + RS, ... of a block
    const int quad = warp & 3;
    bool ok = true;
    uint32_t soff[NI];  // the thread's 16-byte chunks inside a swizzled tile
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int r = rg + RS * i;
      soff[i] = (ch >> 3) * L::kSlab + r * 128 + (((ch & 7) ^ (r & 7)) << 4);
    }
#pragma unroll 1
    for (int bi = grp; bi < nblk && ok; bi += 2) {
      const int s = bi % kAfDepth, hb = bi & 1;
      const int64_t b = bs + bi;
      ok = af_wait(&bars->full[s], (bi / kAfDepth) & 1, bars, a.status);
      if (!ok) break;
      const uint8_t* st_k = ring + s * L::kStage;
      uint4 kreg[NI];
#pragma unroll
      for (int i = 0; i < NI; ++i) kreg[i] = *reinterpret_cast<const uint4*>(st_k + soff[i]);
      if (b * kBlock < a.n0) {
        // block partly filled before this call: only its new rows (and the zero rows past the
        // last token) are written, by hand
        const size_t row_base = (static_cast<size_t>(a.page_table[b]) * a.H + h) * kBlock;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int r = rg + RS * i;
          const int64_t t = b * kBlock + r;
          if (t >= a.n0) {
            const size_t dst = (row_base + r) * D + ch * 8;
            *reinterpret_cast<uint4*>(a.k_pool + dst) = kreg[i];
            *reinterpret_cast<uint4*>(a.v_pool + dst) = *reinterpret_cast<const uint4*>(st_k + L::kTile + soff[i]);
          }
        }
      }
      if (bi >= 2) {
        ok = af_wait(&bars->mma_done[hb], ((bi >> 1) - 1) & 1, bars, a.status);
        if (!ok) break;
      }
      if constexpr (D == 64) {
        // the thread's column sums (rows outside the chunk are zeros) for the key-sum warps
        if (bi >= 2) {
          ok = af_wait(&bars->ks_read[hb], ((bi >> 1) - 1) & 1, bars, a.status);
          if (!ok) break;
        }
        static_assert(NI == 2 && RS * D * 4 * 2 == L::kKsum, "a thread holds two rows of a block");
        const uint32_t* w0 = reinterpret_cast<const uint32_t*>(&kreg[0]);
        const uint32_t* w1 = reinterpret_cast<const uint32_t*>(&kreg[1]);
        float4* dst = reinterpret_cast<float4*>(ones + kAfOnes + 256) + hb * (L::kKsum / 32) + (rg * D + ch * 8) / 4;
#pragma unroll
        for (int e = 0; e < 4; e += 2)
          dst[e / 2] = make_float4(__uint_as_float(w0[e] << 16) + __uint_as_float(w1[e] << 16),
                                   __uint_as_float(w0[e] & 0xffff0000u) + __uint_as_float(w1[e] & 0xffff0000u),
                                   __uint_as_float(w0[e + 1] << 16) + __uint_as_float(w1[e + 1] << 16),
                                   __uint_as_float(w0[e + 1] & 0xffff0000u) + __uint_as_float(w1[e + 1] & 0xffff0000u));
      }
      uint8_t* ph = phi + hb * L::kPhi;
      // rows outside the chunk (only in its first and last block) add nothing to the state
      const bool whole = b * kBlock >= a.n0 && b * kBlock + kBlock <= n_end;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const uint32_t* kw = reinterpret_cast<const uint32_t*>(&kreg[i]);
        uint32_t tw[L::kTerms][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float p0 = af_phi<D, RELU>(__uint_as_float(kw[e] << 16));
          float p1 = af_phi<D, RELU>(__uint_as_float(kw[e] & 0xffff0000u));
#pragma unroll
          for (int t = 0; t < L::kTerms; ++t) {
            tw[t][e] = pack_bf16(p0, p1);
            p0 -= __uint_as_float(tw[t][e] << 16);
            p1 -= __uint_as_float(tw[t][e] & 0xffff0000u);
          }
        }
        if (!whole) {
          const int64_t t = b * kBlock + rg + RS * i;
          if (t < a.n0 || t >= n_end) {
#pragma unroll
            for (int m = 0; m < L::kTerms; ++m)
#pragma unroll
              for (int e = 0; e < 4; ++e) tw[m][e] = 0u;
          }
        }
#pragma unroll
        for (int m = 0; m < L::kTerms; ++m)
          *reinterpret_cast<uint4*>(ph + m * L::kTile + soff[i]) = make_uint4(tw[m][0], tw[m][1], tw[m][2], tw[m][3]);
      }
      fence_proxy_async_smem();  // generic-proxy writes above -> visible to the tensor cores
      mbar_arrive(&bars->phi_ready[hb]);
    }
    // the partial state, once every MMA is done: the last two blocks' barriers, in block order (a
    // group has not watched the other group's barrier, so it must not skip a phase of it)
    for (int bj = max(0, nblk - 2); bj < nblk && ok; ++bj)
      ok = af_wait(&bars->mma_done[bj & 1], (bj >> 1) & 1, bars, a.status);
    tc_fence_after();
    float* out = a.spart + (static_cast<size_t>(h) * a.nsplit + split) * (D * D + D);
    const int row = quad * 32 + lane;
    {
      // TMEM -> shared memory (row pitch D + 4 floats: conflict-free both ways) -> coalesced rows
      float* stage = reinterpret_cast<float*>(phi);
      constexpr int NC = D / 4;  // four warps per lane quadrant, NC columns each
      uint32_t v[NC];
      const int col = ((warp - 2) >> 2) * NC;
      const bool zw = ((warp - 2) >> 2) == 0;  // this warp takes the quadrant's z as well
      uint32_t zv[16];
      zv[0] = 0u;
      if (nblk > 0 && ok) {
        const uint32_t t_row = tmem + (static_cast<uint32_t>(quad * 32) << 16);
        if constexpr (D == 128)
          tmem_ld32(t_row + col, v);
        else
          tmem_ld16(t_row + col, v);
        if (zw) tmem_ld16(t_row + (D == 64 ? kAfColZ64 : kAfColZ), zv);
        tc_wait_ld();
        if constexpr (D == 64) {
          // the other accumulators: (0 + 1) + (2 + 3), the last two only of a second block
          auto add = [](uint32_t x, uint32_t y) { return __float_as_uint(__uint_as_float(x) + __uint_as_float(y)); };
          uint32_t u[3][NC];
#pragma unroll
          for (int m = 0; m < 3; ++m) tmem_ld16(t_row + 64 * (m + 1) + col, u[m]);
          tc_wait_ld();
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            v[i] = add(v[i], u[0][i]);
            if (nblk > 1) v[i] = add(v[i], add(u[1][i], u[2][i]));
          }
          if (zw) {
#pragma unroll
            for (int m = 0; m < 3; ++m) tmem_ld16(t_row + kAfColZ64 + 16 * (m + 1), u[m]);
            tc_wait_ld();
            zv[0] = add(zv[0], u[0][0]);
            if (nblk > 1) zv[0] = add(zv[0], add(u[1][0], u[2][0]));
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < NC; ++i) v[i] = 0u;
      }
      float4* srow = reinterpret_cast<float4*>(stage + row * L::kPitch + col);
#pragma unroll
      for (int i = 0; i < NC / 4; ++i)
        srow[i] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                              __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
      if (zw) {
        if (D == 128)
          out[D * D + row] = __uint_as_float(zv[0]);
        else
          stage[row * L::kPitch + D] = __uint_as_float(zv[0]);
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kAfWorkers) : "memory");
#pragma unroll
      for (int i = 0; i < D * D / 4 / kAfWorkers; ++i) {
        const int f = w + kAfWorkers * i;  // float4 index of the [D][D] partial state
        const int r2 = f / (D / 4), c4 = f % (D / 4);
        float4 o = *reinterpret_cast<const float4*>(stage + r2 * L::kPitch + c4 * 4);
        if (D == 64) {  // lanes 64..127 hold the mid terms
          const float4 m = *reinterpret_cast<const float4*>(stage + (r2 + 64) * L::kPitch + c4 * 4);
          o = make_float4(o.x + m.x, o.y + m.y, o.z + m.z, o.w + m.w);
        }
        reinterpret_cast<float4*>(out)[f] = o;
      }
      if (D == 64 && w < D) out[D * D + w] = stage[w * L::kPitch + D] + stage[(w + 64) * L::kPitch + D];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, L::kTmemCols);
  }
}

namespace {
using AppendKernel = void (*)(AppendArgs, int, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap);
template <int D>
AppendKernel fused_kernel(bool relu) {
  return relu ? append_fused_kernel<D, true> : append_fused_kernel<D, false>;
}
}  // namespace

cudaError_t append_init() {
  cudaError_t e = cudaSuccess;
  for (int relu = 0; relu < 2 && e == cudaSuccess; ++relu) {
    e = cudaFuncSetAttribute(fused_kernel<128>(relu), cudaFuncAttributeMaxDynamicSharedMemorySize, AfSmem<128>::kTotal);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fused_kernel<64>(relu), cudaFuncAttributeMaxDynamicSharedMemorySize, AfSmem<64>::kTotal);
  }
  return e;
}

cudaError_t launch_append(const AppendArgs& a_in, const AppendMaps* maps, cudaStream_t st) {
  AppendArgs a = a_in;
  const int64_t b0 = a.n0 / kBlock;
  const int64_t b1 = (a.n0 + a.n_new - 1) / kBlock;
  cudaError_t e;
  if (a.lin_state) {
    const int nb = static_cast<int>(b1 - b0 + 1);
    const int per = (nb + a.nsplit - 1) / a.nsplit;
    a.nsplit = (nb + per - 1) / per;  // no empty CTAs
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.nsplit, a.H);
    cfg.blockDim = dim3(kAfThreads);
    cfg.dynamicSmemBytes = a.D == 128 ? AfSmem<128>::kTotal : AfSmem<64>::kTotal;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AppendKernel fn = a.D == 128 ? fused_kernel<128>(a.relu) : fused_kernel<64>(a.relu);
    e = cudaLaunchKernelEx(&cfg, fn, a, per, maps->kin, maps->vin, maps->kpool, maps->vpool);
    if (e != cudaSuccess) return e;
  } else {
    dim3 gridA(static_cast<unsigned>(b1 - b0 + 1), a.H);
    cudaLaunchConfig_t cfgA{};
    cfgA.gridDim = gridA;
    cfgA.blockDim = dim3(256);
    cfgA.stream = st;
    cudaLaunchAttribute attrA[1];
    attrA[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrA[0].val.programmaticStreamSerializationAllowed = 1;
    cfgA.attrs = attrA;
    cfgA.numAttrs = a.beside_prior ? 1 : 0;  // (only behind a kernel whose outputs this one leaves alone)
    // All of a thread's rows at once is one round trip to memory instead of four, in 61 registers: four CTAs to an SM.  The loop
    // takes it where it alone runs all CTAs at once (12 heads, 4680 tokens: 7.0 us against 7.5; at 12 x 1560 4.4 against
    // 4.1, at 16 x 4680 10.0 against 8.5), and beside the compression kernel as that kernel's launch says.
    const int64_t ctas = (b1 - b0 + 1) * a.H;
    const bool loop = a.beside_prior ? a.one_row : ctas > 4 * a.nsm && ctas <= kPageCtasPerSm * a.nsm;
    if (a.D == 128)
      e = cudaLaunchKernelEx(&cfgA, loop ? append_pool_ksum_kernel<128, false> : append_pool_ksum_kernel<128, true>, a);
    else
      e = cudaLaunchKernelEx(&cfgA, append_pool_ksum_kernel<64, true>, a);
    return e == cudaSuccess ? cudaGetLastError() : e;
  }
  // The reduction may be scheduled while the kernel before it drains (programmatic dependent
  // launch); it waits for that kernel's results itself before it reads anything.
  const int n = a.D * a.D + a.D;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((n + 255) / 256, a.H);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, a.D == 128 ? state_reduce_kernel<128> : state_reduce_kernel<64>, a);
}

}  // namespace hsa

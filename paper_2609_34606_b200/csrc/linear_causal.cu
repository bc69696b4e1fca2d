// Intra-chunk part of the causal linear branch.  When the query chunk is the most recently
// appended chunk, query i may only see the chunk's own keys up to its position; the state of
// everything before the chunk is applied by the forward kernel, and this kernel supplies
//   num[i,h,:] = sum_{q_pos0 <= j <= q_pos0+i} (phi(q_i).phi(k_j)) v_j,   den[i,h] = sum of weights
// K and V from the pool pages.
//
// phi(K) of the chunk is made first, by a kernel of its own, as bf16 tiles in the workspace (made in the kernel
// of the products it would be made again for every query tile behind a key: that form was bound by it, 42 us
// where this one takes 31 us; and left there by the append, every append would pay for it).
//
// One CTA per (128-row query tile, head), 576 threads:
//   warp 0       TMA producer: Q tile, then, up to the tile's diagonal, phi(K) hi and lo and V (two 64-token
//                pages = 128 keys per step) into rings of four and two 128-key tiles
//   warp 1       tcgen05.mma issuer
//   warps 2..17  phi(Q) once; weights of a step: mask, row sum, hi / lo split
// The map and the weights are fp32 quantities, so each is carried as bf16 hi + lo (about 16 bits):
//   A    = phi(Q)_hi phi(K)_hi^T + phi(Q)_lo phi(K)_hi^T + phi(Q)_hi phi(K)_lo^T      (fp32, TMEM)
//   num += A_hi V + A_lo V   with A masked and split, den from the fp32 A
// Against 64 bits the outputs of a causal forward are off by as much as with fp32 arithmetic
// throughout: the rounding of the result to bf16 is two orders of magnitude larger.
// (A non-finite V reaches every row of its 128-row tile, also those before it: 0 x inf in the product.)
//
// What bounds it: the tensor pipe, 40 products of 128 x 128 x 16 per step = 2560 cycles, with the
// workers' 16384 weights per step beside it.
// Measured, 12 heads of 128, a chunk of 1560 tokens (91 tile pairs per head): 31 us, with the forward
// kernel running on the SMs that are through from 15 us on; one CTA per query and head in fp32 on the
// CUDA cores, which this replaces, took 1678 us.  The longest tile alone is 13 steps of 2 us.
// The steps of a tile grow with its position (chunk of 1560 tokens: 1 to 13), so the longest tiles are
// launched first and the forward kernel behind this one may start on the SMs that are through (see
// hsa_forward_kernel).
// TMEM: num (128 columns) | phi(Q) hi (64) | phi(Q) lo (64) | A, two buffers of 128; the split weights
// overwrite their A buffer, 32 columns of weights as 16 of packed hi and 16 of packed lo.
#include <cuda_bf16.h>

#include "hsa_internal.h"
#include "ptx.cuh"

namespace hsa {

namespace {

constexpr int kClWorkers = 512;
constexpr int kClThreads = 64 + kClWorkers;
constexpr int kClKSlots = 4;  // phi(K) tiles in flight: hi and lo of two steps
constexpr int kClStages = 2;  // V
constexpr uint32_t kClColNum = 0, kClColQh = 128, kClColQl = 192, kClColA = 256;  // A: + 128 * buffer

template <int D>
struct ClSmem {
  static constexpr int kHalf = 128 * 128;    // bytes of one [128 rows x 128 B] slab
  static constexpr int kTile = 128 * D * 2;  // 128 keys (or queries)
  static constexpr int kK = 0;               // phi(K) tiles: slot (2 step + hi / lo) % kClKSlots
  static constexpr int kV = kK + kClKSlots * kTile;
  static constexpr int kQ = kV + kClStages * kTile;
  static constexpr int kBars = kQ + kTile;
  static constexpr int kTotal = kBars + 256 + 1024;
};

struct ClBars {
  uint64_t q_full, q_read;
  uint64_t k_full[kClKSlots], k_empty[kClKSlots];
  uint64_t v_full[kClStages], v_empty[kClStages];
  uint64_t a_full[2], p_full[2];
  uint64_t done;
  uint32_t tmem_base;
  volatile int abort_flag;
};
static_assert(sizeof(ClBars) <= 256, "barrier block must fit its shared-memory slot");

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
// two fp32 values as packed bf16 hi and lo (hi + lo = value to about 16 bits)
__device__ __forceinline__ void cl_split(float a, float b, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16(a, b);
  lo = pack_bf16(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xffff0000u));
}

}  // namespace

// phi(K) of one page of one head: what bounds it is the bytes, 16 KB in and 32 KB out per page at head_dim 128.
template <int D>
__global__ void __launch_bounds__(256) phi_terms_kernel(CausalLinArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int h = blockIdx.y;
  const int64_t b = a.q_pos0 / kBlock + blockIdx.x;
  const uint4* src = reinterpret_cast<const uint4*>(a.k_pool + (static_cast<size_t>(a.page_table[b]) * a.H + h) * kBlock * D);
  uint4* dst = reinterpret_cast<uint4*>(a.phik + (static_cast<size_t>(h) * 2 * a.phik_blocks + blockIdx.x) * kBlock * D);
  const size_t term = static_cast<size_t>(a.phik_blocks) * kBlock * D / 8;  // from one term's tile to the next
#pragma unroll
  for (int i = 0; i < kBlock * D / 8 / 256; ++i) {
    const int c = threadIdx.x + 256 * i;
    const uint4 raw = src[c];
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      cl_split(cl_phi(__uint_as_float(w[e] << 16), a.relu), cl_phi(__uint_as_float(w[e] & 0xffff0000u), a.relu), hi[e], lo[e]);
    dst[c] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    dst[c + term] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

template <int D>
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
    for (int s = 0; s < kClKSlots; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->k_empty[s], 1);
    }
    for (int s = 0; s < kClStages; ++s) {
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->v_empty[s], 1);
      mbar_init(&bars->a_full[s], 1);
      mbar_init(&bars->p_full[s], kClWorkers / 32);
    }
    mbar_init(&bars->done, 1);
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

  // pages of the chunk up to the last token this tile sees
  const int b_first = static_cast<int>(a.q_pos0 / kBlock);
  const int64_t last = a.q_pos0 + min(row0 + kTileM, a.n_q) - 1;
  const int n_pages = static_cast<int>(last / kBlock) - b_first + 1;
  const int nsteps = (n_pages + 1) / 2;
  auto pages_of = [&](int j) { return min(2, n_pages - 2 * j); };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one lane)
    if (elect_one_sync()) {
      mbar_expect_tx(&bars->q_full, L::kTile);
      for (int dh = 0; dh < DH; ++dh) tma_load_3d(smem + L::kQ + dh * L::kHalf, &tm_q, &bars->q_full, dh * 64, h, row0);
      int armed_k = 0, armed_v = 0;  // loads issued per ring, for the drain on abort
      auto load_k = [&](int j, int hl) -> bool {
        const int i = 2 * j + hl, s = i % kClKSlots, npg = pages_of(j);
        if (i >= kClKSlots && !cl_wait(&bars->k_empty[s], ((i / kClKSlots) - 1) & 1, bars, a.status)) return false;
        mbar_expect_tx(&bars->k_full[s], npg * kBlock * D * 2);
        for (int pg = 0; pg < npg; ++pg)
          for (int dh = 0; dh < DH; ++dh)
            tma_load_2d(smem + L::kK + s * L::kTile + dh * L::kHalf + pg * (kBlock * 128), &tm_k, &bars->k_full[s], dh * 64,
                        ((h * 2 + hl) * a.phik_blocks + 2 * j + pg) * kBlock);
        ++armed_k;
        return true;
      };
      auto load_v = [&](int j) -> bool {
        const int s = j % kClStages, npg = pages_of(j);
        int32_t y[2] = {0, 0};  // (looked up ahead of the wait)
        for (int pg = 0; pg < npg; ++pg) y[pg] = (a.page_table[b_first + 2 * j + pg] * a.H + h) * kBlock;
        if (j >= kClStages && !cl_wait(&bars->v_empty[s], ((j / kClStages) - 1) & 1, bars, a.status)) return false;
        mbar_expect_tx(&bars->v_full[s], npg * kBlock * D * 2);
        for (int pg = 0; pg < npg; ++pg)
          for (int dh = 0; dh < DH; ++dh)
            tma_load_2d(smem + L::kV + s * L::kTile + dh * L::kHalf + pg * (kBlock * 128), &tm_v, &bars->v_full[s], dh * 64, y[pg]);
        ++armed_v;
        return true;
      };
      bool ok = true;
      for (int j = 0; j < nsteps && ok; ++j) ok = load_k(j, 0) && load_k(j, 1) && load_v(j);
      if (!ok) {  // let every copy already issued land before the CTA's shared memory goes away
        mbar_wait(&bars->q_full, 0, 1u << 16);
        for (int s = 0; s < kClKSlots; ++s)
          if (armed_k > s) mbar_wait(&bars->k_full[s], ((armed_k - 1 - s) / kClKSlots) & 1, 1u << 16);
        for (int s = 0; s < kClStages; ++s)
          if (armed_v > s) mbar_wait(&bars->v_full[s], ((armed_v - 1 - s) / kClStages) & 1, 1u << 16);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one lane)
    if (elect_one_sync()) {
      constexpr uint32_t kHiSw = desc_hi_sw128(1024);
      auto issue_qk = [&](int j) -> bool {
        const uint32_t d = tmem + kClColA + 128 * (j & 1);
        // (one page in the last step: only its 64 columns are computed)
        const uint32_t idesc = pages_of(j) >= 2 ? idesc_bf16_f32(128, 128, 0, 0) : idesc_bf16_f32(128, 64, 0, 0);
#pragma unroll
        for (int hl = 0; hl < 2; ++hl) {
          const int i = 2 * j + hl, s = i % kClKSlots;
          if (!cl_wait(&bars->k_full[s], (i / kClKSlots) & 1, bars, a.status)) return false;
          tc_fence_after();
          const uint32_t k_lo = desc_lo_sw128(smem_u32(smem + L::kK + s * L::kTile), 16);
#pragma unroll
          for (int qp = 0; qp < 2 - hl; ++qp)  // phi(K) hi meets phi(Q) hi and lo, phi(K) lo meets phi(Q) hi
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t off = ((kk / 4) * L::kHalf + (kk % 4) * 32) >> 4;
              tc_mma_ts_lo(d, tmem + (qp ? kClColQl : kClColQh) + kk * 8, k_lo + off, kHiSw, idesc, (hl > 0 || qp > 0 || kk > 0) ? 1u : 0u);
            }
          tc_commit(&bars->k_empty[s]);
        }
        tc_commit(&bars->a_full[j & 1]);
        return true;
      };
      bool ok = cl_wait(&bars->q_read, 0, bars, a.status);  // phi(Q) is in TMEM
      for (int j = 0; j < min(2, nsteps) && ok; ++j) ok = issue_qk(j);
#pragma unroll 1
      for (int j = 0; j < nsteps && ok; ++j) {
        const int s = j % kClStages;
        ok = cl_wait(&bars->p_full[j & 1], (j >> 1) & 1, bars, a.status) &&
             cl_wait(&bars->v_full[s], (j / kClStages) & 1, bars, a.status);
        if (!ok) break;
        tc_fence_after();
        constexpr uint32_t idesc = idesc_bf16_f32(128, D, 0, 1);
        const uint32_t v_lo = desc_lo_sw128(smem_u32(smem + L::kV + s * L::kTile), L::kHalf);
        const uint32_t p_op = tmem + kClColA + 128 * (j & 1);
        const int nk = 4 * pages_of(j);  // 16 keys each; a page that was not loaded is not touched
        for (int kk = 0; kk < nk; ++kk) {
          const uint32_t p_hi = p_op + 32 * (kk >> 1) + 8 * (kk & 1);
          tc_mma_ts_lo(tmem + kClColNum, p_hi, v_lo + kk * 128, kHiSw, idesc, (j > 0 || kk > 0) ? 1u : 0u);
          tc_mma_ts_lo(tmem + kClColNum, p_hi + 16, v_lo + kk * 128, kHiSw, idesc, 1u);
        }
        tc_commit(&bars->v_empty[s]);
        // the weights of step j + 2 overwrite the ones just consumed: the tensor pipe runs in order
        if (j + 2 < nsteps) ok = issue_qk(j + 2);
      }
      if (ok) tc_commit(&bars->done);
    }
  } else {
    // ------------------------------------------------------------------ weights, result
    const int set = (warp - 2) >> 2;  // 32 of the 128 columns
    const int quad = warp & 3;        // TMEM lane quadrant this warp may access
    const int r = quad * 32 + lane;   // row inside the tile
    const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
    bool ok = __all_sync(0xffffffffu, cl_wait(&bars->q_full, 0, bars, a.status));
    if (ok) {
      if (set * 32 < D) {
        // phi(q) of this thread's row, 32 dims, as the bf16 hi and lo A operands
        const uint8_t* qrow = smem + L::kQ + r * 128;
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cc = set * 4 + c;  // 16-byte chunk of the row
          const uint4 raw = *reinterpret_cast<const uint4*>(qrow + (cc >> 3) * L::kHalf + (((cc & 7) ^ (r & 7)) << 4));
          const uint32_t* qw = reinterpret_cast<const uint32_t*>(&raw);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            cl_split(cl_phi(__uint_as_float(qw[i] << 16), a.relu), cl_phi(__uint_as_float(qw[i] & 0xffff0000u), a.relu),
                     hi[c * 4 + i], lo[c * 4 + i]);
        }
        tmem_st16(tmem + lane_off + kClColQh + set * 16, hi);
        tmem_st16(tmem + lane_off + kClColQl + set * 16, lo);
        tc_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->q_read);
    }
    float den = 0.f;
#pragma unroll 1
    for (int j = 0; j < nsteps && ok; ++j) {
      ok = __all_sync(0xffffffffu, cl_wait(&bars->a_full[j & 1], (j >> 1) & 1, bars, a.status));
      if (!ok) break;
      tc_fence_after();
      const uint32_t buf = tmem + lane_off + kClColA + 128 * (j & 1) + 32 * set;
      uint32_t v[32];
      tmem_ld32(buf, v);
      const int64_t base = static_cast<int64_t>(b_first + 2 * j) * kBlock;  // token of column 0
      const int lo_col = static_cast<int>(a.q_pos0 - base);                 // first visible column (<= 0: all)
      const int hi_col = static_cast<int>(a.q_pos0 + row0 - base);          // last visible column of row 0
      tc_wait_ld();
      if (lo_col > 0 || hi_col < 127) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int c = 32 * set + i;
          if (c < lo_col || c > hi_col + r) v[i] = 0u;
        }
      }
      float s4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t hi[16], lo[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float x0 = __uint_as_float(v[2 * i]), x1 = __uint_as_float(v[2 * i + 1]);
        s4[(2 * i) & 3] += x0;
        s4[(2 * i + 1) & 3] += x1;
        cl_split(x0, x1, hi[i], lo[i]);
      }
      // (over the thread's own columns, which it has read)
      tmem_st16(buf, hi);
      tmem_st16(buf + 16, lo);
      den += (s4[0] + s4[1]) + (s4[2] + s4[3]);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->p_full[j & 1]);
    }
    if (ok) ok = __all_sync(0xffffffffu, cl_wait(&bars->done, 0, bars, a.status));
    tc_fence_after();
    float* dsum = reinterpret_cast<float*>(smem + L::kK);  // [4][128], dead by now
    if (ok) dsum[set * 128 + r] = den;
    // (an aborted wait leaves the loop as well: the barrier takes every worker)
    asm volatile("bar.sync 1, %0;" ::"n"(kClWorkers) : "memory");
    if (ok) {
      const int row = row0 + r;
      if (set * 32 < D) {  // warp-uniform: the load is warp-collective
        uint32_t v[32];
        tmem_ld32(tmem + lane_off + kClColNum + 32 * set, v);
        tc_wait_ld();
        if (row < a.n_q) {
          float4* dst = reinterpret_cast<float4*>(a.lin_num + (static_cast<size_t>(row) * a.H + h) * D + 32 * set);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            dst[i] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]),
                                 __uint_as_float(v[4 * i + 3]));
        }
      }
      if (set == 0 && row < a.n_q) 
        a.lin_den[static_cast<size_t>(row) * a.H + h] = (dsum[r] + dsum[128 + r]) + (dsum[256 + r] + dsum[384 + r]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

cudaError_t causal_linear_init() {
  cudaError_t e = cudaFuncSetAttribute(causal_linear_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, ClSmem<128>::kTotal);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(causal_linear_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, ClSmem<64>::kTotal);
  return e;
}

cudaError_t launch_causal_linear(const CausalLinArgs& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                                 const CUtensorMap& tm_v, cudaStream_t st) {
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
  cfg.gridDim = dim3(static_cast<unsigned>(n_tiles) * a.H);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = a.D == 128 ? ClSmem<128>::kTotal : ClSmem<64>::kTotal;
  if (a.D == 128) return cudaLaunchKernelEx(&cfg, causal_linear_kernel<128>, a, tm_q, tm_k, tm_v);
  return cudaLaunchKernelEx(&cfg, causal_linear_kernel<64>, a, tm_q, tm_k, tm_v);
}

}  // namespace hsa

// Linformer form of the linear branch (Section 3.3 "Linear branch", Eq. 3; Appendix G):
// per appended segment of L tokens and per head, K~ = E_K^T K and V~ = E_V^T V (r rows each) are
// appended to a compressed pool that has the page layout of the main pool, so that the forward
// kernel can run plain softmax attention over it ("every block selected").
//
// One CTA computes a [128 rows of r] x [128 dims] tile of K~ or V~ for one head:
//   C (fp32 in TMEM) = sum over token blocks of  E[tokens, 128 r]^T  X[tokens, 128 d]
// One lane brings the [64 tokens x 128] tiles of E and of X into a ring by TMA (both land
// in the 128-byte-swizzled MN-major layout the tensor cores take as they are; rows past the end of
// the segment arrive as zeros), one lane issues four tcgen05 MMAs per block (K = tokens) and hands the
// stage back, and at the end all warps write the bf16 rows to the compressed pool.
//
// What bounds a tile is what one SM has in flight, a ring of a stream with 1.5 us of latency, so the token blocks of a tile
// of a long segment are split over the 2, 4 or 8 CTAs of a cluster where the device runs that many at once: each leaves its fp32
// sums in its dead ring, and behind a cluster barrier adds up its share of the rows over all of them, in order.  The append
// of a segment (this kernel, launched as a programmatic dependent, and the page write beside it), heads x tokens at
// rank 256, a tile per CTA and a ring of four stages -> now, six stages: 12 x 4680 36.8 -> 27.8 us (144 MB), 16 x 4680 41.1 ->
// 35.4, 2 x 4680 16.9 -> 9.2, 8 x 2000 11.6 -> 9.7, 12 x 1560 11.4 -> 9.7.
// The accumulator of a tile truncates what it adds to, so parts that are added in rounded fp32 are also the more exact: rows
// of 4680 tokens that are not the nearest bf16 0.26 % -> 0.14 %, error against 64 bits 1.65929e-3 (2-norm; rounding alone
// 1.65929e-3), mean magnitude off by -4.8e-6 -> -2.7e-6.
#include <cuda_bf16.h>

#include "hsa_internal.h"
#include "ptx.cuh"

namespace hsa {

namespace {

constexpr int kLcThreads = 512;
constexpr int kLcDepth = 6;
constexpr int kLcTile = 64 * 128 * 2;
constexpr int kLcStage = 2 * kLcTile;  // E tile | X tile
constexpr int kLcSmem = kLcDepth * kLcStage + 256 + 1024;

struct LcBars {
  uint64_t full[kLcDepth];
  uint64_t empty[kLcDepth];
  uint64_t all_done;
  uint32_t tmem_base;
  volatile int abort_flag;
};
constexpr int kLcPitch = 132;  // floats per row of the sums left for the cluster
static_assert(128 * kLcPitch * 4 <= kLcDepth * kLcStage, "the sums fit the ring");
// Which segments are split: the merge of a cluster is 2 us, a token block of a tile 0.15 us while few CTAs stream.  On more than
// half of the SMs the page write beside this kernel is in the way, so only long segments go there.  An append, heads x
// tokens at rank 256, without clusters -> with (2 CTAs unless noted): 4 x 600 6.2 -> 7.0 us, 4 x 1280 7.8 -> 7.8, 4 x 2000 9.5 -> 8.4
// (4 CTAs), 16 x 1024 8.0 -> 9.2, 12 x 2400 12.6 -> 12.8, 12 x 3120 16.8 -> 16.3, 12 x 4680 31.7 -> 28.0.
constexpr int kLcPart = 4;       // token blocks of a part at least
constexpr int kLcShortest = 20;  // token blocks of a segment at least
constexpr int kLcLong = 49;      // the same for clusters on more than half of the SMs

__device__ __forceinline__ bool lc_wait(uint64_t* bar, uint32_t parity, LcBars* bars, int32_t* status) {
  if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t i = 1; i < (1u << 24); ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 1023u) == 0u && bars->abort_flag) return false;
  }
  bars->abort_flag = 1;
  atomicCAS(status, 0, kDevTimeout);
  return false;
}

}  // namespace

template <int C>  // CTAs of a cluster, which share a tile
__global__ void __launch_bounds__(kLcThreads, 1)
linformer_compress_kernel(LinformerArgs a, const __grid_constant__ CUtensorMap tm_ek, const __grid_constant__ CUtensorMap tm_ev,
                          const __grid_constant__ CUtensorMap tm_kin, const __grid_constant__ CUtensorMap tm_vin) {
  constexpr int D = 128;
  extern __shared__ uint8_t lc_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(lc_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  LcBars* bars = reinterpret_cast<LcBars*>(smem + kLcDepth * kLcStage);
  const int h = blockIdx.y;
  const int rtiles = (a.rank + 127) / 128;  // (the last tile may hold 64 rows only: E reads as zeros beyond the rank)
  const int part_c = blockIdx.x % C, tile = blockIdx.x / C;
  const int which = tile / rtiles;  // 0: keys, 1: values
  const int rt = tile % rtiles;
  const CUtensorMap* tm_e = which == 0 ? &tm_ek : &tm_ev;  // [H][seg_tokens][rank], box 64 r x 64 tokens
  const CUtensorMap* tm_x = which == 0 ? &tm_kin : &tm_vin;  // [tokens][H][d], box 64 d x 1 x 64 tokens
  __nv_bfloat16* pool = which == 0 ? a.kc_pool : a.vc_pool;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = (a.seg_tokens + kBlock - 1) / kBlock;
  const int b_lo = blocks * part_c / C, nblk = blocks * (part_c + 1) / C - b_lo;  // this CTA's token blocks

  if (threadIdx.x == 0) {
    for (int s = 0; s < kLcDepth; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    mbar_init(&bars->all_done, 1);
    bars->abort_flag = 0;
    fence_mbar_init();
    // launched as a programmatic dependent: everything before this kernel is complete from here on, for this CTA's
    // loads and, since the trigger comes after the wait, for the page-write kernel of the same append, which is
    // launched behind this one, may run beside it (it touches none of this kernel's outputs) and does not wait itself
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0) a.ccnt[h] = (a.seg_index + 1) * (a.rank / kBlock);  // compressed pages now valid
  }
  if (warp == 0) {
    tmem_alloc(&bars->tmem_base, 128);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  int armed = 0;  // blocks asked for (producer's lane)
  if (warp == 1) {
    // ------------------------------------------------------------------ producer (one lane)
    if (elect_one_sync()) {
      for (int bi = 0; bi < nblk; ++bi) {
        const int s = bi % kLcDepth;
        if (bi >= kLcDepth && !lc_wait(&bars->empty[s], ((bi / kLcDepth) - 1) & 1, bars, a.status)) break;
        ++armed;
        uint8_t* st_e = smem + s * kLcStage;
        uint8_t* st_x = st_e + kLcTile;
        mbar_expect_tx(&bars->full[s], kLcStage);
        for (int half = 0; half < 2; ++half) {
          tma_load_3d(st_e + half * (kLcTile / 2), tm_e, &bars->full[s], rt * 128 + half * 64, (b_lo + bi) * kBlock, h);
          tma_load_3d(st_x + half * (kLcTile / 2), tm_x, &bars->full[s], half * 64, h, (b_lo + bi) * kBlock);
        }
      }
    }
  } else if (warp == 0) {
    // ------------------------------------------------------------------ MMA issuer (one lane)
    if (elect_one_sync()) {
      constexpr uint32_t idesc = idesc_bf16_f32(128, 128, 1, 1);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      bool ok = a.give_up == 0;
      if (!ok) {
        bars->abort_flag = 1;
        atomicCAS(a.status, 0, kDevTimeout);
      }
      for (int bi = 0; bi < nblk && ok; ++bi) {
        const int s = bi % kLcDepth;
        ok = lc_wait(&bars->full[s], (bi / kLcDepth) & 1, bars, a.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t a_lo = desc_lo_sw128(smem_u32(smem + s * kLcStage), kLcTile / 2);
        const uint32_t b_lo = desc_lo_sw128(smem_u32(smem + s * kLcStage + kLcTile), kLcTile / 2);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma_ss_lo(tmem, a_lo + kk * 128, b_lo + kk * 128, hi, idesc, (bi > 0 || kk > 0) ? 1u : 0u);
        tc_commit(&bars->empty[s]);
      }
      tc_commit(&bars->all_done);
    }
  }
  __syncwarp();
  lc_wait(&bars->all_done, 0, bars, a.status);
  __syncthreads();
  const bool ok = bars->abort_flag == 0;  // (one answer for the CTA: all_done alone does not say that every block is in)
  if (!ok) {
    // whoever has given up: the copies issued land before the ring is used for the sums or goes away, and the products end
    // before TMEM goes
    for (int s = 0; s < kLcDepth; ++s)
      if (armed > s) mbar_wait(&bars->full[s], ((armed - 1 - s) / kLcDepth) & 1, 1u << 16);
    if (warp == 0) mbar_wait(&bars->all_done, 0, 1u << 16);
    __syncthreads();
  }
  tc_fence_after();
  const int quad = warp & 3, part = warp >> 2;
  auto out_row = [&](int rr) {  // row of the compressed segment
    const int page = a.seg_index * (a.rank / kBlock) + rr / kBlock;
    return pool + ((static_cast<size_t>(page) * a.H + h) * kBlock + (rr % kBlock)) * D;
  };
  uint32_t v[32];
  if constexpr (C > 1) {
    auto cluster_sync = [] {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    float* sums = reinterpret_cast<float*>(smem);
    float* mine = sums + (quad * 32 + lane) * kLcPitch + part * 32;
    if (ok) {
      tmem_ld32(tmem + (static_cast<uint32_t>(quad * 32) << 16) + part * 32, v);
      tc_wait_ld();
    }
#pragma unroll
    for (int i = 0; i < 32; i += 4)  // (a part that gave up counts for nothing; the status word says so)
      *reinterpret_cast<float4*>(mine + i) = ok ? make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                                                               __uint_as_float(v[i + 3]))
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    cluster_sync();
#pragma unroll
    for (int i = 0; i < 128 / C * 32 / kLcThreads; ++i) {
      const int f = threadIdx.x + kLcThreads * i;  // (row of this CTA's share, four columns)
      const int row = part_c * (128 / C) + f / 32, col = f % 32 * 4;
      float4 x[C];
#pragma unroll
      for (int c = 0; c < C; ++c) x[c] = ld_cluster4(sums + row * kLcPitch + col, c);
      float4 t = x[0];
#pragma unroll
      for (int c = 1; c < C; ++c) t = make_float4(t.x + x[c].x, t.y + x[c].y, t.z + x[c].z, t.w + x[c].w);
      const int rr = rt * 128 + row;
      if (rr < a.rank) *reinterpret_cast<uint2*>(out_row(rr) + col) = make_uint2(pack_bf16(t.x, t.y), pack_bf16(t.z, t.w));
    }
    cluster_sync();  // (nobody leaves while its sums are being read)
  } else {
    const int rr = rt * 128 + quad * 32 + lane;
    if (ok && rr < a.rank) {  // (warp-uniform: the rank is a multiple of 64)
      tmem_ld32(tmem + (static_cast<uint32_t>(quad * 32) << 16) + part * 32, v);
      tc_wait_ld();
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) pk[i] = pack_bf16(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
      __nv_bfloat16* dst = out_row(rr) + part * 32;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        reinterpret_cast<uint4*>(dst)[i] = make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

namespace {
using LcKernel = void (*)(LinformerArgs, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap);
LcKernel lc_kernel(int lg) {
  return lg == 3 ? linformer_compress_kernel<8> : lg == 2 ? linformer_compress_kernel<4> : lg == 1 ? linformer_compress_kernel<2>
                                                                                                   : linformer_compress_kernel<1>;
}
struct LcLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[3];
  LcLaunch(dim3 grid, int cluster, cudaStream_t st, bool room = false) {
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kLcThreads);
    cfg.dynamicSmemBytes = kLcSmem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    int n = 1;
    if (cluster > 1) {
      attr[n].id = cudaLaunchAttributeClusterDimension;
      attr[n].val.clusterDim.x = cluster;
      attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
      ++n;
    }
    if (room) {
      attr[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
      attr[n++].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
  }
};
}  // namespace

cudaError_t linformer_init(int (&clusters)[3]) {
  cudaError_t e = cudaSuccess;
  for (int lg = 0; lg <= 3 && e == cudaSuccess; ++lg)
    e = cudaFuncSetAttribute(lc_kernel(lg), cudaFuncAttributeMaxDynamicSharedMemorySize, kLcSmem);
  for (int lg = 1; lg <= 3 && e == cudaSuccess; ++lg) {
    LcLaunch l(dim3(1 << lg), 1 << lg, nullptr);
    if (cudaOccupancyMaxActiveClusters(&clusters[lg - 1], reinterpret_cast<const void*>(lc_kernel(lg)), &l.cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters[lg - 1] = 0;  // no clusters of this size on this device
    }
  }
  return e;
}

cudaError_t launch_linformer_compress(const LinformerArgs& a, const int (&clusters)[3], int* one_row, const CUtensorMap& tm_ek,
                                      const CUtensorMap& tm_ev, const CUtensorMap& tm_kin, const CUtensorMap& tm_vin,
                                      cudaStream_t st) {
  const int tiles = 2 * ((a.rank + 127) / 128), blocks = (a.seg_tokens + kBlock - 1) / kBlock, items = tiles * a.H;
  int lg = 0;
  while (lg < 3 && items <= clusters[lg] && blocks >= kLcShortest && blocks >> (lg + 1) >= kLcPart) {
    const int ctas = items << (lg + 1);
    if (ctas > a.nsm / 2 && (blocks < kLcLong || (lg > 0 && 3 * ctas > 2 * a.nsm))) break;
    ++lg;
  }
  // The page write beside this kernel, a CTA per block and head, a row of a thread at a time: six CTAs fit an SM that this kernel
  // leaves free, three beside one of its CTAs, but these only if the SM's memory is split for it (the ring alone asks
  // for the next smaller split, all of which it takes).  Where not even that runs all of them at once, they ask for
  // all rows of a thread, four to a free SM, and come in waves.
  const int pages = blocks * a.H, ctas = items << lg, free_ctas = kPageCtasPerSm * (a.nsm - ctas);
  const bool room = pages > free_ctas && pages <= free_ctas + 3 * ctas;
  *one_row = pages <= free_ctas || room;
  LcLaunch l(dim3(tiles << lg, a.H), 1 << lg, st, room);
  return cudaLaunchKernelEx(&l.cfg, lc_kernel(lg), a, tm_ek, tm_ev, tm_kin, tm_vin);
}

}  // namespace hsa

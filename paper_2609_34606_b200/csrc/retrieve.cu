// Page-level retrieval of the hierarchical KV cache (Section 3.2, Stage 2): a KV page is a run of
// kv_page_blocks consecutive 64-token blocks; its score is
//     alpha_j = mean_h( Qbar_h . Kbar_{j,h} ) * scale
// with the chunk's average query and the page's average key, both taken from sums the selection
// path already keeps (query tile sums, per-block key sums), and the top-K_p pages are kept.
#include <cuda_bf16.h>

#include "hsa_internal.h"

namespace hsa {

namespace {

__device__ __forceinline__ uint32_t rt_order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // ascending with the float order
}

// One CTA per (KV page, head, run of kRtRun blocks): fp64 dot of the head's query sum and the run's key sum.
// A warp takes a row of key sums (one block, all dims) at a time, so that every load is a whole row and a
// warp has several in flight; the key sums are asked for ahead of the wait for the query tile sums (that
// kernel writes none of them and has itself waited for everything before it).
// What bounds it: latency (a row per warp and step, ~25 steps at the paper's 195 blocks per page; the
// 13.5 MB of key sums of 2194 blocks x 12 heads take 2 us at the copy bandwidth): the two
// kernels of the retrieval take 13 us behind the tile sums at that size, 4680 queries, against 146 with one
// CTA per KV page whose threads walked the blocks one after another.
constexpr int kRtRun = 256;  // the key-sum workspace (hsa_retrieve_kv_pages) is sized for this

template <int D>
__global__ void __launch_bounds__(256) kv_page_score_kernel(RetrieveArgs a) {
  constexpr int PER = D / 32;  // dims per lane
  constexpr int kRows = 8;     // rows in flight per warp
  __shared__ double qs[256];
  __shared__ double red[8];
  const int j = blockIdx.x, h = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nblk = static_cast<int>((a.n_tokens + kBlock - 1) / kBlock);
  const int64_t page_end = min64(nblk, (static_cast<int64_t>(j) + 1) * a.kv_page_blocks);
  const int64_t b0 = static_cast<int64_t>(j) * a.kv_page_blocks + static_cast<int64_t>(blockIdx.z) * kRtRun;
  const int b1 = static_cast<int>(min64(page_end, b0 + kRtRun));
  double ks[PER];
#pragma unroll
  for (int e = 0; e < PER; ++e) ks[e] = 0.0;
  const float* rows = a.ksum + static_cast<size_t>(h) * a.max_pages * D + lane * PER;
  for (int b = static_cast<int>(b0) + warp; b < b1; b += 8 * kRows) {
    float v[kRows][PER];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int e = 0; e < PER; ++e) v[i][e] = b + 8 * i < b1 ? rows[static_cast<size_t>(b + 8 * i) * D + e] : 0.f;
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int e = 0; e < PER; ++e) ks[e] += static_cast<double>(v[i][e]);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  {
    // the head's query sum: 256 / D threads per column, each an interleaved subset of the tile sums
    constexpr int WAYS = 256 / D;
    const int col = threadIdx.x % D, way = threadIdx.x / D;
    const int n_tiles = (a.n_q + kTileM - 1) / kTileM;
    double s = 0.0;
#pragma unroll 8
    for (int t = way; t < n_tiles; t += WAYS)
      s += static_cast<double>(__ldcg(&a.qpart[(static_cast<size_t>(t) * a.H + h) * D + col]));
    qs[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < D) {
#pragma unroll
      for (int w = 1; w < WAYS; ++w) s += qs[w * D + threadIdx.x];
      qs[threadIdx.x] = s;
    }
    __syncthreads();
  }
  double part = 0.0;
#pragma unroll
  for (int e = 0; e < PER; ++e) part += ks[e] * qs[lane * PER + e];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) red[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w];
    a.part[(static_cast<size_t>(j) * a.H + h) * gridDim.z + blockIdx.z] = t;
  }
}

// One CTA: score of every page (its partial dots in head and run order), rank by (score descending, id
// ascending), keep the first top_kp, ascending ids.
__global__ void __launch_bounds__(256) kv_page_topk_kernel(RetrieveArgs a, int n_pages, int n_part) {
  extern __shared__ uint32_t rkeys[];  // [n_pages] keys, then [n_pages] selected flags
  uint32_t* flag = rkeys + n_pages;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int j = threadIdx.x; j < n_pages; j += 256) {
    double dot = 0.0;
#pragma unroll 8
    for (int i = 0; i < n_part; ++i) dot += __ldcg(&a.part[static_cast<size_t>(j) * n_part + i]);
    const int64_t t0 = static_cast<int64_t>(j) * a.kv_page_blocks * kBlock;
    const int64_t toks = min64(a.n_tokens, t0 + static_cast<int64_t>(a.kv_page_blocks) * kBlock) - t0;
    const float f = static_cast<float>(dot / (static_cast<double>(a.n_q) * static_cast<double>(toks) * a.H) *
                                       static_cast<double>(a.scale));
    rkeys[j] = rt_order_key(f);
    if (a.scores_out) a.scores_out[j] = f;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n_pages; j += 256) {
    const uint32_t kj = rkeys[j];
    int rank = 0;
    for (int i = 0; i < n_pages; ++i) rank += (rkeys[i] > kj) || (rkeys[i] == kj && i < j);
    flag[j] = rank < a.top_kp ? 1u : 0u;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n_pages; j += 256) {
    if (!flag[j]) continue;
    int pos = 0;
    for (int i = 0; i < j; ++i) pos += static_cast<int>(flag[i]);
    a.page_ids[pos] = j;
  }
}

}  // namespace

cudaError_t launch_retrieve(const RetrieveArgs& a, int n_pages, cudaStream_t st) {
  const int n_runs = ((a.kv_page_blocks < a.max_pages ? a.kv_page_blocks : a.max_pages) + kRtRun - 1) / kRtRun;
  // each kernel is a programmatic dependent of the one before it
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_pages, a.H, n_runs);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, a.D == 128 ? kv_page_score_kernel<128> : kv_page_score_kernel<64>, a);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(1);
  cfg.dynamicSmemBytes = static_cast<size_t>(n_pages) * 8;
  return cudaLaunchKernelEx(&cfg, kv_page_topk_kernel, a, n_pages, a.H * n_runs);
}

}  // namespace hsa

// Internal declarations shared by the C-ABI layer and the kernel launchers.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/hsa.h"

namespace hsa {

constexpr int kBlock = HSA_PAGE_TOKENS;  // tokens per KV block = tokens per page
constexpr int kTileM = 128;              // query rows per work item of the forward kernel
constexpr int kStateSplitMax = 16;       // token-axis splits of the state update (per head)
// z as a [16 x 128] bf16 K-major operand image (128-byte swizzle, two slabs of 64 dims): row 0 holds
// the bf16 rounding of z, row 1 the bf16 rounding of the remainder, rows 2..15 are zero, so that
// phi(Q) times it gives the denominator phi(q).z as the sum of two accumulator columns
constexpr int kZopBytes = 4096;
constexpr int kClusterParts = 8;         // CTAs of a cluster that a list of a launch with few items is split over
constexpr int kPhiTerms = 3;             // bf16 terms of phi(K) for the causal products: 24 bits
constexpr int kFwdSplitMax = 16;         // CTAs a long (query tile, head) of the forward kernel is split over

// Parts (their log2) that a list of `steps` two-page steps is cut into by a cluster of 2, 4 or 8 CTAs.  A step takes
// 0.74 us; meeting, dumping and merging cost 6 us and 0.5 us per part (head_dim 128; less at 64).  Forward alone,
// heads x tokens x blocks, whole -> parts: 2 x 256 x 128 55.5 -> 24.0 us (8 parts), 4 x 600 x 128 55.7 -> 27.4 (4),
// 4 x 600 x 32 19.8 -> 18.0, 4 x 2300 x 128 56.7 -> 39.8 (2), 12 x 768 x 64 32.7 -> 27.5; not taken: 4 x 600 x
// 20 15.3 against 18.1, 12 x 768 x 32 20.6 against 22.2.
__host__ __device__ inline int cluster_parts_log2(int cluster, int steps) {
  if (cluster == 2) return steps >= 20 ? 1 : 0;
  return cluster < 4 || steps < 16 ? 0 : cluster >= 8 && steps >= 24 ? 3 : 2;
}

__host__ __device__ inline int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }
__host__ __device__ inline int64_t max64(int64_t a, int64_t b) { return a > b ? a : b; }

// device status word values (match hsa_status)
constexpr int kDevTimeout = HSA_ERR_DEVICE_TIMEOUT;
constexpr int kDevBounds = HSA_ERR_DEVICE_BOUNDS;

struct AppendArgs {
  const __nv_bfloat16* k;
  const __nv_bfloat16* v;
  int n_new;
  int64_t tok_stride, head_stride;
  int64_t n0;  // tokens already in the history
  int H, D, max_pages;
  const int32_t* page_table;
  __nv_bfloat16* k_pool;
  __nv_bfloat16* v_pool;
  float* ksum;      // [H][max_pages][D]
  // The running state lives in two slots that take turns: an append reads slot src_slot and writes
  // slot src_slot ^ 1, which becomes the current one; the other keeps the state before the append
  // (what a causal forward over the appended chunk applies, and what undoing the append returns to).
  float* S[2];          // [H][D][D] per slot
  float* z[2];          // [H][D] per slot
  int src_slot;
  __nv_bfloat16* hilo;  // [H][2 slots][2 hi/lo][D][D]: bf16 hi + lo of S, what the forward kernels read
  uint8_t* zop;         // [H][2 slots][kZopBytes]: z as a tensor-core operand (head_dim 128)
  // key sum the (partly filled) first block of this append had before it: saved here when the append
  // reads it from ksum, read from here instead when the append repeats one that was undone
  float* ksum_saved;    // [H][D]
  int tail_from_saved;
  float* spart;         // [H][nsplit][D*D + D] scratch
  int nsplit;
  int lin_state;  // update the linear state?
  int beside_prior;  // SIMT page write: may run beside the kernel launched just before it (see launch_append)
  int one_row;       // with beside_prior: a row of a thread at a time (see launch_linformer_compress)
  int nsm;           // SMs of the device
  int relu;       // feature map of the state: 0 elu(x) + 1, 1 max(x, 0)
  int32_t* status;  // device status word
};

struct SelectArgs {
  const __nv_bfloat16* q;
  int n_q;
  int64_t tok_stride, head_stride;
  int64_t q_pos0;
  int causal;
  int64_t n_tokens;
  int H, D, max_pages;
  const float* ksum;
  const int32_t* budgets;
  int group_tokens, n_groups;
  float scale;
  float* qpart;  // [n_tiles][H][D] scratch
  uint32_t* keys;  // [H][n_groups][max_pages] scratch: order-preserving score keys
  int32_t* sel_idx;
  int32_t* sel_cnt;
  int kcap;
  int32_t* status;
  unsigned* barrier;  // grid barrier of the single-launch path: {arrive count, generation}, the count
                      // zero when no launch is in flight (null: three launches)
  unsigned long long wait_ns;  // bound of a wait at that barrier
  int use_clusters;            // 1: one thread-block cluster per head (hardware cluster barriers) where the device allows
  // candidate geometry: pages before the first intra-chunk page are selected in runs of inter_pages pages against
  // budgets[], the pages from it on one by one against intra_budgets[] (null: all of them)
  int inter_pages;           // 0 or 1: every page on its own
  int64_t intra_first_page1;  // first intra-chunk page + 1; 0: no intra-chunk region
  const int32_t* intra_budgets;
  // retrieved KV pages (runs of kv_page_blocks blocks): an inter-chunk candidate with a page outside
  // them is no candidate (null: no mask)
  const int32_t* kv_pages;
  int n_kv_pages, kv_page_blocks;
};

struct RetrieveArgs {
  int n_q, H, D, max_pages;
  int64_t n_tokens;
  const float* qpart;  // [tiles][H][D] query tile sums
  const float* ksum;   // [H][max_pages][D]
  int kv_page_blocks, top_kp;
  float scale;
  double* part;        // [pages][H][runs] scratch: partial dots of a page
  float* scores_out;   // [pages] or null
  int32_t* page_ids;   // [min(top_kp, pages)] ascending (output)
};

struct FwdParams {
  int n_q, H;
  int64_t n_tokens;
  int64_t q_pos0;
  int causal;
  const int32_t* sel_idx;
  const int32_t* sel_cnt;
  int kcap, n_groups, group_tokens;
  const int32_t* page_table;
  int n_blocks;
  const float* z;       // [H][D] state the linear branch applies
  const uint8_t* zop;   // [H][2 slots][kZopBytes]: the same z as a tensor-core operand
  int state_slot;       // slot the linear branch applies; row of the hi/lo tensor map = ((h*2 + slot)*2 + hl)*D
  const __nv_bfloat16* g_lin;
  const __nv_bfloat16* g_sp;
  int64_t g_ts, g_hs, g_ds;
  int gate_act;
  int gate_tiles;  // set by the launcher: bit 0 / 1 = the logits of g_lin / g_sp arrive as tiles by TMA
  __nv_bfloat16* out;
  int64_t o_ts, o_hs;
  float scale_log2;  // softmax scale * log2(e)
  uint32_t flags;
  int do_linear, do_sparse;
  const float* lin_num;  // causal intra-chunk partials [n_q][H][D] (or null)
  const float* lin_den;  // [n_q][H]
  int wait_late;         // 1: the kernel before this one wrote lin_num and lin_den and nothing else this one reads
  const __nv_bfloat16* ext_lin;  // linear-branch output computed elsewhere, [n_q][H][D] (or null)
  // Linformer form inside the kernel: the loop first runs over the lf_pages pages of the compressed
  // pool (page ids through lf_table), with an accumulator and row sums of their own (null: none)
  const int32_t* lf_table;
  int lf_pages;
  int relu;  // feature map of the state form: 0 elu(x) + 1, 1 max(x, 0) with 1e-6 added to the denominator
  // split tiles: a (tile, head) with more than split_blocks selected blocks runs as several CTAs
  // (grid z = max_splits); each dumps its unnormalised O, row sums and exponent references, the last
  // one to take a ticket merges them and writes the output
  int max_splits, split_blocks;
  int cluster;           // > 1 (max_splits 1): each (query tile, head) is a cluster of that many CTAs
  int n_tiles, remap;    // set by the launcher: query tiles; 1 = one-dimensional grid, longest lists first
  int nsm;               // SMs of the device (the split rule balances the launch over them)
  float* part_o;         // [slots][D / 4][128][4]: slot (tile H + h) max_splits + part, or the CTA's number (remap)
  float* part_l;         // [slots][128]
  float* part_ref;       // [slots][128]
  int32_t* part_ticket;  // [tiles][H], zero between launches
  int32_t* status;
  // L2 look-ahead of the page gather: the pools themselves (null: none)
  const uint8_t* k_pool;
  const uint8_t* v_pool;
};

constexpr unsigned long long kNoWaitNs = 128;  // wait limits below this: kernels give up at their first wait

struct CausalLinArgs {
  int n_q;
  const int32_t* page_table;
  const __nv_bfloat16* k_pool;
  const __nv_bfloat16* v_pool;
  // workspace: phi(K) of the pages that hold the chunk as bf16 terms, [H][hi/mid/lo][phik_blocks][64][D], block 0
  // being the chunk's first page (its rows before the chunk included)
  __nv_bfloat16* phik;
  int phik_blocks;
  float* sums;     // workspace: sums over groups of pages, [H][sum_groups][...] (causal_sums_bytes; null: none)
  int sum_groups;
  int64_t q_pos0;   // first query position == first token of the intra-chunk part
  int H, D;
  int relu;  // feature map: 0 elu(x) + 1, 1 max(x, 0)
  int nsm;    // SMs of the device
  int alone;  // 1: the forward behind it is the linear branch alone
  int give_up;  // 1: the sums over groups are given up before the first product (a wait limit of next to nothing)
  float* lin_num;
  float* lin_den;
  int32_t* status;  // device status word
};

constexpr int kPageCtasPerSm = 6;  // CTAs of the page write, a row of a thread at a time, on an SM (see launch_append)

struct LinformerArgs {
  const __nv_bfloat16* k;
  const __nv_bfloat16* v;
  int64_t tok_stride, head_stride;
  const __nv_bfloat16* e_k;  // [H][seg_tokens][rank]
  const __nv_bfloat16* e_v;
  __nv_bfloat16* kc_pool;    // [compressed pages][H][64][128]
  __nv_bfloat16* vc_pool;
  int32_t* ccnt;             // [H] number of valid compressed pages
  int H, rank, seg_tokens, seg_index;
  int nsm;                   // SMs of the device
  int give_up;               // 1: the products are given up before the first (a wait limit of next to nothing)
  int32_t* status;
};

// tensor maps of the fused append kernel: the chunk's K and V ([tokens][H][d], box 64 dims x 1 x 64
// tokens) and the two pools ([rows][d], box 64 x 64), all with the 128-byte swizzle
struct AppendMaps {
  CUtensorMap kin, vin, kpool, vpool;
};
cudaError_t launch_append(const AppendArgs& a, const AppendMaps* maps, cudaStream_t st);
// clusters: how many clusters of 2, 4 and 8 CTAs of the compression kernel the device runs at once (linformer_init);
// one_row (output): which form of the page write runs best beside this launch
cudaError_t launch_linformer_compress(const LinformerArgs& a, const int (&clusters)[3], int* one_row, const CUtensorMap& tm_ek,
                                      const CUtensorMap& tm_ev, const CUtensorMap& tm_kin, const CUtensorMap& tm_vin,
                                      cudaStream_t st);
cudaError_t linformer_init(int (&clusters)[3]);
struct AdaptiveArgs {
  double* sorted_w;      // [H][n_groups][max_pages] softmax numerators in sorted order
  int32_t* sorted_idx;   // [H][n_groups][max_pages] block ids in sorted order
  double* gini_part;     // [H][n_groups]
  double* wsum;          // [H][n_groups] sum of the numerators
  float tau_min, tau_max;
  float* gini_out;       // [2][H]: Gini and threshold per head (or null)
};

cudaError_t launch_select(const SelectArgs& a, cudaStream_t st);
cudaError_t launch_qsum(const SelectArgs& a, cudaStream_t st);  // stage 1 alone: query tile sums
cudaError_t launch_retrieve(const RetrieveArgs& a, int n_pages, cudaStream_t st);
cudaError_t launch_select_adaptive(const SelectArgs& a, const AdaptiveArgs& ad, cudaStream_t st);
// tm_kc / tm_vc: maps of the compressed pools, used when p.lf_table is set (else null); tm_gl / tm_gs: maps
// of per-dim gate logits with the geometry of tm_q (null: no such gate, or its strides do not allow one); tm_num: map
// of p.lin_num, box 32 dims x 1 x 128 tokens (head_dim 128, may be null).  (Read by the rows' threads, 64 bytes of lines
// 6 KB apart at a time, the partials took 4 to 6 us of each tile, 12 heads of 128, 1560 tokens; as a tile 2.  Beside per-dim
// gate tiles, in lists split through the workspace and at head_dim 64 they still are.)
cudaError_t launch_forward(const FwdParams& p, int D, const CUtensorMap& tm_q,
                           const CUtensorMap& tm_k, const CUtensorMap& tm_v,
                           const CUtensorMap& tm_state, const CUtensorMap& tm_out, cudaStream_t st,
                           const CUtensorMap* tm_kc = nullptr, const CUtensorMap* tm_vc = nullptr,
                           const CUtensorMap* tm_gl = nullptr, const CUtensorMap* tm_gs = nullptr,
                           const CUtensorMap* tm_num = nullptr);
// tm_q: box of 128 tokens of one head; tm_phik, tm_v: rows of phik and of the V pool, box 64 x 64
cudaError_t launch_causal_linear(const CausalLinArgs& a, const CUtensorMap& tm_q, const CUtensorMap& tm_phik,
                                 const CUtensorMap& tm_v, cudaStream_t st);
cudaError_t causal_linear_init();
int causal_sum_groups(int tokens);
size_t causal_sums_bytes(int heads, int tokens);  // head_dim 128
// linear branch alone (head_dim 128): lean HBM-bound kernel, nsm = SMs of the device
cudaError_t launch_linear_only(const FwdParams& p, int nsm, const CUtensorMap& tm_q, const CUtensorMap& tm_state,
                               const CUtensorMap& tm_out, cudaStream_t st);
cudaError_t linear_only_init();
// clusters: how many clusters of 2, 4 and 8 CTAs of the forward kernel the device runs at once
cudaError_t forward_init(int D, int (&clusters)[3]);
cudaError_t append_init();  // opt in to the shared-memory size the fused append kernel needs

}  // namespace hsa

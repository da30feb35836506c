/* Internal declarations of libmemdecay: workspace layout, launch parameters
 * (passed by value; per-sequence counts come from the exact host mirror) and
 * the launchers of the four kernels. */
#ifndef MD_INTERNAL_H
#define MD_INTERNAL_H

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/memdecay.h"

namespace md {

constexpr int D = MD_HEAD_DIM;
constexpr int GP = MD_MAX_GROUP;            // query heads per KV head, padded
constexpr int PARTIAL_FLOATS = 1088;        // m[8] l[8] O[8][128], padded to 256 B
constexpr int MAX_GRID = 512;               // persistent attention CTAs (>= 2 x SM count)

enum DevStatus { ST_CODE = 0, ST_ABORT = 1, ST_DIAG = 2, ST_WORDS = 8 };

/* A decode step's attention mass per token, summed over layers and query
 * heads, is accumulated in fixed point: u64 with MASS_FRAC_BITS fraction
 * bits.  Integer adds make the sum independent of the order in which the
 * (layer, KV head) items finish.  One token receives at most 1 from each
 * query head, so num_layers * num_q_heads < MASS_MAX_HEADS keeps the sum
 * below 2^64. */
constexpr int MASS_FRAC_BITS = 48;
constexpr float MASS_SCALE = 281474976710656.0f;        // 2^48
constexpr float MASS_UNIT = 3.5527136788005009e-15f;    // 2^-48
constexpr long long MASS_MAX_HEADS = 65536;
constexpr int CALIB_BUCKETS = MD_CALIB_BUCKETS;      // age buckets per region
constexpr int CALIB_WIDTH = MD_CALIB_BUCKET_WIDTH;   // decode steps per bucket

struct RegionTable {
  float base[8];
  float half_life[8];
  int pinned[8];
};

/* Byte offsets of every array inside the caller's workspace. */
struct Layout {
  size_t pool, block_table, page_score, free_stack, region, a, t_ref, t_ins, window, ahat, prio, mass_acc,
      scratch, partials, counters, staging_regions, staging_steps, staging_slots, status,
      calib, page_fill, seq_tokens, io_q, io_k, io_v, io_out, total;
  size_t slots, n_items;
  int scratch_tokens, chunk_stride;
};

size_t compute_layout(const md_config &c, Layout *lay);

/* --------------------------------------------------------- state copy --- */
struct CopyParams {
  const uint4 *src;
  uint4 *dst;
  size_t n;                              // 16-byte pieces, at least 1
};
cudaError_t launch_copy(const CopyParams &p, cudaStream_t s);

/* ------------------------------------------------------------- append --- */
/* The arrays an append writes. */
struct AppendTo {
  uint16_t *pool;
  int32_t *block_table;
  const int32_t *free_stack;
  uint8_t *region;
  float *a, *window, *ahat, *prio;
  int32_t *t_ref, *t_ins;
  uint8_t *page_fill;                    // [max_batch][P_max] tokens per page
  int32_t *seq_tokens;                   // [max_batch] tokens per sequence
  int L, Hkv, ps, P_phys, P_max;
};
/* One new token for each of n_seqs sequences (a decode step's append as a
 * launch of its own), in layers [l0, l0 + L); k_src, v_src are
 * [n_seqs][L][Hkv][D].  Layer 0 opens the pages and starts the tokens' state;
 * later layers find both. */
struct AppendStepParams {
  AppendTo to;
  int l0, L;
  const uint16_t *k_src, *v_src;
  const uint4 *q_src;                    // query rows to bring into the workspace on the way
  uint4 *q_dst;
  unsigned q_n;                          // their 16-byte pieces, or 0
  int n_seqs, insert_step;
  int tok0[MD_MAX_BATCH];                // slot of the token in its sequence
  int pop[MD_MAX_BATCH];                 // free-stack index of the page it opens, or -1
  uint8_t regions[MD_MAX_BATCH];
};
cudaError_t launch_append_step(const AppendStepParams &p, cudaStream_t s);

/* n tokens for one sequence (a prompt, a tool's output); k_src, v_src are
 * [L][Hkv][n][D].  The tokens' labels, insertion steps and slots come as runs
 * in the launch parameters; a text of more runs than fit goes through arrays
 * in the workspace instead (regions_dev, and where needed the others). */
constexpr int MAX_RUNS = 512;
struct AppendRun {
  int start;                             // first token of the run
  int slot;                              // its slot in the sequence (then consecutive)
  int step, region;
};
struct AppendTokensParams {
  AppendTo to;
  const uint16_t *k_src, *v_src;
  const uint8_t *regions_dev;            // per token, or null: runs
  const int32_t *steps_dev;              // per token, or null: insert_step
  const int32_t *slots_dev;              // per token, or null: consecutive from tok0
  int seq, n, tok0, insert_step;
  int pages_before;                      // pages of the sequence before this append
  int pop_base;                          // free-stack index of the first page taken
  int n_runs;
  AppendRun runs[MAX_RUNS];
};
cudaError_t launch_append_tokens(const AppendTokensParams &p, bool aligned, cudaStream_t s);

/* ---------------------------------------------------------- attention --- */
/* The decode step's new tokens, one per sequence, when the attention launch
 * also appends them (free_stack != null): each (sequence, layer, KV head)
 * unit that holds the sequence's last page takes the token's K/V rows from
 * k_new / v_new, writes them into the pool, and uses them in place of the
 * page's stale row.  A page that the step opens is not in the block table
 * yet (tail_pop >= 0): every reader takes its id from the free stack, which
 * nothing changes before the next eviction, and the first layer's KV head 0
 * records it and starts the token's state.  One launch fewer per decode step
 * and per layer call: 32 sequences of 430 tokens, 36 layer calls, 579 -> 454 us;
 * one sequence of 1,700 tokens, 28 layer calls, 408 -> 351 us. */
struct NewTokens {
  const uint16_t *k_new, *v_new;
  long long sb, sl;                      // element strides (sequence, layer) of k_new / v_new
  uint16_t *pool;
  const int32_t *free_stack;             // null: the new tokens are in the pool already
  int32_t *block_table;
  uint8_t *region, *page_fill;
  int32_t *t_ref, *t_ins, *seq_tokens;
  float *a, *window, *ahat, *prio;
  int init_state;                        // this launch's first layer starts the tokens' state
  int insert_step;
  int tail_pop[MD_MAX_BATCH];            // free-stack index of the page the token opens, or -1
  uint8_t tail_fill[MD_MAX_BATCH];       // tokens on the last page, the new one included
  uint8_t tail_region[MD_MAX_BATCH];
};

/* What both attention kernels take. */
struct AttnBase {
  const uint16_t *q;
  uint16_t *out;
  const int32_t *block_table;
  const uint8_t *page_fill;  // [max_batch][P_max] tokens per page, or null: pages are
                             // full up to n_tokens
  unsigned long long *mass_acc;   // [slots] fixed-point mass of the step, or null:
  float *mass;                    // [L*Hkv][slots] one fp32 row per (layer, KV head)
  int *status;         // sticky device status words
  int L, Hq, Hkv, G, ps, P_phys, P_max;   // L: layers of the model
  int l0, L_launch;    // layers [l0, l0 + L_launch) attended by this launch
  int q_layers;        // layers held by the q / out tensors (L or 1)
  long long slots;
  float scale_log2;    // log2(e) / sqrt(D)
  long long spin_limit_ns;
  int n_seqs;
  int n_tokens[MD_MAX_BATCH];
  int n_pages[MD_MAX_BATCH];
  NewTokens nt;
};

/* The persistent kernel (md_attn.cu). */
struct AttnParams : AttnBase {
  float *scratch;      // [grid][2][scratch_tokens][8]
  float *partials;     // [items][chunk_stride][PARTIAL_FLOATS]
  int *counters;       // [items]
  int scratch_tokens;  // scratch row capacity per CTA slot (tokens)
  int chunk_stride;    // partial slots reserved per item
  int extra_arrivals;
  int total_units;
  int units_per_seq;   // > 0: every sequence has this many units (no search)
  int chunks[MD_MAX_BATCH];
  int unit_start[MD_MAX_BATCH + 1];
};

/* The cluster kernel (md_attn_cluster.cu): a cluster of C CTAs of 4 or 8
 * warps per (sequence, layer, KV head), each warp with up to 32 tiles of TILE
 * tokens (more when the scores spill to scratch). */
constexpr int TILE = 16;
constexpr int MAX_CLUSTER = 16;
struct ClusterParams : AttnBase {
  int C;               // CTAs per item
  int warp_tiles;      // most tiles of any warp (sizes the score rows)
  int early;           // K/V copies may start before the kernel ahead has finished
  int out16;           // out is 16-byte aligned
  float *scratch;      // spilled scores [CTA][warp][warp_tiles][TILE][8]
};
struct ClusterPlan {
  int C = 0;           // CTAs per item, or 0: the persistent kernel
  int warps = 4, warp_tiles = 0;
  bool spill = false;  // the scores go to scratch
};
cudaError_t cluster_prepare();
ClusterPlan cluster_plan(const AttnBase &p, size_t scratch_floats);
/* One form (C = 0: the launch cannot take it); p as for cluster_plan. */
ClusterPlan cluster_form(const AttnBase &p, size_t scratch_floats, int C, int warps, bool spill);
cudaError_t launch_cluster(const AttnBase &p, const ClusterPlan &plan, bool early, float *scratch,
                           const CUtensorMap &tmap, cudaStream_t s);
/* The tensor maps of the K/V pool (encode: the driver's cuTensorMapEncodeTiled). */
bool encode_page_map(void *encode, CUtensorMap *m, void *pool, size_t rows, int ps);
bool encode_tile_map(void *encode, CUtensorMap *m, void *pool, size_t rows, int ps);
cudaError_t launch_attention(const AttnParams &p, const CUtensorMap &tmap, int grid,
                             cudaStream_t s);
int attention_grid_limit(int ps);     // CTAs resident at once (0 on error)
cudaError_t attention_prepare(int ps); // one-time function attributes

/* --------------------------------------------------- fold / score ------- */
struct ScoreParams {
  unsigned long long *mass_acc;    // [slots] fixed-point mass of the pending step (read, zeroed)
  float *window, *a, *ahat, *prio, *page_score;
  int32_t *t_ref;
  const int32_t *t_ins;
  const uint8_t *region;
  const int32_t *block_table;
  const uint8_t *page_fill;        // [max_batch][P_max] tokens per page
  const int32_t *seq_tokens;       // [max_batch] |K_t| per sequence
  unsigned long long *calib_sum;   // [8][CALIB_BUCKETS] observed mass, fixed point 2^-32
  unsigned int *calib_cnt;         // [8][CALIB_BUCKETS] observations
  int calib_on;
  long long slots;
  int ps, P_max;
  int fold_only;         // 1: window += the pending step's mass and nothing else
  int observe, mass_pending;
  float norm;            // window steps * L * Hq
  int t;
  float rho, gamma, tau_scale, alpha;
  int score_mode, page_reduce, keep_prio;
  unsigned long long random_seed;
  RegionTable reg;
  int n_seqs, total_pages;
  int n_tokens[MD_MAX_BATCH];
  int n_pages[MD_MAX_BATCH];
  int page_start[MD_MAX_BATCH + 1];
};
cudaError_t launch_score(const ScoreParams &p, cudaStream_t s);

/* ------------------------------------------------------------- select --- */
struct SelectParams {
  const float *page_score;
  int32_t *block_table;
  int32_t *free_stack;
  int32_t *user_evicted;  // optional [n_seqs][P_max]
  uint8_t *page_fill;     // [max_batch][P_max], compacted with the block table
  int32_t *seq_tokens;    // [max_batch], less the evicted pages' tokens
  int *status;
  int P_max, n_seqs, top;
  int n_pages[MD_MAX_BATCH];
  int n_evict[MD_MAX_BATCH];
  int push_off[MD_MAX_BATCH];
};
cudaError_t launch_select(const SelectParams &p, cudaStream_t s);

/* ----------------------------------------- observe (score and select) --- */
/* Most pages and token slots of a sequence: a page's rank reads every key, and
 * a block's 1,024 threads score 4,096 slots in four rounds (about 1 us each);
 * beyond that the grid-wide score kernel is the faster one. */
constexpr int OBSERVE_PAGES = 256, OBSERVE_SLOTS = 4096;
struct ObserveParams {
  ScoreParams s;                         // page_fill, seq_tokens: only with region-aligned pages
  int32_t *block_table, *free_stack, *user_evicted, *seq_tokens;
  uint8_t *page_fill;
  int *status;
  int top;
  int n_evict[MD_MAX_BATCH];
  int push_off[MD_MAX_BATCH];
};
cudaError_t launch_observe(const ObserveParams &p, cudaStream_t s);

/* Launch of a kernel taking one parameter struct, with programmatic stream
 * serialization (the kernel calls pdl_wait() before touching global memory). */
template <class P>
cudaError_t launch_pdl(void (*kernel)(P), int grid, int threads, int smem, cudaStream_t s, const P &p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

/* --------------------------------------------------------------- init --- */
cudaError_t launch_init(int32_t *free_stack, int P_phys, int *status, int *counters,
                        size_t n_items, cudaStream_t s);

}  // namespace md

#endif

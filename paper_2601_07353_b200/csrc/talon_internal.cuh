// Internal declarations shared by the translation units of libtalon (sm_100a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "talon.h"

namespace talon {

// ---- device status bits (ctx->d_status) -----------------------------------------------
constexpr int STATUS_NONFINITE = 1;
constexpr int STATUS_TIMEOUT = 2;
constexpr int STATUS_CAPACITY = 4;

// ---- expansion geometry -----------------------------------------------------------------
constexpr int EXP_THREADS = 256;           // threads per CTA of the row-streaming kernels
constexpr int EXP_WARPS = EXP_THREADS / 32;
constexpr int EXP_VEC = 4;                 // floats per 128-bit load
constexpr int EXP_UNROLL = 4;              // 128-bit loads in flight per thread
constexpr int EXP_TILE = EXP_THREADS * EXP_VEC * EXP_UNROLL;   // 4096 elements per CTA step
constexpr int EXP_CHUNK_ALIGN = EXP_THREADS * EXP_VEC;         // chunk boundaries: 1024 elements
constexpr int EXP_MAX_SPLITS = 32;         // a row is cut into at most this many chunks
constexpr int EXP_CTAS_PER_SM = 4;
constexpr int MAX_BUDGET = 128;
constexpr int MAX_BATCH = 1024;
constexpr int SEL_THREADS = 512;
// chunks and lists of the expansion kernels
constexpr int FX_SURV = 64;                // keys of a row that may pass the merge bound before the slow path
constexpr int FX_MAX_SPLITS = 32;          // chunks per row, at most (one lane per chunk in the merge)
constexpr int FX_LONG_SPLITS = 16;         // the same for lists of more than 16 keys (they are merged in shared memory)

// Order-preserving map fp32 -> u32 (larger float <=> larger integer; -inf > 0).
__host__ __device__ inline uint32_t f32_ord(float f) {
#ifdef __CUDA_ARCH__
  uint32_t b = __float_as_uint(f);
#else
  union { float f; uint32_t u; } c; c.f = f; uint32_t b = c.u;
#endif
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__host__ __device__ inline float f32_unord(uint32_t o) {
  uint32_t b = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  union { float f; uint32_t u; } c; c.u = b; return c.f;
#endif
}
// A candidate key: larger key = larger logit, then lower token id.  Key 0 means "empty".
__host__ __device__ inline uint64_t cand_key(float logit, uint32_t tok) {
  return ((uint64_t)f32_ord(logit) << 32) | (uint64_t)(0xFFFFFFFFu - tok);
}
__host__ __device__ inline float key_logit(uint64_t k) { return f32_unord((uint32_t)(k >> 32)); }
__host__ __device__ inline uint32_t key_tok(uint64_t k) { return 0xFFFFFFFFu - (uint32_t)k; }

// How one expansion layer is cut into work items.  Computed identically (from device data)
// by every CTA of the streaming kernel and by the selection kernel.
struct LayerGeom {
  int total_rows;   // frontier rows over all sequences
  int splits;       // chunks per row
  int chunk_len;    // elements per chunk (multiple of EXP_CHUNK_ALIGN)
};

__host__ __device__ inline LayerGeom make_geom(int total_rows, int vocab, int target_items,
                                               int max_splits = EXP_MAX_SPLITS, int min_chunk = EXP_CHUNK_ALIGN) {
  LayerGeom g;
  g.total_rows = total_rows;
  int want = total_rows > 0 ? (target_items + total_rows - 1) / total_rows : 1;
  if (want < 1) want = 1;
  if (want > max_splits) want = max_splits;
  int len = (vocab + want - 1) / want;
  len = ((len + EXP_CHUNK_ALIGN - 1) / EXP_CHUNK_ALIGN) * EXP_CHUNK_ALIGN;
  if (len < min_chunk) len = min_chunk;
  g.chunk_len = len;
  g.splits = (vocab + len - 1) / len;
  return g;
}

}  // namespace talon

namespace talon {
// A whole step captured as a CUDA graph, keyed by every argument of the call that made it.
constexpr int STEP_GRAPH_SLOTS = 64;
constexpr int STEP_GRAPH_WORDS = 36;
struct StepGraph {
  unsigned long long args[STEP_GRAPH_WORDS];
  cudaGraphExec_t exec;      // null: arguments seen once, nothing captured yet
  long long launches;        // kernels one replay launches
  int layers_run;            // host-side depth counter after the step
  unsigned long long last_use;
  bool used;
};
}  // namespace talon

// The context: parameters, host-side counters, and the device workspace.
struct talon_ctx {
  talon_params p;
  int device;
  int sm_count;
  int W;                  // mask words per node
  int k_cap;              // per-parent candidate cap actually used (cand_topk or N-1)
  int key_stride;         // keys stored per row / per item (k_cap rounded up to 4)
  int B;                  // batch of the current reset
  int layers_run;         // expand calls since reset
  int64_t launches;
  double log_mu;

  void *d_arena;                  // the one allocation behind the pointers below
  int *d_status;                  // the status word; the one after it takes what talon_loop's earlier steps report
  int32_t *d_prefix_len;          // [batch_max]
  // expansion workspace
  int exp_grid;                   // CTAs of the streaming kernel at full width
  int rows_cap;                   // batch_max * (N-1)
  int items_cap;                  // exp_grid + rows_cap
  unsigned long long *d_part_keys;   // [items_cap, key_stride]  per-chunk top-k
  float2 *d_part_ms;                 // [items_cap]              per-chunk (max, sum exp)
  unsigned long long *d_row_keys;    // [rows_cap, key_stride]   per-row top-k
  double *d_row_score;               // [rows_cap, key_stride]   per-row candidate scores (fused kernel, wide frontiers)
  unsigned int *d_row_count;         // [rows_cap]               chunks finished per row, layer by layer (zeroed by a reset)
  unsigned int *d_pass_count;        // [rows_cap]               the same for the row pass (zeroed by the growth kernel after it)
  unsigned int *d_seq_count;         // [batch_max]              chunks finished per sequence (fused kernel)
  int fused_grid;                    // CTAs of the fused kernel at full width
  // whole-step growth (grow_step.cu)
  int ahead;                         // steps of talon_loop whose rows one pass prepares (the workspace holds them)
  int row_grid;                      // CTAs of the row pass at full width
  int32_t *d_growing, *d_depth_at;   // [batch_max] a sequence's tree still grows; layer it stopped at
  unsigned int *d_row_bad;           // [batch_max * N] NaN in a target row (zero between calls)
  int step_rows;                     // 0: whole steps expand layer by layer too
  int step_first_rows;               // > 0: slots per sequence the first round of a step prepares (for experiments)
  int attn_cluster;                  // key ranges of the tensor-core attention merge inside a cluster (1; 2: never more of them than it has CTAs) or in a second kernel (0)
  int attn_clusters[3][9];           // per kind of the tensor-core attention and cluster size: clusters the device holds at once (-1 not asked yet)
  int attn_force_splits;             // > 0: key ranges per (sequence, head, query tiles), for experiments
  int attn_force_tiles;              // 1, 2: query tiles of a CTA, for experiments (1 also where two cannot be had)
  int argmax_oversplit;              // softmax statistics of target rows: chunk rounds per CTA when the rows outnumber the grid
  int expand_max_split;              // fused kernel: chunks a row is cut into at most when the grid has room
  int attn_min_tiles;                // split-KV: key tiles a CTA should at least own
  int pdl;                           // programmatic stream serialization: 1 on, 0 off, -1 on for small batches
  // verification workspace
  unsigned long long *d_argmax;      // [batch_max * N] packed (logit, token) maxima
  int32_t *d_target_tok;             // [batch_max * N]
  unsigned int *d_walk_count;        // [batch_max] what is finished of a sequence's arg-max, or of its commit (zero between calls)
  float2 *d_samp_ms;                 // [batch_max * N, EXP_MAX_SPLITS] per-chunk (max, sum) of target rows
  float *d_attn_o;                   // split-KV partial outputs
  float2 *d_attn_ml;                 // split-KV partial (max, sum)
  size_t attn_o_elems, attn_ml_elems;
  // host-step staging (allocated on first use)
  struct HostStage *stage;
  // per-kernel timing (off unless talon_timing_enable was called)
  cudaEvent_t *ev;                   // [2 * ev_cap] start/stop pairs
  int *ev_kernel;                    // [ev_cap] kernel id of each pair
  int ev_cap, ev_used;
  unsigned ev_mask;                  // kernel families that are timed
  int ev_paused;                     // 1: launches are not bracketed for now
  // talon_step replays (see talon_step)
  int step_graph;                    // 0: never capture
  unsigned long long step_tick;
  talon::StepGraph *graphs;          // [STEP_GRAPH_SLOTS], allocated on first use
};

namespace talon {

// Programmatic dependent launch.  Every kernel of the library starts with pdl_enter(): it lets
// the next kernel of the stream be scheduled at once and then waits until the previous kernel
// has completed and its memory is visible, so only launch latency overlaps, never data.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launches `kernel` so that it may be scheduled while its predecessor in the stream drains
// (the kernel itself waits in pdl_enter()); a plain launch when ctx->pdl is off.  A step is a chain of
// dependent kernels, most of them short, so the overlap of launch latency pays at every batch size
// (sampling verification of 8 sequences: 252 -> 242 us).  The exceptions, chain = false, are launched this way
// up to PDL_AUTO_BATCH sequences only: the row pass of a whole step, whose CTAs, waiting beside the attention of the
// step before, slow that down (270 -> 278 us at the shape with 64 query heads), and an attention that does not start
// beside the growth of the trees, whose CTAs fill SMs and so would take them from the kernel before.
constexpr int PDL_AUTO_BATCH = 4;
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_pdl(const talon_ctx *c, bool chain, void (*kernel)(KArgs...), dim3 grid, dim3 block,
                                     size_t smem, cudaStream_t st, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = (c->pdl == 1 || (c->pdl < 0 && (c->B <= PDL_AUTO_BATCH || chain))) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(const talon_ctx *c, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t st, Args &&...args) {
  return launch_kernel_pdl(c, true, kernel, grid, block, smem, st, static_cast<Args &&>(args)...);
}

// Brackets one kernel launch with a pair of CUDA events on the launching stream when timing
// is on; does nothing otherwise.  Pairs beyond the capacity are silently not timed.
struct LaunchTimer {
  talon_ctx *c;
  cudaStream_t st;
  int slot;
  LaunchTimer(talon_ctx *ctx, int kernel, cudaStream_t stream) : c(ctx), st(stream), slot(-1) {
    if (c->ev && !c->ev_paused && ((c->ev_mask >> kernel) & 1u) && c->ev_used < c->ev_cap) {
      slot = c->ev_used++;
      c->ev_kernel[slot] = kernel;
      cudaEventRecord(c->ev[2 * slot], st);
    }
  }
  ~LaunchTimer() {
    if (slot >= 0) cudaEventRecord(c->ev[2 * slot + 1], st);
  }
};

// Lets `kernel` be launched with as much dynamic shared memory as the device has.  The bound belongs to the kernel, not to
// a context: set to what one context needs, it would refuse the launches of an older one that needs more.
template <typename... KArgs>
inline bool allow_shared_memory(const talon_ctx *c, void (*kernel)(KArgs...)) {
  int most = 0;
  cudaFuncAttributes at;
  return cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) == cudaSuccess &&
         cudaFuncGetAttributes(&at, kernel) == cudaSuccess &&
         cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)at.sharedSizeBytes) == cudaSuccess;
}

// launchers implemented in the .cu files (all asynchronous on `st`).  launch_attention's early_prefix: the
// kernel launched just before is grow_kernel, and this array holds the prefix lengths it copies
talon_status launch_reset(talon_ctx *c, const talon_tree *t, const int32_t *root_tok,
                          const int32_t *prefix_len, int B, cudaStream_t st);
talon_status launch_expand(talon_ctx *c, const talon_tree *t, const float *logits,
                           int64_t row_stride, int rows_per_seq, int layout, cudaStream_t st);
// The draft phase of a whole step (reset, n_layers layers, closing pass) from the draft rows of all node
// slots; k_cap <= 32.  *accepted: the target rows' arg-max and the walk are done as well.
talon_status grow_step_setup(talon_ctx *c);
bool step_rows_pay(const talon_ctx *c, int B, int n_layers);      // false: go layer by layer
talon_status launch_grow_step(talon_ctx *c, const talon_tree *t, const int32_t *root_tok, const int32_t *prefix_len,
                              const float *draft, int64_t draft_stride, int n_layers, const float *target,
                              int64_t target_stride, int32_t *target_tok, int32_t *accept_len, int32_t *accept_nodes,
                              int32_t *bonus_tok, cudaStream_t st, bool *accepted);
// The same for talon_loop, whose steps' rows are all there at the start: rows of `steps` steps (ctx->ahead at most)
// in one pass, then per step the growth and the walk.  False from loop_rows_possible: step by step instead.
bool loop_rows_possible(const talon_ctx *c, int n_layers);
talon_status launch_loop_rows(talon_ctx *c, const float *draft, int64_t draft_stride, int64_t draft_step, int n_layers,
                              const float *target, int64_t target_stride, int64_t target_step, int steps, cudaStream_t st);
talon_status launch_loop_grow(talon_ctx *c, const talon_tree *t, const int32_t *root_tok, const int32_t *prefix_len, int n_layers,
                              int step, int32_t *target_tok, int32_t *accept_len, int32_t *accept_nodes, int32_t *bonus_tok,
                              cudaStream_t st);
talon_status launch_build(talon_ctx *c, const talon_tree *t, uint8_t *dense, cudaStream_t st);
talon_status launch_prune(talon_ctx *c, const talon_tree *t, int keep, cudaStream_t st);
talon_status launch_attention(talon_ctx *c, const talon_tree *t, const void *q, const void *kp,
                              const void *vp, const void *kt, const void *vt,
                              const int64_t *kv_start, const int32_t *block_table, int bt_stride, int64_t kv_tokens,
                              int64_t stride_t, int64_t stride_h,
                              int max_prefix_len, float sm_scale, void *out, cudaStream_t st,
                              const int32_t *early_prefix = nullptr);
bool attention_tc_supported(const talon_ctx *c, int64_t stride_t, int64_t stride_h, float sm_scale);
enum { TC_PAIR = 0, TC_SINGLE = 1, TC_SPLIT_P = 2 };      // query tiles of a CTA; one with P in two bf16 parts
int attention_tc_clusters(talon_ctx *c, int kind, int splits);
talon_status launch_attention_tc(talon_ctx *c, const talon_tree *t, const void *q, const void *kp, const void *vp,
                                 const void *kt, const void *vt, const int64_t *kv_start, const int32_t *block_table,
                                 int bt_stride, int64_t stride_t, int64_t stride_h, int64_t kv_tokens, int max_prefix_len, float sm_scale, void *out,
                                 int splits, int m_blocks, int kind, bool exact_max, cudaStream_t st, int *merged_in_kernel,
                                 const int32_t *early_prefix);
talon_status launch_accept(talon_ctx *c, const talon_tree *t, const float *target_logits,
                           int64_t row_stride, int32_t *target_tok, int32_t *accept_len,
                           int32_t *accept_nodes, int32_t *bonus_tok, cudaStream_t st, bool close_tree = false);
talon_status launch_accept_sample(talon_ctx *c, const talon_tree *t, const float *target_logits, int64_t row_stride,
                                  double temperature, const double *u_accept, const double *u_sample,
                                  int32_t *accept_len, int32_t *accept_nodes, int32_t *out_tok, cudaStream_t st);
talon_status launch_commit(talon_ctx *c, const talon_tree *t, const int32_t *accept_len, const int32_t *accept_nodes,
                           const int32_t *next_tok, const void *k_tree, const void *v_tree, void *k_prefix,
                           void *v_prefix, const int64_t *kv_start, const int64_t *kv_limit, const int32_t *block_table,
                           int bt_stride, const int32_t *n_blocks, int64_t kv_tokens, int64_t stride_t, int64_t stride_h,
                           int32_t *prefix_len, int32_t *root_tok, int64_t *counters, cudaStream_t st);
size_t attention_workspace_elems(const talon_ctx *c, size_t *ml_elems);
talon_status expand_fused_setup(talon_ctx *c);
talon_status launch_expand_fused(talon_ctx *c, const talon_tree *t, const float *logits, int64_t row_stride,
                                 int rows_per_seq, int layout, int rows_bound, cudaStream_t st);

}  // namespace talon

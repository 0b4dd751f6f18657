// The small kernels around the expansion of a draft tree (Algorithm 2 of the paper): initialisation,
// closing pass (positions, sentinels), Top-N prune of the static construction (Algorithm 1).  The layers
// themselves are expand_fused.cu, whole steps grow_step.cu.
#include <math_constants.h>

#include "talon_internal.cuh"

namespace talon {

// ---------------------------------------------------------------------------------------
// Reset and closing pass.
// ---------------------------------------------------------------------------------------
__global__ void reset_kernel(talon_tree t, const int32_t *root_tok, const int32_t *prefix_len,
                             int32_t *prefix_copy, int B, int N, int W, int lo_stride, int *status,
                             unsigned int *row_count, int rows_cap, unsigned int *seq_count) {
  pdl_enter();
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  const int stride = gridDim.x * blockDim.x;
  if (gid == 0) *status = 0;
  for (int i = gid; i < rows_cap; i += stride) row_count[i] = 0u;
  for (int i = gid; i < B; i += stride) seq_count[i] = 0u;
  for (int b = gid; b < B; b += stride) {
    const size_t nb = (size_t)b * N;
    t.n_nodes[b] = 1;
    t.token[nb] = root_tok[b];
    t.parent[nb] = -1;
    t.depth[nb] = 0;
    t.score[nb] = 0.0;
    for (int w = 0; w < W; ++w) t.mask[nb * W + w] = (w == 0) ? 1ull : 0ull;
    t.layer_off[b * lo_stride] = 0;
    t.layer_off[b * lo_stride + 1] = 1;
    prefix_copy[b] = prefix_len[b];
  }
}

__global__ void build_tree_kernel(talon_tree t, const int32_t *prefix_len, uint8_t *dense, int B, int N,
                                  int W, int lo_stride, int layers_run) {
  pdl_enter();
  const int b = blockIdx.x;
  const int n = t.n_nodes[b];
  const size_t nb = (size_t)b * N;
  const int L = prefix_len[b];
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    if (i < n) {
      t.position[nb + i] = L + t.depth[nb + i];
    } else {
      t.token[nb + i] = -1;
      t.parent[nb + i] = -1;
      t.depth[nb + i] = -1;
      t.position[nb + i] = -1;
      t.score[nb + i] = -CUDART_INF;
      for (int w = 0; w < W; ++w) t.mask[(nb + i) * W + w] = ((i >> 6) == w) ? (1ull << (i & 63)) : 0ull;
    }
  }
  for (int i = layers_run + 2 + threadIdx.x; i < lo_stride; i += blockDim.x) t.layer_off[b * lo_stride + i] = n;
  if (dense) {
    __syncthreads();
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) {
      const int i = e / N, j = e - i * N;
      dense[(size_t)b * N * N + e] = (uint8_t)((t.mask[(nb + i) * W + (j >> 6)] >> (j & 63)) & 1ull);
    }
  }
}

// Last step of Algorithm 1 (static tree construction): T <- Top-N(T by p(u)).  One CTA per
// sequence, one thread per node.  A node's rank is the number of nodes with a larger score, or
// the same score and a lower index, so a kept node's parent (score at least as large, index
// lower) is kept too; the survivors keep their order, parents and mask bits are renumbered, the
// layer offsets recounted.  Slots past the new size are left to talon_build_tree.
__global__ void __launch_bounds__(MAX_BUDGET)
prune_tree_kernel(talon_tree t, int B, int N, int W, int lo_stride, int keep) {
  __shared__ double s_score[MAX_BUDGET];
  __shared__ int s_new[MAX_BUDGET];          // new index of a kept node, -1 for a dropped one
  __shared__ int s_depth[MAX_BUDGET];
  __shared__ unsigned s_keep[MAX_BUDGET / 32];
  pdl_enter();
  const int b = blockIdx.x, i = threadIdx.x, lane = i & 31, warp = i >> 5;
  const int n = t.n_nodes[b];
  const size_t nb = (size_t)b * N;
  const bool live = i < n;
  const double sc = live ? t.score[nb + i] : -CUDART_INF;
  const int tok = live ? t.token[nb + i] : -1, par = live ? t.parent[nb + i] : -1, dep = live ? t.depth[nb + i] : -1;
  unsigned long long mk[2] = {0ull, 0ull};
  if (live)
    for (int w = 0; w < W; ++w) mk[w] = t.mask[(nb + i) * W + w];
  s_score[i] = sc;
  __syncthreads();
  int rank = 0;
  for (int j = 0; j < n; ++j) rank += (s_score[j] > sc || (s_score[j] == sc && j < i)) ? 1 : 0;
  const bool kept = live && rank < keep;
  const unsigned bal = __ballot_sync(0xFFFFFFFFu, kept);
  if (lane == 0) s_keep[warp] = bal;
  __syncthreads();
  int before = __popc(bal & ((1u << lane) - 1u));
  for (int w = 0; w < warp; ++w) before += __popc(s_keep[w]);
  int total = 0;
  for (int w = 0; w < MAX_BUDGET / 32; ++w) total += __popc(s_keep[w]);
  s_new[i] = kept ? before : -1;
  s_depth[i] = kept ? dep : 0x7FFFFFFF;
  __syncthreads();
  if (kept) {
    const int ni = before;
    t.token[nb + ni] = tok;
    t.parent[nb + ni] = par < 0 ? -1 : s_new[par];
    t.depth[nb + ni] = dep;
    t.score[nb + ni] = sc;
    unsigned long long nm[2] = {0ull, 0ull};
    for (int w = 0; w < W; ++w) {
      unsigned long long bits = mk[w];
      while (bits) {
        const int j = w * 64 + __ffsll((long long)bits) - 1;
        bits &= bits - 1ull;
        const int nj = s_new[j];
        if (nj >= 0) nm[nj >> 6] |= 1ull << (nj & 63);
      }
    }
    for (int w = 0; w < W; ++w) t.mask[(nb + ni) * W + w] = nm[w];
  }
  // layer_off[d] = kept nodes of depth < d (kept nodes stay sorted by depth)
  for (int d = i; d < lo_stride; d += MAX_BUDGET) {
    int c = 0;
    for (int j = 0; j < n; ++j) c += s_depth[j] < d ? 1 : 0;
    t.layer_off[b * lo_stride + d] = c;
  }
  if (i == 0) t.n_nodes[b] = total;
}

// ---------------------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------------------
talon_status launch_prune(talon_ctx *c, const talon_tree *t, int keep, cudaStream_t st) {
  LaunchTimer lt(c, TALON_K_BUILD, st);
  launch_kernel(c, prune_tree_kernel, dim3(c->B), dim3(MAX_BUDGET), 0, st, *t, c->B, c->p.budget, c->W,
                c->p.max_depth + 2, keep);
  c->launches += 1;
  return cudaGetLastError() == cudaSuccess ? TALON_OK : TALON_ERR_CUDA;
}

static int frontier_upper_bound(const talon_ctx *c, int d) {
  // host-side bound on rows per sequence at layer d (the device knows the real sizes)
  long long f = 1;
  for (int i = 0; i < d; ++i) {
    long long w = (i < c->p.init_layers) ? c->p.root_topk : f * c->k_cap;
    f = w;
    if (f >= c->p.budget - 1) { f = c->p.budget - 1; break; }
  }
  if (f > c->p.budget - 1) f = c->p.budget - 1;
  if (f < 1) f = 1;
  return (int)f;
}

talon_status launch_reset(talon_ctx *c, const talon_tree *t, const int32_t *root_tok,
                          const int32_t *prefix_len, int B, cudaStream_t st) {
  const int threads = 256;
  int blocks = (c->rows_cap + threads - 1) / threads;
  if (blocks > 64) blocks = 64;
  if (blocks < 1) blocks = 1;
  LaunchTimer lt(c, TALON_K_RESET, st);
  launch_kernel(c, reset_kernel, dim3(blocks), dim3(threads), 0, st, *t, root_tok, prefix_len, c->d_prefix_len, B,
                c->p.budget, c->W, c->p.max_depth + 2, c->d_status, c->d_row_count, c->rows_cap, c->d_seq_count);
  c->launches += 1;
  return cudaGetLastError() == cudaSuccess ? TALON_OK : TALON_ERR_CUDA;
}

talon_status launch_expand(talon_ctx *c, const talon_tree *t, const float *logits, int64_t row_stride,
                           int rows_per_seq, int layout, cudaStream_t st) {
  return launch_expand_fused(c, t, logits, row_stride, rows_per_seq, layout, c->B * frontier_upper_bound(c, c->layers_run), st);
}

talon_status launch_build(talon_ctx *c, const talon_tree *t, uint8_t *dense, cudaStream_t st) {
  LaunchTimer lt(c, TALON_K_BUILD, st);
  launch_kernel(c, build_tree_kernel, dim3(c->B), dim3(128), 0, st, *t, c->d_prefix_len, dense, c->B, c->p.budget,
                c->W, c->p.max_depth + 2, c->layers_run);
  c->launches += 1;
  return cudaGetLastError() == cudaSuccess ? TALON_OK : TALON_ERR_CUDA;
}

}  // namespace talon

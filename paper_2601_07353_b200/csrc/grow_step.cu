// The draft phase of a whole step in two kernels (k <= 32), for callers that hand in the draft logits
// of every node slot at once (talon_step, talon_loop, talon_step_host).
//
// What a logit row contributes to the tree -- its k best tokens and their log-probabilities -- does
// not depend on where its node sits in the tree.  Expanding layer by layer (expand_fused.cu) makes
// each layer a dependent chain of launch, DRAM trip, hand-off and merge, about 7 to 12 us however few
// bytes it reads; with all rows at hand that chain is paid once:
//
//   row_pass_kernel : every row of the step, at the streaming rate: k best keys with log P(w | v)
//                     (Eq. 3) per node slot and, when the target rows come along, each target row's
//                     arg-max.  Rows are cut over the grid as in expand_fused.cu, the CTA that
//                     completes a row merges it.
//   grow_kernel     : one CTA per sequence runs Algorithm 2's while-loop on those lists in shared
//                     memory (Top-K of Eq. 5, gate of Eq. 4, truncation to the budget, append) and
//                     closes the tree; with the arg-max of the target rows at hand it walks the
//                     accepted path too.
//
// Rows of slots that the tree turns out not to use, or not to expand, are read for nothing: cheap
// while a step is a few MB, not when it is hundreds.  Large steps therefore go in rounds: a round
// prepares the next rows of the sequences whose trees still grow, then the trees grow as far as those
// rows carry them.
#include "expand_stream.cuh"

namespace talon {

namespace {

struct RowPassArgs {
  const float *draft, *target;        // [B, N] rows; target null: draft rows only
  int64_t draft_stride, target_stride;
  int B, N, V, k, key_stride, max_split;
  int r0, r1;                         // node slots of this round, per sequence
  int t1;                             // target rows of slots r0 .. t1-1 (t1 = r0: none)
  int draft_ctas;                     // CTAs 0 .. draft_ctas-1 take draft rows, the others target rows
  int init_layers;
  double log_mu;
  const int32_t *growing;             // [B] nonzero: this sequence still needs rows; null: all do
  u64 *part_keys; float2 *part_ms;
  u64 *row_keys; double *row_lp;      // [B * N, key_stride]; row_lp slot 0 NaN: row without a softmax
  unsigned int *row_count;            // [B * N] elements of a packed row finished (zero between launches)
  u64 *best; unsigned int *row_bad;   // [B * N] arg-max key and NaN flag of a target row (zero before)
  int *status;
  int clear_status;                   // the step's first launch
};

// Packed rows of the round: the growing sequences' slots one sequence after the other.
struct ActiveSeqs {
  int base_l;            // B <= 32: first packed row of sequence `lane`
  int total;
  const int *s_base;     // B > 32
};

// Block-wide exclusive scan of the row counts of B sequences into s_base[0 .. B].
__device__ void scan_active(const int32_t *growing, int B, int cnt, int *s_base, int *s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int PER = (MAX_BATCH + EXP_THREADS - 1) / EXP_THREADS;
  int f[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int b = tid * PER + i;
    f[i] = (b < B && (!growing || growing[b])) ? cnt : 0;
    sum += f[i];
  }
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  int before = 0, total = 0;
  for (int w = 0; w < EXP_WARPS; ++w) { before += w < warp ? s_warp[w] : 0; total += s_warp[w]; }
  int run = before + inc - sum;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int b = tid * PER + i;
    if (b < B) s_base[b] = run;
    run += f[i];
  }
  if (tid == 0) s_base[B] = total;
  __syncthreads();
}

// Sequence of packed row `row` and the row's index among that sequence's.
__device__ __forceinline__ void locate_active(const RowPassArgs &a, const ActiveSeqs &q, int row, int cnt, int &b, int &j) {
  if (!a.growing) {                      // every sequence has cnt rows
    b = row / cnt;
    j = row - b * cnt;
  } else if (a.B <= 32) {
    const int lane = threadIdx.x & 31;
    b = 31 - __clz(__ballot_sync(FULL, lane < a.B && q.base_l <= row));
    j = row - __shfl_sync(FULL, q.base_l, b);
  } else {
    b = seq_of_row(q.s_base, a.B, row);
    j = row - q.s_base[b];
  }
}

// Arg-max of elements [start, end) of a target row into best[slot] (lowest index among equal maxima,
// a NaN never wins but sets bad[slot]): 16 elements per thread and step, the next step's loads issued
// before the current one is worked on, the index looked for only in a step that raises the maximum.
__device__ __forceinline__ void argmax_chunk(const float *rowp, int start, int end, u64 *best, unsigned int *bad_flag,
                                             u64 *s_key) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float bestv = -CUDART_INF_F;
  uint32_t besti = 0xFFFFFFFFu;
  bool bad = false;
  float4 nx[EXP_UNROLL];
  auto load = [&](int base) {
#pragma unroll
    for (int u = 0; u < EXP_UNROLL; ++u) {
      const int idx = base + u * EXP_CHUNK_ALIGN + tid * EXP_VEC;
      if (idx + EXP_VEC <= end) nx[u] = __ldcs(reinterpret_cast<const float4 *>(rowp + idx));
      else {
        nx[u].x = idx < end ? __ldcs(rowp + idx) : -CUDART_INF_F;
        nx[u].y = idx + 1 < end ? __ldcs(rowp + idx + 1) : -CUDART_INF_F;
        nx[u].z = idx + 2 < end ? __ldcs(rowp + idx + 2) : -CUDART_INF_F;
        nx[u].w = -CUDART_INF_F;
      }
    }
  };
  load(start);
  for (int base = start; base < end; base += EXP_TILE) {
    float v[EXP_UNROLL * EXP_VEC];
#pragma unroll
    for (int u = 0; u < EXP_UNROLL; ++u) { v[4 * u] = nx[u].x; v[4 * u + 1] = nx[u].y; v[4 * u + 2] = nx[u].z; v[4 * u + 3] = nx[u].w; }
    if (base + EXP_TILE < end) load(base + EXP_TILE);
    float bm = -CUDART_INF_F;
#pragma unroll
    for (int e = 0; e < EXP_UNROLL * EXP_VEC; ++e) { bad |= (v[e] != v[e]); bm = fmaxf(bm, v[e]); }
    if (bm > bestv || besti == 0xFFFFFFFFu) {
      uint32_t first = 0xFFFFFFFFu;
#pragma unroll
      for (int e = EXP_UNROLL * EXP_VEC - 1; e >= 0; --e) {
        const int idx = base + (e / EXP_VEC) * EXP_CHUNK_ALIGN + tid * EXP_VEC + e % EXP_VEC;
        if (idx < end && v[e] == bm) first = (uint32_t)idx;
      }
      if (first != 0xFFFFFFFFu) { bestv = bm; besti = first; }
    }
  }
  u64 key = warp_max_u64(besti == 0xFFFFFFFFu ? 0ull : cand_key(bestv, besti));
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(bad_flag, 1u);
  if (lane == 0) s_key[warp] = key;
  __syncthreads();
  if (warp == 0) {
    key = warp_max_u64(lane < EXP_WARPS ? s_key[lane] : 0ull);
    if (lane == 0 && key) atomicMax(best, key);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(EXP_THREADS, 3)
row_pass_kernel(RowPassArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ u64 s_buf[EXP_WARPS][XS_BUF];
  __shared__ u64 s_pool[XS_POOL];
  __shared__ float s_m[EXP_WARPS], s_s[EXP_WARPS], s_wtop[EXP_WARPS], s_wmax[EXP_WARPS];
  __shared__ __align__(8) u64 s_bar[EXP_WARPS][XS_RING];
  __shared__ int s_warp[EXP_WARPS];
  __shared__ int s_pool_n, s_last, s_abort;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = a.k;
  const ChunkShared sh = {reinterpret_cast<float *>(smem_raw) + warp * (XS_RING * XS_WTILE), s_bar[warp], s_buf[warp], s_pool,
                          s_m, s_s, s_wtop, s_wmax, &s_pool_n, &s_abort};
  const ChunkOut res = {a.part_keys, a.part_ms, a.key_stride, a.status};
  u64 *stage = reinterpret_cast<u64 *>(smem_raw + sizeof(float) * EXP_WARPS * XS_RING * XS_WTILE);    // merge of a row
  int *s_base = reinterpret_cast<int *>(stage + stage_words(k));                                       // B > 32, later rounds
  if (lane == 0) {
    for (int i = 0; i < XS_RING; ++i) ring_bar_init(smem_addr(&s_bar[warp][i]));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  chunk_clear(sh);
  if (tid == 0) s_abort = 0;
  pdl_enter();
  if (a.clear_status && blockIdx.x == 0 && tid == 0) *a.status = 0;

  const bool is_draft = (int)blockIdx.x < a.draft_ctas;
  const int cnt = (is_draft ? a.r1 : a.t1) - a.r0;
  ActiveSeqs q = {0, cnt * a.B, s_base};
  if (a.growing) {
    if (a.B <= 32) {
      int inc = (lane < a.B && a.growing[lane]) ? cnt : 0;
      const int own = inc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += t;
      }
      q.base_l = inc - own;
      q.total = __shfl_sync(FULL, inc, 31);
    } else {
      scan_active(a.growing, a.B, cnt, s_base, s_warp);
      q.total = s_base[a.B];
    }
  }
  __syncthreads();

  const int cta = is_draft ? (int)blockIdx.x : (int)blockIdx.x - a.draft_ctas;
  const SpanGeom g = span_geom(q.total, a.V, is_draft ? a.draft_ctas : (int)gridDim.x - a.draft_ctas, a.max_split);
  const unsigned long long line_end = (unsigned long long)q.total * g.pitch;
  const float ln_mu = (float)a.log_mu;
  unsigned wt = 0;

  unsigned long long pos = (unsigned long long)cta * g.span;
  const unsigned long long span_end = min(line_end, pos + g.span);
  int row = pos < span_end ? (int)div_u64(pos, g.pitch) : 0;
  int start = pos < span_end ? (int)(pos - (unsigned long long)row * g.pitch) : 0;
  for (; pos < span_end; ++row, start = 0) {
    const int len = (int)min((unsigned long long)(g.pitch - (unsigned)start), span_end - pos);
    pos += (unsigned)len;
    int b, j;
    locate_active(a, q, row, cnt, b, j);
    const int node = a.r0 + j;
    const size_t slot = (size_t)b * a.N + node;
    const int end = min(a.V, start + len);
    if (!is_draft) {
      if (start < end)
        argmax_chunk(a.target + (int64_t)slot * a.target_stride, start, end, a.best + slot, a.row_bad + slot, s_pool);
      continue;
    }
    // a node below the root is gated when every layer but the first is; deeper Top-K layers are not told apart here
    const bool gated = a.init_layers == 0 || (a.init_layers == 1 && node > 0);
    const int item = cta + row;
    if (!stream_chunk(sh, a.draft + (int64_t)slot * a.draft_stride, start, end, k, k, gated, ln_mu, (size_t)item, res, wt)) return;

    // the barrier orders this CTA's chunk results before thread 0's device-scope release; whoever
    // brings the row's last elements acquires and merges the row
    __syncthreads();
    chunk_clear(sh);
    if (tid == 0) {
      if ((unsigned)len == g.pitch) s_last = 1;
      else {
        cuda::atomic_ref<unsigned int, cuda::thread_scope_device> c(a.row_count[row]);
        const unsigned prev = c.fetch_add((unsigned)len, cuda::memory_order_acq_rel);
        s_last = (prev + (unsigned)len == g.pitch);
        if (s_last) c.store(0u, cuda::memory_order_relaxed);
      }
    }
    __syncthreads();
    if (s_last && warp == 0) {
      u64 key; double lp;
      int item0, S;
      row_chunks(g, row, item0, S);
      const bool finite = merge_row(res, (size_t)item0, S, k, k, 0.0, stage, key, lp);
      if (!finite) lp = lane == 0 ? CUDART_NAN : -CUDART_INF;
      if (lane < k) {
        a.row_keys[slot * a.key_stride + lane] = key;
        a.row_lp[slot * a.key_stride + lane] = lp;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Growing the trees
// ---------------------------------------------------------------------------------------
struct GrowArgs {
  talon_tree t;
  const int32_t *root_tok, *prefix_len;
  int32_t *prefix_copy;
  int lo_stride, B, N, W, k, key_stride, n_layers, max_depth;
  int root_topk, init_layers;
  double log_mu;
  int first;                    // round 0: start from the root
  int rows;                     // row lists of slots 0 .. rows-1 are there
  int group;                    // lanes per row in the selection: k rounded up to a power of two
  const u64 *row_keys; const double *row_lp;
  int32_t *growing, *depth_at;  // [B] out: needs more rows; layer it stopped at
  unsigned int *row_count;      // [B * N] cleared (a row pass that timed out leaves counts behind)
  int *status;
  // accepted path (best null: the target's arg-max is not there yet)
  u64 *best; unsigned int *row_bad;
  int32_t *target_tok, *accept_len, *accept_nodes, *bonus_tok;
};

constexpr int GROW_THREADS = 256;
constexpr int GROW_WARPS = GROW_THREADS / 32;

struct GrowSmem {
  u64 *key;            // [rows][k]
  double *lp;          // [rows][k]
  double *score;       // [N]
  u64 *mask;           // [N][2]
  int *tok, *parent, *depth;   // [N]
  int *off;            // [GROW_WARPS][MAX_BUDGET]  each warp's own copy of the rows' output offsets
  int *cnt;            // [MAX_BUDGET]              candidates of a row still in
};

__host__ __device__ inline size_t grow_smem_bytes(int rows, int k, int N) {
  return (size_t)rows * k * 16 + (size_t)N * (8 + 16 + 12) + GROW_WARPS * MAX_BUDGET * 4 + MAX_BUDGET * 4 + 32;
}

// Exclusive scan of cnt[0 .. F) into this warp's off[]; returns the total.
__device__ __forceinline__ int scan_rows(const int *cnt, int *off, int F, int lane) {
  int v[4], sum = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) { const int jj = lane * 4 + i; v[i] = jj < F ? cnt[jj] : 0; sum += v[i]; }
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += t;
  }
  int run = inc - sum;
  *reinterpret_cast<int4 *>(off + lane * 4) = make_int4(run, run + v[0], run + v[0] + v[1], run + v[0] + v[1] + v[2]);
  __syncwarp();
  return __shfl_sync(FULL, inc, 31);
}

// One CTA per sequence.  A layer is four short phases between barriers: the best candidate of the
// frontier (the gate's anchor), how many candidates of each row pass (they are a prefix: lists are
// sorted), the truncation by rank if more pass than the budget takes, the append.
__global__ void __launch_bounds__(GROW_THREADS)
grow_kernel(GrowArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ u64 s_head[GROW_WARPS];
  GrowSmem sm;
  {
    unsigned char *p = smem_raw;
    sm.key = reinterpret_cast<u64 *>(p);       p += sizeof(u64) * a.rows * a.k;
    sm.lp = reinterpret_cast<double *>(p);     p += sizeof(double) * a.rows * a.k;
    sm.mask = reinterpret_cast<u64 *>(p);      p += sizeof(u64) * 2 * a.N;
    sm.score = reinterpret_cast<double *>(p);  p += sizeof(double) * a.N;
    p = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(p) + 15) & ~(uintptr_t)15);
    sm.off = reinterpret_cast<int *>(p);       p += sizeof(int) * GROW_WARPS * MAX_BUDGET;
    sm.cnt = reinterpret_cast<int *>(p);       p += sizeof(int) * MAX_BUDGET;
    sm.tok = reinterpret_cast<int *>(p);       p += sizeof(int) * a.N;
    sm.parent = reinterpret_cast<int *>(p);    p += sizeof(int) * a.N;
    sm.depth = reinterpret_cast<int *>(p);
  }
  pdl_enter();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x, k = a.k, N = a.N;
  const size_t nb = (size_t)b * N;
  int *off = sm.off + warp * MAX_BUDGET;
  int d = 0, lo = 0, hi = 1;
  if (!a.first) {
    if (!a.growing[b]) return;
    d = a.depth_at[b];
    lo = a.t.layer_off[b * a.lo_stride + d];
    hi = a.t.layer_off[b * a.lo_stride + d + 1];
  }
  const int n_start = hi;                              // nodes that global memory holds already (round 0: only the root, written below)
  const int L = a.prefix_len[b], root = a.root_tok[b];
  // everything the sequence needs: row lists of the slots that can still be expanded, and the nodes' scores and masks
  for (int c = lo * k + tid; c < a.rows * k; c += GROW_THREADS) {
    const int i = c / k;
    const size_t at = (nb + i) * a.key_stride + (c - i * k);
    sm.key[c] = __ldcg(a.row_keys + at);
    sm.lp[c] = __ldcg(a.row_lp + at);
  }
  for (int i = tid; i < N; i += GROW_THREADS) a.row_count[nb + i] = 0u;
  if (a.first) {
    if (tid == 0) {
      sm.score[0] = 0.0; sm.mask[0] = 1ull; sm.mask[1] = 0ull; sm.tok[0] = root; sm.parent[0] = -1; sm.depth[0] = 0;
      a.t.layer_off[b * a.lo_stride] = 0;
      a.t.layer_off[b * a.lo_stride + 1] = 1;
      a.prefix_copy[b] = L;
    }
  } else {
    for (int i = tid; i < hi; i += GROW_THREADS) {
      sm.score[i] = a.t.score[nb + i];
      for (int w = 0; w < 2; ++w) sm.mask[2 * i + w] = w < a.W ? a.t.mask[(nb + i) * a.W + w] : 0ull;
      sm.tok[i] = a.t.token[nb + i];
      sm.parent[i] = a.t.parent[nb + i];
      sm.depth[i] = a.t.depth[nb + i];
    }
  }
  __syncthreads();

  const int G = a.group, gl = lane & (G - 1), gbase = lane & ~(G - 1);     // lanes of one row
  const unsigned gmask = (G == 32 ? FULL : ((1u << G) - 1u)) << gbase;
  const int per_pass = GROW_THREADS / G, my_row = tid / G;
  bool paused = false;
  for (; d < a.n_layers; ++d) {
    const int F = hi - lo, n = hi;
    if (F <= 0 || n >= N) break;
    if (hi > a.rows) { paused = true; break; }          // the frontier's rows are not all there yet
    const int R = N - n, ke = min(k, R);                // a parent can place at most R children
    // ---- the frontier's best candidate; rows without a softmax ----
    int bad = 0;
    u64 head = 0ull;
    if (tid < F) {
      const double lp = sm.lp[(lo + tid) * k];
      bad = lp != lp;
      const double s = sm.score[lo + tid] + lp;
      if (s > -CUDART_INF) head = f64_ord(s);
    }
    if (warp < MAX_BUDGET / 32) {
      head = warp_max_u64(head);
      if (lane == 0) s_head[warp] = head;
    }
    if (__syncthreads_or(bad)) {                        // this sequence adds nothing any more
      if (tid == 0) atomicOr(a.status, STATUS_NONFINITE);
      lo = hi;
      ++d;
      if (tid == 0) a.t.layer_off[b * a.lo_stride + d + 1] = n;
      break;
    }
    const bool init = d < a.init_layers;
    double thr = -CUDART_INF;
    const u64 anchor = umax64(umax64(s_head[0], s_head[1]), umax64(s_head[2], s_head[3]));
    if (!init && anchor != 0ull) thr = a.log_mu + f64_unord(anchor);

    // ---- eligible candidates of each row ----
    for (int j = my_row; j < per_pass * ((F + per_pass - 1) / per_pass); j += per_pass) {
      double s = -CUDART_INF;
      if (j < F && gl < ke) s = sm.score[lo + j] + sm.lp[(lo + j) * k + gl];
      const unsigned m = __ballot_sync(FULL, s > -CUDART_INF && s >= thr) & gmask;
      if (gl == 0 && j < F) sm.cnt[j] = __popc(m);
    }
    __syncthreads();
    const int want = init ? min(a.root_topk, R) : R;
    int total = scan_rows(sm.cnt, off, F, lane);
    if (total > want) {
      // ---- budget truncation: rank by (score desc, parent asc, token asc) among the eligible; rows
      // are sorted that way already, so a rank is a sum of binary searches in the rows' prefixes ----
      int keep[MAX_BUDGET / (GROW_THREADS / 32)];       // of this group's rows, one per pass (32 lanes a row at most)
      int np = 0;
      for (int j0 = 0; j0 < F; j0 += per_pass, ++np) {
        const int j = j0 + my_row;
        bool sel = false;
        if (j < F && gl < sm.cnt[j]) {
          const double s = sm.score[lo + j] + sm.lp[(lo + j) * k + gl];
          int rank = gl;
          for (int o = 0; o < F && rank < want; ++o) {
            int h = sm.cnt[o];
            if (o == j || h == 0) continue;
            const double ps = sm.score[lo + o];
            const double *lp = sm.lp + (lo + o) * k;
            const bool before = o < j;
            int l = 0;
            while (l < h) {
              const int mid = (l + h) >> 1;
              const double v = ps + lp[mid];
              if (v > s || (v == s && before)) l = mid + 1; else h = mid;
            }
            rank += l;
          }
          sel = rank < want;
        }
        const unsigned m = __ballot_sync(FULL, sel) & gmask;
        keep[np & (MAX_BUDGET / (GROW_THREADS / 32) - 1)] = __popc(m);
      }
      __syncthreads();
      np = 0;
      for (int j0 = 0; j0 < F; j0 += per_pass, ++np) {
        const int j = j0 + my_row;
        if (j < F && gl == 0) sm.cnt[j] = keep[np & (MAX_BUDGET / (GROW_THREADS / 32) - 1)];
      }
      __syncthreads();
      total = scan_rows(sm.cnt, off, F, lane);
    }

    // ---- append in storage order: (parent asc, token asc) ----
    for (int j0 = 0; j0 < F; j0 += per_pass) {
      const int j = j0 + my_row;
      const int c = j < F ? sm.cnt[j] : 0;
      const int tok = (gl < c) ? (int)key_tok(sm.key[(lo + j) * k + gl]) : 0x7FFFFFFF;
      int r = 0;
      for (int i = 0; i < G; ++i) r += __shfl_sync(FULL, tok, gbase + i) < tok ? 1 : 0;
      if (gl < c) {
        const int node = n + off[j] + r, par = lo + j;
        sm.tok[node] = tok;
        sm.parent[node] = par;
        sm.depth[node] = d + 1;
        sm.score[node] = sm.score[par] + sm.lp[par * k + gl];
        sm.mask[2 * node] = sm.mask[2 * par] | (node < 64 ? 1ull << node : 0ull);
        sm.mask[2 * node + 1] = sm.mask[2 * par + 1] | (node >= 64 ? 1ull << (node - 64) : 0ull);
      }
    }
    lo = hi;
    hi = n + total;
    if (tid == 0) a.t.layer_off[b * a.lo_stride + d + 2] = hi;
    __syncthreads();
  }

  // ---- the new nodes, and once the tree is finished what closes it (positions, sentinel slots, the
  // unused tail of the layer offsets) ----
  const int n = hi;
  if (tid == 0) {
    a.growing[b] = paused ? 1 : 0;
    a.depth_at[b] = d;
    a.t.n_nodes[b] = n;
  }
  for (int i = (a.first ? 0 : n_start) + tid; i < (paused ? n : N); i += GROW_THREADS) {
    const bool live = i < n;
    a.t.token[nb + i] = live ? sm.tok[i] : -1;
    a.t.parent[nb + i] = live ? sm.parent[i] : -1;
    a.t.depth[nb + i] = live ? sm.depth[i] : -1;
    a.t.position[nb + i] = live ? L + sm.depth[i] : -1;
    a.t.score[nb + i] = live ? sm.score[i] : -CUDART_INF;
    for (int w = 0; w < a.W; ++w)
      a.t.mask[(nb + i) * a.W + w] = live ? sm.mask[2 * i + w] : ((i >> 6) == w ? 1ull << (i & 63) : 0ull);
  }
  if (paused) return;
  for (int i = d + 2 + tid; i < a.lo_stride; i += GROW_THREADS) a.t.layer_off[b * a.lo_stride + i] = n;

  if (!a.best) return;
  // ---- greedy walk over the target's choices (Appendix B, temperature 0) ----
  int *tgt = sm.cnt;                                    // [N]
  int bad = 0;
  for (int i = tid; i < N; i += GROW_THREADS) {
    const u64 key = __ldcg(a.best + nb + i);
    a.best[nb + i] = 0ull;                              // leave the workspace clean
    const int t = (i < n && key != 0ull) ? (int)key_tok(key) : -1;
    tgt[i] = t;
    a.target_tok[nb + i] = t;
    if (a.row_bad[nb + i]) { bad |= i < n; a.row_bad[nb + i] = 0u; }
  }
  if (__syncthreads_or(bad) && tid == 0) atomicOr(a.status, STATUS_NONFINITE);
  if (warp != 0) return;
  int cur = 0, len = 0;
  int32_t *path = a.accept_nodes + (size_t)b * (a.max_depth + 1);
  if (lane == 0) path[0] = 0;
  for (int step = 0; step < a.max_depth; ++step) {
    const int want = tgt[cur];
    int found = -1;
    for (int c0 = (cur + 1) & ~31; c0 < n; c0 += 32) {   // a child comes after its parent
      const int c = c0 + lane;
      const unsigned m = __ballot_sync(FULL, c < n && sm.parent[c] == cur && sm.tok[c] == want);
      if (m) { found = c0 + __ffs(m) - 1; break; }
    }
    if (found < 0) break;
    cur = found;
    ++len;
    if (lane == 0) path[len] = cur;
  }
  for (int i = len + 1 + lane; i <= a.max_depth; i += 32) path[i] = -1;
  if (lane == 0) {
    a.accept_len[b] = len;
    a.bonus_tok[b] = tgt[cur];
  }
}

}  // namespace


static size_t row_pass_smem(const talon_ctx *c, bool scan) {
  return sizeof(float) * EXP_WARPS * XS_RING * XS_WTILE + sizeof(u64) * stage_words(c->k_cap) +
         (scan ? sizeof(int) * (MAX_BATCH + 1) : 0);
}

talon_status grow_step_setup(talon_ctx *c) {
  if (cudaFuncSetAttribute(row_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_pass_smem(c, true)) != cudaSuccess ||
      cudaFuncSetAttribute(grow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)grow_smem_bytes(c->p.budget, c->k_cap, c->p.budget)) != cudaSuccess)
    return TALON_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, row_pass_kernel, EXP_THREADS, row_pass_smem(c, false)) != cudaSuccess ||
      per_sm < 1)
    return TALON_ERR_CUDA;
  if (per_sm > EXP_CTAS_PER_SM) per_sm = EXP_CTAS_PER_SM;
  c->row_grid = c->sm_count * per_sm;
  return TALON_OK;
}

// Host-side bounds: slots that n_layers layers can expand (a full tree is not expanded, so the last
// slot never is), and slots that can hold a node afterwards.
static void step_bounds(const talon_ctx *c, int n_layers, int *expandable, int *nodes) {
  const int N = c->p.budget;
  long long f = 1, sum = 0;
  for (int d = 0; d < n_layers && sum < N; ++d) {
    sum += f;
    f = d < c->p.init_layers ? c->p.root_topk : f * c->k_cap;
    if (f > N) f = N;
  }
  *expandable = (int)(sum < N - 1 ? sum : N - 1);
  *nodes = (int)(sum + f < N ? sum + f : N);
}

talon_status launch_grow_step(talon_ctx *c, const talon_tree *t, const int32_t *root_tok, const int32_t *prefix_len,
                              const float *draft, int64_t draft_stride, int n_layers, const float *target,
                              int64_t target_stride, int32_t *target_tok, int32_t *accept_len, int32_t *accept_nodes,
                              int32_t *bonus_tok, cudaStream_t st, bool *accepted) {
  const talon_params &p = c->p;
  const int B = c->B, N = p.budget, k = c->k_cap;
  int expandable, nodes;
  step_bounds(c, n_layers, &expandable, &nodes);
  const double row_bytes = 4.0 * p.vocab * B;           // of one slot of every sequence
  const bool with_target = target && row_bytes * (expandable + nodes) <= c->step_fuse_mb * 1e6;
  *accepted = with_target;
  int rounds = 1;
  if (!with_target && row_bytes * expandable > c->step_round_mb * 1e6) {
    rounds = c->step_rounds;
    if (rounds > expandable) rounds = expandable;
  }
  RowPassArgs ra;
  ra.draft = draft; ra.draft_stride = draft_stride;
  ra.target = with_target ? target : nullptr; ra.target_stride = target_stride;
  ra.B = B; ra.N = N; ra.V = p.vocab; ra.k = k; ra.key_stride = c->key_stride; ra.max_split = c->expand_max_split;
  ra.init_layers = p.init_layers; ra.log_mu = c->log_mu;
  ra.part_keys = c->d_part_keys; ra.part_ms = c->d_part_ms; ra.row_keys = c->d_row_keys; ra.row_lp = c->d_row_score;
  ra.row_count = c->d_row_count; ra.best = c->d_argmax; ra.row_bad = c->d_row_bad; ra.status = c->d_status;
  GrowArgs ga;
  ga.t = *t; ga.root_tok = root_tok; ga.prefix_len = prefix_len; ga.prefix_copy = c->d_prefix_len;
  ga.lo_stride = p.max_depth + 2; ga.B = B; ga.N = N; ga.W = c->W; ga.k = k; ga.key_stride = c->key_stride;
  ga.n_layers = n_layers; ga.max_depth = p.max_depth; ga.root_topk = p.root_topk; ga.init_layers = p.init_layers;
  ga.log_mu = c->log_mu;
  ga.group = 1;
  while (ga.group < k) ga.group *= 2;
  ga.row_keys = c->d_row_keys; ga.row_lp = c->d_row_score; ga.growing = c->d_growing; ga.depth_at = c->d_depth_at;
  ga.row_count = c->d_row_count; ga.status = c->d_status;
  ga.best = with_target ? c->d_argmax : nullptr; ga.row_bad = c->d_row_bad;
  ga.target_tok = target_tok ? target_tok : c->d_target_tok;
  ga.accept_len = accept_len; ga.accept_nodes = accept_nodes; ga.bonus_tok = bonus_tok;

  int done = 0;
  for (int r = 0; r < rounds; ++r) {
    const int upto = (int)((long long)expandable * (r + 1) / rounds);
    ra.r0 = done; ra.r1 = upto; ra.t1 = with_target ? nodes : done;
    ra.growing = r ? c->d_growing : nullptr;
    ra.clear_status = r == 0;
    // CTAs per row: as many as the grid holds, no row cut into less than a CTA step per chunk
    const long long dr = (long long)B * (upto - done), tr = (long long)B * (ra.t1 - done);
    // (as span_geom cuts them: 4096 elements a chunk at least)
    int cut = (p.vocab + 3) / 4 * 4 / EXP_TILE;
    if (cut > c->expand_max_split) cut = c->expand_max_split;
    if (cut < 1) cut = 1;
    int grid = c->row_grid;
    if (tr == 0) {
      if (dr * cut < grid) grid = (int)(dr * cut);
      ra.draft_ctas = grid;
    } else {
      int gd = (int)(grid * dr / (dr + tr));
      const int target_cut = (p.vocab + 4 * EXP_TILE - 1) / (4 * EXP_TILE);
      if (dr * cut + tr * target_cut <= grid) {
        // small rows: the draft rows are cut as finely as a single layer's would be (the same partial
        // sums, so the same scores to the last bit), the target rows share the rest of the grid
        gd = (int)(dr * cut);
        const int most = (p.vocab + EXP_TILE - 1) / EXP_TILE, st_cut = (int)((grid - gd) / tr);
        grid = gd + (int)(tr * (st_cut < most ? st_cut : most));
      } else if (dr + tr <= grid) {        // whole chunks per row for both kinds
        const int both = (int)(grid / ((dr + tr + 1) / 2));
        int sd = (both + 1) / 2, stt = both / 2;
        if (stt < 1) stt = 1;
        if (sd > cut) sd = cut;
        gd = (int)(dr * sd);
        grid = gd + (int)(tr * stt);
      }
      ra.draft_ctas = gd;
    }
    if (grid < 1) grid = 1;
    {
      LaunchTimer lt(c, TALON_K_EXPAND_ROWS, st);
      launch_kernel(c, row_pass_kernel, dim3(grid), dim3(EXP_THREADS), row_pass_smem(c, r > 0 && B > 32), st, ra);
    }
    if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
    ga.first = r == 0; ga.rows = upto;
    {
      LaunchTimer lt(c, TALON_K_SELECT, st);
      launch_kernel_pdl(c, true, grow_kernel, dim3(B), dim3(GROW_THREADS), grow_smem_bytes(upto, k, N), st, ga);
    }
    if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
    c->launches += 2;
    done = upto;
  }
  c->layers_run = n_layers;
  return TALON_OK;
}

}  // namespace talon

// Adaptive draft-tree expansion (Algorithm 2 of the paper; Eq. 2-5) as ONE kernel per layer,
// for every per-parent candidate cap k (lists of up to 32 keys a row, the paper's K is 10, and wide ones).
//
// Streaming phase: expand_stream.cuh.  The frontier's fp32 logit rows are cut into equal chunks, one
// CTA per chunk at a time; a chunk leaves its k best keys and its share of the normaliser.
//
// Selection phase.  Frontiers of at most sixteen rows: the CTA that finishes a sequence's last chunk
// merges that sequence's rows, one warp per row.  Wider frontiers: the CTA that finishes a row's
// last chunk merges that row (rows of one sequence finish all over the grid, so the merges run in
// parallel), and the CTA that finishes the sequence's last row collects the row results.  Either
// way that CTA then scores the pooled candidates with log p(u) = log p(v) + log P(w | v)
// (Eq. 2-3), applies Top-K (Eq. 5) or the confidence gate p(u) >= mu * max p (Eq. 4), truncates
// to the remaining budget, and appends the survivors with parent links, depths, scores and
// ancestor-mask rows.  Nothing returns to the host in between.
#include <algorithm>
#include "expand_stream.cuh"

namespace talon {

namespace {

// Frontiers wider than this merge their rows all over the grid.  Up to two rows per warp the CTA that
// completes the sequence is quicker: no second hand-off, no row results to publish and collect (2 us).
// (Lists of more than 8, whose merge takes twice as long, gain a little from one row per warp where rows are long: nine layers of four
// static trees, ten rows of 128256 each, 145.7 -> 144.9 us; one tree of five layers of nine rows of 31152 loses: 90.3 -> 92.9.)
constexpr int XS_TWO_LEVEL = 2 * EXP_WARPS;

struct FusedArgs {
  const float *logits;
  int64_t row_stride;
  int rows_per_seq, layout;
  talon_tree t;
  int lo_stride;
  int B, N, W, V, d, k, key_stride, base_offset, pool_cap;
  int root_topk, init_layers;
  int prefetch_rows;       // most rows the CTAs ask L2 for before the layer before has finished (0: none)
  double log_mu;
  SpanTable spans;
  u64 *part_keys;          // [items, key_stride]  per-chunk top-k, descending
  float2 *part_ms;         // [items]              per-chunk (max, sum of exp)
  u64 *row_keys;           // [rows, key_stride]   per-row top-k (wide frontiers)
  double *row_score;       // [rows, key_stride]   log p(u) of those candidates; slot 0 NaN: row not finite
  unsigned int *row_count; // [rows]               chunks finished per row (zero between layers)
  unsigned int *seq_count; // [B]                  chunks or rows finished per sequence (zero between layers)
  int *status;
};

// Exclusive scan of the per-sequence frontier sizes: s_base[b] = first packed row of sequence
// b, s_base[B] = total rows.  A sequence whose tree is full has no rows.  The tree's size before
// this layer is layer_off[d + 1], which this launch never writes (n_nodes changes under it).
__device__ void frontier_bases(const FusedArgs &a, int *s_base, int *s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int PER = (MAX_BATCH + EXP_THREADS - 1) / EXP_THREADS;
  int f[PER];
  int sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int b = tid * PER + i;
    int v = 0;
    if (b < a.B) {
      const int lo = a.t.layer_off[b * a.lo_stride + a.d], hi = a.t.layer_off[b * a.lo_stride + a.d + 1];
      v = hi < a.N ? max(hi - lo, 0) : 0;
    }
    f[i] = v;
    sum += v;
  }
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < EXP_WARPS ? s_warp[lane] : 0;
    int winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, winc, o);
      if (lane >= o) winc += t;
    }
    if (lane < EXP_WARPS) s_warp[lane] = winc - w;
    if (lane == EXP_WARPS - 1) s_base[a.B] = winc;
  }
  __syncthreads();
  int run = s_warp[warp] + inc - sum;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int b = tid * PER + i;
    if (b < a.B) s_base[b] = run;
    run += f[i];
  }
  __syncthreads();
}

// Where a packed frontier row lives: sequence, index inside that sequence's frontier, tree
// node, frontier size and first packed row of the sequence.
struct RowLoc { int b, j, node, F, row0; };

// Frontier geometry of the layer.  For B <= 32 every warp holds it in registers (lane b = sequence
// b) and needs no shared memory or barrier; larger batches use a block-wide scan.
struct Frontier {
  int base_l, f_l, lo_l;     // B <= 32: this lane's sequence
  int total;
  bool in_regs;
  const int *s_base;
};

__device__ inline RowLoc locate_row(const FusedArgs &a, const Frontier &fr, int row) {
  RowLoc r;
  const int lane = threadIdx.x & 31;
  if (fr.in_regs) {
    // the last sequence whose first row is <= row (bases never decrease, empty sequences share
    // their base with the next one)
    const unsigned m = __ballot_sync(FULL, lane < a.B && fr.base_l <= row);
    r.b = 31 - __clz(m);
    r.row0 = __shfl_sync(FULL, fr.base_l, r.b);
    r.F = __shfl_sync(FULL, fr.f_l, r.b);
    r.j = row - r.row0;
    r.node = __shfl_sync(FULL, fr.lo_l, r.b) + r.j;
  } else {
    r.b = seq_of_row(fr.s_base, a.B, row);
    r.row0 = fr.s_base[r.b];
    r.F = fr.s_base[r.b + 1] - r.row0;
    r.j = row - r.row0;
    r.node = a.t.layer_off[r.b * a.lo_stride + a.d] + r.j;
  }
  return r;
}

// ---------------------------------------------------------------------------------------
// Selection phase
// ---------------------------------------------------------------------------------------
// Shared-memory carve-up of the selection phase (it reuses the streaming ring).
struct TailSmem {
  u64 *stage;        // [EXP_WARPS][stage_words(k)]  chunk lists of the row a warp is merging, survivors, result
  u64 *row_keys;     // [N-1][k]               per-row top-k keys, descending
  double *score;     // [N-1][k]               log p(u) of each pooled candidate
  u64 *row_mask;     // [N-1][W]               ancestor mask of the row's parent
  int *row_cnt, *row_off;   // [N-1]
  unsigned char *state;     // [N-1][k]        bit0 eligible, bit2 selected
};

// Gate, budget truncation and append for one sequence, from the pooled candidates in shared
// memory (sm.row_keys / sm.score: F rows of k, each row descending; sm.row_mask: the parents'
// mask rows).  n is the tree's size before the layer, k the pitch of the rows.
__device__ void select_and_append(const FusedArgs &a, const TailSmem &sm, int b, int lo, int F, int n, int k,
                                  u64 *s_anchor, int *s_cnt) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int R = a.N - n;
  const int ke = min(a.k, R);               // a parent can place at most R children
  const size_t nb = (size_t)b * a.N;
  const int C = F * k;

  // ---- eligibility: Top-K layers take every candidate, gated layers Eq. 4 ----
  const bool init = a.d < a.init_layers;
  double thr = -CUDART_INF;
  if (!init && *s_anchor != 0ull) thr = a.log_mu + f64_unord(*s_anchor);
  int local = 0;
  for (int c = tid; c < C; c += EXP_THREADS) {
    const double s = sm.score[c];
    unsigned char stt = (s > -CUDART_INF) ? 1 : 0;
    if (stt && !init && !(s >= thr)) stt = 0;
    sm.state[c] = stt;
    local += stt;
  }
  for (int j = tid; j < F; j += EXP_THREADS) sm.row_cnt[j] = 0;
#pragma unroll
  for (int o = 16; o; o >>= 1) local += __shfl_xor_sync(FULL, local, o);
  if (lane == 0 && local) atomicAdd(s_cnt, local);
  __syncthreads();
  const int eligible = *s_cnt;
  const int want = init ? min(a.root_topk, R) : R;
  const int n_sel = min(eligible, want);

  // ---- budget truncation: rank among all candidates by (score desc, parent asc, token asc).
  // Every row is sorted that way already, so a rank is a sum of binary searches. ----
  for (int c = tid; c < C; c += EXP_THREADS) {
    if (!sm.state[c]) continue;
    bool sel = true;
    if (eligible > want) {
      const int j = c / k, i = c - j * k;
      const double s = sm.score[c];
      int rank = i;
      for (int o = 0; o < F && rank < want; ++o) {
        if (o == j) continue;
        const double *sc = sm.score + o * k;
        const bool before = o < j;
        int l = 0, h = ke;
        while (l < h) {
          const int mid = (l + h) >> 1;
          const double v = sc[mid];
          if (v > s || (v == s && before)) l = mid + 1; else h = mid;
        }
        rank += l;
      }
      sel = rank < want;
    }
    if (sel) {
      sm.state[c] = 5;
      atomicAdd(&sm.row_cnt[c / k], 1);
    }
  }
  __syncthreads();

  // ---- append in storage order: (parent asc, token asc) ----
  if (warp == 0) {
    int v[4], sum = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) { const int jj = lane * 4 + i; v[i] = jj < F ? sm.row_cnt[jj] : 0; sum += v[i]; }
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    int run = inc - sum;
#pragma unroll
    for (int i = 0; i < 4; ++i) { const int jj = lane * 4 + i; if (jj < F) sm.row_off[jj] = run; run += v[i]; }
  }
  __syncthreads();
  for (int c = tid; c < C; c += EXP_THREADS) {
    if (!(sm.state[c] & 4)) continue;
    const int j = c / k;
    const int tok = (int)key_tok(sm.row_keys[c]);
    int r = 0;
#pragma unroll 4
    for (int i = 0; i < ke; ++i) {
      const int o = j * k + i;
      r += ((sm.state[o] & 4) && (int)key_tok(sm.row_keys[o]) < tok) ? 1 : 0;
    }
    const int node = n + sm.row_off[j] + r;
    a.t.token[nb + node] = tok;
    a.t.parent[nb + node] = lo + j;
    a.t.depth[nb + node] = a.d + 1;
    a.t.score[nb + node] = sm.score[c];
    for (int w = 0; w < a.W; ++w) {
      u64 m = sm.row_mask[j * a.W + w];
      if ((node >> 6) == w) m |= 1ull << (node & 63);
      a.t.mask[(nb + node) * a.W + w] = m;
    }
  }
  if (tid == 0) {
    a.t.n_nodes[b] = n + n_sel;
    a.t.layer_off[b * a.lo_stride + a.d + 2] = n + n_sel;
  }
}

// While the layer before is still merging and selecting, DRAM idles: one warp asks for the logit rows this layer
// will most likely read.  Only a hint to L2, so it may run before the wait, on sizes that are not final and rows
// that are still being written (L2 is where those writes arrive too); whatever it reads is clamped to the caller's rows.
// Four sequences of ten rows of 128256: a layer's data is there 3.8 us after the wait, 4.8 without (234 -> 227 us a step).
__device__ void prefetch_rows(const FusedArgs &a) {
  const int lane = threadIdx.x & 31;
  int lo = 0, f = 0;
  if (lane < a.B) {
    const int *off = a.t.layer_off + lane * a.lo_stride + a.d;
    f = a.d == 0 ? 1 : a.root_topk;
    if (a.d >= 2 && a.d >= a.init_layers) f = __ldcg(off) - __ldcg(off - 1);       // as many as the layer before had
    if (a.layout == TALON_ROWS_BY_NODE && a.d > 0) lo = min(max(__ldcg(off), 0), a.rows_per_seq);
    f = min(max(f, 0), a.rows_per_seq - lo);
  }
  int inc = f;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += t;
  }
  const int total = min(__shfl_sync(FULL, inc, 31), a.prefetch_rows);
  if (total <= 0) return;
  const int per_row = max(1, (int)gridDim.x / total), step = max(1, (int)gridDim.x / per_row);
  const int piece = ((a.V + per_row - 1) / per_row + 3) & ~3;
  const int start = (int)(blockIdx.x % per_row) * piece, n = min(piece, a.V - start);
  for (int row = blockIdx.x / per_row; row < total; row += step) {
    const int b = __ffs(__ballot_sync(FULL, inc > row)) - 1;
    const int j = row - __shfl_sync(FULL, inc - f, b), base = __shfl_sync(FULL, lo, b);
    if (lane == 0 && n > 0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                   ::"l"(a.logits + ((int64_t)b * a.rows_per_seq + base + j) * a.row_stride + start), "r"((n * 4 + 15) & ~15) : "memory");
  }
}

// WIDE: k above 32 (see expand_stream.cuh); a row is then merged by the whole CTA that completes it,
// whatever the width of the frontier.
template <int KMAX>          // k rounded up to 8, 16, 32 or 128 (WIDE)
__global__ void __launch_bounds__(EXP_THREADS, KMAX > 32 ? 2 : 3)
expand_fused_kernel(FusedArgs a) {
  constexpr bool WIDE = KMAX > 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ u64 s_buf[EXP_WARPS][ListSize<WIDE>::BUF];          // per-warp buffers of keys that reached the threshold
  __shared__ u64 s_pool[ListSize<WIDE>::POOL];                   // the chunk's candidates, all warps
  __shared__ int s_warp[EXP_WARPS];
  __shared__ float s_m[EXP_WARPS], s_s[EXP_WARPS];
  __shared__ __align__(8) u64 s_bar[EXP_WARPS][XS_RING];   // "tile landed" barriers, per warp
  __shared__ float s_wtop[EXP_WARPS];               // each warp's ceil(k/8)-th largest lane maximum
  __shared__ float s_wmax[EXP_WARPS];               // each warp's largest
  __shared__ u64 s_anchor;
  __shared__ int s_pool_n, s_last, s_last_seq, s_ecnt, s_bad, s_abort;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = a.k;
  if (lane == 0) {
    for (int i = 0; i < XS_RING; ++i) ring_bar_init(smem_addr(&s_bar[warp][i]));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_wtop[warp] = -CUDART_INF_F;
    s_wmax[warp] = -CUDART_INF_F;
  }
  if (tid == 0) {
    s_pool_n = 0; s_abort = 0;
    s_anchor = 0ull; s_ecnt = 0; s_bad = 0;
  }
  __syncthreads();                 // (here, not on the way from the previous layer to the first byte)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (a.prefetch_rows > 0 && warp == EXP_WARPS - 1) prefetch_rows(a);
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // ---- frontier geometry (from layer_off[d], layer_off[d + 1]: never written by this launch) ----
  Frontier fr;
  fr.in_regs = a.B <= 32;
  // batches above 32 keep their frontier bases behind the ring (the launch adds the room)
  int *s_base = reinterpret_cast<int *>(smem_raw + a.base_offset);
  fr.s_base = s_base;
  fr.base_l = fr.f_l = fr.lo_l = 0;
  if (fr.in_regs) {
    if (lane < a.B) {
      fr.lo_l = a.t.layer_off[lane * a.lo_stride + a.d];
      const int hi = a.t.layer_off[lane * a.lo_stride + a.d + 1];
      fr.f_l = hi < a.N ? max(hi - fr.lo_l, 0) : 0;
      if (fr.f_l == 0 && blockIdx.x == 0 && warp == 0)        // nothing to expand: close the layer
        a.t.layer_off[lane * a.lo_stride + a.d + 2] = hi;
    }
    int inc = fr.f_l;
#pragma unroll
    for (int o = 1; o < a.B; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    fr.base_l = inc - fr.f_l;
    fr.total = __shfl_sync(FULL, inc, a.B - 1);
  } else {
    frontier_bases(a, s_base, s_warp);
    fr.total = s_base[a.B];
    if (blockIdx.x == 0)
      for (int b = tid; b < a.B; b += EXP_THREADS)
        if (s_base[b + 1] == s_base[b])
          a.t.layer_off[b * a.lo_stride + a.d + 2] = a.t.layer_off[b * a.lo_stride + a.d + 1];
  }
  const SpanGeom g = span_geom(fr.total, a.V, (int)gridDim.x, a.spans);
  const unsigned long long line_end = (unsigned long long)fr.total * g.pitch;
  const bool gated = a.d >= a.init_layers;
  const float ln_mu = (float)a.log_mu;
  unsigned wt = 0;                 // tiles this warp has taken from its ring so far
  const ChunkShared sh = {reinterpret_cast<float *>(smem_raw) + warp * (XS_RING * XS_WTILE), s_bar[warp], s_buf[warp], s_pool,
                          s_m, s_s, s_wtop, s_wmax, &s_pool_n, &s_abort};
  const ChunkOut res = {a.part_keys, a.part_ms, a.key_stride, a.status};

  unsigned long long pos = (unsigned long long)blockIdx.x * g.span;
  const unsigned long long span_end = min(line_end, pos + g.span);
  int row = pos < span_end ? (g.per_row ? (int)div_small(blockIdx.x, g.per_row) : (int)div_u64(pos, g.pitch)) : 0;
  int start = pos < span_end ? (int)(pos - (unsigned long long)row * g.pitch) : 0;
  for (; pos < span_end; ++row, start = 0) {
    // ---- one chunk: elements [start, start + len) of packed row `row` ----
    const int len = (int)min((unsigned long long)(g.pitch - (unsigned)start), span_end - pos);
    pos += (unsigned)len;
    const int item = (int)blockIdx.x + row;
    const RowLoc rl = locate_row(a, fr, row);
    int rsel = (a.layout == TALON_ROWS_BY_NODE) ? rl.node : rl.j;
    if (rsel >= a.rows_per_seq) {               // caller reserved too few rows: stay in bounds, report
      rsel = a.rows_per_seq - 1;
      if (tid == 0) atomicOr(a.status, STATUS_CAPACITY);
    }
    const float *rowp = a.logits + ((int64_t)rl.b * a.rows_per_seq + rsel) * a.row_stride;
    const int end = min(a.V, start + len);        // (an empty chunk past the row's end still reports in)
    const int lo = rl.node - rl.j;               // first frontier node of the sequence
    const int n_before = lo + rl.F;              // the tree's size before this layer
    const int ke = min(k, a.N - n_before);       // a parent can place at most N - |T| children
    if (!stream_chunk<WIDE>(sh, rowp, start, end, k, ke, gated, ln_mu, (size_t)item, res, wt)) return;

    // ---- hand-off.  The barrier orders this CTA's writes before thread 0's device-scope
    // release; the last arrival acquires.  Narrow frontiers count chunks per sequence, wide ones
    // chunks per row and then rows per sequence. ----
    const bool two_level = WIDE || rl.F > XS_TWO_LEVEL;
    __syncthreads();
    chunk_clear(sh);
    if (tid == 0) {
      if (two_level && (unsigned)len == g.pitch) {
        s_last = 1;                                               // the row's only chunk
      } else {
        // the counters add up elements of the line: a row is done at pitch, a narrow frontier at F * pitch
        cuda::atomic_ref<unsigned int, cuda::thread_scope_device> c(two_level ? a.row_count[row] : a.seq_count[rl.b]);
        const unsigned target = two_level ? g.pitch : (unsigned)rl.F * g.pitch;
        const unsigned prev = c.fetch_add((unsigned)len, cuda::memory_order_acq_rel);
        s_last = (prev + (unsigned)len == target);
        if (s_last) c.store(0u, cuda::memory_order_relaxed);      // ready for the next layer
      }
    }
    __syncthreads();
    if (!s_last) continue;

    TailSmem sm;
    const int rows_max = a.N - 1;
    // pitch of the pooled rows; WIDE rows are packed at the ke children a parent can still place, which
    // bounds the pool by rows x remaining budget
    const int kp = WIDE ? ke : k;
    // (the others lie candidate by candidate, a row per lane)
    const int pitch = rows_max | 1;
    const int pool_cap = WIDE ? a.pool_cap : pitch * k;
    {
      unsigned char *p = smem_raw;
      sm.stage = reinterpret_cast<u64 *>(p);            p += WIDE ? 0 : sizeof(u64) * EXP_WARPS * stage_words(k);
      sm.row_keys = reinterpret_cast<u64 *>(p);         p += sizeof(u64) * pool_cap;
      sm.score = reinterpret_cast<double *>(p);         p += sizeof(double) * pool_cap;
      sm.row_mask = reinterpret_cast<u64 *>(p);         p += sizeof(u64) * rows_max * a.W;
      sm.row_cnt = reinterpret_cast<int *>(p);          p += sizeof(int) * rows_max;
      sm.row_off = reinterpret_cast<int *>(p);          p += sizeof(int) * rows_max;
      sm.state = p;
    }
    const size_t nb = (size_t)rl.b * a.N;
    if (two_level) {
      // ---- this CTA finished a row of a wide frontier: one warp merges it, publishes the result
      // and counts the row; the CTA that counts the sequence's last row goes on ----
      if (WIDE) {
        int item0, S;
        row_chunks(g, row, item0, S);
        merge_row_wide(res, (size_t)item0, S, k, ke, a.t.score[nb + rl.node], reinterpret_cast<u64 *>(smem_raw),
                       a.row_keys + (size_t)row * a.key_stride, a.row_score + (size_t)row * a.key_stride, a.status);
        __syncthreads();
      }
      if (warp == 0) {
        if (!WIDE) {
          u64 key; double sc;
          int item0, S;
          row_chunks(g, row, item0, S);
          const double ps = a.t.score[nb + rl.node];
          const bool finite = merge_row<KMAX>(res, (size_t)item0, S, k, ke, ps, sm.stage, key, sc);
          if (!finite) {
            sc = lane == 0 ? CUDART_NAN : -CUDART_INF;
            if (lane == 0) atomicOr(a.status, STATUS_NONFINITE);
          }
          if (lane < k) {
            a.row_keys[(size_t)row * a.key_stride + lane] = key;
            a.row_score[(size_t)row * a.key_stride + lane] = sc;
          }
        }
        __syncwarp();
        if (lane == 0) {
          cuda::atomic_ref<unsigned int, cuda::thread_scope_device> c(a.seq_count[rl.b]);
          const unsigned prev = c.fetch_add(1u, cuda::memory_order_acq_rel);
          s_last_seq = (prev == (unsigned)rl.F - 1u);
          if (s_last_seq) c.store(0u, cuda::memory_order_relaxed);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // the merge wrote where copies will land
      __syncthreads();
      if (!s_last_seq) continue;
      // ---- collect the sequence's row results and the parents' mask rows: four loads per thread
      // go to registers before the first store, so that they share one trip to L2 ----
      const int C = rl.F * kp;
      for (int c0 = 0; c0 < C; c0 += 4 * EXP_THREADS) {
        u64 key[4]; double sc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = c0 + u * EXP_THREADS + tid;
          const int j = c / kp, i = c - j * kp;
          key[u] = c < C ? __ldcg(a.row_keys + (size_t)(rl.row0 + j) * a.key_stride + i) : 0ull;
          sc[u] = c < C ? __ldcg(a.row_score + (size_t)(rl.row0 + j) * a.key_stride + i) : -CUDART_INF;
        }
        const int mi = c0 / 4 + tid;                 // the mask words ride along, EXP_THREADS per round
        const u64 mword = mi < rl.F * a.W ? a.t.mask[(nb + lo) * a.W + mi] : 0ull;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = c0 + u * EXP_THREADS + tid;
          if (c >= C) continue;
          const int at = WIDE ? c : (c % kp) * pitch + c / kp;
          sm.row_keys[at] = key[u];
          if (sc[u] != sc[u]) { s_bad = 1; sm.score[at] = -CUDART_INF; }
          else {
            sm.score[at] = sc[u];
            // rows are sorted: heads carry the maxima
            if (WIDE && c % kp == 0 && sc[u] > -CUDART_INF) atomicMax(&s_anchor, f64_ord(sc[u]));
          }
        }
        if (mi < rl.F * a.W) sm.row_mask[mi] = mword;
      }
      for (int mi = (C + 4 * EXP_THREADS - 1) / (4 * EXP_THREADS) * EXP_THREADS + tid; mi < rl.F * a.W; mi += EXP_THREADS)
        sm.row_mask[mi] = a.t.mask[(nb + lo) * a.W + mi];
    } else if (!WIDE) {
      // ---- this CTA finished the sequence: one warp per row ----
      for (int j = warp; j < rl.F; j += EXP_WARPS) {
        u64 key; double sc;
        int item0, S;
        row_chunks(g, rl.row0 + j, item0, S);
        const double ps = a.t.score[nb + lo + j];
        const u64 pmask = lane < a.W ? a.t.mask[(nb + lo + j) * a.W + lane] : 0ull;     // the parent's ancestor-mask row
        const bool finite = merge_row<KMAX>(res, (size_t)item0, S, k, ke, ps, sm.stage + warp * stage_words(k), key, sc);
        if (!finite && lane == 0) { s_bad = 1; atomicOr(a.status, STATUS_NONFINITE); }
        if (lane < k) {
          sm.row_keys[lane * pitch + j] = key;
          sm.score[lane * pitch + j] = sc;
        }
        if (lane < a.W) sm.row_mask[j * a.W + lane] = pmask;
      }
    }
    __syncthreads();
    if (s_bad) {             // a frontier row was not finite: this sequence adds nothing
      if (tid == 0) a.t.layer_off[rl.b * a.lo_stride + a.d + 2] = n_before;
    } else {
      if (WIDE) {
        select_and_append(a, sm, rl.b, lo, rl.F, n_before, kp, &s_anchor, &s_ecnt);
      } else {
        auto append = [&](int slot, int j, int, int tok, double score) {
          const int node = n_before + slot;
          a.t.token[nb + node] = tok;
          a.t.parent[nb + node] = lo + j;
          a.t.depth[nb + node] = a.d + 1;
          a.t.score[nb + node] = score;
          for (int w = 0; w < a.W; ++w) {
            u64 m = sm.row_mask[j * a.W + w];
            if ((node >> 6) == w) m |= 1ull << (node & 63);
            a.t.mask[(nb + node) * a.W + w] = m;
          }
        };
        auto score = [&](int j, int i) { return sm.score[i * pitch + j]; };
        auto tok = [&](int j, int i) { return (int)key_tok(sm.row_keys[i * pitch + j]); };
        const bool init = !gated;
        const int R = a.N - n_before, want = init ? min(a.root_topk, R) : R;
        constexpr int KN = WIDE ? 32 : KMAX;
        const int total = rl.F <= 32 ? layer_select<1, KN, EXP_THREADS>(rl.F, k, ke, want, init, a.log_mu, sm.row_cnt, score, tok, append)
                                     : layer_select<4, KN, EXP_THREADS>(rl.F, k, ke, want, init, a.log_mu, sm.row_cnt, score, tok, append);
        if (tid == 0) {
          a.t.n_nodes[rl.b] = n_before + total;
          a.t.layer_off[rl.b * a.lo_stride + a.d + 2] = n_before + total;
        }
      }
    }
    // the next chunk's bulk copies land in the memory the selection phase just used
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) { s_anchor = 0ull; s_ecnt = 0; s_bad = 0; }
  }
}

// Largest pool of a layer: F rows of min(k, N - 1 - F) candidates (the tree holds F + 1 nodes at least;
// the root's layer: one row of up to N - 1).
int pool_capacity(const talon_ctx *c) {
  int best = 1;
  for (int f = 1; f <= c->p.budget - 1; ++f) {
    const int r = f == 1 ? c->p.budget - 1 : c->p.budget - 1 - f;
    const int ke = c->k_cap < r ? c->k_cap : r;
    if (f * ke > best) best = f * ke;
  }
  return best;
}

size_t fused_smem_bytes(const talon_ctx *c) {
  const size_t rows = c->p.budget - 1, k = c->k_cap, W = c->W;
  const bool wide = c->k_cap > 32;
  const size_t pool = wide ? pool_capacity(c) : (rows | 1) * k;
  const size_t tail = (wide ? 0 : sizeof(u64) * EXP_WARPS * stage_words(k)) + pool * (8 + 8 + 1) + rows * (8 * W + 4 + 4) + 16;
  size_t bytes = sizeof(float) * EXP_WARPS * XS_RING * XS_WTILE;            // the two phases share the space
  if (bytes < tail) bytes = tail;
  if (wide && bytes < sizeof(u64) * WIDE_STAGE_WORDS) bytes = sizeof(u64) * WIDE_STAGE_WORDS;
  return (bytes + 15) & ~(size_t)15;
}

// batches above 32 sequences keep the frontier bases in dynamic shared memory behind that
size_t fused_base_bytes(int B) { return B > 32 ? sizeof(int) * (MAX_BATCH + 1) : 0; }

void (*fused_kernel_for(const talon_ctx *c))(FusedArgs) {
  return c->k_cap <= 8 ? expand_fused_kernel<8>
                       : (c->k_cap <= 16 ? expand_fused_kernel<16> : (c->k_cap <= 32 ? expand_fused_kernel<32> : expand_fused_kernel<128>));
}

}  // namespace

talon_status expand_fused_setup(talon_ctx *c) {
  const size_t bytes = fused_smem_bytes(c);
  if (!allow_shared_memory(c, fused_kernel_for(c))) return TALON_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fused_kernel_for(c), EXP_THREADS, bytes) !=
      cudaSuccess || per_sm < 1)
    return TALON_ERR_CUDA;
  if (per_sm > EXP_CTAS_PER_SM) per_sm = EXP_CTAS_PER_SM;
  c->fused_grid = c->sm_count * per_sm;
  return TALON_OK;
}

talon_status launch_expand_fused(talon_ctx *c, const talon_tree *t, const float *logits, int64_t row_stride,
                                 int rows_per_seq, int layout, int rows_bound, cudaStream_t st) {
  FusedArgs a;
  a.logits = logits; a.row_stride = row_stride; a.rows_per_seq = rows_per_seq; a.layout = layout;
  a.t = *t; a.lo_stride = c->p.max_depth + 2;
  a.B = c->B; a.N = c->p.budget; a.W = c->W; a.V = c->p.vocab; a.d = c->layers_run; a.k = c->k_cap;
  a.key_stride = c->key_stride;
  a.pool_cap = pool_capacity(c);
  a.spans = span_table(c->p.vocab, c->k_cap, c->expand_max_split);
  long long max_items = (long long)rows_bound * FX_MAX_SPLITS;
  int grid = c->fused_grid;
  if (max_items < grid) grid = (int)max_items;
  if (grid < 1) grid = 1;
  // Below 4.5 MB (0.7 us of DRAM) a layer's rows land as fast as they are asked for, and the hint costs a trip to
  // the tree; more than 8 MB does not arrive before the wait ends (24 and 48 MB: no better, 229 us).
  const long long row_bytes = 4ll * a.V, likely = (a.d == 0 ? 1ll : c->p.root_topk) * a.B * row_bytes;
  a.prefetch_rows = a.B <= 32 && likely >= 4500000 ? (int)std::max(1ll, 8000000 / row_bytes) : 0;
  a.root_topk = c->p.root_topk; a.init_layers = c->p.init_layers; a.log_mu = c->log_mu;
  a.part_keys = c->d_part_keys; a.part_ms = c->d_part_ms; a.row_keys = c->d_row_keys; a.row_score = c->d_row_score;
  a.row_count = c->d_row_count; a.seq_count = c->d_seq_count; a.status = c->d_status;
  {
    LaunchTimer lt(c, TALON_K_EXPAND_ROWS, st);
    a.base_offset = (int)fused_smem_bytes(c);
    launch_kernel_pdl(c, true, fused_kernel_for(c), dim3(grid), dim3(EXP_THREADS), fused_smem_bytes(c) + fused_base_bytes(c->B), st, a);
  }
  if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
  c->launches += 1;
  return TALON_OK;
}

}  // namespace talon

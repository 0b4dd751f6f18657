// Tree attention (verification forward of Appendix B) -- warp-MMA implementation.
//
// For sequence b and kv head h the g = Hq/Hkv query heads of all N tree nodes are packed
// into one [g*N, 128] query matrix (row r = node * g + head-in-group), so each K/V tile is
// read once for the whole group.  The key axis (L_b prefix keys followed by the N tree keys)
// is cut into 64-key tiles and the tiles are divided over `splits` CTAs (split-KV); every
// CTA keeps a running (max, sum, O) per query row and a second kernel merges the splits
// with the log-sum-exp rule.  Prefix keys are visible to every node; a tree key j is visible
// to node i iff bit j of the node's ancestor-mask row is set.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>

#include "talon_internal.cuh"

namespace talon {

constexpr int AT_THREADS = 256;
constexpr int AT_BM = 128;     // packed query rows per CTA (16 per warp)
constexpr int AT_BN = 64;      // keys per tile
constexpr int AT_D = 128;      // head dimension
constexpr int AT_TILE_BYTES = AT_BN * AT_D * 2;
constexpr int AT_SMEM = AT_BM * AT_D * 2 + 4 * AT_TILE_BYTES;   // Q + 2 stages of (K, V)

struct AttnArgs {
  const __nv_bfloat16 *q, *kp, *vp, *kt, *vt;
  const int64_t *kv_start;
  int64_t stride_t, stride_h;
  const int32_t *prefix_len, *n_nodes;
  const unsigned long long *mask;
  int B, N, W, Hq, Hkv, g;
  int npt;                    // combine kernel: nodes per query tile of the partials (0: rows packed without gaps)
  float scale_log2;
  int splits, m_blocks;
  __nv_bfloat16 *out;
  float *part_o;
  float2 *part_ml;
};

__device__ inline void cp_async16(void *smem, const void *gmem, bool pred) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  const int sz = pred ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(sz));
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ inline void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ inline void ldsm_x4(unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3, const void *p) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(s));
}
__device__ inline void ldsm_x4_t(unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3, const void *p) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(s));
}
__device__ inline void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ inline unsigned pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned *>(&v);
}
// byte offset of 16-byte chunk c of row r in a [rows][128] bf16 tile, XOR-swizzled
__device__ inline int swz(int r, int c) { return r * 256 + ((c ^ (r & 7)) << 4); }

// copy a [64 keys][128] tile: key t0+row of a source with `nvalid` keys, `stride` elements apart
__device__ inline void load_kv_tile(unsigned char *dst, const __nv_bfloat16 *src, int64_t stride, int t0,
                                    int nvalid, int tid) {
#pragma unroll
  for (int i = 0; i < (AT_BN * 16) / AT_THREADS; ++i) {
    const int id = tid + i * AT_THREADS;
    const int row = id >> 4, c = id & 15;
    const bool ok = (t0 + row) < nvalid;
    const __nv_bfloat16 *g = ok ? src + (int64_t)(t0 + row) * stride + c * 8 : src;
    cp_async16(dst + swz(row, c), g, ok);
  }
}

__global__ void __launch_bounds__(AT_THREADS, 1)
tree_attention_mma_kernel(AttnArgs a) {
  pdl_enter();
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char *s_q = smem;
  unsigned char *s_kv = smem + AT_BM * AT_D * 2;     // stage s: K at s*2*TILE, V at (s*2+1)*TILE

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int mblk = blockIdx.x, split = blockIdx.y;
  const int bh = blockIdx.z, b = bh / a.Hkv, kvh = bh - b * a.Hkv;
  const int n = a.n_nodes[b];
  const int L = a.prefix_len[b];
  const int rows_valid = a.g * n;                // packed rows that hold real nodes
  const int rows_total = a.g * a.N;

  // ---- Q tile -> shared -> A fragments ----
#pragma unroll
  for (int i = 0; i < (AT_BM * 16) / AT_THREADS; ++i) {
    const int id = tid + i * AT_THREADS;
    const int rl = id >> 4, c = id & 15;
    const int r = mblk * AT_BM + rl;
    const bool ok = r < rows_valid;
    const int node = ok ? r / a.g : 0, qh = ok ? r - node * a.g : 0;
    const __nv_bfloat16 *gp = a.q + (((int64_t)b * a.N + node) * a.Hq + kvh * a.g + qh) * AT_D + c * 8;
    cp_async16(s_q + swz(rl, c), gp, ok);
  }
  cp_async_commit();

  const int nP = (L + AT_BN - 1) / AT_BN;
  const int nT = (a.N + AT_BN - 1) / AT_BN;
  const int tt = nP + nT;
  const int tps = (tt + a.splits - 1) / a.splits;
  const int t_begin = split * tps;
  const int t_end = min(tt, t_begin + tps);

  const __nv_bfloat16 *kp = a.kp + a.kv_start[b] * a.stride_t + (int64_t)kvh * a.stride_h;
  const __nv_bfloat16 *vp = a.vp + a.kv_start[b] * a.stride_t + (int64_t)kvh * a.stride_h;
  const int64_t tree_stride = (int64_t)a.Hkv * AT_D;
  const __nv_bfloat16 *kt = a.kt + ((int64_t)b * a.N * a.Hkv + kvh) * AT_D;
  const __nv_bfloat16 *vt = a.vt + ((int64_t)b * a.N * a.Hkv + kvh) * AT_D;

  auto issue_tile = [&](int tg, int stage) {
    unsigned char *ks = s_kv + (stage * 2) * AT_TILE_BYTES;
    unsigned char *vs = ks + AT_TILE_BYTES;
    if (tg < nP) {
      load_kv_tile(ks, kp, a.stride_t, tg * AT_BN, L, tid);
      load_kv_tile(vs, vp, a.stride_t, tg * AT_BN, L, tid);
    } else {
      load_kv_tile(ks, kt, tree_stride, (tg - nP) * AT_BN, a.N, tid);
      load_kv_tile(vs, vt, tree_stride, (tg - nP) * AT_BN, a.N, tid);
    }
  };
  if (t_begin < t_end) issue_tile(t_begin, 0);
  cp_async_commit();

  cp_async_wait<1>();      // Q has landed
  __syncthreads();
  unsigned qf[8][4];
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
    ldsm_x4(qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3],
            s_q + swz(warp * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), kk * 2 + (lane >> 4)));

  // rows owned by this thread: r0 and r0 + 8
  const int r0 = mblk * AT_BM + warp * 16 + (lane >> 2);
  unsigned long long mrow[2][2] = {{0ull, 0ull}, {0ull, 0ull}};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = r0 + h * 8;
    if (r < rows_valid) {
      const int node = r / a.g;
      for (int w = 0; w < a.W; ++w) mrow[h][w] = a.mask[((int64_t)b * a.N + node) * a.W + w];
    }
  }

  float oacc[16][4];
#pragma unroll
  for (int i = 0; i < 16; ++i) { oacc[i][0] = oacc[i][1] = oacc[i][2] = oacc[i][3] = 0.f; }
  float m_i[2] = {-CUDART_INF_F, -CUDART_INF_F}, l_i[2] = {0.f, 0.f};

  int it = 0;
  for (int tg = t_begin; tg < t_end; ++tg, ++it) {
    const int stage = it & 1;
    if (tg + 1 < t_end) {
      issue_tile(tg + 1, stage ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const unsigned char *ks = s_kv + (stage * 2) * AT_TILE_BYTES;
    const unsigned char *vs = ks + AT_TILE_BYTES;

    float sacc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) { sacc[i][0] = sacc[i][1] = sacc[i][2] = sacc[i][3] = 0.f; }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
#pragma unroll
      for (int nj = 0; nj < 4; ++nj) {
        unsigned b0, b1, b2, b3;
        ldsm_x4(b0, b1, b2, b3, ks + swz(nj * 16 + (lane >> 4) * 8 + (lane & 7), kk * 2 + ((lane >> 3) & 1)));
        mma_bf16(sacc[2 * nj], qf[kk], b0, b1);
        mma_bf16(sacc[2 * nj + 1], qf[kk], b2, b3);
      }
    }

    // ---- scale, mask, online softmax (base-2 exponent domain) ----
    const bool tree_tile = tg >= nP;
    const int key0 = tree_tile ? (tg - nP) * AT_BN : tg * AT_BN;
    float rmax[2] = {-CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int h = c >> 1;
        const int key = key0 + nt * 8 + (lane & 3) * 2 + (c & 1);
        bool vis;
        if (tree_tile) vis = key < a.N && ((mrow[h][key >> 6] >> (key & 63)) & 1ull);
        else vis = key < L;
        const float x = vis ? sacc[nt][c] * a.scale_log2 : -CUDART_INF_F;
        sacc[nt][c] = x;
        rmax[h] = fmaxf(rmax[h], x);
      }
    }
    float alpha[2], muse[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xFFFFFFFFu, rmax[h], 1));
      rmax[h] = fmaxf(rmax[h], __shfl_xor_sync(0xFFFFFFFFu, rmax[h], 2));
      const float mnew = fmaxf(m_i[h], rmax[h]);
      muse[h] = (mnew == -CUDART_INF_F) ? 0.f : mnew;
      alpha[h] = exp2f(m_i[h] - muse[h]);
      m_i[h] = mnew;
    }
    float rsum[2] = {0.f, 0.f};
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int h = c >> 1;
        const float p = exp2f(sacc[nt][c] - muse[h]);
        sacc[nt][c] = p;
        rsum[h] += p;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) l_i[h] = l_i[h] * alpha[h] + rsum[h];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      oacc[i][0] *= alpha[0]; oacc[i][1] *= alpha[0];
      oacc[i][2] *= alpha[1]; oacc[i][3] *= alpha[1];
    }

    // ---- O += P V ----
#pragma unroll
    for (int kk2 = 0; kk2 < 4; ++kk2) {
      unsigned pa[4];
      pa[0] = pack_bf16(sacc[2 * kk2][0], sacc[2 * kk2][1]);
      pa[1] = pack_bf16(sacc[2 * kk2][2], sacc[2 * kk2][3]);
      pa[2] = pack_bf16(sacc[2 * kk2 + 1][0], sacc[2 * kk2 + 1][1]);
      pa[3] = pack_bf16(sacc[2 * kk2 + 1][2], sacc[2 * kk2 + 1][3]);
#pragma unroll
      for (int dj = 0; dj < 8; ++dj) {
        unsigned b0, b1, b2, b3;
        ldsm_x4_t(b0, b1, b2, b3, vs + swz(kk2 * 16 + ((lane >> 3) & 1) * 8 + (lane & 7), dj * 2 + (lane >> 4)));
        mma_bf16(oacc[2 * dj], pa, b0, b1);
        mma_bf16(oacc[2 * dj + 1], pa, b2, b3);
      }
    }
    __syncthreads();
  }
  cp_async_wait<0>();

#pragma unroll
  for (int h = 0; h < 2; ++h) {
    l_i[h] += __shfl_xor_sync(0xFFFFFFFFu, l_i[h], 1);
    l_i[h] += __shfl_xor_sync(0xFFFFFFFFu, l_i[h], 2);
  }

  if (a.splits == 1) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = r0 + h * 8;
      if (r >= rows_total) continue;
      const int node = r / a.g, qh = r - node * a.g;
      const bool live = r < rows_valid && l_i[h] > 0.f;
      const float inv = live ? 1.f / l_i[h] : 0.f;
      __nv_bfloat16 *op = a.out + (((int64_t)b * a.N + node) * a.Hq + kvh * a.g + qh) * AT_D + (lane & 3) * 2;
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) {
        const __nv_bfloat162 v = __floats2bfloat162_rn(oacc[nt][2 * h] * inv, oacc[nt][2 * h + 1] * inv);
        *reinterpret_cast<__nv_bfloat162 *>(op + nt * 8) = v;
      }
    }
  } else {
    const int mpad = a.m_blocks * AT_BM;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = r0 + h * 8;
      const int64_t prow = ((int64_t)bh * a.splits + split) * mpad + r;
      float *op = a.part_o + prow * AT_D + (lane & 3) * 2;
#pragma unroll
      for (int nt = 0; nt < 16; ++nt)
        *reinterpret_cast<float2 *>(op + nt * 8) = make_float2(oacc[nt][2 * h], oacc[nt][2 * h + 1]);
      if ((lane & 3) == 0) a.part_ml[prow] = make_float2(m_i[h], l_i[h]);
    }
  }
}

// merge the split-KV partials: one warp per packed query row
__global__ void attention_combine_kernel(AttnArgs a) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int mpad = a.m_blocks * AT_BM;
  const int rows_total = a.g * a.N;
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t total = (int64_t)a.B * a.Hkv * rows_total;
  if (gw >= total) return;
  const int bh = (int)(gw / rows_total), r = (int)(gw - (int64_t)bh * rows_total);
  const int b = bh / a.Hkv, kvh = bh - b * a.Hkv;
  const int node = r / a.g, qh = r - node * a.g;
  const int pr = a.npt ? node / a.npt * AT_BM + node % a.npt * a.g + qh : r;      // the packed row
  __nv_bfloat16 *op = a.out + (((int64_t)b * a.N + node) * a.Hq + kvh * a.g + qh) * AT_D + lane * 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float lsum = 0.f;
  if (r < a.g * a.n_nodes[b]) {
    float mx = -CUDART_INF_F;
    for (int s = 0; s < a.splits; ++s) mx = fmaxf(mx, a.part_ml[((int64_t)bh * a.splits + s) * mpad + pr].x);
    for (int s = 0; s < a.splits; ++s) {
      const int64_t prow = ((int64_t)bh * a.splits + s) * mpad + pr;
      const float2 ml = a.part_ml[prow];
      if (ml.x == -CUDART_INF_F) continue;
      const float w = exp2f(ml.x - mx);
      const float4 o = *reinterpret_cast<const float4 *>(a.part_o + prow * AT_D + lane * 4);
      acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
      lsum += w * ml.y;
    }
  }
  const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
  const __nv_bfloat162 v0 = __floats2bfloat162_rn(acc.x * inv, acc.y * inv);
  const __nv_bfloat162 v1 = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
  *reinterpret_cast<__nv_bfloat162 *>(op) = v0;
  *reinterpret_cast<__nv_bfloat162 *>(op + 2) = v1;
}

static int attn_m_blocks(const talon_ctx *c) {
  const int g = c->p.n_q_heads / c->p.n_kv_heads;
  return (g * c->p.budget + AT_BM - 1) / AT_BM;
}
// the tensor-core kernel packs whole nodes into a query tile
static int attn_tc_blocks(const talon_ctx *c) {
  const int g = c->p.n_q_heads / c->p.n_kv_heads;
  if (g > AT_BM) return attn_m_blocks(c);
  const int npt = AT_BM / g;
  return (c->p.budget + npt - 1) / npt;
}

size_t attention_workspace_elems(const talon_ctx *c, size_t *ml_elems) {
  const int mb = attn_tc_blocks(c);
  long long ctas = 2LL * c->p.batch_max * c->p.n_kv_heads * mb;       // room for two key ranges per CTA slot
  if (ctas < 2LL * c->sm_count) ctas = 2LL * c->sm_count;
  *ml_elems = (size_t)ctas * AT_BM;
  return (size_t)ctas * AT_BM * AT_D;
}

talon_status attention_mma_setup() {
  return cudaFuncSetAttribute(tree_attention_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AT_SMEM) ==
                 cudaSuccess ? TALON_OK : TALON_ERR_CUDA;
}

// How the tensor-core kernel is launched: its kind, the key ranges, and whether the reference follows the maximum.
struct AttnPlan { int kind, splits; bool exact_max; };
static AttnPlan plan_attention(talon_ctx *c, const AttnArgs &a, int tiles, bool early, bool split_p) {
  const int heads = c->B * a.Hkv;
  const bool only_one = split_p || a.m_blocks == 1 || c->attn_force_tiles == 1;
  const int ctas = only_one ? a.m_blocks * heads : (a.m_blocks + 1) / 2 * heads;
  bool one = only_one;
  int sp = 1;
  // How exact the rounding of P to bf16 is hangs on the ranges: a row's largest probability in the first tile of
  // each is 1 and so exact, and its neighbours round with half the error.  `usual`: as many ranges as the SMs and two
  // tiles a range allow (eight rather than nine or more, where a cluster has enough rows to merge).  With fewer the
  // reference follows every growth of the maximum (exact_max), which comes closer to 64 bits than the usual number
  // does (512 keys 2.20e-3 of the norm against 2.25e-3, 2048 keys 2.23e-3 against 2.28e-3; without it 2.30e-3
  // and 2.33e-3) for a rescale of O now and then, 0.15 us a key tile with one query tile and 0.3 with two.
  int usual = 1;
  if (!split_p && ctas < c->sm_count) {
    usual = std::max(1, std::min(c->sm_count / ctas, (tiles + c->attn_min_tiles - 1) / c->attn_min_tiles));
    if (usual > 8 && c->attn_cluster && heads * a.g * a.N >= 1024) usual = 8;
  }
  if (ctas < c->sm_count) {
    // Room for key ranges, or for a CTA per query tile instead of two tiles: the cheapest by a model in
    // microseconds, fitted to 1 to 4 sequences of 1-3 query tiles over 2048 tokens.  A key tile takes a CTA
    // 1.2 with one query tile and 1.6 with two, all before the first another 2.6; writing the result of one
    // range 1.6 a query tile.  Merging ranges in a cluster moves a CTA's partial result, 64 KB a query
    // tile, between SMs; the second kernel (more ranges than a cluster has CTAs) 8 and 11.  Clusters whose
    // CTAs fill SMs only fit a GPC at a time, so the device says how many it holds: a second round of them
    // doubles the time.  Started beside the growth of the trees (about 1.2 a layer), the work on the prefix
    // counts only where it takes longer than that.
    const float growing = early ? 1.2f * c->layers_run : 0.f;
    auto cost = [&](bool single, int s) {
      const int n = single ? a.m_blocks * heads : ctas;
      const int held = s >= 2 && s <= 8 && c->attn_cluster ? attention_tc_clusters(c, split_p ? TC_SPLIT_P : single ? TC_SINGLE : TC_PAIR, s) : 0;
      const int slots = held > 0 ? held : std::max(c->sm_count / s, 1);
      const float end = s == 1 ? (single ? 1.6f : 3.2f) : held == 0 ? (single ? 8.f : 11.f)
                        : s <= 4 ? (single ? 4.9f : 7.3f) : (single ? 5.9f : 9.f);
      const float tile = split_p ? 1.4f : single ? 1.2f : 1.6f, rescale = s < usual ? (single ? 0.15f : 0.3f) : 0.f;
      const float before = 2.6f + ((tiles + s - 1) / s - 1) * (tile + rescale);
      return (n + slots - 1) / slots * (std::max(before, growing) + tile) + end;
    };
    const int most = std::min((tiles + c->attn_min_tiles - 1) / c->attn_min_tiles, c->attn_cluster == 2 ? 8 : c->sm_count);
    float best = cost(one, 1);
    for (int single = only_one; single <= (c->attn_force_tiles != 2 || only_one); ++single)
      for (int s = 1; s <= std::min(most, c->sm_count / (single ? a.m_blocks * heads : ctas)); ++s) {
        const float t = cost(single, s);
        if (t < best) { best = t; sp = s; one = single; }
      }
  } else if (ctas % c->sm_count) {
    // More CTAs than SMs and a ragged last wave: halving the key ranges can fill it (512 CTAs on
    // 148 SMs are 4 waves of 257 tiles, 1024 half CTAs are 7 waves of 129).  Cost model in key
    // tiles: waves x (tiles per CTA + 2 for the prologue and epilogue), plus what merging the
    // partial results costs, about one tile per 24 CTAs per SM.
    const long long sm = c->sm_count;
    auto cost = [&](int s) {
      const long long n = (long long)ctas * s;
      const long long waves = (n + sm - 1) / sm;
      return waves * ((tiles + s - 1) / s + 2) + (s > 1 ? n / (24 * sm) + 3 : 0);
    };
    if (tiles >= 32 && cost(2) < cost(1)) sp = 2;
  }
  if (c->attn_force_splits > 0) sp = c->attn_force_splits;
  if (c->attn_force_tiles == 2) one = only_one;
  while (sp > 1 && (size_t)a.m_blocks * c->B * a.Hkv * sp * AT_BM > c->attn_ml_elems) --sp;
  return {split_p ? TC_SPLIT_P : one ? TC_SINGLE : TC_PAIR, sp, sp < usual};
}

talon_status launch_attention(talon_ctx *c, const talon_tree *t, const void *q, const void *kp, const void *vp,
                              const void *kt, const void *vt, const int64_t *kv_start, const int32_t *block_table,
                              int bt_stride, int64_t kv_tokens,
                              int64_t stride_t, int64_t stride_h, int max_prefix_len, float sm_scale, void *out,
                              cudaStream_t st, const int32_t *early_prefix) {
  AttnArgs a;
  a.q = (const __nv_bfloat16 *)q; a.kp = (const __nv_bfloat16 *)kp; a.vp = (const __nv_bfloat16 *)vp;
  a.kt = (const __nv_bfloat16 *)kt; a.vt = (const __nv_bfloat16 *)vt;
  a.kv_start = kv_start; a.stride_t = stride_t; a.stride_h = stride_h;
  a.prefix_len = c->d_prefix_len; a.n_nodes = t->n_nodes; a.mask = (const unsigned long long *)t->mask;
  a.B = c->B; a.N = c->p.budget; a.W = c->W; a.Hq = c->p.n_q_heads; a.Hkv = c->p.n_kv_heads;
  a.g = a.Hq / a.Hkv;
  a.scale_log2 = sm_scale * 1.4426950408889634f;
  a.m_blocks = attn_m_blocks(c);
  a.npt = 0;
  a.out = (__nv_bfloat16 *)out; a.part_o = c->d_attn_o; a.part_ml = c->d_attn_ml;

  if (attention_tc_supported(c, stride_t, stride_h, sm_scale)) {
    // tensor-core path: CTAs own two 128-row query tiles and 128-key tiles
    a.m_blocks = attn_tc_blocks(c);
    a.npt = AT_BM / a.g;
    const int tiles = (max_prefix_len + 127) / 128 + (a.N + 127) / 128, heads = c->B * a.Hkv;
    const bool odd = AT_BM % a.g != 0;
    AttnPlan plan = plan_attention(c, a, tiles, early_prefix != nullptr, false);
    plan.exact_max |= odd;
    if (odd) {
      // Query groups that do not divide 128 ran on the warp-MMA kernel once.  Its 64-key tiles, and up to `finer` ranges,
      // make more of the largest probabilities exact: 2.06e-3 to 2.30e-3 of the norm, and up to 6 % more in 128-key tiles
      // even if the reference follows every growth.  With sixteen tiles a range and no more than twice our ranges there,
      // the two are within 0.2 % (two seeds differ by 0.5); elsewhere P goes in as two parts (1.66e-3), 0 to 30 % more
      // time for a step of 100 to 700 keys.  At 2000 keys and 8 sequences two parts cost 46 %, following the maximum 4 %.
      const int blocks = attn_m_blocks(c) * heads, keys64 = (max_prefix_len + AT_BN - 1) / AT_BN + (a.N + AT_BN - 1) / AT_BN;
      const int finer = blocks < c->sm_count ? std::max(1, std::min(c->sm_count / blocks, keys64)) : 1;
      if (tiles < 16 * plan.splits || finer > 2 * plan.splits) plan = plan_attention(c, a, tiles, early_prefix != nullptr, true);
    }
    a.splits = plan.splits;
    int merged = 0;
    talon_status r = launch_attention_tc(c, t, q, kp, vp, kt, vt, kv_start, block_table, bt_stride, stride_t, stride_h, kv_tokens,
                                         max_prefix_len, sm_scale, out, plan.splits, a.m_blocks, plan.kind, plan.exact_max, st, &merged,
                                         early_prefix);
    if (r != TALON_OK) return r;
    if (plan.splits > 1 && !merged) {
      const int64_t rows = (int64_t)c->B * a.Hkv * a.g * a.N;
      const int wpb = 8;
      LaunchTimer lt(c, TALON_K_COMBINE, st);
      launch_kernel(c, attention_combine_kernel, dim3((unsigned)((rows + wpb - 1) / wpb)), dim3(wpb * 32), 0, st, a);
      if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
      c->launches += 1;
    }
    return TALON_OK;
  }

  if (block_table) return TALON_ERR_UNSUPPORTED;     // the warp-MMA kernel reads contiguous blocks only
  const int base = a.m_blocks * c->B * a.Hkv;
  const int max_tiles = (max_prefix_len + AT_BN - 1) / AT_BN + (a.N + AT_BN - 1) / AT_BN;
  int splits = 1;
  if (base < c->sm_count) {
    splits = c->sm_count / base;
    if (splits > max_tiles) splits = max_tiles;
    if (splits < 1) splits = 1;
  }
  // stay inside the partial workspace sized at creation
  while (splits > 1 && (size_t)base * splits * AT_BM > c->attn_ml_elems) --splits;
  a.splits = splits;

  dim3 grid(a.m_blocks, splits, c->B * a.Hkv);
  {
    LaunchTimer lt(c, TALON_K_ATTENTION, st);
    launch_kernel(c, tree_attention_mma_kernel, grid, dim3(AT_THREADS), AT_SMEM, st, a);
  }
  if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
  c->launches += 1;
  if (splits > 1) {
    const int64_t rows = (int64_t)c->B * a.Hkv * a.g * a.N;
    const int wpb = 8;
    LaunchTimer lt(c, TALON_K_COMBINE, st);
    launch_kernel(c, attention_combine_kernel, dim3((unsigned)((rows + wpb - 1) / wpb)), dim3(wpb * 32), 0, st, a);
    if (cudaGetLastError() != cudaSuccess) return TALON_ERR_CUDA;
    c->launches += 1;
  }
  return TALON_OK;
}

}  // namespace talon

// Row-wise kernels between the GEMMs: embedding lookup, residual add + RMSNorm, rotary
// embedding + KV-cache append, SiLU gating, per-row top-k with log-sum-exp.
// Model definition (pre-norm blocks, RMSNorm, half-split rotary pairs, gated SiLU MLP) is the
// reading taken for the architecture details the paper leaves to the target VLMs (Section 4).
#pragma once
#include "common.cuh"

// ---------------------------------------------------------------------------------------
// x[r] = embed[tok[r]] (fp32 residual stream).  tok < 0 leaves a zero row.  One thread per four
// elements: grid (rows, ceil(d / 1024)).  The first block of a row also copies the rotary factors of the
// row's position for every layer of the call: rope_tab[r][i] = rope_pos[pos[r]][i], i < half.
template <typename T>
__global__ void k_embed(const T *__restrict__ embed, const int *__restrict__ tok, float *x, int d,
                        int vocab, int *status, const int *__restrict__ pos, const float2 *__restrict__ rope_pos, int n_pos,
                        float2 *rope_tab, int half) {
  kernel_entry(TR_k_embed);
  int r = blockIdx.x, t = tok[r];
  if (blockIdx.y == 0)
    for (int i = threadIdx.x; i < half; i += blockDim.x) rope_tab[(long long)r * half + i] = rope_pos[(long long)min(pos[r], n_pos - 1) * half + i];
  int i = (blockIdx.y * blockDim.x + threadIdx.x) * 4;
  if (t >= vocab) { if (threadIdx.x == 0 && blockIdx.y == 0) atomicMax(status, DREAM_DEV_BAD_INDEX); t = -1; }
  if (i >= d) return;
  *reinterpret_cast<float4 *>(x + (long long)r * d + i) = t >= 0 ? ld_f4(embed + (long long)t * d + i) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// Prompt input rows of the prefill: visual embeddings inside [vis_start, vis_start+v),
// token embeddings elsewhere.  Writes the running residual x and a kept copy x0.
template <typename T>
__global__ void k_build_prompt(const T *__restrict__ embed, const T *__restrict__ visual,
                               const int *__restrict__ ids, int vis_start, int v, float *x,
                               float *x0, int d, int vocab, int *status) {
  kernel_entry(TR_k_build_prompt);
  int r = blockIdx.x;
  const T *src;
  if (r >= vis_start && r < vis_start + v) src = visual + (long long)(r - vis_start) * d;
  else {
    int t = ids[r < vis_start ? r : r - v];
    if (t < 0 || t >= vocab) { if (threadIdx.x == 0) atomicMax(status, DREAM_DEV_BAD_INDEX); t = 0; }
    src = embed + (long long)t * d;
  }
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    float f = to_f(src[i]);
    x[(long long)r * d + i] = f;
    x0[(long long)r * d + i] = f;
  }
}

// ---------------------------------------------------------------------------------------
// Per row: x += (GEMM output, if any); xn = RMSNorm(x) * gain as the next GEMM's input.
// Optional side outputs of the updated residual: `copy` (fp32; when tap_state is given the
// row is copied only if its sequence's tap layer equals `layer`) and `raw` (element type,
// unnormalised: the memory side of Eq. 1 takes features without a norm).
// A row is a cluster of blocks, 4 TH NV columns each, grid (blocks of a row, rows); they exchange their sums of
// squares through distributed shared memory, before anything is stored (a cluster barrier behind stores to
// global memory waits for them).  Bound by latency in a decode round, by memory in a prompt.
// Decode rows: 512 threads with one group of four columns each and at most 64 registers, so that a block is
// resident beside a GEMM's CTA before that ends and the next GEMM's CTAs start filling their rings when it does
// (a block of 1024 threads per row kept those out until the norm was done).  Round, SmolVLM-shaped / LLaVA-7B-shaped:
// 2339 / 4878 us; with 256 threads, twice the cluster, 2392 / 4923; with 256 threads of two groups 2371 / 4946.
// Prompt rows, many waves of blocks: 256 threads with two groups, half the barriers per row: SmolVLM-shaped request
// 11137 us, against 11205 with the decode form; four blocks per SM (64 registers) instead of three: Pixtral-shaped request 75.1 -> 74.0 ms.
template <typename T, int TH, int NV>
__global__ void __launch_bounds__(TH, 1024 / TH)
k_resid(float *x, GemmOut gin, int has_in, const T *__restrict__ gain, float eps, int d, T *xn, float *copy, const int *row_seq,
        const int *tap_state, int layer, T *raw, XLayout lay) {
  __shared__ float warp_ss[TH / 32], block_ss[2];
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.y, i0 = (blockIdx.x * NV * TH + threadIdx.x) * 4, n = gridDim.x;
  // the gains are weights: they can be fetched before the predecessor has finished
  float4 g[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) g[j] = xn && i0 + j * 4 * TH < d ? ld_f4(gain + i0 + j * 4 * TH) : make_float4(0.f, 0.f, 0.f, 0.f);
  float *xr = x + (long long)r * d;
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    const bool live = warm_pass(pass, tr, TR_k_resid);
    float4 v[NV];
    float ss = 0.f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int i = i0 + j * 4 * TH;
      const bool on = live && i < d;
      v[j] = on ? *reinterpret_cast<const float4 *>(xr + i) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (has_in) add4(v[j], gemm_val4<5>(gin, r, i, on));
      ss += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
    }
    bool do_copy = copy != nullptr && live;
    if (tap_state && do_copy) do_copy = tap_state[row_seq[r]] == layer;
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) warp_ss[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = warp_ss[0];
#pragma unroll
    for (int k = 1; k < TH / 32; ++k) tot += warp_ss[k];
    if (n > 1) {                                             // the row's blocks in ascending order
      if (threadIdx.x == 0) block_ss[pass] = tot;
      cluster_sync_all();
      tot = 0.f;
      for (int k = 0; k < n; ++k) tot += ld_cluster(mapa(smem_u32(block_ss + pass), k));
    } else __syncthreads();
    const float inv = 1.f / sqrtf(tot / (float)d + eps);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int i = i0 + j * 4 * TH;
      if (!live || i >= d) continue;
      if (has_in) *reinterpret_cast<float4 *>(xr + i) = v[j];
      if (do_copy) *reinterpret_cast<float4 *>(copy + (long long)r * d + i) = v[j];
      if (raw) store_split4<T>(raw + r * lay.row_stride + i, lay.lo_delta, v[j]);
      if (xn) store_split4<T>(xn + r * lay.row_stride + i, lay.lo_delta,
                              make_float4(v[j].x * inv * g[j].x, v[j].y * inv * g[j].y, v[j].z * inv * g[j].z, v[j].w * inv * g[j].w));
    }
  }
  if (n > 1) cluster_sync_relaxed();                         // no block leaves while another may still read its sum
}

// ---------------------------------------------------------------------------------------
// Rotary factors of every position a sequence can reach, made once: rope_pos[pos][i] = (cos, sin)(pos * theta^(-2i/hd)).
// The inverse frequency and the product are taken in double and reduced to [-pi, pi] before
// the single-precision sincos, so long prefixes lose no phase accuracy.  (Computed per row, head and layer, the
// double arithmetic took a third of a prompt's k_qkv_post_target.)  grid (n_pos).
__global__ void k_rope_table(float2 *rope_pos, int hd, float theta) {
  const int pos = blockIdx.x, half = hd / 2;
  for (int i = threadIdx.x; i < half; i += blockDim.x) {
    double a = (double)pos * exp2(-2.0 * (double)i / (double)hd * log2((double)theta));
    const double two_pi = 6.283185307179586476925286766559;
    a -= two_pi * rint(a / two_pi);
    float c, s;
    sincosf((float)a, &s, &c);
    rope_pos[(long long)pos * half + i] = make_float2(c, s);
  }
}

// (cos, sin) of four neighbouring rotary indices i..i+3 (i a multiple of 4) of a row of a rotary table.
__device__ __forceinline__ void rope_cs4(const float2 *tab, int row, int half, int i, float4 &cs01, float4 &cs23) {
  const float4 *t = reinterpret_cast<const float4 *>(tab + (long long)row * half + i);
  cs01 = t[0]; cs23 = t[1];
}

// Where a row's K/V go.  Target cache: pages [layer][2][page][H_kv][page_tokens][hd].
struct PagedKV {
  void *base;                    // this layer's K pool; V pool = base + kv_stride elements
  long long kv_stride;           // elements between the K pool and the V pool of one layer
  const int *page_table;         // [max_batch][pages_per_seq]
  int pages_per_seq, page_tokens, page_shift, hkv, hd;
  __device__ __forceinline__ long long off(int seq, int slot, int kvh) const {
    int pg = page_table[seq * pages_per_seq + (slot >> page_shift)];
    return (((long long)pg * hkv + kvh) * page_tokens + (slot & (page_tokens - 1))) * hd;
  }
};

// Rotary on four neighbouring pairs (a: columns i.., b: columns i + half..).
__device__ __forceinline__ void rotate4(float4 &a, float4 &b, const float4 &cs01, const float4 &cs23) {
  const float c0 = cs01.x, s0 = cs01.y, c1 = cs01.z, s1 = cs01.w, c2 = cs23.x, s2 = cs23.y, c3 = cs23.z, s3 = cs23.w;
  const float4 ra = make_float4(a.x * c0 - b.x * s0, a.y * c1 - b.y * s1, a.z * c2 - b.z * s2, a.w * c3 - b.w * s3);
  b = make_float4(b.x * c0 + a.x * s0, b.y * c1 + a.y * s1, b.z * c2 + a.z * s2, b.w * c3 + a.w * s3);
  a = ra;
}

// Column of the first value of pair `a` of column tile ct in the paired order of a GEMM with a fused epilogue
// (gemm_tc.cuh): 16 first and 16 second values alternate.
__device__ __forceinline__ int paired_col(int ct, int a) { return ct * 256 + (a >> 6) * 128 + ((a & 63) >> 4) * 32 + (a & 15); }
__device__ __forceinline__ int gemm_tile(const GemmOut &g, int r, int c) { return (c >> 8) * g.n_tt + div_small(r, g.inv_tile); }

// After the QKV GEMM of target rows: rotary on q and k (row r of rope_tab), q -> qbuf,
// k, v -> the paged cache at (row_seq, row_slot).  grid (rows, ceil(items / 256)); a work item
// is four neighbouring rotary pairs of one head, read and written as 128-bit words.  PAIRED: only what the GEMM's own
// epilogue has left (its stream-K tiles, in paired columns), from head hh0 on.
template <typename T, bool PAIRED>
__global__ void __launch_bounds__(256, 5)
k_qkv_post_target(GemmOut g, const int *__restrict__ row_seq, const int *__restrict__ row_slot,
                  int row0, int hh0, void *qbuf, PagedKV kv, int H, const float2 *__restrict__ rope_tab) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.x + row0, lr = blockIdx.x;
  const int hd = kv.hd, half = hd >> 1, q4_log2 = 28 - __clz(hd), Hkv = kv.hkv;     // hd / 8 items per head
  const int w = blockIdx.y * 256 + threadIdx.x, hw = w >> q4_log2, hh = hh0 + hw, i = (w - (hw << q4_log2)) * 4;
  const int ca = PAIRED ? paired_col(hh * hd >> 8, ((hh * hd & 255) >> 1) + i) : hh * hd + i, cb = ca + (PAIRED ? 16 : half);
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    const bool live = warm_pass(pass, tr, TR_k_qkv_post_target);
    bool on = live && hh < H + 2 * Hkv;
    if (PAIRED) on = on && gemm_tile(g, lr, ca) >= g.n_full;
    const int seq = on ? row_seq[r] : 0, slot = on ? row_slot[r] : 0;
    if (hh >= H && slot < 0) on = false;               // an idle row (malformed tree node) stores no K/V
    float4 cs01 = make_float4(1.f, 0.f, 1.f, 0.f), cs23 = cs01;
    if (on && hh < H + Hkv) rope_cs4(rope_tab, r, half, i, cs01, cs23);      // fetched along with the slots
    float4 a = gemm_val4<3>(g, lr, ca, on), b = gemm_val4<3>(g, lr, cb, on);
    rotate4(a, b, cs01, cs23);
    if (!on) continue;
    if (hh < H) {
      q_store4(qbuf, sizeof(T) == 2, (long long)r * H + hh, hd, i, a);
      q_store4(qbuf, sizeof(T) == 2, (long long)r * H + hh, hd, i + half, b);
    } else {
      const int v = hh >= H + Hkv ? 1 : 0;
      T *dst = (T *)kv.base + (v ? kv.kv_stride : 0) + kv.off(seq, slot, hh - H - (v ? Hkv : 0)) + i;
      store_split4<T>(dst, 0, a);
      store_split4<T>(dst + half, 0, b);
    }
  }
}

// Draft caches are flat per sequence and hold 4 bytes per element (they are small):
// [seq][2][H_kv][cap] rows of hd floats (fp32 configurations), or of 2 * hd bf16 = a high row
// then a low row (bf16 configurations: what the tensor-core attention reads directly).
struct FlatKV {
  void *base;
  int cap, hkv, hd, split;
  __device__ __forceinline__ long long off(int seq, int kv, int kvh, int row) const {
    return ((((long long)seq * 2 + kv) * hkv + kvh) * cap + row) * (split ? 2 : 1) * hd;
  }
  __device__ __forceinline__ void store4(long long o, int e, float4 v) const {
    if (split) store_split4<bf16>((bf16 *)base + o + e, hd, v);
    else *reinterpret_cast<float4 *>((float *)base + o + e) = v;
  }
};

// After a draft QKV GEMM (has_q: the GEMM produced q columns first, then K, then V; otherwise
// K then V only): rotary, q -> qbuf (when has_q), k/v -> draft self-attention cache row
// row_dst[r] (skipped when < 0).  The rotary table is by row, or by position.  Work items and grid as in k_qkv_post_target.
__global__ void __launch_bounds__(256, 5)
k_qkv_post_draft(GemmOut g, const int *__restrict__ row_seq, const int *__restrict__ row_pos, const int *__restrict__ row_dst,
                 int has_q, void *qbuf, FlatKV kv, int H, const float2 *__restrict__ rope_tab, int by_pos) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.x;
  const int hd = kv.hd, half = hd >> 1, q4_log2 = 28 - __clz(hd), Hkv = kv.hkv, Hq = has_q ? H : 0;
  const int w = blockIdx.y * 256 + threadIdx.x, hh = w >> q4_log2, i = (w - (hh << q4_log2)) * 4;
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    const bool live = warm_pass(pass, tr, TR_k_qkv_post_draft);
    bool on = live && hh < Hq + 2 * Hkv;
    const int dst = on ? row_dst[r] : 0, seq = on ? row_seq[r] : 0, tab_row = on && by_pos ? row_pos[r] : r;
    if (hh >= Hq && dst < 0) on = false;
    float4 cs01 = make_float4(1.f, 0.f, 1.f, 0.f), cs23 = cs01;
    if (on && hh < Hq + Hkv) rope_cs4(rope_tab, tab_row, half, i, cs01, cs23);
    float4 a = gemm_val4<3>(g, r, hh * hd + i, on), b = gemm_val4<3>(g, r, hh * hd + i + half, on);
    rotate4(a, b, cs01, cs23);
    if (!on) continue;
    if (hh < Hq) {
      q_store4(qbuf, kv.split, (long long)r * H + hh, hd, i, a);
      q_store4(qbuf, kv.split, (long long)r * H + hh, hd, i + half, b);
    } else {
      const int v = hh >= Hq + Hkv ? 1 : 0;
      const long long o = kv.off(seq, v, hh - Hq - (v ? Hkv : 0), dst);
      kv.store4(o, i, a);
      kv.store4(o, i + half, b);
    }
  }
}

// A GEMM output [rows][H * hd] becomes the query rows of the cross-attention (no rotary).
// grid (rows, ceil(H * hd / 1024)).
__global__ void __launch_bounds__(256)
k_gemm_to_q(GemmOut g, void *qbuf, int H, int hd, int split) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.x, i = (blockIdx.y * 256 + threadIdx.x) * 4, hd_log2 = 31 - __clz(hd), h = i >> hd_log2;
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    const bool live = warm_pass(pass, tr, TR_k_gemm_to_q), on = live && h < H;
    float4 v = gemm_val4<6>(g, r, i, on);
    if (on) q_store4(qbuf, split, (long long)r * H + h, hd, i - (h << hd_log2), v);
  }
}

// Cross-attention memory rows (Eq. 1: K = S W_K, V = S W_V): GEMM output [rows][2 H_kv hd]
// -> memory cache row of sequence row_seq[r]: row_dst[r] when nperm is null, else the
// tree-region row nperm[seq] + row_in[r].  Negative indices skip the row.
// grid (rows, ceil(2 H_kv hd / 1024)).
__global__ void __launch_bounds__(256)
k_mem_append(GemmOut g, const int *__restrict__ row_seq, const int *__restrict__ row_dst, const int *__restrict__ row_in,
             const int *__restrict__ nperm, FlatKV kv) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.x, i = (blockIdx.y * 256 + threadIdx.x) * 4, hd_log2 = 31 - __clz(kv.hd), hh = i >> hd_log2;
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    bool on = warm_pass(pass, tr, TR_k_mem_append) && hh < 2 * kv.hkv;
    const int seq = on ? row_seq[r] : 0;
    int dst = on ? (nperm ? row_in : row_dst)[r] : 0;
    if (dst < 0) on = false;
    if (nperm && on) dst += nperm[seq];
    const float4 v = gemm_val4<6>(g, r, i, on);
    const int which = hh >= kv.hkv ? 1 : 0;
    if (on) kv.store4(kv.off(seq, which, hh - which * kv.hkv, dst), i - (hh << hd_log2), v);
  }
}

// act = silu(gate) * up, from a GEMM output whose columns are [gate(ff) | up(ff)].
// grid (ceil(ff / 1024), rows).  PAIRED: only what the GEMM's own epilogue has left, from gate column i0 on.
template <typename T, bool PAIRED>
__global__ void __launch_bounds__(256, 8)
k_silu_mul(GemmOut g, T *act, int ff, int i0, XLayout lay) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  const int r = blockIdx.y, i = i0 + (blockIdx.x * 256 + threadIdx.x) * 4;
  const int ca = PAIRED ? paired_col(i >> 7, i & 127) : i, cb = ca + (PAIRED ? 16 : ff);
#pragma unroll 1
  for (int pass = warm_first(); pass < 2; ++pass) {
    const bool live = warm_pass(pass, tr, TR_k_silu_mul), on = live && i < ff && (!PAIRED || gemm_tile(g, r, ca) >= g.n_full);
    float4 a = gemm_val4<2>(g, r, ca, on), b = gemm_val4<2>(g, r, cb, on);
    const float4 o = make_float4(a.x / (1.f + __expf(-a.x)) * b.x, a.y / (1.f + __expf(-a.y)) * b.y,
                                 a.z / (1.f + __expf(-a.z)) * b.z, a.w / (1.f + __expf(-a.w)) * b.w);
    if (on) store_split4<T>(act + r * lay.row_stride + i, lay.lo_delta, o);
  }
}

// Gather fp32 rows into element-type GEMM input rows: dst[r] = src[idx[r]] (idx < 0 -> zeros).
template <typename T>
__global__ void k_gather_rows(const float *__restrict__ src, const int *__restrict__ idx, T *dst,
                              int d, const int *layer_ptr, int layer_lo, long long layer_stride,
                              XLayout lay) {
  kernel_entry(TR_k_gather_rows);
  int r = blockIdx.x, s = idx[r];
  if (layer_ptr) src += (long long)(*layer_ptr - layer_lo) * layer_stride;
  for (int i = threadIdx.x * 4; i < d; i += blockDim.x * 4)
    store_split4<T>(dst + r * lay.row_stride + i, lay.lo_delta,
                    s >= 0 ? ld_f4(src + (long long)s * d + i) : make_float4(0.f, 0.f, 0.f, 0.f));
}

// ---------------------------------------------------------------------------------------
// Per row of a [rows][V] GEMM output: the KTOP largest logits (ties -> lower id), in
// descending order, and the log-sum-exp of the row.  grid (rows, nsplit): block (r, sp) scans
// columns [sp * NV * 256, (sp + 1) * NV * 256), NV (4 or 16) per thread held in registers, and leaves a
// sorted partial list and an (m, z) pair; the block that finishes a row last merges the partials,
// always in the same order.  Selection is KTOP rounds of "best remaining" (topk_warp, topk_block).
#define TOPK_MAX 16
#define TOPK_THREADS 256
#define TOPK_COLS 4096
#define TOPK_PER_THREAD (TOPK_COLS / TOPK_THREADS)
struct TopkScratch {
  float *pv;       // [rows][nsplit][TOPK_MAX] partial values
  int *pi;         // [rows][nsplit][TOPK_MAX] partial ids
  float *pm, *pz;  // [rows][nsplit] running max and sum of exp
  int *counter;    // [rows] blocks done; zero between launches
};

// A float as an unsigned key of the same order (-0 = +0); 0 is below every number and stands for nothing (and NaN).
__device__ __forceinline__ uint32_t topk_key(float v) {
  const uint32_t u = __float_as_uint(v + 0.f);
  return v == v ? u ^ (u & 0x80000000u ? 0xffffffffu : 0x80000000u) : 0u;
}
__device__ __forceinline__ float topk_value(uint32_t k) {
  return k ? __uint_as_float(k ^ (k & 0x80000000u ? 0x80000000u : 0xffffffffu)) : -INFINITY;
}
// The ktop best of a warp's candidates (key[j] with id(j), NV per lane), larger key first, then lower id, to out_k, out_i.
// A lane keeps its best at hand and looks for the next one only after it has won a round, and a round is two
// warp reductions in hardware (five shuffle steps of a pair and a scan in every lane: three times as long).
template <int NV, typename Id>
__device__ __forceinline__ void topk_warp(uint32_t (&key)[NV], Id id, int ktop, uint32_t *out_k, int *out_i) {
  uint32_t bk = 0u;
  int bi = 0x7fffffff;
  auto scan = [&]() {
    bk = 0u; bi = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < NV; ++j)
      if (key[j] > bk || (key[j] == bk && bk && id(j) < bi)) { bk = key[j]; bi = id(j); }
  };
  scan();
#pragma unroll 1
  for (int round = 0; round < ktop; ++round) {
    const uint32_t wk = __reduce_max_sync(0xffffffffu, bk);
    const int wi = __reduce_min_sync(0xffffffffu, bk == wk ? bi : 0x7fffffff);
    if ((threadIdx.x & 31) == 0) { out_k[round] = wk; out_i[round] = wi; }
    if (bk == wk && bi == wi && wk) {
#pragma unroll
      for (int j = 0; j < NV; ++j) if (id(j) == wi) key[j] = 0u;
      scan();
    }
    __syncwarp();
  }
}
// ... of a block's candidates, to out_v, out_i: every warp selects its own ktop, then warp 0 selects from the warps' lists.
// sh_* hold TOPK_THREADS / 32 * TOPK_MAX entries.
template <int NV, typename Id>
__device__ __forceinline__ void topk_block(uint32_t (&key)[NV], Id id, int ktop, float *out_v, int *out_i, uint32_t *sh_k, int *sh_i) {
  constexpr int NW = TOPK_THREADS / 32, NC = NW * TOPK_MAX / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  topk_warp<NV>(key, id, ktop, sh_k + warp * TOPK_MAX, sh_i + warp * TOPK_MAX);
  __syncthreads();
  if (warp == 0) {
    uint32_t ck[NC];
    int ci[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      const int e = j * 32 + lane, k = e % TOPK_MAX;          // entry k of list e / TOPK_MAX
      ck[j] = k < ktop ? sh_k[e] : 0u;
      ci[j] = k < ktop ? sh_i[e] : 0x7fffffff;
    }
    __syncwarp();
    topk_warp<NC>(ck, [&](int j) { return ci[j]; }, ktop, sh_k, sh_i);
    if (lane < ktop) { out_v[lane] = topk_value(sh_k[lane]); out_i[lane] = sh_i[lane]; }
  }
  __syncthreads();
}

template <int NV>
__global__ void __launch_bounds__(TOPK_THREADS)
k_topk_lse(GemmOut g, int V, int ktop, int nsplit, TopkScratch ts, float *top_val, int *top_id, float *lse,
           float *logits_out) {
  __shared__ float red[33];
  __shared__ uint32_t sh_k[TOPK_THREADS / 32 * TOPK_MAX];
  __shared__ int sh_i[TOPK_THREADS / 32 * TOPK_MAX];
  __shared__ int is_last;
  kernel_entry(TR_k_topk_lse);
  int r = blockIdx.x, sp = blockIdx.y, tid = threadIdx.x;
  int c0 = sp * (NV * TOPK_THREADS);
  float v[NV];
  const bool vec = (V & 3) == 0;
  // column of a thread's candidate j (ascending in j)
  auto id = [&](int j) { return vec ? c0 + ((j >> 2) * TOPK_THREADS + tid) * 4 + (j & 3) : c0 + j * TOPK_THREADS + tid; };
  if (vec) {
    float4 q[NV / 4];
#pragma unroll
    for (int j = 0; j < NV / 4; ++j) {
      int c = c0 + (j * TOPK_THREADS + tid) * 4;
      q[j] = gemm_val4<2>(g, r, c, c < V);
      if (c >= V) q[j] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    }
#pragma unroll
    for (int j = 0; j < NV / 4; ++j) {
      int c = c0 + (j * TOPK_THREADS + tid) * 4;
      if (logits_out && c < V) *reinterpret_cast<float4 *>(logits_out + (long long)r * V + c) = q[j];
      v[4 * j] = q[j].x; v[4 * j + 1] = q[j].y; v[4 * j + 2] = q[j].z; v[4 * j + 3] = q[j].w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      int c = c0 + j * TOPK_THREADS + tid;
      v[j] = c < V ? gemm_val(g, r, c) : -INFINITY;
      if (logits_out && c < V) logits_out[(long long)r * V + c] = v[j];
    }
  }
  // (m, z) of this block's columns, combined in a fixed order
  float m = -INFINITY;
#pragma unroll
  for (int j = 0; j < NV; ++j) m = fmaxf(m, v[j]);
  float bm = warp_max(m);
  if ((tid & 31) == 0) red[tid >> 5] = bm;
  __syncthreads();
  if (tid < 32) { float t = tid < TOPK_THREADS / 32 ? red[tid] : -INFINITY; t = warp_max(t); if (tid == 0) red[32] = t; }
  __syncthreads();
  float gm = red[32];
  float z = 0.f;
#pragma unroll
  for (int j = 0; j < NV; ++j) z += __expf(v[j] - gm);        // exp(-inf) = 0 for padding
  float tot = block_sum(z, red);
  long long po = (long long)r * nsplit + sp;
  if (tid == 0) { ts.pm[po] = gm; ts.pz[po] = tot; }
  uint32_t key[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) key[j] = id(j) < V ? topk_key(v[j]) : 0u;
  topk_block<NV>(key, id, ktop, ts.pv + po * TOPK_MAX, ts.pi + po * TOPK_MAX, sh_k, sh_i);
  // the last block of the row merges
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    int old = atomicAdd(ts.counter + r, 1);
    is_last = old == nsplit - 1;
    if (is_last) ts.counter[r] = 0;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // candidates: nsplit lists of ktop entries, up to 4 per thread (nsplit * ktop <= 1024)
  uint32_t ck[4];
  int ci[4];
  int ncand = nsplit * ktop;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    int e = j * TOPK_THREADS + tid;
    bool ok = e < ncand;
    int q = ok ? e / ktop : 0, w = ok ? e - q * ktop : 0;
    ci[j] = ok ? __ldcg(ts.pi + ((long long)r * nsplit + q) * TOPK_MAX + w) : 0x7fffffff;
    const float cv = ok ? __ldcg(ts.pv + ((long long)r * nsplit + q) * TOPK_MAX + w) : 0.f;
    ck[j] = ok && ci[j] != 0x7fffffff ? topk_key(cv) : 0u;
  }
  if (tid < 32) {                 // log-sum-exp of the row from the blocks' (max, sum) pairs, one warp, fixed order
    float pm[8], pz[8];           // up to 256 blocks
    float mm = -INFINITY;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      int q = k * 32 + tid;
      pm[k] = q < nsplit ? __ldcg(ts.pm + (long long)r * nsplit + q) : -INFINITY;
      pz[k] = q < nsplit ? __ldcg(ts.pz + (long long)r * nsplit + q) : 0.f;
      mm = fmaxf(mm, pm[k]);
    }
    mm = warp_max(mm);
    float zz = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) zz += pz[k] * __expf(pm[k] - mm);         // exp(-inf) = 0 for the padding
    zz = warp_sum(zz);
    if (tid == 0) lse[r] = mm + logf(zz);
  }
  topk_block<4>(ck, [&](int j) { return ci[j]; }, ktop, top_val + (long long)r * ktop, top_id + (long long)r * ktop, sh_k, sh_i);
}

// Attention kernels of the fp32 configurations:
//   - causal prefill attention with the entropy accumulators of Eq. 2 fused in,
//   - visual-token importance (column sums of the attention matrix, Section 3.3),
//   - tree-masked verification attention over the paged prefix plus the tree tail,
//   - the draft's self- and cross-attention (Eq. 1) over flat caches plus tree rows.
// Every lane holds HD/32 consecutive elements of q, k and v; a key costs one coalesced
// row load, HD/32 FMAs and a butterfly reduction.  Softmax runs online in fp32.
#pragma once
#include "common.cuh"
#include "rows.cuh"

template <int EPL> struct RowLoad {
  static __device__ __forceinline__ void ld(const float *p, int lane, float (&o)[EPL]) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) o[e] = p[lane * EPL + e];
  }
};

// Online-softmax state of one (row, head): running max m, Z = sum e^{s-m}, the weighted
// value sum, and U = sum e^{s-m}(s-m) for the entropy  H = ln Z - U/Z  (Eq. 2, inner sum).
template <int EPL> struct Soft {
  float m, z, u, acc[EPL];
  __device__ __forceinline__ void init() {
    m = -INFINITY; z = 0.f; u = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
  }
  template <bool ENT>
  __device__ __forceinline__ void push(float s, const float (&v)[EPL]) {
    if (s > m) {
      float delta = s - m;                    // may be +inf on the first key
      float sc = __expf(-delta);              // 0 when m was -inf
      if (ENT) u = z > 0.f ? sc * (u - delta * z) : 0.f;
      z *= sc;
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] *= sc;
      m = s;
    }
    float p = __expf(s - m);
    z += p;
    if (ENT) u += p * (s - m);
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] += p * v[e];
  }
};

template <int EPL>
__device__ __forceinline__ float dot_lane(const float (&a)[EPL], const float (&b)[EPL]) {
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < EPL; ++e) s += a[e] * b[e];
  return warp_sum(s);
}

#define ATT_WARPS 8

// ---------------------------------------------------------------------------------------
// Causal self-attention of the n prompt rows at one layer.  A warp owns ATT_PF_ROWS consecutive
// rows of one head, so a key/value row fetched from the cache serves all of them; two keys are
// in flight at a time (their loads and butterfly reductions overlap) and each row's softmax state
// takes its keys one by one in ascending order.  grid (ceil(n / (8 * ATT_PF_ROWS)), H).
// Outputs: attn_out, rows of H*hd values (input of the O projection); lse [H][n] (row
// log-sum-exp of the scaled scores, for the importance pass), ent [H][n] row entropies.
#define ATT_PF_ROWS 4
template <int HD>
__global__ void __launch_bounds__(ATT_WARPS * 32)
k_attn_prefill(const float *__restrict__ qbuf, PagedKV kv, int seq, int n, int H, float scale,
               float *attn_out, float *lse, float *ent) {
  constexpr int EPL = HD / 32, RW = ATT_PF_ROWS;
  kernel_entry(TR_k_attn_prefill);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int i0 = (blockIdx.x * ATT_WARPS + w) * RW, h = blockIdx.y;
  if (i0 >= n) return;
  const int nr = min(RW, n - i0);
  int kvh = h / (H / kv.hkv);
  const float *Kp = (const float *)kv.base, *Vp = Kp + kv.kv_stride;
  float q[RW][EPL];
  Soft<EPL> st[RW];
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    RowLoad<EPL>::ld(qbuf + ((long long)min(i0 + r, n - 1) * H + h) * HD, lane, q[r]);
#pragma unroll
    for (int e = 0; e < EPL; ++e) q[r][e] *= scale;
    st[r].init();
  }
  const int jmax = i0 + nr - 1;
  for (int j = 0; j <= jmax; j += 2) {
    float k0[EPL], v0[EPL], k1[EPL], v1[EPL], s0[RW], s1[RW];
    const bool two = j + 1 <= jmax;
    long long o0 = kv.off(seq, j, kvh), o1 = kv.off(seq, two ? j + 1 : j, kvh);
    RowLoad<EPL>::ld(Kp + o0, lane, k0);
    RowLoad<EPL>::ld(Vp + o0, lane, v0);
    RowLoad<EPL>::ld(Kp + o1, lane, k1);
    RowLoad<EPL>::ld(Vp + o1, lane, v1);
#pragma unroll
    for (int r = 0; r < RW; ++r) { s0[r] = dot_lane<EPL>(q[r], k0); s1[r] = dot_lane<EPL>(q[r], k1); }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      if (r < nr && j <= i0 + r) st[r].template push<true>(s0[r], v0);
      if (r < nr && two && j + 1 <= i0 + r) st[r].template push<true>(s1[r], v1);
    }
  }
#pragma unroll
  for (int r = 0; r < RW; ++r) {
    if (r >= nr) break;
    const int i = i0 + r;
    float inv = 1.f / st[r].z;
#pragma unroll
    for (int e = 0; e < EPL; ++e) attn_out[((long long)i * H + h) * HD + lane * EPL + e] = st[r].acc[e] * inv;
    if (lane == 0) {
      lse[(long long)h * n + i] = st[r].m + logf(st[r].z);
      ent[(long long)h * n + i] = logf(st[r].z) - st[r].u / st[r].z;
    }
  }
}

// AE(l) = mean over rows and heads of the row entropies (Eq. 2), all layers at once: a block per layer, fixed order.
// sum_out (may be null) receives the sums themselves: the start of the running form of Eq. 2.
__global__ void k_entropy_mean(const float *__restrict__ ent, long long layer_stride, int count, float *out, float *sum_out) {
  __shared__ float sh[33];
  kernel_entry(TR_k_entropy_mean);
  const float *e = ent + blockIdx.x * layer_stride;
  float s = 0.f;
  for (int i = threadIdx.x; i < count; i += blockDim.x) s += e[i];
  float t = block_sum(s, sh);
  if (threadIdx.x == 0) { out[blockIdx.x] = t / (float)count; if (sum_out) sum_out[blockIdx.x] = t; }
}

// Importance of visual token j at the tapped layer (Section 3.3): the attention weight it receives,
// summed over the later query rows (and its own row when include_self) and over heads.
// One warp per (visual column, head), grid (ceil(v / 8), H): rows ascending, four in flight at a
// time, added in row order; k_colsum_heads then adds the heads in ascending order: a fixed order.  Queries and
// log-sum-exps are kept for every candidate layer (q_stride, lse_stride apart), the layer is known on the device.
template <int HD>
__global__ void __launch_bounds__(ATT_WARPS * 32)
k_colsum(const float *__restrict__ qbuf, long long q_stride, PagedKV kv, long long layer_stride, int seq, int n, int H, float scale,
         const float *__restrict__ lse, long long lse_stride, const int *__restrict__ tap, int tap_lo, int vis_start, int v, int include_self,
         float *part /* [H][v] */) {
  constexpr int EPL = HD / 32;
  kernel_entry(TR_k_colsum);
  qbuf += (*tap - tap_lo) * q_stride; lse += (*tap - tap_lo) * lse_stride;
  const float *K = (const float *)kv.base + (*tap - 1) * layer_stride;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int jv = blockIdx.x * ATT_WARPS + w, h = blockIdx.y;
  if (jv >= v) return;
  int j = vis_start + jv;
  int kvh = h / (H / kv.hkv);
  float k[EPL];
  RowLoad<EPL>::ld(K + kv.off(seq, j, kvh), lane, k);
  const float *lse_h = lse + (long long)h * n;
  float hs = 0.f;
  int i = include_self ? j : j + 1;
  for (; i + 3 < n; i += 4) {
    float q0[EPL], q1[EPL], q2[EPL], q3[EPL];
    RowLoad<EPL>::ld(qbuf + ((long long)i * H + h) * HD, lane, q0);
    RowLoad<EPL>::ld(qbuf + ((long long)(i + 1) * H + h) * HD, lane, q1);
    RowLoad<EPL>::ld(qbuf + ((long long)(i + 2) * H + h) * HD, lane, q2);
    RowLoad<EPL>::ld(qbuf + ((long long)(i + 3) * H + h) * HD, lane, q3);
    float l0 = lse_h[i], l1 = lse_h[i + 1], l2 = lse_h[i + 2], l3 = lse_h[i + 3];
    float s0 = dot_lane<EPL>(q0, k), s1 = dot_lane<EPL>(q1, k), s2 = dot_lane<EPL>(q2, k), s3 = dot_lane<EPL>(q3, k);
    hs += __expf(s0 * scale - l0);
    hs += __expf(s1 * scale - l1);
    hs += __expf(s2 * scale - l2);
    hs += __expf(s3 * scale - l3);
  }
  for (; i < n; ++i) {
    float q[EPL];
    RowLoad<EPL>::ld(qbuf + ((long long)i * H + h) * HD, lane, q);
    hs += __expf(dot_lane<EPL>(q, k) * scale - lse_h[i]);
  }
  if (lane == 0) part[(long long)h * v + jv] = hs;
}

// score[jv] = sum over heads, ascending, of the per-head column sums.
__global__ void k_colsum_heads(const float *__restrict__ part, int H, int v, float *score) {
  kernel_entry(TR_k_colsum);
  int jv = blockIdx.x * blockDim.x + threadIdx.x;
  if (jv >= v) return;
  float tot = 0.f;
  for (int h = 0; h < H; ++h) tot += part[(long long)h * v + jv];
  score[jv] = tot;
}

// ---------------------------------------------------------------------------------------
// Few query rows (tree nodes, draft rows): a block per (row, head).  Its warps take the keys in turn, four
// in flight each, and their softmax states meet in shared memory, warps in ascending order: one warp
// walking 96..160 keys one by one is a chain of as many loads and reductions (verify 34 us and draft 15 us a
// launch; 7.8 and 4.6 us so).
template <int EPL, bool ENT, typename Off>
__device__ __forceinline__ void push_keys(Soft<EPL> &st, const float (&q)[EPL], const float *K, const float *V, int lane, int w, int n, Off off) {
  for (int j0 = w; j0 < n; j0 += 4 * ATT_WARPS) {
    float k[4][EPL], v[4][EPL], s[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const long long o = off(min(j0 + c * ATT_WARPS, n - 1));
      RowLoad<EPL>::ld(K + o, lane, k[c]);
      RowLoad<EPL>::ld(V + o, lane, v[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) s[c] = dot_lane<EPL>(q, k[c]);
#pragma unroll
    for (int c = 0; c < 4; ++c) if (j0 + c * ATT_WARPS < n) st.template push<ENT>(s[c], v[c]);
  }
}
// Merges the warps' states; the row's output goes to out[0 .. HD), its entropy (if asked for) to *ent.
// A row without any key is zero.
template <int EPL>
__device__ __forceinline__ void merge_states(const Soft<EPL> &st, int lane, int w, float *out, float *ent) {
  __shared__ float sm[ATT_WARPS], sz[ATT_WARPS], su[ATT_WARPS], sa[ATT_WARPS][EPL * 32];
  if (lane == 0) { sm[w] = st.m; sz[w] = st.z; su[w] = st.u; }
#pragma unroll
  for (int e = 0; e < EPL; ++e) sa[w][lane * EPL + e] = st.acc[e];
  __syncthreads();
  float m = sm[0];
#pragma unroll
  for (int i = 1; i < ATT_WARPS; ++i) m = fmaxf(m, sm[i]);
  float z = 0.f, u = 0.f, f[ATT_WARPS];
#pragma unroll
  for (int i = 0; i < ATT_WARPS; ++i) {
    f[i] = sz[i] > 0.f ? __expf(sm[i] - m) : 0.f;
    z += f[i] * sz[i];
    if (f[i] > 0.f) u += f[i] * (su[i] + (sm[i] - m) * sz[i]);
  }
  const float inv = z > 0.f ? 1.f / z : 0.f;
  for (int e = threadIdx.x; e < EPL * 32; e += ATT_WARPS * 32) {
    float a = 0.f;
#pragma unroll
    for (int i = 0; i < ATT_WARPS; ++i) a += f[i] * sa[i][e];
    out[e] = a * inv;
  }
  if (ent && threadIdx.x == 0) *ent = logf(z) - u * inv;
}

// Tree-masked verification attention (Section 3.1).  Row r = tree node of sequence
// row_seq[r]; it sees prefix slots [0, P) and tail slots P + j for every j in its
// ancestor-or-self bit set.  grid (R, H).
// row_ent (ENT only): [R][H] entropy of the row's attention distribution.
template <int HD, bool ENT>
__global__ void __launch_bounds__(ATT_WARPS * 32)
k_attn_tree(const float *__restrict__ qbuf, PagedKV kv, const int *__restrict__ row_seq, const int *__restrict__ P_state,
            const uint32_t *__restrict__ mask, int T_nodes, int H, float scale, float *attn_out, float *row_ent) {
  constexpr int EPL = HD / 32;
  kernel_entry(TR_k_attn_tree);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = blockIdx.x, h = blockIdx.y;
  const int seq = row_seq[r], P = P_state[seq], kvh = h / (H / kv.hkv);
  const float *K = (const float *)kv.base, *V = K + kv.kv_stride;
  float q[EPL];
  RowLoad<EPL>::ld(qbuf + ((long long)r * H + h) * HD, lane, q);
#pragma unroll
  for (int e = 0; e < EPL; ++e) q[e] *= scale;
  Soft<EPL> st;
  st.init();
  push_keys<EPL, ENT>(st, q, K, V, lane, w, P, [&](int j) { return kv.off(seq, j, kvh); });
  const uint32_t *mr = mask + (long long)r * 4;
  for (int j = w; j < T_nodes; j += ATT_WARPS) {
    if (!((mr[j >> 5] >> (j & 31)) & 1u)) continue;
    const long long o = kv.off(seq, P + j, kvh);
    float k[EPL], v[EPL];
    RowLoad<EPL>::ld(K + o, lane, k);
    RowLoad<EPL>::ld(V + o, lane, v);
    st.template push<ENT>(dot_lane<EPL>(q, k), v);
  }
  merge_states<EPL>(st, lane, w, attn_out + ((long long)r * H + h) * HD, ENT ? row_ent + (long long)r * H + h : nullptr);
}

// ---------------------------------------------------------------------------------------
// Draft attention over a flat cache: permanent rows [0, nperm[seq]) are all visible, then
// tree-region rows nperm + j for each j in the row's ancestor set (self excluded when
// strict: cross-attention reads the draft features of strict ancestors only, Section 3.1).
// Rows with row_in < 0 are idle, unless row_vis is given and holds v >= 0 for the row: such a row
// sees the rows [0, v) and nothing else (none at all when v = 0: its output is zero).  grid (R, H).
template <int HD>
__global__ void __launch_bounds__(ATT_WARPS * 32)
k_attn_draft(const float *__restrict__ qbuf, FlatKV kv, const int *__restrict__ row_seq,
             const int *__restrict__ row_in, const int *__restrict__ row_vis, const int *__restrict__ nperm,
             const unsigned long long *__restrict__ anc, int anc_stride, int strict, int H,
             float scale, float *attn_out) {
  constexpr int EPL = HD / 32;
  kernel_entry(TR_k_attn_draft);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = blockIdx.x, h = blockIdx.y;
  const int in = row_in ? row_in[r] : 0, rv = row_vis ? row_vis[r] : -1;
  if (in < 0 && rv < 0) return;
  const int seq = row_seq[r], np = rv >= 0 ? rv : nperm[seq], kvh = h / (H / kv.hkv);
  const float *K = (const float *)kv.base + kv.off(seq, 0, kvh, 0), *V = (const float *)kv.base + kv.off(seq, 1, kvh, 0);
  float q[EPL];
  RowLoad<EPL>::ld(qbuf + ((long long)r * H + h) * HD, lane, q);
#pragma unroll
  for (int e = 0; e < EPL; ++e) q[e] *= scale;
  Soft<EPL> st;
  st.init();
  push_keys<EPL, false>(st, q, K, V, lane, w, np, [&](int j) { return (long long)j * HD; });
  unsigned long long bits = rv >= 0 ? 0ull : anc[(long long)seq * anc_stride + in];
  if (strict && rv < 0) bits &= ~(1ull << in);
  for (int i = 0; bits; ++i) {
    const int j = __ffsll((long long)bits) - 1;
    bits &= bits - 1;
    if (i % ATT_WARPS != w) continue;
    float k[EPL], v[EPL];
    RowLoad<EPL>::ld(K + (long long)(np + j) * HD, lane, k);
    RowLoad<EPL>::ld(V + (long long)(np + j) * HD, lane, v);
    st.template push<false>(dot_lane<EPL>(q, k), v);
  }
  merge_states<EPL>(st, lane, w, attn_out + ((long long)r * H + h) * HD, nullptr);
}

// Shared device helpers of the DREAM hot path: element conversion, deterministic block
// reductions, the split-output descriptor every GEMM consumer reads through.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

typedef __nv_bfloat16 bf16;

#define DREAM_MAX_BATCH 8          // sequences one call may list

#define DREAM_DEV_OK 0
#define DREAM_DEV_TIMEOUT 1
#define DREAM_DEV_BAD_INDEX 2
#define DREAM_DEV_LAYOUT 3             // a block's shared memory does not start where its kernel needs it (dream_init checks; see attn_tc.cuh)
// The waits that can expire, as the second status word names the first one that did.
enum {
  WAIT_none = 0,
  WAIT_gemm_peer, WAIT_gemm_w_ring, WAIT_gemm_w_last, WAIT_gemm_x_ring, WAIT_gemm_operands, WAIT_gemm_acc_empty, WAIT_gemm_acc_last, WAIT_gemm_acc_full,
  WAIT_attn_k_ring, WAIT_attn_v_ring, WAIT_attn_q, WAIT_attn_p_v, WAIT_attn_k_s, WAIT_attn_softmax, WAIT_attn_last,
  WAIT_colsum_q_ring, WAIT_colsum_k, WAIT_colsum_operands, WAIT_colsum_scores, WAIT_colsum_last,
  WAIT_probe
};
#define DREAM_WAIT_NAMES {"none", "k_gemm_tc: partner's TMEM", "k_gemm_tc: weight ring", "k_gemm_tc: last weight stages", "k_gemm_tc: token ring", "k_gemm_tc: operands", "k_gemm_tc: accumulator emptied", "k_gemm_tc: last accumulators emptied", "k_gemm_tc: accumulator complete", "k_attn_tc: key ring", "k_attn_tc: value ring", "k_attn_tc: queries", "k_attn_tc: probabilities and values", "k_attn_tc: keys and score buffer", "k_attn_tc: softmax", "k_attn_tc: last releases", "k_colsum_tc: query ring", "k_colsum_tc: keys", "k_colsum_tc: queries and accumulator", "k_colsum_tc: scores", "k_colsum_tc: last releases", "k_wait_probe"}

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

// Programmatic dependent launch: a kernel may start while its predecessor in the stream is still
// running; pdl_wait() blocks until the predecessor has completed and its writes are visible, and
// pdl_trigger() lets the successor start early.  Every kernel of the library calls pdl_wait()
// before it touches memory another kernel writes (weights never change and may be read earlier).
// Both are no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Optional timeline of a stream: when a trace buffer is installed (dream_trace), thread 0 of block
// 0 of every kernel appends (kernel id, %globaltimer) right after its grid dependency resolved,
// i.e. when its predecessor has completed.  Differences between consecutive entries are the
// critical-path time of each kernel as it runs in the stream, overlap included.  Layout of the
// buffer: word 0 = entries written, word 1 = capacity, then pairs (id, nanoseconds).
__device__ unsigned long long *g_dream_trace;
enum {
  TR_none = 0,
  TR_k_embed,
  TR_k_build_prompt,
  TR_k_resid,
  TR_k_qkv_post_target,
  TR_k_qkv_post_draft,
  TR_k_gemm_to_q,
  TR_k_mem_append,
  TR_k_silu_mul,
  TR_k_gather_rows,
  TR_k_topk_lse,
  TR_k_attn_prefill,
  TR_k_entropy_mean,
  TR_k_colsum,
  TR_k_attn_tree,
  TR_k_attn_draft,
  TR_k_attn_tc,
  TR_k_attn_combine,
  TR_k_draft_begin,
  TR_k_tree_expand,
  TR_k_tree_finalize,
  TR_k_verify_setup,
  TR_k_accept,
  TR_k_compact_kv,
  TR_k_accept_rows,
  TR_k_select_tap,
  TR_k_select_visual,
  TR_k_ctx_rows,
  TR_k_gemm_simt,
  TR_k_iota_rows,
  TR_k_set_seq,
  TR_k_set_int,
  TR_k_set_pages,
  TR_k_first_token,
  TR_k_argmax_out,
  TR_k_copy_f32,
  TR_k_split_rows,
  TR_k_gemm_collect,
  TR_k_gemm_tc,
  TR_count
};
#define DREAM_TRACE_NAMES {"none", "k_embed", "k_build_prompt", "k_resid", "k_qkv_post_target", "k_qkv_post_draft", "k_gemm_to_q", "k_mem_append", "k_silu_mul", "k_gather_rows", "k_topk_lse", "k_attn_prefill", "k_entropy_mean", "k_colsum", "k_attn_tree", "k_attn_draft", "k_attn_tc", "k_attn_combine", "k_draft_begin", "k_tree_expand", "k_tree_finalize", "k_verify_setup", "k_accept", "k_compact_kv", "k_accept_rows", "k_select_tap", "k_select_visual", "k_ctx_rows", "k_gemm_simt", "k_iota_rows", "k_set_seq", "k_set_int", "k_set_pages", "k_first_token", "k_argmax_out", "k_copy_f32", "k_split_rows", "k_gemm_collect", "k_gemm_tc"}
// The buffer's address is asked for at a kernel's entry, by the one thread that will use it (trace_open), and looked at behind the grid
// dependency.  Asked for behind the dependency, as it first was, every kernel began with a round trip to L2 or, behind a GEMM's weight
// stream, to HBM, in the block that the others then waited for (SmolVLM-shaped round 2315 -> 2290 us, fp32 toy request 4900 -> 4856).
__device__ __forceinline__ unsigned long long *trace_open(bool me) { return me ? g_dream_trace : nullptr; }
__device__ __forceinline__ unsigned long long *trace_open() {
  return trace_open(blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0);
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void trace_stamp(unsigned long long *tr, int id, unsigned long long t) {
  unsigned long long i = atomicAdd(tr, 1ull);
  if (i < tr[1]) { tr[2 + 2 * i] = (unsigned long long)id; tr[3 + 2 * i] = t; }
}
__device__ __forceinline__ void trace_stamp(unsigned long long *tr, int id) {
  if (tr) trace_stamp(tr, id, global_ns());
}
// Entry of every kernel of the library: let the successor start, wait for the predecessor.
__device__ __forceinline__ void kernel_entry(int id) {
  pdl_trigger();
  unsigned long long *tr = trace_open();
  pdl_wait();
  trace_stamp(tr, id);
}

// A kernel whose code has left the instruction caches fetches it line by line, a few hundred nanoseconds each,
// and the short kernels between two GEMMs are then mostly that.  So they run their body twice: a first time
// with every load and store switched off, while they wait for their predecessor anyway, and then for real:
//   pdl_trigger();
//   unsigned long long *tr = trace_open();
//   for (int pass = warm_first(); pass < 2; ++pass) { const bool live = warm_pass(pass, tr, id); ... }
// live is false the first time; the compiler does not know.  LLaVA-7B-shaped round 5.22 -> 5.07 ms, SmolVLM-shaped
// 2.64 -> 2.56 ms.  A grid of many waves skips it: its later blocks find the code there, and would run it
// twice for nothing (LLaVA-7B-shaped request 29.4 -> 30.0 ms).
#define WARM_BLOCKS 740
__device__ __forceinline__ int warm_first() { return gridDim.x * gridDim.y * gridDim.z <= WARM_BLOCKS ? 0 : 1; }
__device__ __forceinline__ bool warm_pass(int pass, unsigned long long *tr, int id) {
  if (pass) {
    pdl_wait();
    trace_stamp(tr, id);
  }
  int live = pass;
  asm volatile("" : "+r"(live));
  return live != 0;
}

// A bf16 GEMM input row is stored as two bf16 rows, hi = bf16(v) and lo = bf16(v - hi), so the
// tensor cores see the activation to ~16 mantissa bits while the weights stream once.  fp32
// inputs have no lo part.  XLayout says where the rows of such a buffer live: token t starts at
// element t * row_stride, and its lo part lo_delta elements further on (0 = no lo part).
struct XLayout {
  long long row_stride;
  long long lo_delta;
};
template <typename T> __device__ __forceinline__ void store_split(T *p, long long lo_delta, float v);
template <> __device__ __forceinline__ void store_split<float>(float *p, long long, float v) { *p = v; }
template <> __device__ __forceinline__ void store_split<bf16>(bf16 *p, long long lo_delta, float v) {
  bf16 hi = __float2bfloat16_rn(v);
  *p = hi;
  if (lo_delta) p[lo_delta] = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// Output of a GEMM: [rows][ld].  The stream-K part of the tensor-core kernel (tiles n_full and up) leaves
// up to ceil(kb / units per worker) + 1 partial sums per tile, slot_stride floats apart; its full waves and
// the SIMT kernel leave one.
struct GemmOut {
  const float *base;
  long long slot_stride;   // floats between consecutive slots
  int ld;                  // floats between consecutive rows (tokens)
  int kb;                  // k-panels per tile
  int n_full, n_tt;        // tiles with a single slot; token tiles per 256 columns
  float inv_upc, inv_tile; // 1 / work units (tile, k-panel) per worker (0: nothing has more slots); 1 / tokens per tile (0: one token tile)
};
// a / b of small non-negative integers (below 2^21) from 1 / b: the half keeps the product a half of 1 / b away from
// the next integer, which its rounding does not bridge.  An integer division is thirty instructions of code that
// every launch fetches anew.
__device__ __forceinline__ int div_small(int a, float inv_b) { return (int)(((float)a + 0.5f) * inv_b); }

__device__ __forceinline__ int gemm_extra_slots(const GemmOut &g, int r, int c) {
  const int tile = (c >> 8) * g.n_tt + div_small(r, g.inv_tile) - g.n_full, u0 = max(tile, 0) * g.kb;
  return tile < 0 ? 0 : div_small(u0 + g.kb - 1, g.inv_upc) - div_small(u0, g.inv_upc);
}
__device__ __forceinline__ float gemm_val(const GemmOut &g, int r, int c) {
  const float *p = g.base + (long long)r * g.ld + c;
  float s = *p;
  const int extra = gemm_extra_slots(g, r, c);
  for (int i = 1; i <= extra; ++i) s += p[(long long)i * g.slot_stride];
  return s;
}

// Four consecutive columns c..c+3 (c a multiple of 4: they share a tile, hence a slot count), zero unless `on`.
// The slots are added in slot order, MAXS extra ones fetched per round trip.
__device__ __forceinline__ void add4(float4 &s, const float4 &t) { s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w; }
template <int MAXS>
__device__ __forceinline__ float4 gemm_val4(const GemmOut &g, int r, int c, bool on = true) {
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 *p = reinterpret_cast<const float4 *>(g.base + (long long)r * g.ld + c);
  float4 s = on ? *p : zero;
  const int extra = on ? gemm_extra_slots(g, r, c) : 0;
  const long long st4 = g.slot_stride >> 2;
  int i = 1;
  do {                                          // at least one round: the code is the same whatever `on` says
    float4 t[MAXS];
#pragma unroll
    for (int k = 0; k < MAXS; ++k) t[k] = i + k <= extra ? p[(long long)(i + k) * st4] : zero;
#pragma unroll
    for (int k = 0; k < MAXS; ++k) add4(s, t[k]);
    i += MAXS;
  } while (i <= extra);
  return s;
}

// Four consecutive elements of a GEMM input row, high (and low) parts, as 8-byte stores.
template <typename T> __device__ __forceinline__ void store_split4(T *p, long long lo_delta, float4 v);
template <> __device__ __forceinline__ void store_split4<float>(float *p, long long, float4 v) {
  *reinterpret_cast<float4 *>(p) = v;
}
template <> __device__ __forceinline__ void store_split4<bf16>(bf16 *p, long long lo_delta, float4 v) {
  __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
  uint2 hv = make_uint2(*reinterpret_cast<uint32_t *>(&h0), *reinterpret_cast<uint32_t *>(&h1));
  *reinterpret_cast<uint2 *>(p) = hv;
  if (lo_delta) {
    float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2bfloat162_rn(v.z - f1.x, v.w - f1.y);
    *reinterpret_cast<uint2 *>(p + lo_delta) = make_uint2(*reinterpret_cast<uint32_t *>(&l0), *reinterpret_cast<uint32_t *>(&l1));
  }
}
__device__ __forceinline__ float4 ld_f4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ld_f4(const bf16 *p) {
  uint2 u = *reinterpret_cast<const uint2 *>(p);
  float2 a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// Query rows between the QKV post-processing and the attention kernels: one block of hd
// values per (row, head): fp32 (fp32 configurations), or hd high parts then hd low parts in bf16
// (bf16 configurations: what the tensor-core attention copies straight into shared memory).
// Four bytes per element either way.  rh = row * H + head.
__device__ __forceinline__ void q_store4(void *qbuf, int split, long long rh, int hd, int i, float4 v) {
  if (split) store_split4<bf16>((bf16 *)qbuf + rh * 2 * hd + i, hd, v);
  else *reinterpret_cast<float4 *>((float *)qbuf + rh * hd + i) = v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// ---- thread-block clusters
__device__ __forceinline__ uint32_t cluster_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r)); return r; }
// Address of this shared-memory location in the CTA of the given rank.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed;\n barrier.cluster.wait;" ::: "memory");
}
// Reads from the shared memory of a CTA of this cluster (addresses from mapa).
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

// Sum over a block of up to 1024 threads, same value returned to every thread; the order
// of additions is fixed, so results are reproducible run to run.
__device__ __forceinline__ float block_sum(float v, float *sh /* >= 33 floats */) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    float t = lane < nw ? sh[lane] : 0.f;
    t = warp_sum(t);
    if (lane == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

// (value, index) ordering used by every top-k / argmax: larger value first, then lower index.
__device__ __forceinline__ bool better(float va, int ia, float vb, int ib) {
  return va > vb || (va == vb && ia < ib);
}

// Few-query attention on the tcgen05 tensor cores for sm_100a: the tree-masked verification
// over the paged target cache (Section 3.1), the draft's self- and cross-attention over its flat
// caches (Eq. 1), and the causal prefill attention with the row entropies of Eq. 2.
//
// A CTA owns one tile of 64 query entries (entry = (row, query head of one KV-head group)), one KV
// head and one chunk of keys.  Queries carry ~16 mantissa bits as a high and a low bf16 row, so
// the tile is the MMA's M = 128: eight entries' high parts, then their low parts, then the next eight entries.  A warp reads its
// accumulators as 16 lanes x 8 columns fragments (tcgen05.ld.16x256b), in which lanes i and i + 8 come to the same thread: the two
// products of an entry are added without a shuffle.  (High and low part in neighbouring lanes, two shuffles and four selects per pair of
// keys, was half of the softmax's instructions.)  Keys are walked in blocks of 64:
//   S_b = Q K_b^T        tcgen05.mma 128 x 64 x 16 over head_dim, A = Q and B = K_b from shared memory
//                        (K-major, 128-byte swizzle, TMA-fed), fp32 accumulators in a TMEM ring, as far
//                        ahead of the softmax as the rings allow;
//   softmax              eight warps, each eight entries: the four lanes of a quad take 16 of the block's keys each for one entry, so
//                        a row's maximum and sums are two shuffles and nothing is exchanged between warps.  One pass: the block's row
//                        maximum, then P = 2^(s - m), its row sum, and P's high and low bf16 parts to the entry's two rows
//                        of a shared-memory tile in the operand layout.   m is any
//                        reference near the maximum: it follows the maximum only when that has outgrown it by 2^8, so
//                        the O accumulator is hardly ever rescaled (in TMEM, tcgen05.ld / tcgen05.st);
//   O += P_b V_b         tcgen05.mma 128 x head_dim x 16 steps over the block's keys, A = P_b (K-major)
//                        and B = V_b as stored ([key][head_dim]: an MN-major operand).
// K/V blocks arrive through two TMA rings; during verification the blocks below the verified prefix
// are requested before the grid dependency resolves.  Each CTA of a split tile keeps
// its (m, l, O) in its shared memory, and after a cluster barrier every CTA merges a share of the rows, reading
// the others' through distributed shared memory (a merge kernel behind partials in global memory costs 4 us more
// per launch, most of it the kernel boundary; it stays for tiles whose many chunks no cluster holds).  The
// prefill has one chunk and also leaves each row's log-sum-exp and entropy.  Warp roles: 0 = TMA producer, 1 = S issuer and TMEM owner,
// 2..9 = softmax and epilogue, 10 = O issuer.  One warp issuing both products spent 2.1k cycles per block at head_dim 256, 1.3k of them the
// matrix instructions' own time and the rest its waits in turn for P, V, K and a free S; of the 2.3k cycles of a block the softmax waited 0.9k.
// In-stream time per layer, one issuer and rows in pairs -> now, us: prompts of 832 rows, 32 heads of 128 52 -> 29 (two CTAs per SM: half of a
// CTA's 25k cycles is start, first fetch and end), 1152 rows, 32 heads of 64 45 -> 34, 4352 rows, 16 heads of 256 on 8 KV heads 502 -> 405 (bound by
// the MMA of N = 64, whose A operand's shared-memory reads take half again its own time); verification of 61 rows behind 832, 32 heads of
// 128 13.6 -> 12.7, of 81 rows behind 4352 at head_dim 256 22.5 -> 19.8 and its merge; draft, 32 heads of 128 10.2 -> 9.9.
// The loops are kept compact on purpose: this kernel's code is
// fetched anew at almost every launch (the weight stream between two launches pushes it out of the
// caches), and straight-line code then costs its own fetch (a fully unrolled version of the same
// loops ran four times slower).  Every mbarrier wait is bounded (mbar_wait, gemm_tc.cuh); a CTA of a cluster that gives
// up still meets the others at the merge, and they finish with what it left.
#pragma once
#include <map>
#include <vector>

#include "attn_merge.cuh"
#include "common.cuh"
#include "gemm_tc.cuh"
#include "q_tile.cuh"
#include "rows.cuh"

#define AT_THREADS 352
#define AT_RESCALE 8.f                 // the maximum may outgrow its reference by this power of two
#define AT_KBLK 64
#define AT_QTILE (128 * 64 * 2)        // one 64-column panel of the query tile (128 rows)
#define AT_KVTILE (64 * 64 * 2)        // one 64-column panel of a 64-key block
#define AT_PTILE (128 * 64 * 2)        // probabilities of one block (128 rows x 64 keys)

#define AT_MAX_CHUNKS 32               // most key chunks of a tile
#define AT_MAX_CLUSTER 16              // ... that are a cluster

enum { AT_VERIFY = 0, AT_DRAFT = 1, AT_PREFILL = 2 };

// Two floats -> packed bf16 pair (high parts) and the packed pair of the remainders.
__device__ __forceinline__ void split_pair(float x, float y, uint32_t &hi, uint32_t &lo) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  float2 f = __bfloat1622float2(h);
  __nv_bfloat162 l = __floats2bfloat162_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<uint32_t *>(&h);
  lo = *reinterpret_cast<uint32_t *>(&l);
}

// Ring depths: what shared memory (K and V blocks stay until their MMAs ran) and the TMEM columns
// (head_dim for O, 64 per S_b) hold.  PF: the prefill's form.
template <int HD, bool FLAT, bool PF = false> struct AtShape {
  static constexpr int PLANES = FLAT ? 2 : 1;
  // head_dim 64 over the paged cache, and a prompt's head_dim 128, take fewer blocks, so that O and S fit 256 TMEM columns and two
  // CTAs (98 and 113 KB of shared memory each) share an SM: twice the key chunks in flight per layer; in a prompt, one walks its keys while the
  // other starts or ends
  static constexpr bool SMALL = PF && HD == 128;
  static constexpr int STAGES = SMALL ? 2 : HD == 64 ? (FLAT ? 4 : 3) : (HD == 128 ? (FLAT ? 2 : 5) : (FLAT ? 1 : 2));   // K (and V) blocks
  static constexpr int S_BUFS = SMALL ? 2 : HD == 64 ? 3 : 4;        // S blocks in TMEM
  static constexpr int P_BUFS = SMALL ? 1 : 2;                       // blocks of probabilities
  static constexpr int TMEM_COLS = HD + S_BUFS * 64 <= 256 ? 256 : 512;
  static constexpr int CTAS_PER_SM = (HD == 64 && !FLAT) || SMALL ? 2 : 1;
  static constexpr int KP = HD / 64;                                 // 64-column panels per row
  static constexpr int KV_STAGE = PLANES * KP * AT_KVTILE;           // one block of K (or of V)
  static constexpr int Q_BYTES = KP * AT_QTILE;
  static constexpr int O_LD = HD + 8;                                // floats per row of the merge's O tile (over the K/V rings)
  static constexpr size_t SMEM = (SMALL ? 0 : 1024) + Q_BYTES + 2 * STAGES * KV_STAGE + P_BUFS * AT_PTILE + 384;
};

struct AttnTcArgs {
  int mode;                         // AT_*
  int slot_seq[DREAM_MAX_BATCH];    // sequence of each grid-z slot
  const int *prefix_len;            // by sequence: keys [0, prefix) are visible to every row (verify, draft)
  const int *row_in;                // [R] or null: rows with a negative entry are idle; index into anc (draft)
  const int *row_vis;               // [R] or null (draft): an entry >= 0 makes the row see keys [0, entry) and no tail key
  const uint32_t *mask;             // [R][4] visible tail keys (verify)
  const unsigned long long *anc;    // [seq][anc_stride] ancestor-or-self bits over tail keys (draft)
  int anc_stride, strict;
  int rows_per_seq, tail_len, H, G; // query rows per sequence slot, tail keys, query heads, heads per KV head
  int n_keys;                       // prefill: keys in the sequence (row i sees keys 0..i)
  float scale_log2;
  int n_chunks, blocks_per_chunk, n_rt;
  void *out;                        // [R][H*hd] rows in GEMM-input layout
  XLayout lay;
  int out_chunk_rows;               // prefill: the output rows are laid out per chunk of this many rows ...
  long long out_chunk_stride;       // ... this many elements apart (0: one chunk)
  float *lse, *ent;                 // prefill: [H][n] row log-sum-exp and entropy, or null
  float *row_ent;                   // verify: [R][H] entropy of every tree row's attention distribution, or null
  float *part_o, *part_ml, *part_u; // null: the chunks are a cluster; else the partials [slot][chunk][kvh][rt][64][hd], [..][64][2], [..][64] (with row_ent)
  // where the K/V blocks live, as rows of the K and V tensor maps
  const int *page_table;            // paged: [max_batch][pages_per_seq]
  int pages_per_seq, page_tokens, page_shift, hkv;
  long long flat_rows_per_head;     // flat: cap (rows per (sequence, K|V, KV head))
  int *status;
};

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, int w, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w), "l"(policy) : "memory");
}
__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z, int w, int v, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6, %7}], [%2], %8;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v), "l"(policy) : "memory");
}
// 16 TMEM lanes x 64 columns, as the accumulator fragment of a warp-level MMA: lane 4 i + j of the warp gets columns 8 c + 2 j and 8 c + 2 j + 1
// of TMEM lane i in r[4 c] and r[4 c + 1], of TMEM lane i + 8 in r[4 c + 2] and r[4 c + 3].
__device__ __forceinline__ void tmem_ld16x64(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16x64(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Makes this thread's shared-memory stores visible to the asynchronous proxy (the MMA reads P through it).
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared-memory descriptor of an MN-major operand with 128-byte swizzle: 64 elements of the MN axis
// are contiguous (one 128-byte row per K index), 8 K-rows form a 1024-byte group, and the next 64
// MN elements start lbo_bytes further on.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t saddr, uint32_t lbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(lbo_bytes >> 4) << 16;          // leading byte offset: between 64-element MN blocks
  d |= (uint64_t)(1024 >> 4) << 32;               // stride byte offset: between groups of 8 K-rows
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// 2^x for x <= 8 or so, subnormal results as zero.
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Pairs of keys, added and scaled one by one (the packed instructions give the same values and cost more in packing than they save).
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 d) { return make_float2(fmaf(a.x, b.x, d.x), fmaf(a.y, b.y, d.y)); }
// w[i] of the four lanes of a quad: lane j ends up with the quad's words j, in lane order.
__device__ __forceinline__ void quad_transpose(uint32_t (&w)[4], int lane) {
#pragma unroll
  for (int o = 1; o < 4; o <<= 1)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (!(j & o)) {
        const bool up = (lane & o) != 0;
        const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? w[j] : w[j | o], o);
        if (up) w[j] = got; else w[j | o] = got;
      }
}

template <int HD, bool FLAT, bool PF>
__global__ void __launch_bounds__(AT_THREADS, (AtShape<HD, FLAT, PF>::CTAS_PER_SM))
k_attn_tc(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
          const __grid_constant__ AttnTcArgs a) {
  using Sh = AtShape<HD, FLAT, PF>;
  constexpr int STAGES = Sh::STAGES, S_BUFS = Sh::S_BUFS, P_BUFS = Sh::P_BUFS, KP = Sh::KP, PLANES = Sh::PLANES;
  extern __shared__ __align__(1024) uint8_t at_smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)at_smem_raw + 1023) & ~(uintptr_t)1023);
  if (Sh::SMALL && smem != at_smem_raw) {                   // no room to align by hand: two CTAs fill an SM's shared memory (attn_tc_setup checks too)
    if (threadIdx.x == 0) atomicMax(a.status, DREAM_DEV_LAYOUT);
    return;
  }
  uint8_t *q_s = smem, *k_s = q_s + Sh::Q_BYTES, *v_s = k_s + STAGES * Sh::KV_STAGE, *p_s = v_s + STAGES * Sh::KV_STAGE;
  float *o_s = (float *)k_s, *ml_s = o_s + 64 * Sh::O_LD;     // merge: O of the 64 entries, then (m, l, u, -) of each
  uint64_t *bars = (uint64_t *)(p_s + P_BUFS * AT_PTILE);
  uint64_t *q_full = bars, *k_full = q_full + 1, *k_empty = k_full + STAGES, *v_full = k_empty + STAGES, *v_empty = v_full + STAGES;
  uint64_t *s_full = v_empty + STAGES, *s_free = s_full + S_BUFS, *p_full = s_free + S_BUFS, *p_empty = p_full + P_BUFS;
  uint32_t *tmem_base_p = (uint32_t *)(p_empty + P_BUFS);
  volatile int *abort_flag = (volatile int *)(tmem_base_p + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  // (prefill: the tiles with the most keys first, so that the last wave is short)
  const int chunk = blockIdx.x, slot = blockIdx.z;
  const int kvh = PF ? blockIdx.y % a.hkv : blockIdx.y / a.n_rt, rt = PF ? a.n_rt - 1 - blockIdx.y / a.hkv : blockIdx.y - kvh * a.n_rt;
  const int seq = a.slot_seq[slot];
  unsigned long long *tr = trace_open();
  if (warp == 0) {      // a lane per ring stage: the set-up is a few instructions deep instead of a loop
    if (lane < STAGES) { mbar_init(k_full + lane, 1); mbar_init(k_empty + lane, 1); mbar_init(v_full + lane, 1); mbar_init(v_empty + lane, 1); }
    else if (lane >= 8 && lane < 8 + S_BUFS) { mbar_init(s_full + lane - 8, 1); mbar_init(s_free + lane - 8, 8); }
    else if (lane >= 16 && lane < 16 + P_BUFS) { mbar_init(p_full + lane - 16, 8); mbar_init(p_empty + lane - 16, 1); }
    else if (lane == 24) { mbar_init(q_full, 1); *abort_flag = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_p)), "r"((uint32_t)Sh::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_base_p;
  int gave_up = WAIT_none;                                  // the wait of this warp that ran out
  // Verification reads the verified prefix and its length, which were written rounds ago (hundreds
  // of kernels back in the stream): its K/V blocks below the prefix length are fetched before the
  // grid dependency resolves.  Everything else is an output of the immediate predecessors.
  const bool early = a.mode == AT_VERIFY;
  if (!early) pdl_wait();

  // ---- the chunk's blocks
  const int rows_total = a.rows_per_seq * a.G;              // entries of this sequence slot
  const int e_base = rt * 64;                               // first entry of the tile
  int total_keys, P = 0;
  if (PF) {
    // causal: nothing beyond the tile's last row is visible to any of its rows
    int last_node = min(rows_total - 1, e_base + 63) / a.G;
    total_keys = min(a.n_keys, last_node + 1);
  } else {
    P = a.prefix_len[seq];
    total_keys = P + a.tail_len;
  }
  const int nb = (total_keys + AT_KBLK - 1) / AT_KBLK;
  const int b0 = chunk * a.blocks_per_chunk, b1 = min(nb, b0 + a.blocks_per_chunk);
  const int n_blk = max(0, b1 - b0);

  // K (which = 0) or V (1) of the chunk's block `it` into ring stage `st` (the whole producer warp)
  const uint64_t pol_kv = policy_evict_first();
  auto issue = [&](int which, int it, int st) {
    const int j0 = (b0 + it) * AT_KBLK;
    uint8_t *dst = (which ? v_s : k_s) + st * Sh::KV_STAGE;
    uint64_t *full = (which ? v_full : k_full) + st;
    const CUtensorMap *map = which ? &map_v : &map_k;
    if (elect_one()) mbar_expect_tx(full, (uint32_t)Sh::KV_STAGE);
    if (FLAT) {
      // rows of the map: (sequence, K | V, KV head, key); the second coordinate selects the plane
      const long long rk = (((long long)seq * 2 + which) * a.hkv + kvh) * a.flat_rows_per_head + j0;
      if (elect_one())
        for (int pp = 0; pp < PLANES * KP; ++pp) tma_load_3d(dst + pp * AT_KVTILE, map, full, (pp % KP) * 64, pp / KP, (int)rk, pol_kv);
    } else {
      const int sub_rows = min(64, a.page_tokens), n_sub = 64 / sub_rows;
      for (int sub = 0; sub < n_sub; ++sub) {
        const int j = min(j0 + sub * sub_rows, a.pages_per_seq * a.page_tokens - 1);
        const int pg = a.page_table[seq * a.pages_per_seq + (j >> a.page_shift)];
        const int row = (pg * a.hkv + kvh) * a.page_tokens + (j & (a.page_tokens - 1));
        if (elect_one())
          for (int kp = 0; kp < KP; ++kp) tma_load_2d(dst + kp * AT_KVTILE + sub * sub_rows * 128, map, full, kp * 64, row, pol_kv);
      }
    }
    __syncwarp();
  };
  int n_pre = 0;                                            // blocks of the first ring filling already under way
  if (early) {
    if (warp == 0 && n_blk > 0) {
      if (lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
      }
      __syncwarp();
      while (n_pre < min(n_blk, STAGES) && (b0 + n_pre + 1) * AT_KBLK <= P) { issue(0, n_pre, n_pre); issue(1, n_pre, n_pre); ++n_pre; }
    }
    pdl_wait();
  }
  trace_stamp(tr, TR_k_attn_tc);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (n_blk > 0) {
      const uint64_t pol_q = policy_evict_last();
      if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_q) : "memory");
      __syncwarp();
      // queries: boxes of 64 columns, whose rows come as the tile has them
      int c2, c4;
      q_tile_start(a.G, slot * a.rows_per_seq + e_base / a.G, c2, c4);
      if (elect_one()) {
        mbar_expect_tx(q_full, (uint32_t)Sh::Q_BYTES);
        for (int kp = 0; kp < KP; ++kp) tma_load_5d(q_s + kp * AT_QTILE, &map_q, q_full, kp * 64, kvh * a.G, c2, 0, c4, pol_q);
      }
      __syncwarp();
      // K runs one block ahead of V: its stage is free as soon as S was computed, V's only after O
      int ks = n_pre % STAGES, vs = ks;
      uint32_t kph = n_pre >= STAGES ? 0u : 1u, vph = kph;    // parity of the stage's last release (1: none needed yet)
      for (int it = n_pre; it <= n_blk; ++it) {
        if (it < n_blk) {
          if (!mbar_wait_warp(k_empty + ks, kph, abort_flag)) { gave_up = WAIT_attn_k_ring; break; }
          issue(0, it, ks);
          if (++ks == STAGES) { ks = 0; kph ^= 1u; }
        }
        if (it > n_pre) {
          if (!mbar_wait_warp(v_empty + vs, vph, abort_flag)) { gave_up = WAIT_attn_v_ring; break; }
          issue(1, it - 1, vs);
          if (++vs == STAGES) { vs = 0; vph ^= 1u; }
        }
      }
      // Until the last releases have arrived (the commits that nothing else waits for): one that came in after this CTA has
      // left would land in the shared memory of the CTA that follows it on the SM.
#pragma unroll 1
      for (int i = 0; i < STAGES && !gave_up; ++i) {
        if (!mbar_wait_warp(k_empty + ks, kph, abort_flag) || !mbar_wait_warp(v_empty + vs, vph, abort_flag)) gave_up = WAIT_attn_last;
        if (++ks == STAGES) { ks = 0; kph ^= 1u; }
        if (++vs == STAGES) { vs = 0; vph ^= 1u; }
      }
      // (parity of the last phase of a barrier used n times: n - 1; never used: 1)
      for (int b = 0; b < P_BUFS && !gave_up; ++b)
        if (!mbar_wait_warp(p_empty + b, (uint32_t)((n_blk + P_BUFS - 1 - b) / P_BUFS + 1) & 1u, abort_flag)) gave_up = WAIT_attn_last;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ S issuer: the whole warp, an elected
    // lane for the tcgen05 instructions (as in the GEMM).  fp32 accumulate, bf16 operands, M = 128, N = 64, both K-major
    if (n_blk > 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t s_addr0 = tmem_base + HD;
      const uint64_t qd = smem_desc(smem_u32(q_s)), kd = smem_desc(smem_u32(k_s));
      if (!mbar_wait_warp(q_full, 0, abort_flag)) gave_up = WAIT_attn_q;
      int ks = 0, sb = 0;                                    // ring positions of K and S
      uint32_t kph = 0, sph = 1;
#pragma unroll 1
      for (int it = 0; it < n_blk && !gave_up; ++it) {
        if (!__all_sync(0xffffffffu, mbar_wait(s_free + sb, sph, abort_flag) && mbar_wait(k_full + ks, kph, abort_flag))) { gave_up = WAIT_attn_k_s; break; }
        tc_fence_after();
        if (elect_one()) {
#pragma unroll 1
          for (int pp = 0; pp < PLANES * KP; ++pp) {
            const uint64_t ad = qd + (uint64_t)((pp % KP) * (AT_QTILE >> 4)), bd = kd + (uint64_t)((ks * Sh::KV_STAGE + pp * AT_KVTILE) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k) mma_bf16(s_addr0 + (uint32_t)(sb * 64), ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), idesc, (pp > 0 || k > 0) ? 1u : 0u);
          }
          mma_commit(k_empty + ks);
          mma_commit(s_full + sb);
        }
        __syncwarp();
        if (++ks == STAGES) { ks = 0; kph ^= 1u; }
        if (++sb == S_BUFS) { sb = 0; sph ^= 1u; }
      }
    }
  } else if (warp == 10) {
    // ------------------------------------------------------------------ O issuer: N = head_dim, B MN-major
    if (n_blk > 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t o_addr = tmem_base;
      const uint64_t pd = smem_desc(smem_u32(p_s)), vd = smem_desc_mn(smem_u32(v_s), AT_KVTILE);
      int vs = 0;
      uint32_t vph = 0;
#pragma unroll 1
      for (int it = 0; it < n_blk; ++it) {
        const int pb = it % P_BUFS;
        if (!__all_sync(0xffffffffu, mbar_wait(v_full + vs, vph, abort_flag) && mbar_wait(p_full + pb, (uint32_t)(it / P_BUFS) & 1u, abort_flag))) { gave_up = WAIT_attn_p_v; break; }
        tc_fence_after();
        const uint64_t ad = pd + (uint64_t)(pb * (AT_PTILE >> 4));
        if (elect_one()) {
#pragma unroll
          for (int pl = 0; pl < PLANES; ++pl) {
            const uint64_t bd = vd + (uint64_t)((vs * Sh::KV_STAGE + pl * KP * AT_KVTILE) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k)                                 // 16 keys = two groups of 8 K-rows = 2048 bytes
              mma_bf16(o_addr, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 128), idesc, (it > 0 || pl > 0 || k > 0) ? 1u : 0u);
          }
          mma_commit(p_empty + pb);
          mma_commit(v_empty + vs);
        }
        __syncwarp();
        if (++vs == STAGES) { vs = 0; vph ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax and epilogue: warps 2..5 and 6..9 each take 16
    // lanes of a quarter, that is eight entries; the four lanes of a quad share an entry
    const int q = warp & 3, half = warp >= 6 ? 1 : 0;          // TMEM lane quarter this warp may access, its half of it
    const int quad = lane >> 2, ql = lane & 3;
    const int ei = q * 16 + half * 8 + quad, row = q * 32 + half * 16 + quad, e = e_base + ei;      // entry of the tile; its high parts' row (low parts: + 8)
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32 + half * 16) << 16);
    // what this row sees: keys below `vis_end`, plus tail key j (key index tail0 + j) for the bits of mw
    int r = -1, h = 0, vis_end = 0, tail0 = 0;
    uint32_t mw[4] = {0u, 0u, 0u, 0u};
    if (e < rows_total) {
      const int node = e / a.G;
      r = slot * a.rows_per_seq + node; h = kvh * a.G + (e - node * a.G);
      if (PF) vis_end = node + 1;
      else {
        vis_end = P; tail0 = P;
        if (a.mode == AT_VERIFY) {
          for (int wd = 0; wd < 4; ++wd) mw[wd] = a.mask[(long long)r * 4 + wd];
        } else {
          const int in = a.row_in ? a.row_in[r] : 0;
          const int rv = a.row_vis ? a.row_vis[r] : -1;
          if (rv >= 0) vis_end = rv;
          else if (in < 0) r = -1;
          else {
            unsigned long long bits = a.anc[(long long)seq * a.anc_stride + in];
            if (a.strict) bits &= ~(1ull << in);
            mw[0] = (uint32_t)bits; mw[1] = (uint32_t)(bits >> 32);
          }
        }
      }
    }
    // Everything the loops below read sits in registers (the argument block is read through memory),
    // and the loops are kept small on purpose: the kernel's code is fetched anew at every launch
    // (the weight stream has pushed it out of L2 by then), so straight-line code costs its fetch.
    const float scale = a.scale_log2;
    const int tail_len = PF ? 0 : a.tail_len;
    const unsigned long long mlo = (unsigned long long)mw[0] | ((unsigned long long)mw[1] << 32),
                             mhi = (unsigned long long)mw[2] | ((unsigned long long)mw[3] << 32);
    // visibility of the 64 keys j0 .. j0 + 63 as a bit mask
    auto vis64 = [=](int j0) -> unsigned long long {
      const int npre = min(64, max(0, vis_end - j0));
      unsigned long long m = npre >= 64 ? ~0ull : (1ull << npre) - 1ull;
      if (npre < 64 && tail_len > 0) {
        const int sh = j0 - tail0;                             // tail key index of bit 0
        if (sh < 0) m |= sh > -64 ? mlo << (-sh) : 0ull;
        else if (sh < 64) m |= (mlo >> sh) | (sh ? mhi << (64 - sh) : 0ull);
        else m |= sh < 128 ? mhi >> (sh - 64) : 0ull;
      }
      return m;
    };
    // A wait that runs out (or finds that another warp's did) clears ok.  The warp then walks on to the end, its waits skipped.
    bool ok = true;
    auto wait = [&](uint64_t *bar, uint32_t parity) {            // one lane polls for the warp
      int w = 1;
      if (lane == 0 && (!ok || !mbar_wait(bar, parity, abort_flag))) w = 0;
      if (!__shfl_sync(0xffffffffu, w, 0) && ok) {
        ok = false;
        if (lane == 0) wait_expired(a.status, WAIT_attn_softmax, abort_flag, -1);
      }
    };
    float m_ref = -INFINITY;                                   // exp2 domain
    float2 l2 = make_float2(0.f, 0.f), u2 = l2;                // this lane's share of l = sum p and of u = sum p (s - m) for the entropy
    const bool want_ent = a.ent != nullptr || a.row_ent != nullptr;
    const float2 scale2 = make_float2(scale, scale);
    // where the lane's pairs of probabilities go: rows of 128 bytes, 16-byte pieces swizzled like the MMA expects a K-major operand
    // (piece ^ (row & 7)); low parts eight rows further on
    const uint32_t p_off = (uint32_t)(row * 128 + (quad << 4) + ql * 4);
    int sb = 0;
    uint32_t sph = 0;
#pragma unroll 1
    for (int it = 0; it < n_blk; ++it) {
      const int pb = it % P_BUFS, j0 = (b0 + it) * AT_KBLK;
      const bool all = __all_sync(0xffffffffu, vis_end >= j0 + AT_KBLK);
      wait(s_full + sb, sph);
      tc_fence_after();
      uint32_t sr[32];
      tmem_ld16x64(lane_addr + (uint32_t)(HD + sb * 64), sr);
      tmem_ld_wait();
      tc_fence_before();
      if (lane == 0) mbar_arrive(s_free + sb);
      if (++sb == S_BUFS) { sb = 0; sph ^= 1u; }
      // the products of the entry's high and low query parts; this lane's keys are 8 c + 2 ql and the next one
      float2 t[8];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        t[c] = add2(make_float2(__uint_as_float(sr[4 * c]), __uint_as_float(sr[4 * c + 1])), make_float2(__uint_as_float(sr[4 * c + 2]), __uint_as_float(sr[4 * c + 3])));
      if (!all) {
        const unsigned long long vm = vis64(j0) >> (2 * ql);
        const uint32_t v0 = (uint32_t)vm, v1 = (uint32_t)(vm >> 32);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t v = c < 4 ? v0 >> (8 * c) : v1 >> (8 * c - 32);
          t[c].x = v & 1u ? t[c].x : -INFINITY;
          t[c].y = v & 2u ? t[c].y : -INFINITY;
        }
      }
      float bm = fmaxf(t[0].x, t[0].y), bn = fmaxf(t[1].x, t[1].y);
#pragma unroll
      for (int c = 2; c < 8; c += 2) { bm = fmaxf(bm, fmaxf(t[c].x, t[c].y)); bn = fmaxf(bn, fmaxf(t[c + 1].x, t[c + 1].y)); }
      bm = fmaxf(bm, bn);
      bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
      bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2)) * scale;        // the block's row maximum, the same in the four lanes of the quad
      const bool grow = bm > m_ref + AT_RESCALE && m_ref != -INFINITY;
      if (__any_sync(0xffffffffu, grow)) {
        // ---- the accumulator takes the new reference (behind the O of every earlier block)
        wait(p_empty + (it - 1) % P_BUFS, (uint32_t)((it - 1) / P_BUFS) & 1u);
        tc_fence_after();
        const float corr = grow ? ex2(m_ref - bm) : 1.f;
#pragma unroll 1
        for (int c0 = 0; c0 < HD; c0 += 64) {
          uint32_t orr[32];
          tmem_ld16x64(lane_addr + (uint32_t)c0, orr);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 32; ++c) orr[c] = __float_as_uint(__uint_as_float(orr[c]) * corr);
          tmem_st16x64(lane_addr + (uint32_t)c0, orr);
        }
        tmem_st_wait();
        if (grow) {
          const float dm = bm - m_ref;
          u2 = make_float2(corr * (u2.x - dm * l2.x), corr * (u2.y - dm * l2.y));
          l2 = make_float2(l2.x * corr, l2.y * corr);
          m_ref = bm;
        }
      }
      if (m_ref == -INFINITY) m_ref = bm;
      const float base = m_ref == -INFINITY ? 0.f : m_ref;
      const float2 nbase2 = make_float2(-base, -base);
      if (it >= P_BUFS) wait(p_empty + pb, (uint32_t)(it / P_BUFS - 1) & 1u);
      // ---- probabilities, row sum, P's high and low parts into shared memory
      uint8_t *p_buf = p_s + pb * AT_PTILE;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float2 d = fma2(t[c], scale2, nbase2);
        const float2 p = make_float2(ex2(d.x), ex2(d.y));      // a masked key: 2^-inf = 0
        l2 = add2(l2, p);
        if (want_ent) u2 = fma2(p, make_float2(fmaxf(d.x, -1024.f), fmaxf(d.y, -1024.f)), u2);      // (p is 0 far above that)
        uint32_t hi, lo;
        split_pair(p.x, p.y, hi, lo);
        uint8_t *w = p_buf + (p_off ^ (uint32_t)(c << 4));
        *reinterpret_cast<uint32_t *>(w) = hi;
        *reinterpret_cast<uint32_t *>(w + 1024) = lo;
      }
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full + pb);
    }
    // ---- epilogue: the entry's accumulator (TMEM lanes i and i + 8 added), partial or finished.  What does not need the accumulator stands before
    // the wait for it: this code too is fetched at every launch, and as long as it stood behind, the CTA waited for O first and
    // then for the code.  From the last P to the end a draft launch at head_dim 128 took 7.2k cycles of 16.0k, now 5.4k of 14.0k (two blocks of keys);
    // LLaVA-7B-shaped round with all options 5160 -> 5115 us, SmolVLM-shaped 2290 -> 2260, LLaVA-7B-shaped 4897 -> 4857.
    float l_run = l2.x + l2.y, u_run = u2.x + u2.y;            // each of the quad's lanes summed a quarter of the keys
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    u_run += __shfl_xor_sync(0xffffffffu, u_run, 1);
    u_run += __shfl_xor_sync(0xffffffffu, u_run, 2);
    const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
    const long long pbase = ((((long long)slot * a.n_chunks + chunk) * a.hkv + kvh) * a.n_rt + rt) * 64 + ei;
    float *po = PF || a.n_chunks == 1 ? nullptr : a.part_o ? a.part_o + pbase * HD : o_s + ei * Sh::O_LD;
    bf16 *out = reinterpret_cast<bf16 *>(a.out) + h * HD;
    if (a.out_chunk_stride) out += (long long)(r / a.out_chunk_rows) * a.out_chunk_stride + (long long)(r % a.out_chunk_rows) * a.lay.row_stride;
    else out += (long long)r * a.lay.row_stride;
    if (n_blk > 0) wait(p_empty + (n_blk - 1) % P_BUFS, (uint32_t)((n_blk - 1) / P_BUFS) & 1u);
    pdl_trigger();                                            // the keys are done: the kernel that follows may take the SMs
    if (ok) {
      tc_fence_after();
#pragma unroll 1
      for (int c0 = 0; c0 < HD; c0 += 64) {
        uint32_t orr[32];
        if (n_blk > 0) { tmem_ld16x64(lane_addr + (uint32_t)c0, orr); tmem_ld_wait(); }
        else {
#pragma unroll
          for (int c = 0; c < 32; ++c) orr[c] = 0u;
        }
        // columns c0 + 8 c + 2 ql and the next one
        float2 v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
          v[c] = add2(make_float2(__uint_as_float(orr[4 * c]), __uint_as_float(orr[4 * c + 1])), make_float2(__uint_as_float(orr[4 * c + 2]), __uint_as_float(orr[4 * c + 3])));
        if (!PF && a.n_chunks > 1) {
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<float2 *>(po + c0 + 8 * c + 2 * ql) = v[c];
        } else {
          // turned within the quad: a lane stores eight consecutive columns
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) split_pair(v[4 * g + c].x * inv, v[4 * g + c].y * inv, hi[c], lo[c]);
            quad_transpose(hi, lane);
            quad_transpose(lo, lane);
            if (r >= 0) {
              bf16 *o = out + c0 + 32 * g + 8 * ql;
              *reinterpret_cast<uint4 *>(o) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
              if (a.lay.lo_delta) *reinterpret_cast<uint4 *>(o + a.lay.lo_delta) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
          }
        }
      }
      if (!PF && a.n_chunks > 1 && ql == 0) {
        if (a.part_o) {
          *reinterpret_cast<float2 *>(a.part_ml + pbase * 2) = make_float2(m_ref, l_run);
          if (a.row_ent) a.part_u[pbase] = u_run;
        } else *reinterpret_cast<float4 *>(ml_s + ei * 4) = make_float4(m_ref, l_run, u_run, 0.f);
      }
      if (r >= 0 && ql == 0 && (PF || a.n_chunks == 1)) {
        if (a.row_ent) {
          a.row_ent[(long long)r * a.H + h] = l_run > 0.f ? logf(l_run) - u_run * 0.6931471805599453f / l_run : 0.f;
        }
        if (a.lse) {
          // natural-log units: lse = m ln 2 + ln l;  H = ln l - u ln 2 / l
          const int node = r - slot * a.rows_per_seq;
          const float ln2 = 0.6931471805599453f;
          a.lse[(long long)h * a.n_keys + node] = m_ref * ln2 + logf(l_run);
          if (a.ent) a.ent[(long long)h * a.n_keys + node] = logf(l_run) - u_run * ln2 / l_run;
        }
      }
    }
  }
  if (gave_up && lane == 0) wait_expired(a.status, gave_up, abort_flag, -1);
  drain_if_aborted(abort_flag);
  tc_fence_before();
  if (!PF && a.n_chunks > 1 && !a.part_o) {
    // ---- merge: out = sum_c w_c O_c / sum_c w_c l_c with w_c = 2^(m_c - max m), chunks in ascending order; this CTA's
    // share of the (entry, four columns) items
    __syncwarp();
    cluster_sync_all();
    const uint32_t o_addr = smem_u32(o_s), ml_addr = smem_u32(ml_s);
    const int n = a.n_chunks;
    bf16 *out = reinterpret_cast<bf16 *>(a.out);
#pragma unroll 1
    for (int i = chunk * AT_THREADS + (int)threadIdx.x; i < 64 * (HD / 4); i += n * AT_THREADS) {
      const int en = i / (HD / 4), c4 = (i % (HD / 4)) * 4, e = e_base + en;
      if (e >= rows_total) continue;
      float M = -INFINITY, L = 0.f, U = 0.f;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
      for (int c = 0; c < n; c += 4) {
        float4 ml[4], o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ml[k] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
          o[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (c + k < n) { ml[k] = ld_cluster4(mapa(ml_addr + en * 16, c + k)); o[k] = ld_cluster4(mapa(o_addr + (en * Sh::O_LD + c4) * 4, c + k)); }
        }
        // A chunk without a visible key has no weight, but what was read of it enters the sums all the same: the closing
        // barrier does not wait for a read whose value nobody uses, and its CTA might leave before the read gets there.
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool on = ml[k].x != -INFINITY;
          const float Mn = fmaxf(M, ml[k].x), sc = on ? ex2(M - Mn) : 1.f, w = on ? ex2(ml[k].x - Mn) : 0.f;       // 2^-inf = 0 on the first live chunk
          // u relative to the new reference: sum p' (s - Mn) with p' = p 2^(m - Mn)
          U = on ? (L > 0.f ? sc * (U + (M - Mn) * L) : 0.f) + w * (ml[k].z + (ml[k].x - Mn) * ml[k].y) : U;
          L = L * sc + ml[k].y * w;
          acc.x = acc.x * sc + (on ? o[k].x : 0.f) * w; acc.y = acc.y * sc + (on ? o[k].y : 0.f) * w;
          acc.z = acc.z * sc + (on ? o[k].z : 0.f) * w; acc.w = acc.w * sc + (on ? o[k].w : 0.f) * w;
          M = Mn;
        }
      }
      const float inv = L > 0.f ? 1.f / L : 0.f;
      const int node = e / a.G, r = slot * a.rows_per_seq + node, h = kvh * a.G + (e - node * a.G);
      if (a.row_ent && c4 == 0) a.row_ent[(long long)r * a.H + h] = L > 0.f ? logf(L) - U * 0.6931471805599453f * inv : 0.f;
      store_split4<bf16>(out + (long long)r * a.lay.row_stride + h * HD + c4, a.lay.lo_delta, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
    }
    __syncwarp();
    cluster_sync_relaxed();                     // no CTA leaves while another may still read its shared memory
  } else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Sh::TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------ host side

// Tensor maps of the attention operands, cached by everything that defines them.
struct AtMapCache { std::map<std::vector<unsigned long long>, CUtensorMap> maps; };

// bf16 tensor of `rank` dimensions (innermost first), 128-byte swizzle, zero fill beyond the extents.
static inline bool at_map(GemmTcPlan *pl, AtMapCache *cache, const void *ptr, int rank, const unsigned long long *dims,
                          const unsigned long long *strides_bytes, const unsigned *box, CUtensorMap *out) {
  std::vector<unsigned long long> key;
  key.push_back((unsigned long long)(uintptr_t)ptr);
  key.push_back((unsigned long long)rank);
  for (int i = 0; i < rank; ++i) { key.push_back(dims[i]); key.push_back(box[i]); if (i) key.push_back(strides_bytes[i - 1]); }
  auto it = cache->maps.find(key);
  if (it != cache->maps.end()) { *out = it->second; return true; }
  cuuint64_t d[5], st[4];
  cuuint32_t b[5], es[5];
  for (int i = 0; i < rank; ++i) { d[i] = dims[i]; b[i] = box[i]; es[i] = 1; if (i) st[i - 1] = strides_bytes[i - 1]; }
  CUtensorMap m;
  CUresult r = pl->encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(ptr), d, st, b, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (cache->maps.size() > 4096) cache->maps.clear();
  cache->maps[key] = m;
  *out = m;
  return true;
}

// The query rows as the tiles take them (q_tile.cuh).
static inline bool attn_q_map(GemmTcPlan *pl, AtMapCache *cache, const void *q, int rows, int H, int G, int hd, CUtensorMap *out) {
  const QTileMap m = q_tile_map(rows, H, G, hd);
  return at_map(pl, cache, q, 5, m.dims, m.strides, m.box, out);
}

template <int HD, bool FLAT, bool PF>
static inline void attn_tc_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr, cudaStream_t stream, int use_pdl, int n_chunks, int cluster, int tiles, int n_slots) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(n_chunks, tiles, n_slots); cfg->blockDim = dim3(AT_THREADS);
  cfg->dynamicSmemBytes = AtShape<HD, FLAT, PF>::SMEM; cfg->stream = stream;
  int n = 0;
  if (cluster) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)n_chunks; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (use_pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg->attrs = attr; cfg->numAttrs = n;
}

// max_tiles[n]: tiles of n chunks (clusters of n CTAs) that are resident at once.
template <int HD, bool FLAT, bool PF>
static inline const char *attn_tc_setup(int *max_tiles, int n_sms) {
  auto *kernel = k_attn_tc<HD, FLAT, PF>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AtShape<HD, FLAT, PF>::SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return "cannot raise the attention kernel's shared memory or cluster limit";
  if (AtShape<HD, FLAT, PF>::SMALL) {          // dynamic shared memory lies behind the system's and the kernel's own
    int dev = 0, reserved = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, kernel) != cudaSuccess)
      return "cannot read the attention kernel's shared memory layout";
    if (reserved % 1024 || fa.sharedSizeBytes % 1024) return "the prompt's attention needs shared memory that starts on a multiple of 1024 bytes";
  }
  if (PF) return nullptr;                      // one chunk, no clusters
  max_tiles[0] = 0;
  max_tiles[1] = n_sms * AtShape<HD, FLAT, PF>::CTAS_PER_SM;
  for (int n = 2; n <= AT_MAX_CLUSTER; ++n) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    attn_tc_config<HD, FLAT, PF>(&cfg, attr, nullptr, 0, n, 1, 1, 1);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); clusters = 0; }
    max_tiles[n] = clusters;
  }
  return nullptr;
}

// Enqueue one attention launch: grid (a.n_chunks, H_kv * a.n_rt, n_slots), the chunks of a tile a cluster unless
// there are partials.
template <int HD, bool FLAT, bool PF>
static inline cudaError_t attn_tc_launch(cudaStream_t stream, int use_pdl, const CUtensorMap &mq, const CUtensorMap &mk, const CUtensorMap &mv,
                                         const AttnTcArgs &a, int n_slots) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  attn_tc_config<HD, FLAT, PF>(&cfg, attr, stream, use_pdl, a.n_chunks, a.n_chunks > 1 && !a.part_o, (a.H / a.G) * a.n_rt, n_slots);
  return cudaLaunchKernelEx(&cfg, k_attn_tc<HD, FLAT, PF>, mq, mk, mv, a);
}

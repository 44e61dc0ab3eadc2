// Weight-streaming GEMM on pairs of SMs for sm_100a:  out[t][c] = sum_k X[t][k] * W[c][k].
//
// A decode call has few tokens (1..256 rows), so this is a stream of W from HBM; a prompt has hundreds,
// and the tensor cores bound it.  Design:
//   * a cluster of two CTAs on neighbouring SMs works on one tile: 256 weight rows are the MMA's M
//     (tcgen05.mma.cta_group::2, 128 rows and 128 TMEM lanes per CTA) and up to 256 token rows its N, of
//     which each CTA stages one half.  Half as many workers as SMs also means half as many partial
//     sums per tile for the consumers to add;
//   * activations carry ~16 mantissa bits as two bf16 rows per token, kept as two planes (high parts,
//     then low parts lo_rows further on):
//       - up to 128 tokens (TC_X_CONCAT): both planes side by side are one N = 2 x tokens operand (the
//         first CTA stages the high plane, the second the low plane), the epilogue adds column t and
//         column tokens + t.  The weight panel is read from shared memory once;
//       - more tokens (TC_X_TWO): two MMAs per k-step, high then low, into the same columns;
//   * the tensor core adds into its accumulator with truncation, about half a unit in the last place
//     per MMA and always towards zero, so chains of MMAs into one accumulator are kept short: CONCAT deals
//     its k-steps out to as many accumulators as fit, TWO changes the accumulator every few panels (TcParams::chain)
//     and the epilogue warps carry the sums in registers;
//   * two shared-memory rings fed by TMA (cp.async.bulk.tensor.2d, 128-byte swizzle, no multicast), wp
//     panels of 64 k per stage: W (128 rows, 16 KB a panel) and X.  W gets all the room X leaves: it is
//     what a CTA can fetch before its grid dependency resolves.  One commit per stage frees both: the X
//     producer waits on the W stage that went with the X stage it reuses;
//   * tiles are 256 weight rows x up to 256 tokens, the token tiles of one weight tile next to each other.
//     With several token tiles, full waves of tiles come first, one tile per pair, so that neighbouring pairs read the same weight
//     panels at the same time (one HBM read serves them all).  The rest, between one and two waves of tiles
//     (or all of them when there are fewer than two), is stream-K: its (tile, panel) units are dealt
//     out in equal contiguous ranges, each inside one tile where tiles are few; a pair that covers part of a tile writes a partial sum to its own
//     slot and the consumer adds the slots in a fixed order;
//   * a prompt's gate/up and QKV projections finish in the epilogue (TC_EPI_SILU, TC_EPI_ROPE): their weight rows
//     are loaded in pairs (gate and up of a column; the two halves of a rotary pair), 16 rows of one kind and
//     16 of the other per TMEM lane quarter, so that one shuffle brings a pair together, and the
//     finished values go where the next kernel reads them.  Only the stream-K tiles still leave partial
//     sums (in the same paired column order) for the row kernel;
//   * programmatic dependent launch: W never changes, so its ring fills before the grid
//     dependency resolves; only the X producer and the epilogue wait for the previous kernel;
//   * the MMA issuer and the producers are whole warps that run their loops together and elect a lane for
//     the asynchronous instructions.  Run by one lane of a diverged warp, their operands are moved to uniform
//     registers one by one: measured 180..380 cycles of issue per MMA against 48..128 (its own time) so;
//   * warp roles: 0 = W producer, 1 = MMA issuer (first CTA of the pair) and TMEM owner, 2 = X producer,
//     4..11 = epilogue.  A TMEM lane is an output column c, so a warp's store of one token covers 128
//     contiguous bytes without a transpose; two TMEM accumulators alternate so that the epilogue of
//     one segment overlaps the MMAs of the next;
//   * every mbarrier wait is bounded, see mbar_wait.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <map>
#include <tuple>

#include "common.cuh"
#include "rows.cuh"

#define TC_BN 256               // weight rows per tile (MMA M, both CTAs)
#define TC_BK 64                // k elements per panel (128 bytes: one swizzle row)
#define TC_THREADS 384          // 12 warps, see the roles above
#define TC_WPANEL (128 * TC_BK * 2)          // one CTA's half of a weight panel
#define TC_MAX_STAGES 12
#define TC_EVEN 4               // units a pair may walk further for a share that lies in one tile

// How the token rows lie in the X buffer.  PLAIN: one bf16 row per token.  PLANAR: high parts, then
// the low parts lo_rows rows further on.
enum { TC_X_PLAIN = 0, TC_X_PLANAR = 1 };
// How the MMA takes them (see above).
// TILES: TWO over several token tiles, with full waves of tiles; a form of its own because the decode forms'
// code is fetched anew at every launch and each division in it shows (one kernel for all: rounds 4 % slower).
enum { TC_X_ONE = 0, TC_X_CONCAT = 1, TC_X_TWO = 2, TC_X_TILES = 3 };

enum { TC_EPI_STORE = 0, TC_EPI_SILU = 1, TC_EPI_ROPE = 2 };

// What a fused epilogue needs besides the sums.
struct TcEpi {
  bf16 *dst;                    // SILU: act rows (row_stride, lo_delta apart).  ROPE: query rows [row][head][hi | lo][hd]
  XLayout lay;
  int ff;                       // SILU: real gate columns
  int H, row0, seq;             // ROPE: query heads; the prompt row of token 0 (its position and cache slot)
  const float2 *rope_pos;
  PagedKV kv;
};

struct TcParams {
  float *out;
  long long slot_stride;        // floats between partial-sum slots
  int N, KB, ld;                // output columns, k panels, floats between token rows
  int kbu;                      // work units per tile: KB, or more so that every pair's share lies in one tile
  int n_pairs, n_waves, n_full; // pairs, full waves, tiles in them (n_pairs * n_waves)
  int sk_units, upc;            // stream-K part: units = tiles x panels, units per pair
  float inv_kbu, inv_upc;       // reciprocals, for div_small
  int n_tt, tile_t, mma_n;      // token tiles, tokens per tile, N of an MMA
  int chain;                    // TWO / TILES: panels per accumulator
  int n_sub;                    // CONCAT / ONE: accumulators the k-steps of a segment are dealt out to (1, 2 or 4)
  int n_tok;                    // real token rows
  int lo_rows;                  // row of the first low part in the X tensor map
  int wp, w_stages, x_stages;   // panels per stage, ring depths
  int *status;
  TcEpi epi;
};

// ------------------------------------------------------------------------------------------ PTX wrappers

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// ---- bounded waits.  A wait gives up WAIT_LIMIT_NS after it first found its phase incomplete, or as soon as the CTA's abort
// flag is set; the warp that gives up first names the wait in the status words and sets the flag in every CTA that depends on
// its own (wait_expired), and all leave within a millisecond or so.  (A limit that counts attempts is no limit: each may
// suspend the thread for as long as the hardware likes.)  No wait starts before the kernel's grid dependency has
// resolved, so that the limit covers this kernel's own work, milliseconds at most, however long its predecessors take.
// What has no limit: griddepcontrol.wait, whose predecessors end by the same rule; cluster and named barriers, which every
// thread of the CTAs concerned reaches whatever its waits said; the TMEM allocation, which waits for CTAs that
// hold some on the same SM, and these wait for no allocation any more.
#define WAIT_LIMIT_NS 1000000000ull
#define WAIT_SUSPEND_NS 1000000u         // an attempt suspends the thread no longer than this
#define WAIT_DRAIN_NS 1000000ull
__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done) : "r"(addr), "r"(parity), "r"(WAIT_SUSPEND_NS) : "memory");
  return done != 0;
}
// Waits for a phase parity; false when the limit ran out or the abort flag is set.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const volatile int *abort_flag, unsigned long long limit_ns = WAIT_LIMIT_NS) {
  const uint32_t addr = smem_u32(bar);
  if (mbar_try(addr, parity)) return true;
  const unsigned long long t0 = global_ns();
  do {
    if (mbar_try(addr, parity)) return true;
    if (*abort_flag) return false;
  } while (global_ns() - t0 < limit_ns);
  return false;
}
// One thread of a warp whose wait gave up.  peer: the CTA of the cluster that depends on this one (none: -1); it cannot
// have left, the closing barrier needs this thread too.
__device__ __forceinline__ void wait_expired(int *status, int where, volatile int *abort_flag, int peer) {
  if (*abort_flag) return;                     // somebody else's wait was the first
  *abort_flag = 1;
  atomicCAS(status + 1, 0, where);
  atomicMax(status, DREAM_DEV_TIMEOUT);
  if (peer >= 0)
    asm volatile("{\n .reg .b32 a;\n mapa.shared::cluster.u32 a, %0, %1;\n st.relaxed.cluster.shared::cluster.u32 [a], 1;\n fence.acq_rel.cluster;\n}"
                 ::"r"((uint32_t)__cvta_generic_to_shared((const void *)abort_flag)), "r"(peer) : "memory");
}
// Before a CTA that gave up leaves: its copies and matrix instructions under way land within microseconds.
__device__ __forceinline__ void drain_if_aborted(const volatile int *abort_flag) {
  if (!*abort_flag) return;
  for (const unsigned long long t0 = global_ns(); global_ns() - t0 < WAIT_DRAIN_NS;) {}
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_normal() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes,
// 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);        // start address
  d |= (uint64_t)1 << 16;                         // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;               // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                         // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                         // 128-byte swizzle
  return d;
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}

// One lane of a converged warp (always the same one).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0;
}
// The bounded wait made by a whole warp, which stays together whatever its lanes see.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, const volatile int *abort_flag, unsigned long long limit_ns = WAIT_LIMIT_NS) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, limit_ns));
}

// ---- pairs of CTAs (cluster of two; the even rank leads)
// Releases nothing: what it hands over is TMEM, ordered by the tcgen05 fences.  (An arrive with release at cluster
// scope waits until the thread's stores to global memory have been performed, 1.5 us behind an epilogue.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// A load into this CTA's shared memory that completes on the pair leader's barrier.
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, uint32_t leader_bar, int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(leader_bar), "r"(x), "r"(y), "l"(policy) : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}

// The segments (tile, panels [k0, k1)) of one pair, in order.  TILES: full waves first.
template <bool TILES> struct TcWalk {
  int pair, w, u, u_end;
  __device__ __forceinline__ TcWalk(const TcParams &p, int pair_) : pair(pair_), w(0) { u = pair * p.upc; u_end = min(u + p.upc, p.sk_units); }
  __device__ __forceinline__ bool next(const TcParams &p, int &tile, int &k0, int &k1) {
    if (TILES && w < p.n_waves) { tile = w * p.n_pairs + pair; k0 = 0; k1 = p.KB; ++w; return true; }
    if (u >= u_end) return false;
    tile = div_small(u, p.inv_kbu); k0 = u - tile * p.kbu; k1 = min(p.kbu, k0 + u_end - u);
    u += k1 - k0;
    k1 = min(k1, p.KB);
    if (TILES) tile += p.n_full;
    return true;
  }
};

// Eight lanes hold one column each of eight rows (v[j]: row j): turned so that lane m of the eight stores 8 consecutive
// columns of row m in one piece per part, high parts at d and (lo_delta != 0) low parts lo_delta behind.  (Stored one
// by one as 2-byte words the epilogue outlasted the MMAs of the next tile: 6 % of a request.)
__device__ __forceinline__ void tc_store8(const float (&v)[8], int lane, bool on, bf16 *d, long long lo_delta) {
  uint32_t w[8];                               // high part | low part
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const bf16 h = __float2bfloat16_rn(v[j]), l = __float2bfloat16_rn(v[j] - __bfloat162float(h));
    w[j] = (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(l) << 16);
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1)
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (!(j & o)) {
        const bool up = (lane & o) != 0;
        const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? w[j] : w[j | o], o);
        if (up) w[j] = got; else w[j | o] = got;
      }
  if (!on) return;
  *reinterpret_cast<uint4 *>(d) = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410), __byte_perm(w[4], w[5], 0x5410), __byte_perm(w[6], w[7], 0x5410));
  if (lo_delta)
    *reinterpret_cast<uint4 *>(d + lo_delta) = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632), __byte_perm(w[4], w[5], 0x7632), __byte_perm(w[6], w[7], 0x7632));
}

// Weight rows of pair `a` (0..127, a multiple of 16) of column tile ct.
template <int EPI>
__device__ __forceinline__ void tc_pair_rows(const TcEpi &e, int ct, int a, int &ya, int &yb) {
  if (EPI == TC_EPI_SILU) { ya = ct * 128 + a; yb = e.ff + ya; }
  else {
    const int half_log2 = 30 - __clz(e.kv.hd), half = 1 << half_log2;
    ya = ct * TC_BN + (a >> half_log2) * e.kv.hd + (a & (half - 1));
    yb = ya + half;
  }
}

// ------------------------------------------------------------------------------------------ kernel
// Dynamic shared memory (1024-byte aligned): W ring [w_stages][wp][16 KB], X ring [x_stages][wp][panel], barriers.
// Registers: the decode forms are held to 64, so that the row kernel that waits for this launch is resident beside
// it as a whole (its blocks have started, hence the next GEMM's CTAs can start as soon as these leave).
template <int FORM, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TC_THREADS, FORM >= TC_X_TWO ? 1 : 2)
k_gemm_tc(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // bytes of token rows one CTA stages per k panel
  const uint32_t xtile_bytes = (uint32_t)(FORM == TC_X_CONCAT ? p.tile_t : p.mma_n >> 1) * 128u;
  const uint32_t xpanel_bytes = FORM >= TC_X_TWO ? 2u * xtile_bytes : xtile_bytes;
  const uint32_t wstage_bytes = (uint32_t)p.wp * TC_WPANEL, xstage_bytes = (uint32_t)p.wp * xpanel_bytes;
  uint8_t *wring = smem, *xring = smem + (size_t)p.w_stages * wstage_bytes;
  uint64_t *bars = (uint64_t *)(xring + (size_t)p.x_stages * xstage_bytes);
  uint64_t *full_w = bars, *empty_w = full_w + TC_MAX_STAGES, *full_x = empty_w + TC_MAX_STAGES;
  uint64_t *acc_full = full_x + TC_MAX_STAGES, *acc_empty = acc_full + 2;
  uint64_t *peer_tmem = acc_empty + 2;            // first CTA: the second one has its TMEM
  uint32_t *tmem_base_p = (uint32_t *)(peer_tmem + 1);
  volatile int *abort_flag = (volatile int *)(tmem_base_p + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform for the compiler too
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  unsigned long long *tr = trace_open(blockIdx.x == 0 && lane == 0 && (warp == 0 || warp == 2));
  const unsigned long long t_start = blockIdx.x == 0 && threadIdx.x == 0 ? global_ns() : 0ull;
  if (warp == 0) {      // a lane per barrier: the set-up is a few instructions deep instead of a loop
    if (lane < TC_MAX_STAGES) { mbar_init(full_w + lane, 1); mbar_init(empty_w + lane, 1); }
    else if (lane < 2 * TC_MAX_STAGES) mbar_init(full_x + lane - TC_MAX_STAGES, 1);
    else if (lane < 2 * TC_MAX_STAGES + 2) { mbar_init(acc_full + lane - 2 * TC_MAX_STAGES, 1); mbar_init(acc_empty + lane - 2 * TC_MAX_STAGES, 16); }
    else if (lane == 31) { mbar_init(peer_tmem, 1); *abort_flag = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Both CTAs run from here on, and their barriers are initialised.  The allocation is an act of the pair: issued before its
  // partner was known to run it hung, once in some ten million launches (the first CTA's had come back, the second's never did).
  cluster_sync_all();
  if (warp == 1) {      // all 512 TMEM columns (two accumulators of 256), allocated by one full warp of each CTA
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_p)), "r"(512u) : "memory");
    tc_fence_before();
    if (rank == 1 && lane == 0) mbar_arrive_cluster(mapa(smem_u32(peer_tmem), 0));
  }
  pdl_trigger();
  uint32_t tmem_base = 0;
  if (warp == 1 || warp >= 4) {                  // the warps that use them
    asm volatile("bar.sync 1, 288;" ::: "memory");
    tc_fence_after();
    tmem_base = *tmem_base_p;
  }
  int tile, k0, k1;
  constexpr bool TILES = FORM == TC_X_TILES;
  TcWalk<TILES> walk(p, pair);
  int gave_up = WAIT_none;                       // the wait of this warp that ran out

  if (warp == 0) {
    // ------------------------------------------------------------------ W producer: weights are
    // constant, so nothing here waits for anything but ring space
    const uint64_t pol = TILES ? policy_evict_normal() : policy_evict_first();     // several token tiles read a weight panel
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
    __syncwarp();
    const uint32_t bar0 = mapa(smem_u32(full_w), 0);
    int s = 0;
    uint32_t ph = 1;
    while (!gave_up && walk.next(p, tile, k0, k1)) {
      const int y = (TILES ? tile / p.n_tt : tile) * TC_BN + (int)rank * 128;
      for (int kb = k0; kb < k1; kb += p.wp) {
        const int np = min(p.wp, k1 - kb);
        if (!mbar_wait_warp(empty_w + s, ph, abort_flag)) { gave_up = WAIT_gemm_w_ring; break; }
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full_w + s, 2u * (uint32_t)np * TC_WPANEL);
          uint8_t *dst = wring + (size_t)s * wstage_bytes;
          if (EPI == TC_EPI_STORE) {
            for (int i = 0; i < np; ++i) tma_load_2d_pair(dst + (size_t)i * TC_WPANEL, &map_w, bar0 + 8u * s, (kb + i) * TC_BK, y, pol);
          } else {                               // pairs of 16 rows (one panel per stage)
#pragma unroll 1
            for (int g = 0; g < 4; ++g) {
              int ya, yb;
              tc_pair_rows<EPI>(p.epi, tile / p.n_tt, (int)rank * 64 + g * 16, ya, yb);
              tma_load_2d_pair(dst + g * 4096, &map_w, bar0 + 8u * s, kb * TC_BK, ya, pol);
              tma_load_2d_pair(dst + g * 4096 + 2048, &map_w, bar0 + 8u * s, kb * TC_BK, yb, pol);
            }
          }
        }
        __syncwarp();
        if (++s == p.w_stages) { s = 0; ph ^= 1; pdl_wait(); }      // (a stage is released only behind the dependency)
      }
    }
    pdl_wait();
    if (tr) trace_stamp(tr, TR_none, t_start);                    // CTA start, before any dependency
    // Until the last releases have arrived, which the pair's first CTA signals across: an arrival that comes in after this
    // CTA has left would land in the shared memory of the CTA that follows it on the SM.
    for (int i = 0; !gave_up && i < p.w_stages; ++i) {
      if (!mbar_wait_warp(empty_w + s, ph, abort_flag)) gave_up = WAIT_gemm_w_last;
      if (++s == p.w_stages) { s = 0; ph ^= 1; }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ X producer: waits until the
    // input exists (previous kernel), then feeds one X stage per W stage
    const uint64_t pol = policy_evict_last();
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
    __syncwarp();
    bool more = walk.next(p, tile, k0, k1);
    pdl_wait();
    trace_stamp(tr, TR_k_gemm_tc);
    __syncwarp();
    const uint32_t bar0 = mapa(smem_u32(full_x), 0);
    const int y_off = FORM == TC_X_CONCAT ? (int)rank * p.lo_rows : (int)rank * (p.mma_n >> 1);   // first token row this CTA stages, from the tile's
    int s = 0, n_free = p.x_stages, ws = 0;      // unused X stages left; W stage that went with the X stage to reuse
    uint32_t wph = 0;
    for (; !gave_up && more; more = walk.next(p, tile, k0, k1)) {
      const int y = (TILES ? tile % p.n_tt * p.tile_t : 0) + y_off;
      for (int kb = k0; kb < k1; kb += p.wp) {
        const int np = min(p.wp, k1 - kb);
        if (n_free > 0) --n_free;
        else {
          if (!mbar_wait_warp(empty_w + ws, wph, abort_flag)) { gave_up = WAIT_gemm_x_ring; break; }
          if (++ws == p.w_stages) { ws = 0; wph ^= 1; }
        }
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full_x + s, 2u * (uint32_t)np * xpanel_bytes);
          for (int i = 0; i < np; ++i) {
            uint8_t *dst = xring + (size_t)s * xstage_bytes + (size_t)i * xpanel_bytes;
            tma_load_2d_pair(dst, &map_x, bar0 + 8u * s, (kb + i) * TC_BK, y, pol);
            if (FORM >= TC_X_TWO) tma_load_2d_pair(dst + xtile_bytes, &map_x, bar0 + 8u * s, (kb + i) * TC_BK, p.lo_rows + y, pol);
          }
        }
        __syncwarp();
        if (++s == p.x_stages) s = 0;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the pair's first CTA)
    if (rank == 0) {
      // instruction descriptor: fp32 accumulate, bf16 A and B, both K-major, M = 256
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.mma_n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const uint64_t wdesc = smem_desc(smem_u32(wring)), xdesc = smem_desc(smem_u32(xring));
      const int w_stages = p.w_stages, x_stages = p.x_stages, wp = p.wp;
      const uint32_t sub_n = (uint32_t)p.mma_n, sub_mask = (uint32_t)p.n_sub - 1u;
      int ws = 0, xs = 0;
      uint32_t wph = 0, xph = 0, fill = 0;                            // fill counts accumulator fills
      k0 = k1 = 0;
      pdl_wait();
      if (!mbar_wait_warp(peer_tmem, 0, abort_flag)) gave_up = WAIT_gemm_peer;
      while (!gave_up && (k0 < k1 || walk.next(p, tile, k0, k1))) {
        const int fill_end = FORM >= TC_X_TWO ? min(k1, k0 + p.chain) : k1;
        const uint32_t buf = fill & 1u, use = fill >> 1;              // use: earlier fills of this accumulator
        ++fill;
        if (!mbar_wait_warp(acc_empty + buf, (use & 1u) ^ 1u, abort_flag)) { gave_up = WAIT_gemm_acc_empty; break; }
        tc_fence_after();
        const uint32_t d_addr = tmem_base + buf * 256u;
        uint32_t begun = 0u;                                          // 0: the first MMA of an accumulator overwrites it
        while (k0 < fill_end) {
          const int np = min(wp, fill_end - k0);
          if (!__all_sync(0xffffffffu, mbar_wait(full_w + ws, wph, abort_flag) && mbar_wait(full_x + xs, xph, abort_flag))) { gave_up = WAIT_gemm_operands; break; }
          tc_fence_after();
          for (int i = 0; i < np; ++i) {
            const uint64_t ad = wdesc + (uint64_t)((ws * wp + i) * (TC_WPANEL >> 4));
            const uint64_t bd = xdesc + (uint64_t)((uint32_t)(xs * wp + i) * (xpanel_bytes >> 4));
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < TC_BK / 16; ++k) {
                if (FORM >= TC_X_TWO) {
                  mma_bf16_pair(d_addr, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), idesc, k ? 1u : begun);
                  mma_bf16_pair(d_addr, ad + (uint64_t)(k * 2), bd + (uint64_t)((xtile_bytes >> 4) + k * 2), idesc, 1u);
                } else {
                  const uint32_t sub = (uint32_t)k & sub_mask;
                  mma_bf16_pair(d_addr + sub * sub_n, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), idesc, (uint32_t)k > sub_mask ? 1u : begun);
                }
              }
            }
            begun = 1u;
          }
          if (elect_one()) mma_commit_pair(empty_w + ws);             // frees both stages in both CTAs once these MMAs have read them
          k0 += np;
          if (++ws == w_stages) { ws = 0; wph ^= 1; }
          if (++xs == x_stages) { xs = 0; xph ^= 1; }
        }
        if (!gave_up && elect_one()) mma_commit_pair(acc_full + buf);       // accumulator complete
        __syncwarp();
      }
      // as above for the second CTA's arrivals: both accumulators emptied (they are relaxed, and the barrier at the end
      // does not wait for them).  The decode forms send only the arrivals that the loop above has waited for.
      for (uint32_t buf = 0; FORM >= TC_X_TWO && !gave_up && buf < 2u; ++buf)
        if (!mbar_wait_warp(acc_empty + buf, (((fill + 1u - buf) >> 1) & 1u) ^ 1u, abort_flag)) gave_up = WAIT_gemm_acc_last;
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ epilogue: this CTA's 128 output
    // columns of every segment, one per TMEM lane; warps 4..7 and 8..11 take token groups in turn
    const int q = warp & 3, half = warp >= 8 ? 1 : 0;       // TMEM lane quarter this warp may read; its token groups
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    const uint32_t done_bar = mapa(smem_u32(acc_empty), 0);
    pdl_wait();                               // the output buffer belongs to earlier kernels
    uint32_t fill = 0;
    const uint32_t n_seg = FORM >= TC_X_TWO || walk.u >= walk.u_end ? 0u : (uint32_t)(div_small(walk.u_end - 1, p.inv_kbu) - div_small(walk.u, p.inv_kbu) + 1);
    bool ok = true;
    auto wait_full = [&](uint32_t buf, uint32_t use) {
      int w = 1;
      if (lane == 0) w = mbar_wait(acc_full + buf, use & 1u, abort_flag) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, w, 0) != 0;
      if (!ok) gave_up = WAIT_gemm_acc_full;
      tc_fence_after();
    };
    while (ok && walk.next(p, tile, k0, k1)) {
      const int sk_tile = TILES ? tile - p.n_full : tile, slot = TILES && sk_tile < 0 ? 0 : pair - div_small(sk_tile * p.kbu, p.inv_upc);
      const int ct = TILES ? tile / p.n_tt : tile, tok0 = TILES ? (tile - ct * p.n_tt) * p.tile_t : 0, nt = min(p.tile_t, p.n_tok - tok0);
      const int c = ct * TC_BN + (int)rank * 128 + q * 32 + lane;
      float *dst = p.out + (long long)slot * p.slot_stride + (long long)tok0 * p.ld + c;
      if (FORM >= TC_X_TWO) {
        // token groups of 16: half 0 takes groups 0, 2, .., half 1 groups 1, 3, ..
        float run[128];
#pragma unroll
        for (int j = 0; j < 128; ++j) run[j] = 0.f;
        for (; k0 < k1; k0 += p.chain) {
          const uint32_t buf = fill & 1u;
          wait_full(buf, fill >> 1);
          ++fill;
          if (!ok) break;
          const uint32_t taddr = lane_addr + buf * 256u + (uint32_t)(half * 16);
#pragma unroll
          for (int g = 0; g < 8; ++g)
            if ((2 * g + half) * 16 < nt) {
              uint32_t r[16];
              tmem_ld16(taddr + (uint32_t)(g * 32), r);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) run[g * 16 + j] += __uint_as_float(r[j]);
            }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(done_bar + 8u * buf);
        }
        if (EPI != TC_EPI_STORE && sk_tile < 0) {
          // lanes l and l + 16 hold the two columns of a pair; each takes 8 of a group's 16 tokens
          const TcEpi &e = p.epi;
          const int a0 = (int)rank * 64 + q * 16 + (lane & 15), hi16 = lane >> 4;       // pair index in the tile
          int ya, yb;
          tc_pair_rows<EPI>(e, ct, a0, ya, yb);
          const int hd_log2 = EPI == TC_EPI_ROPE ? 31 - __clz(e.kv.hd) : 0, hh = ya >> hd_log2, i = ya - (hh << hd_log2), hkv = e.kv.hkv;
          const bool col_ok = EPI == TC_EPI_SILU ? ya < e.ff : hh < e.H + 2 * hkv;
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            if ((2 * g + half) * 16 >= nt) continue;                                    // (warp-uniform)
            // the 8 tokens from t0 on, in the column this lane holds
            const int t0 = (2 * g + half) * 16 + hi16 * 8;
            float va[8], vb[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float lo8 = run[g * 16 + j], hi8 = run[g * 16 + 8 + j];
              const float other = __shfl_xor_sync(0xffffffffu, hi16 ? lo8 : hi8, 16);
              va[j] = hi16 ? other : lo8; vb[j] = hi16 ? hi8 : other;
            }
            const int t = t0 + (lane & 7);                    // the token this lane stores
            const bool st = ok && col_ok && t < nt;
            if (EPI == TC_EPI_SILU) {
#pragma unroll
              for (int j = 0; j < 8; ++j) va[j] = va[j] / (1.f + __expf(-va[j])) * vb[j];
              tc_store8(va, lane, st, e.dst + (long long)(tok0 + t) * e.lay.row_stride + (ya & ~7), e.lay.lo_delta);
            } else {
              const int r0 = e.row0 + tok0 + t0, r = e.row0 + tok0 + t;
              const bool rot = hh < e.H + hkv, is_q = hh < e.H;
              const int v = rot ? 0 : 1;
              bf16 *d = !st ? e.dst
                        : is_q ? e.dst + (((long long)r * e.H + hh) << (hd_log2 + 1)) + (i & ~7)
                               : (bf16 *)e.kv.base + (v ? e.kv.kv_stride : 0) + e.kv.off(e.seq, r, hh - e.H - (v ? hkv : 0)) + (i & ~7);
              float2 cs[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) cs[j] = rot && t0 + j < nt ? e.rope_pos[(long long)(r0 + j) * (e.kv.hd >> 1) + i] : make_float2(1.f, 0.f);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float x = va[j], y = vb[j];
                va[j] = x * cs[j].x - y * cs[j].y;
                vb[j] = y * cs[j].x + x * cs[j].y;
              }
              tc_store8(va, lane, st, d, is_q ? e.kv.hd : 0);
              tc_store8(vb, lane, st, d + (e.kv.hd >> 1), is_q ? e.kv.hd : 0);
            }
          }
        } else if (ok && c < p.N) {
#pragma unroll
          for (int g = 0; g < 8; ++g)
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int t = (2 * g + half) * 16 + j;
              if (t < nt) dst[(long long)t * p.ld] = run[g * 16 + j];
            }
        }
      } else {
        const uint32_t buf = fill & 1u;
        wait_full(buf, fill >> 1);
        ++fill;
        if (!ok) break;
        const uint32_t taddr = lane_addr + buf * 256u;
        // the parts of a sum: accumulators, and within each (CONCAT) the high and the low plane's columns
        const int n_part = p.n_sub * (FORM == TC_X_CONCAT ? 2 : 1), part_n = FORM == TC_X_CONCAT ? p.tile_t : p.mma_n;
#pragma unroll 1
        for (int t0 = half * 16; t0 < nt; t0 += 32) {
          float v[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = 0.f;
#pragma unroll 1
          for (int i = 0; i < n_part; ++i) {
            uint32_t r[16];
            tmem_ld16(taddr + (uint32_t)(i * part_n + t0), r);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += __uint_as_float(r[j]);
          }
          if (c < p.N) {
            float *d = dst + (long long)t0 * p.ld;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              if (t0 + j < nt) *d = v[j];
              d += p.ld;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && fill + 1u < n_seg) mbar_arrive_cluster(done_bar + 8u * buf);      // the accumulator is filled again
      }
    }
  }
  if (gave_up && lane == 0) wait_expired(p.status, gave_up, abort_flag, (int)(rank ^ 1u));
  drain_if_aborted(abort_flag);
  __syncwarp();
  if (warp == 1) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");     // the pair's too: both have allocated
  tc_fence_before();
  __syncthreads();
  cluster_sync_relaxed();                      // neither CTA leaves while its peer may still signal it or read its operands
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    __syncwarp();
  }
  // Freeing is an act of the pair too: both have freed before either leaves.  (0.2 to 0.5 % of a round.)
  cluster_sync_relaxed();
}

// ------------------------------------------------------------------------------------------ host side

struct GemmTcPlan {
  PFN_cuTensorMapEncodeTiled_v12000 encode;
  int n_sms;
  int max_smem;
  int use_pdl;
  int *status;
  std::map<std::tuple<const void *, int, int, int>, CUtensorMap> maps;
};

static inline const char *gemm_tc_plan_init(GemmTcPlan *pl, int *status, int use_pdl) {
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult qr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr) != cudaSuccess || !fn)
    return "cuTensorMapEncodeTiled not available";
  pl->encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&pl->n_sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&pl->max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  bool ok = true;
  auto raise = [&](auto *kernel) { ok = ok && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, pl->max_smem) == cudaSuccess; };
  raise(k_gemm_tc<TC_X_ONE, TC_EPI_STORE>); raise(k_gemm_tc<TC_X_CONCAT, TC_EPI_STORE>); raise(k_gemm_tc<TC_X_TWO, TC_EPI_STORE>);
  raise(k_gemm_tc<TC_X_TILES, TC_EPI_STORE>); raise(k_gemm_tc<TC_X_TILES, TC_EPI_SILU>); raise(k_gemm_tc<TC_X_TILES, TC_EPI_ROPE>);
  if (!ok)
    return "cannot raise the dynamic shared memory limit";
  pl->status = status;
  pl->use_pdl = use_pdl;
  return nullptr;
}

#define TC_TOKENS 256           // most tokens of a tile

static inline bool gemm_tc_supported(int N, int K) {
  return K % TC_BK == 0 && K >= TC_BK && N % 8 == 0 && N >= 8;
}

// bf16 row-major [rows][K] matrix, box = 64 x box_rows, 128-byte swizzle.  Rows of a box that lie
// beyond `rows` read as zero.
// The encoded map is copied to *out: the cache may drop its entries at any later call.
static inline bool tc_map(GemmTcPlan *pl, const void *ptr, int rows, int K, int box_rows, CUtensorMap *out) {
  auto key = std::make_tuple(ptr, rows, K, box_rows);
  auto it = pl->maps.find(key);
  if (it != pl->maps.end()) { *out = it->second; return true; }
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  cuuint32_t box[2] = {TC_BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = pl->encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (pl->maps.size() > 8192) pl->maps.clear();
  pl->maps[key] = m;
  *out = m;
  return true;
}

// How a launch of `rows` token rows is cut (see the head of the file).
struct TcSplit { int n_tt, tile_t, n_pairs, n_waves, kbu, sk_units, upc, slots; };
static inline TcSplit gemm_tc_split(int n_sms, int rows, int N, int K) {
  TcSplit t;
  const int KB = K / TC_BK;
  t.n_tt = (rows + TC_TOKENS - 1) / TC_TOKENS;
  // tokens in 16s (the N of an MMA over both CTAs); up to 128 rows both planes share an MMA, so 8s do
  t.tile_t = t.n_tt > 1 || rows > 128 ? ((rows + t.n_tt - 1) / t.n_tt + 15) & ~15 : (rows + 7) & ~7;
  const int pairs = n_sms / 2 > 0 ? n_sms / 2 : 1, tiles = (N + TC_BN - 1) / TC_BN * t.n_tt;
  // full waves, less one when the rest alone is so small that a tile would be shared by many pairs
  t.n_waves = t.n_tt > 1 ? tiles / pairs : 0;
  if (t.n_waves && tiles % pairs && 4 * (tiles % pairs) < pairs) --t.n_waves;
  // Few tiles: every pair a share of one tile, where that is at most TC_EVEN units longer than dealing all units out evenly.
  // A share that crosses a tile's end empties two accumulators, and its tiles have one or two more slots for
  // the next kernel to read.  Rounds, spread -> whole: SmolVLM-shaped 2321 -> 2222 us, LLaVA-7B-shaped 4719 -> 4701, four of it
  // 9458 -> 9370, Pixtral- 7992 -> 7924, Gemma-shaped 10984 -> 10860; five units (172 panels: 43 instead of 38) lose 7 us.
  // Between a half and two thirds as many tiles as pairs, three pairs per two tiles in the same way (LLaVA-7B-shaped QKV, 48 tiles: the
  // rotary kernel adds two slots instead of three): round 4711 -> 4669 us, chain 4318 -> 4279, four sequences 9435 -> 9324.
  const int left = tiles - t.n_waves * pairs, share = left > 0 ? pairs / left : 0;      // whole pairs per tile
  const bool three = share == 1 && 3 * left <= 2 * pairs && KB > (KB + 2) / 3 * 2;        // three pairs per two tiles, no share empty
  const int spread = (left * KB + pairs - 1) / pairs, even = share > 1 ? (KB + share - 1) / share : three ? (KB + 2) / 3 * 2 : 0;
  const bool whole = even && even <= spread + TC_EVEN;
  t.upc = whole ? even : left ? spread : 1;
  t.kbu = !whole ? KB : three ? even / 2 * 3 : (KB + even - 1) / even * even;
  t.sk_units = left * t.kbu;
  t.n_pairs = t.n_waves ? pairs : (t.sk_units + t.upc - 1) / t.upc;
  t.slots = whole ? (t.kbu + t.upc - 1) / t.upc : left ? (KB + t.upc - 1) / t.upc + 1 : 1;      // a tile is shared by at most as many pairs
  return t;
}
// Where the partial sums lie.  One token tile or no full wave: slots of rows x N.  Behind full waves only the columns
// from c0 on have further slots, and a row holds them behind its N columns: five slots of everything were
// 0.8 GB at 1280 rows of a gate/up projection of 30720 columns, this is 0.2.
struct TcOut { long long slot_stride, floats; int ld; };
static inline TcOut gemm_tc_out(const TcSplit &t, int rows, int N) {
  TcOut o;
  o.ld = N; o.slot_stride = (long long)rows * N;
  if (t.n_waves) {
    const int left = N - t.n_pairs * t.n_waves / t.n_tt * TC_BN;
    o.ld = N + (t.slots - 1) * left; o.slot_stride = left;
  }
  o.floats = t.n_waves ? (long long)rows * o.ld : t.slots * o.slot_stride;
  return o;
}
// Floats a launch of up to `rows` rows may write on a device of up to n_sms SMs (the split follows the SMs, not monotonically).
static inline long long gemm_tc_room(int n_sms, int rows, int N, int K) {
  long long most = 0;
  for (int r = TC_TOKENS; r < rows + TC_TOKENS; r += TC_TOKENS)
    for (int sms = 2; sms <= n_sms; sms += 2) {
      const int n = r < rows ? r : rows;
      const long long f = gemm_tc_out(gemm_tc_split(sms, n, N, K), n, N).floats;
      if (f > most) most = f;
    }
  return most;
}

// Enqueue one GEMM of `rows` token rows.
//   X: bf16, row-major, K columns.  TC_X_PLAIN (up to 128 rows): row t = token t.  TC_X_PLANAR: row t =
//   high part, row lo_rows + t = low part.
// *g receives the descriptor consumers read the result through.  Returns false if the launch could
// not be made.
//   epi / e: a fused epilogue (launches of several token tiles only).  The sums of the stream-K tiles (n_full and up) then
//   lie in pairs: N counts 256 columns per column tile of 128 pairs.
static inline bool gemm_tc_launch(GemmTcPlan *pl, cudaStream_t stream, const void *W, const void *X, int x_mode, int lo_rows,
                                  int rows, int N, int K, float *out, long long out_floats, GemmOut *g, int epi = TC_EPI_STORE, const TcEpi *e = nullptr) {
  const int w_rows = N;
  if (epi == TC_EPI_SILU) N = (e->ff + 127) / 128 * TC_BN;
  if (epi == TC_EPI_ROPE) N = (N + TC_BN - 1) / TC_BN * TC_BN;
  if (epi != TC_EPI_STORE && rows <= TC_TOKENS) return false;
  if (rows < 1 || (x_mode == TC_X_PLAIN && rows > 128)) return false;
  const TcSplit t = gemm_tc_split(pl->n_sms, rows, N, K);
  if (t.sk_units + t.kbu >= 1 << 21) return false;          // div_small
  TcParams p;
  p.n_tok = rows; p.lo_rows = lo_rows;
  p.N = N; p.KB = K / TC_BK;
  p.n_pairs = t.n_pairs; p.n_waves = t.n_waves; p.n_full = t.n_pairs * t.n_waves; p.sk_units = t.sk_units; p.upc = t.upc;
  p.n_tt = t.n_tt; p.tile_t = t.tile_t;
  p.kbu = t.kbu; p.inv_kbu = 1.f / (float)t.kbu; p.inv_upc = 1.f / (float)p.upc;
  // N of an MMA is a multiple of 16 and each CTA stages half of it (8-row groups)
  int form;
  if (x_mode == TC_X_PLAIN) { form = TC_X_ONE; p.tile_t = p.mma_n = (rows + 15) & ~15; }
  else if (rows <= 128) { form = TC_X_CONCAT; p.mma_n = 2 * p.tile_t; }
  else { form = p.n_tt > 1 ? TC_X_TILES : TC_X_TWO; p.mma_n = p.tile_t; }
  // Every eight MMAs of a chain (a panel) add 1.7e-7 of bias to sums of one sign, and emptying an accumulator costs time: at most
  // eight panels, fewer where K is small, so that no width is less exact than when 148 CTAs shared the panels.  K 2048, 200
  // rows, relative L2 against float64: eight panels 2.68e-6, four 2.51e-6 (as before); four everywhere: prompts 3 % slower.
  p.chain = p.KB / 8 < 4 ? 4 : p.KB / 8 > 8 ? 8 : p.KB / 8;
  p.n_sub = p.mma_n <= 64 ? 4 : p.mma_n <= 128 ? 2 : 1;
  p.out = out;
  const TcOut o = gemm_tc_out(t, rows, N);
  p.slot_stride = o.slot_stride; p.ld = o.ld;
  if (o.floats > out_floats) return false;
  CUtensorMap mw, mx;
  const int x_rows = x_mode == TC_X_PLANAR ? lo_rows + rows : rows;
  const int x_box = form == TC_X_CONCAT ? p.tile_t : p.mma_n / 2;
  if (!tc_map(pl, W, w_rows, K, epi == TC_EPI_STORE ? 128 : 16, &mw) || !tc_map(pl, X, x_rows, K, x_box, &mx)) return false;
  g->base = p.out; g->slot_stride = p.slot_stride; g->ld = o.ld; g->kb = t.kbu; g->n_full = p.n_full; g->n_tt = p.n_tt;
  g->inv_upc = p.inv_upc; g->inv_tile = p.n_tt > 1 ? 1.f / (float)p.tile_t : 0.f;
  // Stages of two panels halve the waits and commits per panel (61 rows, 12288 x 4096: 22.2 -> 20.9 us) as
  // long as five fit; where a token panel is larger than a weight panel (244 rows: 38.3 against 39.4 us) the
  // rings are deeper with one
  const int xpanel = x_box * 128 * (form >= TC_X_TWO ? 2 : 1);
  p.wp = xpanel <= TC_WPANEL / 2 ? 2 : 1;
  if (e) p.epi = *e;
  if (epi != TC_EPI_STORE) p.wp = 1;
  const int xstage = p.wp * xpanel, wstage = p.wp * TC_WPANEL;
  // a few KB stay free for the blocks of the row kernel that waits beside this launch (1 KB each)
  const int room = pl->max_smem - 2048 - 4096;
  p.x_stages = xpanel < TC_WPANEL ? 6 / p.wp : xpanel == TC_WPANEL ? 4 : room / (xstage + wstage);
  p.w_stages = (room - p.x_stages * xstage) / wstage;
  if (p.w_stages > TC_MAX_STAGES) p.w_stages = TC_MAX_STAGES;
  if (p.w_stages < 2 || p.x_stages < 2) return false;
  p.status = pl->status;
  size_t smem = (size_t)p.w_stages * wstage + (size_t)p.x_stages * xstage + 2048;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * p.n_pairs); cfg.blockDim = dim3(TC_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pl->use_pdl ? 1 : 0;
  auto *kernel = form == TC_X_CONCAT ? k_gemm_tc<TC_X_CONCAT, TC_EPI_STORE> : form == TC_X_TWO ? k_gemm_tc<TC_X_TWO, TC_EPI_STORE> : form == TC_X_ONE ? k_gemm_tc<TC_X_ONE, TC_EPI_STORE>
               : epi == TC_EPI_SILU ? k_gemm_tc<TC_X_TILES, TC_EPI_SILU> : epi == TC_EPI_ROPE ? k_gemm_tc<TC_X_TILES, TC_EPI_ROPE> : k_gemm_tc<TC_X_TILES, TC_EPI_STORE>;
  return cudaLaunchKernelEx(&cfg, kernel, mw, mx, p) == cudaSuccess;
}

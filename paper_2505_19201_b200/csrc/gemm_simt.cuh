// Plain CUDA-core GEMM  out[r][c] = sum_k X[r][k] W[c][k]  with fp32 accumulation.
// It serves the fp32 (toy) configuration, whose tolerances rule out tf32 tensor-core
// rounding; bf16 configurations always take the tensor-core kernel.
//
// At these sizes (1..96 rows, K = 256 or 1024, weights in L2) a launch is a chain of latencies, so the work
// is cut into many short warps: a warp owns TR rows x 4 columns and one slice of k, its lanes hold four
// consecutive k each, and all loads of a 128-k step are in flight at once.  The lanes' sums meet in a halving
// butterfly (31 shuffles leave output i in lane i), the slices in shared memory, in a fixed order.  The
// first step's weights are fetched before the grid dependency resolves.  Mean launch of the toy request (539
// launches, 1..96 rows): 25.6 us with 64 x 64 block tiles and 16-k steps, 2.8 us so.
#pragma once
#include "common.cuh"

#define SG_TC 4          // columns per warp
#define SG_WARPS 8
#define SG_STEP 128      // k per step of a warp

// Four consecutive elements of a row of K, zero beyond its end.  VEC: 16-byte aligned rows, K a multiple of 4.
template <bool VEC>
__device__ __forceinline__ float4 sg_ld(const float *row, int k, int K) {
  if (k >= K) return make_float4(0.f, 0.f, 0.f, 0.f);
  if (VEC) return ld_f4(row + k);
  return make_float4(row[k], k + 1 < K ? row[k + 1] : 0.f, k + 2 < K ? row[k + 2] : 0.f, k + 3 < K ? row[k + 3] : 0.f);
}

// Halving butterfly over a warp: after the step of offset O a lane keeps the half of the N values its bit O
// selects; the lanes of one remaining value add it up.
template <int O, int N, int NA>
__device__ __forceinline__ void sg_reduce(float (&acc)[NA], int lane) {
  if constexpr (O > 0) {
    if constexpr (N > 1) {
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        const float send = (lane & O) ? acc[i] : acc[N / 2 + i], mine = (lane & O) ? acc[N / 2 + i] : acc[i];
        acc[i] = mine + __shfl_xor_sync(0xffffffffu, send, O);
      }
      sg_reduce<O / 2, N / 2>(acc, lane);
    } else {
      acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], O);
      sg_reduce<O / 2, 1>(acc, lane);
    }
  }
}

// grid (ceil(N / (4 * 8 / ks)), ceil(rows / TR)); ks k-slices (1, 2, 4 or 8) per output tile.
template <int TR, bool VEC>
__global__ void __launch_bounds__(SG_WARPS * 32)
k_gemm_simt(const float *__restrict__ X, const float *__restrict__ W, float *__restrict__ out, int rows,
            int N, int K, int ldo, int ks) {
  __shared__ float part[SG_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slice = warp & (ks - 1), c0 = (blockIdx.x * (SG_WARPS / ks) + warp / ks) * SG_TC, r0 = blockIdx.y * TR;
  const int k_first = slice * SG_STEP + lane * 4, k_step = ks * SG_STEP;
  float4 w[SG_TC];
#pragma unroll
  for (int c = 0; c < SG_TC; ++c) w[c] = sg_ld<VEC>(W + (long long)min(c0 + c, N - 1) * K, k_first, K);
  kernel_entry(TR_k_gemm_simt);
  float acc[TR * SG_TC] = {};
  for (int k = k_first; k - lane * 4 < K; k += k_step) {
    float4 x[TR];
#pragma unroll
    for (int r = 0; r < TR; ++r) x[r] = sg_ld<VEC>(X + (long long)min(r0 + r, rows - 1) * K, k, K);
#pragma unroll
    for (int r = 0; r < TR; ++r)
#pragma unroll
      for (int c = 0; c < SG_TC; ++c) {
        float a = acc[r * SG_TC + c];
        a = fmaf(x[r].x, w[c].x, a); a = fmaf(x[r].y, w[c].y, a); a = fmaf(x[r].z, w[c].z, a); a = fmaf(x[r].w, w[c].w, a);
        acc[r * SG_TC + c] = a;
      }
    if (k - lane * 4 + k_step < K) {
#pragma unroll
      for (int c = 0; c < SG_TC; ++c) w[c] = sg_ld<VEC>(W + (long long)min(c0 + c, N - 1) * K, k + k_step, K);
    }
  }
  constexpr int NA = TR * SG_TC;
  sg_reduce<16, NA>(acc, lane);
  float v = acc[0];
  if (ks > 1) {
    part[warp][lane] = v;
    __syncthreads();
    if (slice) return;
    for (int i = 1; i < ks; ++i) v += part[warp + i][lane];
  }
  const int idx = lane * NA / 32, r = r0 + idx / SG_TC, c = c0 + idx % SG_TC;
  if (lane * NA % 32 == 0 && r < rows && c < N) out[(long long)r * ldo + c] = v;
}

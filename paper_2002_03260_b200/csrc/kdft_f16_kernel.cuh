// What the KDFT kernels with fp16 pieces share: the pieces, the stage sizes and the reduction that finds the scale.
//
// The split x = hi + lo, W = W_hi + W_lo uses fp16 pieces (11-bit significands, like TF32) and
// tcgen05.mma kind::f16, which contracts K = 16 per instruction at twice the TF32 rate: half the MMAs and half
// the table bytes for the same three products (hi*hi, lo*hi, hi*lo) and the same fp32 accumulation.
//
// fp16 has a narrow exponent range, so the operands are scaled by powers of two (exact):
//   * the table holds 1024 * W (entries in [-1024, 1024]; the lo piece of all but vanishing entries stays normal);
//   * the data is multiplied by 2^k with k chosen from the largest input magnitude, which every pass records for
//     its successor (amax_out) and a small reduction kernel provides for the first pass; the largest scaled value
//     lies in [2^13, 2^14).  An entry more than 2^18 below the largest loses relative precision (its lo piece
//     becomes subnormal: absolute error 2^-25 of a scaled unit, i.e. 2^-38 of the largest entry), which is far
//     below fp32 rounding in the norm-wise sense the transform is judged in.
//   The epilogue multiplies by 2^-10 * 2^-k (and 1/n for a scaled inverse).
// A stage covers 64 reals of the contraction (128-byte rows of the fp16 table); the raw fp32 data stage is 32 KB.
#pragma once
#include <cuda_fp16.h>
#include "kdft_kernel.cuh"
#include "split_f16.cuh"

namespace dft3d {

constexpr int kF16BlockK = 64;          // reals of the contraction per pipeline stage
constexpr int kF16BytesStageA = kTileM * kF16BlockK * 4;   // raw fp32 data of one stage: 32 KB

struct KdftF16Params {
  int k2, bn, n_tiles, chunk_kb;        // as KdftParams; chunk_kb counts 64-real stages
  long long m_tiles, rows, batches, C;
  int lpb, bpt;
  long long c_tiles;
  float* out;
  unsigned int* status;
  long long* profile;
  float out_mul;                        // 2^-10, times 1/n for a scaled inverse
  int n_group;                          // table panels (n-tiles) that are live at a time; the tiles go
                                        // panel group by panel group, all lines within a group (0 or n_tiles: one group)
  const unsigned int* amax_in;          // float bits: largest |input| (an upper bound is enough)
  unsigned int* amax_out;               // float bits: receives the largest |output| (atomic max)
  WaitControl wc;
};

// |v|, or 0 for an infinity or NaN: a line that holds one has no finite result whatever the scale, and the other lines
// need the scale of the finite data
__device__ __forceinline__ float finite_magnitude(float v) {
  const float a = fabsf(v);
  return a <= 3.402823466e38f ? a : 0.0f;
}

// Largest finite magnitude of a float array -> words[0]; words[1..clear] (those of the passes that follow) are set to zero.
// Every block leaves its maximum in `scratch`, the last one to finish reduces them: no word has to be cleared before the
// launch.  scratch[0] counts the finished blocks and wraps to zero by itself.
constexpr int kAmaxThreads = 256, kAmaxUnroll = 4;
__global__ void __launch_bounds__(kAmaxThreads) amax_kernel(const float4* x, long long n4, unsigned int* words, int clear,
                                                            unsigned int* scratch) {
  __shared__ unsigned int part[kAmaxThreads / 32];
  __shared__ bool last;
  ptx::griddep_launch();
  ptx::griddep_wait();
  float m = 0.0f;
  const long long step = (long long)gridDim.x * kAmaxThreads;
  for (long long i = blockIdx.x * (long long)kAmaxThreads + threadIdx.x; i < n4; i += step * kAmaxUnroll) {
    float4 v[kAmaxUnroll];
#pragma unroll
    for (int u = 0; u < kAmaxUnroll; ++u) v[u] = i + u * step < n4 ? x[i + u * step] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kAmaxUnroll; ++u)
      m = fmaxf(fmaxf(m, fmaxf(finite_magnitude(v[u].x), finite_magnitude(v[u].y))),
                fmaxf(finite_magnitude(v[u].z), finite_magnitude(v[u].w)));
  }
  // non-negative floats compare like their bits
  unsigned int r = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kAmaxThreads / 32; ++w) r = max(r, part[w]);
    scratch[1 + blockIdx.x] = r;
    __threadfence();
    last = atomicInc(scratch, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  r = 0;
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += kAmaxThreads) r = max(r, __ldcg(scratch + 1 + b));
  r = __reduce_max_sync(0xffffffffu, r);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kAmaxThreads / 32; ++w) r = max(r, part[w]);
    words[0] = r;
    for (int w = 1; w <= clear; ++w) words[w] = 0;
  }
}

}  // namespace dft3d

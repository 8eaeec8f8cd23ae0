// FP64 block and grid reductions shared by the kernel files: warp shuffles, a block
// reduction of NV values (sum, max or min), and the last-block pattern (every block writes
// its partials and takes a ticket; the last block reduces the partials in block order, so the
// result is bit-reproducible).
#pragma once
#include <math.h>

#include "otgb_internal.cuh"

namespace otgb {

// doubles as integers of the same order (not for NaN), and tests on the bits: comparisons on the
// integer pipe
__device__ __forceinline__ long long ordered_bits(long long b) {
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ long long ordered_key(double x) {
  return ordered_bits(__double_as_longlong(x));
}
__device__ __forceinline__ double key_value(long long k) {
  return __longlong_as_double(ordered_bits(k));
}
__device__ __forceinline__ bool finite_key(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool nan_key(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// ---------------------------------------------------------------------------------------
// block reductions
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Reduce NV values per thread over the block (kind: 0 sum, 1 max, 2 min per value);
// result valid in thread 0.  Needs blockDim.x a multiple of 32 and <= 1024.
template <int NV>
__device__ void block_reduce(double (&v)[NV], const int (&kind)[NV]) {
  __shared__ double red[32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int a = 0; a < NV; ++a)
    v[a] = kind[a] == 0 ? warp_sum(v[a]) : (kind[a] == 1 ? warp_max(v[a]) : warp_min(v[a]));
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int a = 0; a < NV; ++a) red[wid][a] = v[a];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      double init = kind[a] == 0 ? 0.0 : (kind[a] == 1 ? -INFINITY : INFINITY);
      double x = lane < nw ? red[lane][a] : init;
      v[a] = kind[a] == 0 ? warp_sum(x) : (kind[a] == 1 ? warp_max(x) : warp_min(x));
    }
  }
  __syncthreads();
}

// Sums of NV <= 16 values per thread over a block of 256: the lanes of a warp exchange halves of
// the values, so that a warp takes NP + 4 - log2(NP) FP64 additions (NP: NV rounded up to a power
// of two) where a shuffle tree per value takes 5 NV; FP64 starts one warp instruction per 16
// clocks and SM here.  Thread 8 a (a < NV) receives sum a; true in those threads.
template <int NV>
__device__ bool block_fold(const double (&v)[NV], double& sum) {
  constexpr int NP = NV > 8 ? 16 : (NV > 4 ? 8 : (NV > 2 ? 4 : NV));
  __shared__ double red[8][NP];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double x[NP];
#pragma unroll
  for (int a = 0; a < NP; ++a) x[a] = a < NV ? v[a] : 0.0;
  int o = 16;
#pragma unroll
  for (int h = NP / 2; h > 0; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int a = 0; a < h; ++a)
      x[a] = (up ? x[a + h] : x[a]) + __shfl_xor_sync(0xffffffffu, up ? x[a] : x[a + h], o);
  }
#pragma unroll
  for (; o > 0; o /= 2) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
  if (lane % (32 / NP) == 0) red[wid][lane / (32 / NP)] = x[0];
  __syncthreads();
  const int a = threadIdx.x >> 3;
  if (wid * 4 >= NV) return false;  // (whole warps)
  double s = a < NV ? red[threadIdx.x & 7][a] : 0.0;
  s += __shfl_xor_sync(0xffffffffu, s, 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  sum = s;
  return (threadIdx.x & 7) == 0 && a < NV;
}

// Write the block's partials, take a ticket; returns true in the (whole) last block,
// after which `partials` of all blocks are visible.
template <int NV>
__device__ bool publish_partials(const double (&v)[NV], double* partials, unsigned int* ticket) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    const size_t bid = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    for (int a = 0; a < NV; ++a) partials[bid * NV + a] = v[a];
    __threadfence();
    unsigned int nb = gridDim.x * gridDim.y;
    unsigned int k = atomicAdd(ticket, 1u);
    last = (k == nb - 1);
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// In the last block: reduce the per-block partials in block order (each thread a strided
// subset, then a block reduction).
template <int NV>
__device__ void reduce_partials(double (&v)[NV], const int (&kind)[NV], const double* partials,
                                unsigned int nb) {
#pragma unroll
  for (int a = 0; a < NV; ++a) v[a] = kind[a] == 0 ? 0.0 : (kind[a] == 1 ? -INFINITY : INFINITY);
  for (unsigned int b = threadIdx.x; b < nb; b += blockDim.x) {
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      double x = ((volatile const double*)partials)[(size_t)b * NV + a];
      v[a] = kind[a] == 0 ? v[a] + x : (kind[a] == 1 ? fmax(v[a], x) : fmin(v[a], x));
    }
  }
  block_reduce<NV>(v, kind);
}

}  // namespace otgb

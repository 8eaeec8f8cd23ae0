// Training of the learned warm start's network (FP32): loss and gradient of one minibatch, and
// the Adam step.  The network 16 -> 128 -> 128 -> 128 -> 1 acts row by row, so one kernel takes a
// block's rows through the forward and the backward pass in shared memory and adds up the weight
// gradients in registers; a second one adds the blocks' sums.
//
// What bounds it: FP32 FMAs, 102,600 per row (35,000 forward, 33,000 for the data gradients,
// 35,000 for the weight gradients): 83 us for 32,768 rows at 128 FMA per clock and SM.  Layout:
//   - W1 and W2 stay in shared memory (rows of 132 floats: a warp reads 16 bytes of 32 rows, or 32
//     consecutive floats of one, without bank conflicts), with the activations A0, A1 and one
//     gradient buffer of R = 8 RW rows; a pair of warps owns RW rows through all layers, a lane
//     two of their columns, so the layers of a pair follow each other without a block barrier;
//     16 warps of 128 registers, since 8 of 255 left half of the issue slots empty;
//   - the products run on packed FP32 pairs (fma.rn.f32x2): pairs along k in the layers, whose
//     operands come out of 16-byte loads as pairs, and along the second index in the weight
//     gradients, of which a thread keeps 8 x 4 of each 128 x 128 matrix for the block's lifetime;
//   - per 4 k and warp a layer reads 8 wavefronts of weights and RW of activations for 32 RW
//     FMAs: RW = 7 (56 rows, all of shared memory) balances the two, 4 and 2 serve small batches,
//     where the number of blocks counts more.
// Measured on one GB300 (gradient call, us, with the gradient in pinned host memory; before: 25
// launches of 64 x 64-tile GEMMs through global memory, column sums and a one-thread loss sum):
//   32,768 rows 1937 -> 236, 1,024 rows 723 -> 56.
#include <math.h>
#include <stdint.h>

#include "f32x2.cuh"
#include "otgb_internal.cuh"
#include "spectral.cuh"  // prepare_launch

namespace otgb {
namespace {

using pair::fma2;
using pair::pk;
using pair::u64;
using pair::upk;

constexpr int K = OTGB_WS_K, H = OTGB_WS_H;
constexpr int HH = H * H, WS = H + 4;  // shared-memory row stride of W1, W2
// offsets in the flat parameter vector
constexpr int oW0 = 0, ob0 = oW0 + H * K, oW1 = ob0 + H, ob1 = oW1 + HH, oW2 = ob1 + H,
              ob2 = oW2 + HH, ow3 = ob2 + H, ob3 = ow3 + H;
constexpr int kPartStride = (ob3 + 1 + 3) / 4 * 4;  // floats of one block's partial sums
constexpr int kThreads = 512, kPairs = kThreads / 64;

template <int RW>
struct Smem {
  static constexpr int R = kPairs * RW;
  float w[2][H * WS];         // W1, W2
  float a0[R * H], a1[R * H], d[R * H];
  float x[2][R * K], t[2][R];  // this chunk's rows and the next one's
  float w3[H];
  float y[2][R];               // the output's two column halves
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src));
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src));
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ float pair_sum(u64 v) {
  float lo, hi;
  upk(v, lo, hi);
  return lo + hi;
}

// acc[r][c] += sum_k a[r][k] W[col + 32 c][k] (the forward product), a: the pair's RW rows
template <int RW>
__device__ __forceinline__ void mul_rows(const float* a, const float* W, int col,
                                         u64 (&acc)[RW][2]) {
  const float* wl = W + col * WS;
#pragma unroll 2
  for (int k = 0; k < H; k += 4) {
    ulonglong2 w[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) w[c] = *reinterpret_cast<const ulonglong2*>(wl + 32 * c * WS + k);
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(a + r * H + k);
#pragma unroll
      for (int c = 0; c < 2; ++c) acc[r][c] = fma2(x.y, w[c].y, fma2(x.x, w[c].x, acc[r][c]));
    }
  }
}
// acc[r][c] += sum_k a[r][k] W[k][col + 32 c] (the data gradient)
template <int RW>
__device__ __forceinline__ void mul_cols(const float* a, const float* W, int col,
                                         u64 (&acc)[RW][2]) {
  const float* wl = W + col;
#pragma unroll 2
  for (int k = 0; k < H; k += 4) {
    u64 w[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      w[c][0] = pk(wl[k * WS + 32 * c], wl[(k + 1) * WS + 32 * c]);
      w[c][1] = pk(wl[(k + 2) * WS + 32 * c], wl[(k + 3) * WS + 32 * c]);
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(a + r * H + k);
#pragma unroll
      for (int c = 0; c < 2; ++c) acc[r][c] = fma2(x.y, w[c][1], fma2(x.x, w[c][0], acc[r][c]));
    }
  }
}
// g[i][j] += sum_r a[r][4 lane + i] d[r][8 wid + 2 j, + 1]
__device__ __forceinline__ void add_outer(const float* d, const float* a, int rows, int wid,
                                          int lane, u64 (&g)[4][4]) {
#pragma unroll 2
  for (int r = 0; r < rows; ++r) {
    const float4 x = *reinterpret_cast<const float4*>(a + r * H + 4 * lane);
    const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(d + r * H + 8 * wid),
                     q = *reinterpret_cast<const ulonglong2*>(d + r * H + 8 * wid + 4);
    const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const u64 xx = pk(xv[i], xv[i]);
      g[i][0] = fma2(xx, p.x, g[i][0]);
      g[i][1] = fma2(xx, p.y, g[i][1]);
      g[i][2] = fma2(xx, q.x, g[i][2]);
      g[i][3] = fma2(xx, q.y, g[i][3]);
    }
  }
}
// a thread's 8 x 4 of a weight gradient to out (rows 8 wid + ., columns 4 lane + .)
__device__ __forceinline__ void store_outer(float* out, int wid, int lane, const u64 (&g)[4][4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) upk(g[i][j], lo[i], hi[i]);
    float4* p = reinterpret_cast<float4*>(out + (8 * wid + 2 * j) * H + 4 * lane);
    p[0] = make_float4(lo[0], lo[1], lo[2], lo[3]);
    p[H / 4] = make_float4(hi[0], hi[1], hi[2], hi[3]);
  }
}
// sum of column tid % 128 over every fourth row
__device__ __forceinline__ float col_sum(const float* d, int rows, int tid) {
  float s = 0.f;
  for (int r = tid >> 7; r < rows; r += 4) s += d[r * H + (tid & 127)];
  return s;
}

__device__ __forceinline__ void silu(float z, float& a, float& da) {
  const float s = 1.0f / (1.0f + expf(-z));
  a = z * s;
  da = s * (1.0f + z * (1.0f - s));
}

// The gradient sums of rows [blockIdx.x rpb, + rpb) of the minibatch, in chunks of `chunk` <=
// 8 RW rows, to part[blockIdx.x], and their squared errors' sum to loss_part.  scr: SiLU' of the
// first two layers (written and read by the same thread).
template <int RW>
__global__ void __launch_bounds__(kThreads, 1)
    k_ws_train(const float* __restrict__ params, const float* __restrict__ X,
               const float* __restrict__ t, const long long* __restrict__ idx, int B, int rpb,
               int chunk, float* __restrict__ scr, float* __restrict__ part,
               double* __restrict__ loss_part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<RW>& S = *reinterpret_cast<Smem<RW>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int pr = wid >> 1, col = 64 * (wid & 1) + lane;  // the warp's pair, the lane's columns
  auto pair_sync = [&]() {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + pr) : "memory");
  };
  const int r0 = blockIdx.x * rpb, r1 = min(B, r0 + rpb);
  // stage row c0 + row of the minibatch (thread 4 row + q: 16 bytes of it); rows past the
  // chunk's end are zero and drop out of every sum below
  auto row_of = [&](int c0) -> long long {
    const int r = c0 + (tid >> 2);
    return (tid >> 2) < chunk && r < r1 ? idx[r] : -1;
  };
  auto stage_row = [&](int c0, long long src, int b) {
    const int row = tid >> 2, q = tid & 3;
    if (row >= Smem<RW>::R) return;
    if (src >= 0) {
      cp_async16(&S.x[b][row * K + 4 * q], X + src * K + 4 * q);
      if (q == 0) cp_async4(&S.t[b][row], t + src);
    } else {
      *reinterpret_cast<float4*>(&S.x[b][row * K + 4 * q]) = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q == 0) S.t[b][row] = 0.f;
    }
  };
  stage_row(r0, row_of(r0), 0);
  for (int e = tid; e < 2 * HH / 4; e += kThreads) {
    const int m = e / (HH / 4), f = e % (HH / 4);  // matrix, float4 of it
    cp_async16(&S.w[m][(f / (H / 4)) * WS + 4 * (f % (H / 4))], params + (m ? oW2 : oW1) + 4 * f);
  }
  if (tid < H) S.w3[tid] = params[ow3 + tid];
  const float b3 = params[ob3];

  u64 g1[4][4], g2[4][4];  // dW1, dW2
  float g0[4];             // dW0: unit tid % 128, inputs 4 (tid / 128) .. + 3
  float gw3[2] = {0.f, 0.f}, gb[3] = {0.f, 0.f, 0.f}, gb3 = 0.f;
  double loss = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g0[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) g1[i][j] = g2[i][j] = 0ull;
  }

  float* sc0 = scr + ((size_t)blockIdx.x * 2 * RW * 2) * kThreads + tid;
  float* sc1 = sc0 + RW * 2 * kThreads;
  float *A0 = S.a0 + pr * RW * H, *A1 = S.a1 + pr * RW * H, *D = S.d + pr * RW * H;
  int b = 0;
  for (int c0 = r0; c0 < r1; c0 += chunk, b ^= 1) {
    const int rows = min(chunk, r1 - c0);  // (block-uniform)
    cp_async_wait();
    __syncthreads();  // this chunk's rows; the last chunk's readers of D
    const long long next = c0 + chunk < r1 ? row_of(c0 + chunk) : -1;
    u64 acc[RW][2];
    // layer 0
    {
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) acc[r][c] = 0ull;
#pragma unroll
      for (int k = 0; k < K; k += 4) {
        ulonglong2 w[2];
#pragma unroll
        for (int c = 0; c < 2; ++c)
          w[c] = __ldg(reinterpret_cast<const ulonglong2*>(params + oW0 + (col + 32 * c) * K + k));
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const ulonglong2 x =
              *reinterpret_cast<const ulonglong2*>(&S.x[b][(pr * RW + r) * K + k]);
#pragma unroll
          for (int c = 0; c < 2; ++c) acc[r][c] = fma2(x.y, w[c].y, fma2(x.x, w[c].x, acc[r][c]));
        }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float bias = __ldg(params + ob0 + col + 32 * c);
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          float a, da;
          silu(pair_sum(acc[r][c]) + bias, a, da);
          A0[r * H + col + 32 * c] = a;
          sc0[(r * 2 + c) * kThreads] = da;
          acc[r][c] = 0ull;
        }
      }
      pair_sync();
    }
    // layer 1
    mul_rows<RW>(A0, S.w[0], col, acc);
    if (c0 + chunk < r1) stage_row(c0 + chunk, next, b ^ 1);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float bias = __ldg(params + ob1 + col + 32 * c);
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        float a, da;
        silu(pair_sum(acc[r][c]) + bias, a, da);
        A1[r * H + col + 32 * c] = a;
        sc1[(r * 2 + c) * kThreads] = da;
        acc[r][c] = 0ull;
      }
    }
    pair_sync();
    // layer 2, the output, its gradient
    mul_rows<RW>(A1, S.w[1], col, acc);
    {
      float y[RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) y[r] = 0.f;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float bias = __ldg(params + ob2 + col + 32 * c), w3 = S.w3[col + 32 * c];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          float a, da;
          silu(pair_sum(acc[r][c]) + bias, a, da);
          y[r] = fmaf(a, w3, y[r]);
          acc[r][c] = pk(a, w3 * da);
        }
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) y[r] += __shfl_xor_sync(0xffffffffu, y[r], o);
        if (lane == 0) S.y[wid & 1][pr * RW + r] = y[r];
      }
      pair_sync();
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const int row = pr * RW + r;
        const float e = row < rows ? S.y[0][row] + S.y[1][row] + b3 - S.t[b][row] : 0.f;
        const float dy = 2.0f * e / (float)B;
        if (tid % 64 == 0) {
          loss += (double)e * (double)e;
          gb3 += dy;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float a, w3da;
          upk(acc[r][c], a, w3da);
          gw3[c] = fmaf(a, dy, gw3[c]);
          D[r * H + col + 32 * c] = dy * w3da;
          acc[r][c] = 0ull;
        }
      }
    }
    __syncthreads();
    // layer 2's weights, and the gradient at layer 1
    add_outer(S.d, S.a1, rows, wid, lane, g2);
    gb[2] += col_sum(S.d, rows, tid);
    mul_cols<RW>(D, S.w[1], col, acc);
    __syncthreads();  // every reader of A1 is done: dZ1 takes its place
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        A1[r * H + col + 32 * c] = pair_sum(acc[r][c]) * sc1[(r * 2 + c) * kThreads];
        acc[r][c] = 0ull;
      }
    __syncthreads();
    // layer 1's weights, and the gradient at layer 0 (into D, whose readers are done)
    add_outer(S.a1, S.a0, rows, wid, lane, g1);
    gb[1] += col_sum(S.a1, rows, tid);
    mul_cols<RW>(A1, S.w[0], col, acc);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int r = 0; r < RW; ++r)
        D[r * H + col + 32 * c] = pair_sum(acc[r][c]) * sc0[(r * 2 + c) * kThreads];
    __syncthreads();
    // layer 0's weights
    gb[0] += col_sum(S.d, rows, tid);
    {
      const float* x = &S.x[b][4 * (tid >> 7)];
      for (int r = 0; r < rows; ++r) {
        const float dz = S.d[r * H + (tid & 127)];
        const float4 p = *reinterpret_cast<const float4*>(x + r * K);
        g0[0] = fmaf(dz, p.x, g0[0]);
        g0[1] = fmaf(dz, p.y, g0[1]);
        g0[2] = fmaf(dz, p.z, g0[2]);
        g0[3] = fmaf(dz, p.w, g0[3]);
      }
    }
  }

  // the block's sums
  float* out = part + (size_t)blockIdx.x * kPartStride;
  store_outer(out + oW1, wid, lane, g1);
  store_outer(out + oW2, wid, lane, g2);
  *reinterpret_cast<float4*>(out + oW0 + (tid & 127) * K + 4 * (tid >> 7)) =
      make_float4(g0[0], g0[1], g0[2], g0[3]);
  __syncthreads();
  // the biases' four parts and w3's eight pairs, in a fixed order (in the gradient buffer)
  float* red = S.d;
#pragma unroll
  for (int l = 0; l < 3; ++l) red[(l * 4 + (tid >> 7)) * H + (tid & 127)] = gb[l];
  __syncthreads();
  if (tid < 3 * H) {
    const float* q = red + (tid >> 7) * 4 * H + (tid & 127);
    const int o = (tid >> 7) == 0 ? ob0 : ((tid >> 7) == 1 ? ob1 : ob2);
    out[o + (tid & 127)] = (q[0] + q[H]) + (q[2 * H] + q[3 * H]);
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 2; ++c) red[pr * H + col + 32 * c] = gw3[c];
  double* redl = reinterpret_cast<double*>(red + kPairs * H);
  float* red3 = red + kPairs * H + 2 * kPairs;
  if (tid % 64 == 0) {
    redl[pr] = loss;
    red3[pr] = gb3;
  }
  __syncthreads();
  if (tid < H) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kPairs; ++w) s += red[w * H + tid];
    out[ow3 + tid] = s;
  } else if (tid == H) {
    float s = 0.f;
    double l = 0.0;
#pragma unroll
    for (int w = 0; w < kPairs; ++w) {
      s += red3[w];
      l += redl[w];
    }
    out[ob3] = s;
    for (int q = ob3 + 1; q < kPartStride; ++q) out[q] = 0.f;
    loss_part[blockIdx.x] = l;
  }
}

// grad = the sum of the blocks' partials (16 bytes per thread of 32 columns x 16 groups of blocks,
// fixed order; a thread's ten loads of a full grid are in flight together), loss = the mean
// squared error
__global__ void __launch_bounds__(512)
    k_ws_train_sum(const float* __restrict__ part, const double* __restrict__ loss_part, int nb,
                   double inv_b, float* __restrict__ grad, double* __restrict__ loss) {
  __shared__ float4 red[16][32];
  const int col = blockIdx.x * 32 + (threadIdx.x & 31), grp = threadIdx.x >> 5;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (col < kPartStride / 4) {
    const float4* p = reinterpret_cast<const float4*>(part) + col;
#pragma unroll 10
    for (int k = grp; k < nb; k += 16) {
      const float4 v = __ldg(p + (size_t)k * (kPartStride / 4));
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
  }
  red[grp][threadIdx.x & 31] = s;
  __syncthreads();
  if (threadIdx.x < 128) {
    const int c = threadIdx.x;
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) v += reinterpret_cast<const float*>(red[k])[c];
    const int o = blockIdx.x * 128 + c;
    if (o <= ob3) grad[o] = v;
  } else if (blockIdx.x == 0 && threadIdx.x < 160) {
    double v = 0.0;
    for (int k = threadIdx.x - 128; k < nb; k += 32) v += loss_part[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 128) *loss = v * inv_b;
  }
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, long n, float lr, float b1, float b2,
                       float c1, float c2, float eps) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n;
       q += (long)gridDim.x * blockDim.x) {
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.0f - b1) * gq;
    const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    p[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
  }
}

// How a minibatch of B rows is split: RW rows per warp, rows per block, rows per chunk, blocks.
// The cheapest by the clocks of a chunk: four layer products of 32 steps, each bound by shared
// memory (16 (8 + RW) wavefronts) or by FMAs (32 RW), the weight gradients (2 x 8 RW rows of 128
// clocks) and the rest (activations, barriers).
// A block per SM at most, except that none sums over more than 2048 rows (FP32 sums).
struct Split {
  int rw, rpb, chunk, nb;
};
int max_blocks(int B, int sms) { return (B + 2047) / 2048 > sms ? (B + 2047) / 2048 : sms; }
Split split_rows(int B, int sms) {
  Split best{0, 0, 0, 0};
  long cost = 0;
  const int most = max_blocks(B, sms);
  for (int rw : {7, 4, 2}) {
    const int R = kPairs * rw, nb = (B + R - 1) / R < most ? (B + R - 1) / R : most;
    const int rpb = (B + nb - 1) / nb, n = (rpb + R - 1) / R;
    const int step = 16 * (8 + rw) > 32 * rw ? 16 * (8 + rw) : 32 * rw;
    const long c = (long)n * (4 * 32 * step + 2 * R * 128 + 700 * rw + 3000);
    if (!best.rw || c < cost) {
      cost = c;
      best = Split{rw, rpb, (rpb + n - 1) / n, (B + rpb - 1) / rpb};
    }
  }
  return best;
}

template <int RW>
cudaError_t train_launch(const Split& s, const float* params, const float* X, const float* t,
                         const long long* idx, int B, WsTrainBuffers& tb, cudaStream_t st) {
  const size_t sm = sizeof(Smem<RW>);
  const cudaError_t e = prepare_launch(k_ws_train<RW>, kThreads, sm);
  if (e != cudaSuccess) return e;
  k_ws_train<RW><<<s.nb, kThreads, sm, st>>>(params, X, t, idx, B, s.rpb, s.chunk, tb.scr,
                                             tb.part, tb.loss_part);
  return cudaGetLastError();
}

}  // namespace

int ws_train_blocks(int B, int sms) { return max_blocks(B, sms); }
size_t ws_train_scratch_floats() { return (size_t)2 * 7 * 2 * kThreads; }
size_t ws_train_part_floats() { return kPartStride; }

// gradient and loss of one minibatch (the trainer adds Adam)
cudaError_t launch_ws_grad(const float* params, const float* X, const float* t,
                           const long long* idx, int B, WsTrainBuffers& tb, cudaStream_t st) {
  const Split s = split_rows(B, tb.sms);
  cudaError_t e;
  if (s.rw == 7)
    e = train_launch<7>(s, params, X, t, idx, B, tb, st);
  else if (s.rw == 4)
    e = train_launch<4>(s, params, X, t, idx, B, tb, st);
  else
    e = train_launch<2>(s, params, X, t, idx, B, tb, st);
  if (e != cudaSuccess) return e;
  k_ws_train_sum<<<(kPartStride / 4 + 31) / 32, 512, 0, st>>>(tb.part, tb.loss_part, s.nb,
                                                              1.0 / (double)B, tb.grad, tb.loss);
  return cudaGetLastError();
}

cudaError_t launch_ws_adam(float* p, float* m, float* v, const float* g, long n, float lr,
                           int t, cudaStream_t st) {
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = (float)(1.0 - pow(b1, t)), c2 = (float)(1.0 - pow(b2, t));
  k_adam<<<(int)((n + 255) / 256), 256, 0, st>>>(p, m, v, g, n, lr, (float)b1, (float)b2, c1, c2,
                                                 1e-8f);
  return cudaGetLastError();
}

}  // namespace otgb

// Nonlinear residual + linearised coefficients (Eq. ma2, linearmaeq, translation), input
// translation, and the GMRES(m) kernels (Sec. 4.2) of the damped-Newton solver.
//
// Reductions: every block writes its partials to a scratch array; the last block to take
// a ticket reduces them in block order and finalises the scalars in DevScalars.  The
// order is fixed, so results are bit-reproducible from run to run.
#include <math.h>
#include <string.h>

#include "dd.cuh"
#include "dd2.cuh"
#include "otgb_internal.cuh"
#include "gmres_dev.cuh"
#include "reduce.cuh"

namespace otgb {

#define RTX 32  // residual tile width (x / columns); 8 warps

// Block sum of NV floats (result valid in thread 0).
template <int NV>
__device__ void block_sum_f(float (&v)[NV]) {
  __shared__ float redf[32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int a = 0; a < NV; ++a)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[a] += __shfl_xor_sync(0xffffffffu, v[a], o);
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int a = 0; a < NV; ++a) redf[wid][a] = v[a];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      float x = lane < nw ? redf[lane][a] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      v[a] = x;
    }
  }
  __syncthreads();
}

// FP32 sum of NV values over the grid (1-D grid), for the FP32 Krylov vectors of the mixed
// mode: block tree sums, per-block partials, and the last block to take a ticket sums them
// in block order (fixed order: bit-reproducible).  Returns true in that block, with the
// totals in thread 0.  GB300 runs FP32 at ~60x its FP64 rate, and FP64 tree reductions
// (shuffle + add per level) had become a visible part of these short kernels.
template <int NV>
__device__ bool grid_sum_f(float (&v)[NV], double* partials, unsigned int* ticket) {
  __shared__ bool last;
  float* pf = reinterpret_cast<float*>(partials);
  block_sum_f<NV>(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) pf[(size_t)blockIdx.x * NV + a] = v[a];
    __threadfence();
    const unsigned int k = atomicAdd(ticket, 1u);
    last = (k == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int a = 0; a < NV; ++a) v[a] = 0.f;
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] += ((volatile const float*)pf)[(size_t)b * NV + a];
  block_sum_f<NV>(v);
  return true;
}

// Double-float reductions (dd.cuh) of NV values with kinds 0 sum, 1 max, 2 min, on the FP32
// pipes: the FP64-accuracy grid reductions of the mixed-mode residual.
__device__ __forceinline__ dd dd_combine(dd a, dd b, int kind) {
  if (kind == 0) return dd_add(a, b);
  if (kind == 1) return dd_gt(b, a) ? b : a;
  return dd_gt(a, b) ? b : a;
}
__device__ __forceinline__ dd dd_identity(int kind) {
  return kind == 0 ? dd{0.f, 0.f} : (kind == 1 ? dd{-INFINITY, 0.f} : dd{INFINITY, 0.f});
}
__device__ __forceinline__ dd warp_reduce_dd(dd v, int kind) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const dd w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    v = dd_combine(v, w, kind);
  }
  return v;
}
// result valid in thread 0 (all of warp 0)
template <int NV>
__device__ void block_reduce_dd(dd (&v)[NV], const int (&kind)[NV]) {
  __shared__ float2 redd[32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int a = 0; a < NV; ++a) v[a] = warp_reduce_dd(v[a], kind[a]);
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int a = 0; a < NV; ++a) redd[wid][a] = make_float2(v[a].hi, v[a].lo);
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      const dd x = lane < nw ? dd{redd[lane][a].x, redd[lane][a].y} : dd_identity(kind[a]);
      v[a] = warp_reduce_dd(x, kind[a]);
    }
  }
  __syncthreads();
}
// grid-wide: per-block (hi, lo) partials, the last block to take a ticket combines them in
// block order; true in that block, totals in thread 0 (2-D grids allowed)
template <int NV>
__device__ bool grid_reduce_dd(dd (&v)[NV], const int (&kind)[NV], double* partials,
                               unsigned int* ticket) {
  __shared__ bool last;
  float2* pf = reinterpret_cast<float2*>(partials);
  const unsigned int nb = gridDim.x * gridDim.y;
  block_reduce_dd<NV>(v, kind);
  if (threadIdx.x == 0) {
    const size_t bid = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
#pragma unroll
    for (int a = 0; a < NV; ++a) pf[bid * NV + a] = make_float2(v[a].hi, v[a].lo);
    __threadfence();
    const unsigned int k = atomicAdd(ticket, 1u);
    last = (k == nb - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int a = 0; a < NV; ++a) v[a] = dd_identity(kind[a]);
  for (unsigned int b = threadIdx.x; b < nb; b += blockDim.x)
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      const volatile float2* q = (const volatile float2*)pf + (size_t)b * NV + a;
      v[a] = dd_combine(v[a], dd{q->x, q->y}, kind[a]);
    }
  block_reduce_dd<NV>(v, kind);
  return true;
}

// ---------------------------------------------------------------------------------------
// Input translation (Eq. translation applied to both densities, as for the images of
// Sec. 5.2): d <- d - mean(d) + 1; rejects non-finite input or a non-positive result.
// ---------------------------------------------------------------------------------------
// block sums of v, minima of kf and kg (ordered_key) and counts bf, bg, in thread 0 of 256
__device__ __forceinline__ void input_reduce(double (&v)[2], long long& kf, long long& kg, int& bf,
                                             int& bg) {
  __shared__ double ss[2];
  __shared__ long long sk[8][2];
  __shared__ int sb[8][2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    kf = min(kf, __shfl_xor_sync(0xffffffffu, kf, o));
    kg = min(kg, __shfl_xor_sync(0xffffffffu, kg, o));
  }
  bf = __reduce_add_sync(0xffffffffu, bf);
  bg = __reduce_add_sync(0xffffffffu, bg);
  if (lane == 0) {
    sk[wid][0] = kf;
    sk[wid][1] = kg;
    sb[wid][0] = bf;
    sb[wid][1] = bg;
  }
  double s;
  if (block_fold<2>(v, s)) ss[threadIdx.x >> 3] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    v[0] = ss[0];
    v[1] = ss[1];
    for (int w = 1; w < 8; ++w) {
      kf = min(kf, sk[w][0]);
      kg = min(kg, sk[w][1]);
      bf += sb[w][0];
      bg += sb[w][1];
    }
  }
  __syncthreads();
}

__global__ void k_input_stats(const double* __restrict__ f, const double* __restrict__ g,
                              long P, double* partials, DevScalars* sc, Bat bat) {
  f = badv(f, bat);
  g = badv(g, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  // per thread: the sums in FP64, minima and counts on the integer pipe (FP64 starts two
  // instructions per clock and SM on this GPU); four loads of each plane in flight
  double v[2] = {0.0, 0.0};
  long long kf = ordered_key(INFINITY), kg = kf;
  int bf = 0, bg = 0;
  const long nth = (long)gridDim.x * blockDim.x;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P; p += 4 * nth) {
    double a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = p + k * nth < P;
      a[k] = in ? f[p + k * nth] : 0.0;
      b[k] = in ? g[p + k * nth] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (p + k * nth >= P) break;
      v[0] += a[k];
      v[1] += b[k];
      bf += !finite_key(a[k]);
      bg += !finite_key(b[k]);
      if (!nan_key(a[k])) kf = min(kf, ordered_key(a[k]));
      if (!nan_key(b[k])) kg = min(kg, ordered_key(b[k]));
    }
  }
  input_reduce(v, kf, kg, bf, bg);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    double* q = partials + (size_t)blockIdx.x * 6;
    q[0] = v[0];
    q[1] = v[1];
    q[2] = __longlong_as_double(kf);
    q[3] = __longlong_as_double(kg);
    q[4] = __longlong_as_double(bf);
    q[5] = __longlong_as_double(bg);
    __threadfence();
    last = atomicAdd(&sc->ticket[TK_INPUT], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  v[0] = v[1] = 0.0;
  kf = kg = ordered_key(INFINITY);
  bf = bg = 0;
  for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    const double* q = partials + (size_t)b * 6;
    v[0] += __ldcg(q);
    v[1] += __ldcg(q + 1);
    kf = min(kf, __double_as_longlong(__ldcg(q + 2)));
    kg = min(kg, __double_as_longlong(__ldcg(q + 3)));
    bf += (int)__double_as_longlong(__ldcg(q + 4));
    bg += (int)__double_as_longlong(__ldcg(q + 5));
  }
  input_reduce(v, kf, kg, bf, bg);
  if (threadIdx.x == 0) {
    const double fmin = key_value(kf), gmin = key_value(kg);
    sc->in_mean[0] = v[0] / (double)P;
    sc->in_mean[1] = v[1] / (double)P;
    sc->in_min[0] = fmin;
    sc->in_min[1] = gmin;
    sc->in_nonfinite[0] = bf;
    sc->in_nonfinite[1] = bg;
    // translated inputs must be positive after the translation, inputs used as given
    // (in_plain) as they are
    const double sf = sc->in_plain ? 0.0 : 1.0 - sc->in_mean[0];
    const double sg = sc->in_plain ? 0.0 : 1.0 - sc->in_mean[1];
    const bool bad = bf > 0 || bg > 0 || !(fmin + sf > 0.0) || !(gmin + sg > 0.0);
    sc->in_bad = bad ? 1 : 0;
    sc->ticket[TK_INPUT] = 0;
  }
}

// the translated inputs; in the mixed mode also f as (hi, lo) floats, and for the learned start's
// features log f - log g with FP32 logarithms: one pass, where the two were passes of their own
// over f and g (6.0 and 5.4 us at 512x512 beside 6.8 us, cold caches)
__global__ void k_input_apply(const double* __restrict__ f, const double* __restrict__ g,
                              double* __restrict__ ft, double* __restrict__ gt,
                              float2* __restrict__ fdd, float* __restrict__ src, long P,
                              const DevScalars* __restrict__ sc, Bat bat) {
  f = badv(f, bat);
  g = badv(g, bat);
  ft = badv(ft, bat);
  gt = badv(gt, bat);
  fdd = badv(fdd, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  const double sf = 1.0 - sc->in_mean[0], sg = 1.0 - sc->in_mean[1];
  const long nth = (long)gridDim.x * blockDim.x;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P; p += 4 * nth) {
    double a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = p + k * nth < P;
      a[k] = in ? f[p + k * nth] : 0.0;
      b[k] = in ? g[p + k * nth] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long q = p + k * nth;
      if (q >= P) break;
      a[k] += sf;
      b[k] += sg;
      ft[q] = a[k];
      gt[q] = b[k];
      if (fdd) {
        const dd v = dd_from_double(a[k]);
        fdd[q] = make_float2(v.hi, v.lo);
        if (src) src[q] = logf(v.hi) - logf(dd_from_double(b[k]).hi);
      }
    }
  }
}

// blocks of a grid reduction or an elementwise pass over P points: 1024 points each, at most two
// blocks per SM
static int reduce_blocks(long P) {
  static int nb = 0;
  if (nb == 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    nb = (sms > 0 ? sms : 148) * 2;
  }
  return (int)(P < 1024L * nb ? (P + 1023) / 1024 : nb);
}

cudaError_t launch_input_stats(const double* f, const double* g, int N, int M,
                               double* partials, DevScalars* sc, cudaStream_t st, Bat bat) {
  const long P = (long)N * M;
  k_input_stats<<<bgrid(dim3(reduce_blocks(P)), bat), 256, 0, st>>>(f, g, P, partials, sc, bat);
  return cudaGetLastError();
}

// %globaltimer: the GPU's nanosecond clock (PTX special register)
__global__ void k_stamp(DevScalars* sc, int cls) {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  const int prev = sc->stamp_cls;
  if (prev >= 0 && prev < PH_COUNT && t > sc->stamp_t) sc->phase_ns[prev] += t - sc->stamp_t;
  if (prev >= 100 && prev < 116 && t > sc->stamp_t) sc->class_ns[prev - 100] += t - sc->stamp_t;
  sc->stamp_t = t;
  sc->stamp_cls = cls;
}

cudaError_t launch_stamp(DevScalars* sc, int cls, cudaStream_t st) {
  k_stamp<<<1, 1, 0, st>>>(sc, cls);
  return cudaGetLastError();
}

cudaError_t launch_translate_inputs(const double* f, const double* g, double* ft, double* gt,
                                    int N, int M, double* partials, DevScalars* sc,
                                    cudaStream_t st, Bat bat, float2* fdd, float* src) {
  const long P = (long)N * M;
  const dim3 nb = bgrid(dim3(reduce_blocks(P)), bat);
  k_input_stats<<<nb, 256, 0, st>>>(f, g, P, partials, sc, bat);
  k_input_apply<<<nb, 256, 0, st>>>(f, g, ft, gt, fdd, src, P, sc, bat);
  return cudaGetLastError();
}

// indices modulo L
__device__ __forceinline__ int wrapi(int a, int L) {
  int r = a % L;
  return r < 0 ? r + L : r;
}

__device__ __forceinline__ int wrap_near(int a, int L) {  // a in [-L, 2L)
  return a < 0 ? a + L : (a >= L ? a - L : a);
}

// ---------------------------------------------------------------------------------------
// Mixed-mode residual + coefficients (FP64: residual_f64.cu).  u is staged in shared memory with a
// periodic halo of 2 for the 4th-order centred stencils; every FP64-accuracy quantity (the stencils
// of u, the displaced point, the B-spline value gather, det, f_n and F) is in double-float
// arithmetic on the FP32 pipes (dd.cuh, unit round-off 2^-48), the Jacobian coefficients,
// the interpolant's gradient and the Simpson sums in FP32.  Inputs: u (FP64), f and c
// pre-split into (hi, lo) float pairs; output F_raw in FP64.
// ---------------------------------------------------------------------------------------
struct ResidConstsDD {
  dd Mh, Nh, Mh2, Nh2, MNh;  // M/12, N/12, M^2/12, N^2/12, MN/144
  dd inv36;                  // 1/36 (the value weights are computed x6 per axis)
  float M, N;
  float w3M, w3N;            // 1/(3M), 1/(3N)
  int nob;                   // 1: the simplified operator (b = 0)
  // interpolation of g: 0 cubic B-spline; 1 bilinear, 2 nearest node (then cdd = g as (hi, lo) pairs)
  int interp;
  const float* gx;           // grid gradient of g (FP32: the Jacobian only)
  const float* gy;
};

__device__ __forceinline__ dd ldd(const float2* __restrict__ a, size_t i) {
  const float2 v = __ldg(a + i);
  return dd{v.x, v.y};
}

// 6 x the cubic B-spline value weights at t in [0, 1) (taps -1, 0, 1, 2) for two positions: s^3,
// 3 t^3 - 6 t^2 + 4, 6 - (the other three), t^3, with s = 1 - t; all coefficients exact
__device__ __forceinline__ void bspline6_dd2(pair::D2 t, pair::D2 w[4]) {
  using namespace pair;
  const D2 s = d2_sub(D2{pk(1.0f, 1.0f), 0ull}, t);
  const u64 nt = neg2(t.h);
  const D2 t2 = d2_mul_n(t, t, nt), t3 = d2_mul_n(t2, t, nt);
  const u64 ns = neg2(s.h);
  w[0] = d2_mul_n(d2_mul_n(s, s, ns), s, ns);
  w[1] = d2_add_f(d2_sub(d2_mul_f(t3, pk(3.0f, 3.0f)), d2_mul_f(t2, pk(6.0f, 6.0f))),
                  pk(4.0f, 4.0f));
  w[3] = t3;
  w[2] = d2_sub(D2{pk(6.0f, 6.0f), 0ull}, d2_add(d2_add(w[0], w[1]), w[3]));
}
// the FP32 weights and their derivatives for two positions (the Jacobian's)
__device__ __forceinline__ void bspline_w2(pair::u64 t, pair::u64 w[4], pair::u64 dw[4]) {
  using namespace pair;
  auto c = [](float x) { return pk(x, x); };
  const u64 s = sub2(c(1.0f), t), t2 = mul2(t, t), s2 = mul2(s, s);
  const float sixth = 1.0f / 6.0f;
  w[0] = mul2(mul2(s2, s), c(sixth));
  w[1] = fma2(t2, fma2(t, c(0.5f), c(-1.0f)), c(4.0f * sixth));
  w[2] = fma2(t, fma2(t, fma2(t, c(-0.5f), c(0.5f)), c(0.5f)), c(sixth));
  w[3] = mul2(mul2(t2, t), c(sixth));
  dw[0] = mul2(s2, c(-0.5f));
  dw[1] = mul2(c(0.5f), fma2(c(3.0f), t2, mul2(c(-4.0f), t)));
  dw[3] = mul2(t2, c(0.5f));
  // (their sum is zero: a rounding error of it enters G_x times M)
  dw[2] = neg2(add2(add2(dw[0], dw[3]), dw[1]));
}

// floor of a dd position p (|p| < 2^23): integer part k and fraction t in [0, 1) as dd.
// p.hi - floor(p.hi) is not exact for -1 < p.hi < 0 (the result needs more bits than
// p.hi), so the subtraction is an error-free dd add.
__device__ __forceinline__ int dd_floor(dd p, dd* t) {
  float fl = floorf(p.hi);
  dd fr = dd_add_f(p, -fl);
  if (fr.hi < 0.0f) {
    fl -= 1.0f;
    fr = dd_add_f(fr, 1.0f);
  } else if (fr.hi >= 1.0f) {
    fl += 1.0f;
    fr = dd_add_f(fr, -1.0f);
  }
  *t = fr;
  return (int)fl;
}

// the scalars of a residual from its ten totals
__device__ __forceinline__ void residual_close(DevScalars* sc, const double (&v)[10], int N,
                                               int M) {
  const double Pd = (double)N * (double)M;
  const double mean_fn = v[0] / Pd;
  const double shift = mean_fn - 1.0;
  sc->mean_fn = mean_fn;
  sc->shift = shift;
  sc->res_inf = fmax(fabs(v[6] + shift), fabs(v[7] + shift));
  for (int a = 0; a < 5; ++a) sc->abar[a] = v[1 + a];
  sc->min_det = v[8];
  sc->k1_nonfinite = (int)v[9];
  sc->admissible = (v[9] == 0.0 && isfinite(sc->res_inf) && v[8] > 0.0) ? 1 : 0;
  sc->ticket[TK_RESID] = 0;
}

// Nearest-node and bilinear interpolation (a block covers 32 columns x 8 RPT rows, RPT rows per
// thread)
template <int RPT>
__global__ void __launch_bounds__(8 * RTX, 3)
    k_residual_dd(const float2* __restrict__ fdd, const float2* __restrict__ cdd,
                  const double* __restrict__ ua, const double* __restrict__ ub, int sel, int N,
                  int M, ResidConstsDD K, double* __restrict__ Fraw, float* __restrict__ coef,
                  double* partials, DevScalars* sc, Bat bat) {
  constexpr int RTY = 8 * RPT;
  __shared__ dd tile[RTY + 4][RTX + 4];
  __shared__ dd dyt[RTY][RTX + 4];  // unscaled y-difference of u (halo 2 in x)
  fdd = badv(fdd, bat);
  cdd = badv(cdd, bat);
  ua = badv(ua, bat);
  ub = badv(ub, bat);
  Fraw = badv(Fraw, bat);
  coef = badv(coef, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  const double* __restrict__ u = (ub && ((sc->upar ^ sel) & 1)) ? ub : ua;
  const int bx = blockIdx.x * RTX, by = blockIdx.y * RTY;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < (RTY + 4) * (RTX + 4); idx += blockDim.x) {
    const int r = idx / (RTX + 4), cc = idx - r * (RTX + 4);
    int gi = by + r - 2, gj = bx + cc - 2;
    while (gi < 0) gi += N;
    while (gi >= N) gi -= N;
    while (gj < 0) gj += M;
    while (gj >= M) gj -= M;
    tile[r][cc] = dd_from_double_cvt(u[(size_t)gi * M + gj]);
  }
  __syncthreads();
  for (int idx = tid; idx < RTY * (RTX + 4); idx += blockDim.x) {
    const int r = idx / (RTX + 4), cc = idx - r * (RTX + 4);
    // (u[+2] - u[-2]) is subtracted from 8 (u[+1] - u[-1]), all in y
    dyt[r][cc] = dd_sub(dd_scale2(dd_sub(tile[r + 3][cc], tile[r + 1][cc]), 8.0f),
                        dd_sub(tile[r + 4][cc], tile[r][cc]));
  }
  __syncthreads();
  // partials: sum fn (dd), max Fraw, min Fraw (dd), min det (dd), non-finite count
  dd sum_fn = dd{0.f, 0.f}, fmax_ = dd{-INFINITY, 0.f}, fmin_ = dd{INFINITY, 0.f},
     dmin = dd{INFINITY, 0.f};
  float nonfinite = 0.f;
  float simp[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  const int tx = tid % RTX, ty0 = tid / RTX;
  const int j = bx + tx;
  const size_t P = (size_t)N * M;
  const float wx = ((j & 1) ? 4.0f : 2.0f) * K.w3M;
#pragma unroll 1
  for (int rr = 0; rr < RPT; ++rr) {
    const int ty = ty0 + rr * 8;
    const int i = by + ty;
    if (i >= N || j >= M) continue;
    const int r = ty + 2, q = tx + 2;
    const dd c0 = tile[r][q];
    const dd xp1 = tile[r][q + 1], xm1 = tile[r][q - 1], xp2 = tile[r][q + 2],
             xm2 = tile[r][q - 2];
    const dd ux =
        dd_mul(dd_sub(dd_scale2(dd_sub(xp1, xm1), 8.0f), dd_sub(xp2, xm2)), K.Mh);
    const dd uy = dd_mul(dyt[ty][q], K.Nh);
    // 16 (u[+1] + u[-1]) - (u[+2] + u[-2]) - 30 u
    const dd uxx = dd_mul(dd_sub(dd_sub(dd_scale2(dd_add(xp1, xm1), 16.0f), dd_add(xp2, xm2)),
                                 dd_mul_f(c0, 30.0f)),
                          K.Mh2);
    const dd yp1 = tile[r + 1][q], ym1 = tile[r - 1][q], yp2 = tile[r + 2][q],
             ym2 = tile[r - 2][q];
    const dd uyy = dd_mul(dd_sub(dd_sub(dd_scale2(dd_add(yp1, ym1), 16.0f), dd_add(yp2, ym2)),
                                 dd_mul_f(c0, 30.0f)),
                          K.Nh2);
    const dd uxy = dd_mul(dd_sub(dd_scale2(dd_sub(dyt[ty][q + 1], dyt[ty][q - 1]), 8.0f),
                                 dd_sub(dyt[ty][q + 2], dyt[ty][q - 2])),
                          K.MNh);
    // displaced point in grid units and the periodic cubic B-spline value there
    dd tx_, ty_;
    const int fj = dd_floor(dd_add_f(dd_mul_f(ux, K.M), (float)j), &tx_);
    const int fi = dd_floor(dd_add_f(dd_mul_f(uy, K.N), (float)i), &ty_);
    const int j0 = wrapi(fj, M), i0 = wrapi(fi, N);
    int jj[4], ii[4];
    jj[0] = j0 == 0 ? M - 1 : j0 - 1;
    jj[1] = j0;
    jj[2] = wrap_near(j0 + 1, M);
    jj[3] = wrap_near(j0 + 2, M);
    ii[0] = i0 == 0 ? N - 1 : i0 - 1;
    ii[1] = i0;
    ii[2] = wrap_near(i0 + 1, N);
    ii[3] = wrap_near(i0 + 2, N);
    dd G;
    float Gx, Gy;
    if (K.interp == 2) {  // nearest node (round half up on the fraction)
      const bool upx = tx_.hi > 0.5f || (tx_.hi == 0.5f && tx_.lo >= 0.0f);
      const bool upy = ty_.hi > 0.5f || (ty_.hi == 0.5f && ty_.lo >= 0.0f);
      const int jn = wrapi(fj + (upx ? 1 : 0), M);
      const int in = wrapi(fi + (upy ? 1 : 0), N);
      const size_t q = (size_t)in * M + jn;
      G = ldd(cdd, q);
      Gx = __ldg(K.gx + q);
      Gy = __ldg(K.gy + q);
    } else {  // bilinear on the cell (i0, j0) .. (i0 + 1, j0 + 1)
      const dd sx = dd_add_f(dd{-tx_.hi, -tx_.lo}, 1.0f), sy = dd_add_f(dd{-ty_.hi, -ty_.lo}, 1.0f);
      const size_t q00 = (size_t)ii[1] * M + jj[1], q01 = (size_t)ii[1] * M + jj[2];
      const size_t q10 = (size_t)ii[2] * M + jj[1], q11 = (size_t)ii[2] * M + jj[2];
      const dd r0 = dd_fma(ldd(cdd, q01), tx_, dd_mul(ldd(cdd, q00), sx));
      const dd r1 = dd_fma(ldd(cdd, q11), tx_, dd_mul(ldd(cdd, q10), sx));
      G = dd_fma(r1, ty_, dd_mul(r0, sy));
      const float ax = tx_.hi, ay = ty_.hi;
      const float w00 = (1.f - ax) * (1.f - ay), w01 = ax * (1.f - ay), w10 = (1.f - ax) * ay,
                  w11 = ax * ay;
      Gx = w00 * __ldg(K.gx + q00) + w01 * __ldg(K.gx + q01) + w10 * __ldg(K.gx + q10) +
           w11 * __ldg(K.gx + q11);
      Gy = w00 * __ldg(K.gy + q00) + w01 * __ldg(K.gy + q01) + w10 * __ldg(K.gy + q10) +
           w11 * __ldg(K.gy + q11);
    }
    const dd det = dd_sub(dd_mul(dd_add_f(uxx, 1.0f), dd_add_f(uyy, 1.0f)), dd_mul(uxy, uxy));
    const dd fn = dd_mul(G, det);
    const size_t p = (size_t)i * M + j;
    const dd fr = dd_sub(ldd(fdd, p), fn);
    Fraw[p] = (double)fr.hi + (double)fr.lo;
    // coefficients of the linearisation (Jacobian only), FP32
    const float Gt = G.hi, dett = det.hi;
    const float a11 = Gt * (1.0f + uyy.hi), a12 = -Gt * uxy.hi, a22 = Gt * (1.0f + uxx.hi);
    const float b1 = K.nob ? 0.0f : dett * Gx, b2 = K.nob ? 0.0f : dett * Gy;
    coef[p] = a11;
    coef[P + p] = a12;
    coef[2 * P + p] = a22;
    coef[3 * P + p] = b1;
    coef[4 * P + p] = b2;
    const float w = ((i & 1) ? 4.0f : 2.0f) * K.w3N * wx;
    simp[0] += w * a11;
    simp[1] += w * a12;
    simp[2] += w * a22;
    simp[3] += w * b1;
    simp[4] += w * b2;
    if (isfinite(fn.hi) && isfinite(fn.lo)) {
      sum_fn = dd_add(sum_fn, fn);
      if (dd_gt(fr, fmax_)) fmax_ = fr;
      if (dd_gt(fmin_, fr)) fmin_ = fr;
    } else {
      nonfinite += 1.0f;
    }
    if (dd_gt(dmin, det)) dmin = det;
  }
  // grid reductions in double-float (sum f_n, the five Simpson sums, max F, min F, min det,
  // the non-finite count)
  dd r[10] = {sum_fn,
              dd{simp[0], 0.f},
              dd{simp[1], 0.f},
              dd{simp[2], 0.f},
              dd{simp[3], 0.f},
              dd{simp[4], 0.f},
              fmax_,
              fmin_,
              dmin,
              dd{nonfinite, 0.f}};
  const int kind[10] = {0, 0, 0, 0, 0, 0, 1, 2, 2, 0};
  if (!grid_reduce_dd<10>(r, kind, partials, &sc->ticket[TK_RESID])) return;
  if (threadIdx.x == 0) {
    double v[10];
    for (int a = 0; a < 10; ++a) v[a] = (double)r[a].hi + (double)r[a].lo;
    residual_close(sc, v, N, M);
  }
}

// ---------------------------------------------------------------------------------------
// The cubic-spline residual on two points per thread, rows ty and ty + RB of a tile of 2 RB RT x 32
// points, held in the two lanes of packed FP32 pairs (dd2.cuh): every double-float operation is one
// packed instruction for both points.  The kernel is bound by instruction issue and the latency of
// the double-float chains (16 warps per SM: a point pair fills 128 registers), not by its 52 bytes
// a point: with one point per thread 1650 instructions a point, 1120 here, a tenth of the former
// the block sums' shuffle trees.  These are folded: eight values' halves change lanes together, and
// maxima and minima go as ordered integers through the warp reduction instructions.  1024^2: 75.5
// -> 63.6 us, 256^2 15.1 -> 11.0.  (80 registers for 24 warps per SM: 79 us, spills.)
// ---------------------------------------------------------------------------------------
struct ResidSums {
  dd s[6];            // sum of f_n, the five Simpson sums
  dd fmax, fmin, dmin;
  int bad;
};
__device__ __forceinline__ int ordered32(float x) {
  const int b = __float_as_int(x);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unordered32(int k) {
  return __int_as_float(k ^ ((k >> 31) & 0x7fffffff));
}
// smallest dd of the lanes in mask (largest: of the negated one; no lane holds a NaN)
__device__ __forceinline__ dd warp_min_dd(dd v, unsigned mask) {
  const int h = ordered32(v.hi), m = __reduce_min_sync(mask, h);
  const int l = __reduce_min_sync(mask, h == m ? ordered32(v.lo) : 0x7fffffff);
  return dd{unordered32(m), unordered32(l)};
}
// the block's ten values to dst (the order of k_residual_dd's partials); NW (4 or 8) warps
template <int NW>
__device__ __forceinline__ void resid_block_sums(const ResidSums& r, float2* dst) {
  __shared__ float2 ws[NW][8], we[3][NW];
  __shared__ int wb[NW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto shfl = [](dd v, int o) {
    return dd{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
  };
  dd x[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) x[a] = a < 6 ? r.s[a] : dd{0.f, 0.f};
  int o = 16;
#pragma unroll
  for (int h = 4; h > 0; h /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int a = 0; a < h; ++a)
      x[a] = dd_add(up ? x[a + h] : x[a], shfl(up ? x[a] : x[a + h], o));
  }
  x[0] = dd_add(x[0], shfl(x[0], 2));
  x[0] = dd_add(x[0], shfl(x[0], 1));
  const dd mx = warp_min_dd(dd_neg(r.fmax), 0xffffffffu), mn = warp_min_dd(r.fmin, 0xffffffffu),
           md = warp_min_dd(r.dmin, 0xffffffffu);
  const int nb = __reduce_add_sync(0xffffffffu, r.bad);
  if (lane % 4 == 0) ws[wid][lane / 4] = make_float2(x[0].hi, x[0].lo);
  if (lane == 0) {
    we[0][wid] = make_float2(mx.hi, mx.lo);
    we[1][wid] = make_float2(mn.hi, mn.lo);
    we[2][wid] = make_float2(md.hi, md.lo);
    wb[wid] = nb;
  }
  __syncthreads();
  if (threadIdx.x < 8 * NW) {  // (groups of NW lanes: value threadIdx.x / NW)
    const int a = threadIdx.x / NW;
    const float2 q = ws[threadIdx.x % NW][a];
    dd s = dd{q.x, q.y};
#pragma unroll
    for (int m = NW / 2; m > 0; m /= 2) s = dd_add(s, shfl(s, m));
    if (threadIdx.x % NW == 0 && a < 6) dst[a] = make_float2(s.hi, s.lo);
  } else if (wid == NW - 1 && lane < NW) {
    constexpr unsigned mask = (1u << NW) - 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float2 q = we[a][lane];
      dd m = warp_min_dd(dd{q.x, q.y}, mask);
      if (a == 0) m = dd_neg(m);
      if (lane == 0) dst[6 + a] = make_float2(m.hi, m.lo);
    }
    const int n = __reduce_add_sync(mask, wb[lane]);
    if (lane == 0) dst[9] = make_float2((float)n, 0.f);
  }
}

template <int RB, int RT, int BPS>
__global__ void __launch_bounds__(RB * RTX, BPS)
    k_residual_dd2(const float2* __restrict__ fdd, const float2* __restrict__ cdd,
                   const double* __restrict__ ua, const double* __restrict__ ub, int sel, int N,
                   int M, ResidConstsDD K, double* __restrict__ Fraw, float* __restrict__ coef,
                   double* partials, DevScalars* sc, Bat bat) {
  using namespace pair;
  constexpr int RTY = 2 * RB * RT, W = RTX + 4;
  __shared__ float th[RTY + 4][W], tl[RTY + 4][W];  // u with a halo of 2, high and low words
  __shared__ float yh[RTY][W], yl[RTY][W];          // its unscaled y-difference
  fdd = badv(fdd, bat);
  cdd = badv(cdd, bat);
  ua = badv(ua, bat);
  ub = badv(ub, bat);
  Fraw = badv(Fraw, bat);
  coef = badv(coef, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  const double* __restrict__ u = (ub && ((sc->upar ^ sel) & 1)) ? ub : ua;
  const int bx = blockIdx.x * RTX, by = blockIdx.y * RTY;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < (RTY + 4) * W; idx += RB * RTX) {
    const int r = idx / W, cc = idx - r * W;
    int gi = wrap_near(by + r - 2, N), gj = wrap_near(bx + cc - 2, M);
    if (gi >= N) gi %= N;  // (a grid smaller than the tile)
    if (gj >= M) gj %= M;
    const dd v = dd_from_double_cvt(u[(size_t)gi * M + gj]);
    th[r][cc] = v.hi;
    tl[r][cc] = v.lo;
  }
  __syncthreads();
  for (int idx = tid; idx < RTY / 2 * W; idx += RB * RTX) {  // rows r and r + RTY / 2
    constexpr int H = RTY / 2;
    const int r = idx / W, c = idx - r * W;
    auto T = [&](int d) {
      return D2{pk(th[r + d][c], th[r + H + d][c]), pk(tl[r + d][c], tl[r + H + d][c])};
    };
    const D2 v = d2_sub(d2_scale2(d2_sub(T(3), T(1)), 8.0f), d2_sub(T(4), T(0)));
    upk(v.h, yh[r][c], yh[r + H][c]);
    upk(v.l, yl[r][c], yl[r + H][c]);
  }
  __syncthreads();
  ResidSums acc;
  acc.fmax = dd{-INFINITY, 0.f};
  acc.fmin = acc.dmin = dd{INFINITY, 0.f};
  acc.bad = 0;
  D2 sfn{0ull, 0ull};
  float simp[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  const int tx = tid % RTX, ty0 = tid / RTX;
  const int j = bx + tx;
  const size_t P = (size_t)N * M;
  const float wx = ((j & 1) ? 4.0f : 2.0f) * K.w3M;
  const u64 one = pk(1.0f, 1.0f);
  auto bc = [](dd c) { return D2{pk(c.hi, c.hi), pk(c.lo, c.lo)}; };
#pragma unroll 1
  for (int rr = 0; rr < RT; ++rr) {
    const int ty = ty0 + 2 * RB * rr;
    const int i = by + ty;
    if (i >= N || j >= M) continue;
    const bool two = i + RB < N;  // (a missing second row is computed on the wrapped rows)
    const int q = tx + 2;
    auto T = [&](int dr, int dc) {
      const int r = ty + 2 + dr;
      return D2{pk(th[r][q + dc], th[r + RB][q + dc]), pk(tl[r][q + dc], tl[r + RB][q + dc])};
    };
    auto Y = [&](int dc) {
      return D2{pk(yh[ty][q + dc], yh[ty + RB][q + dc]), pk(yl[ty][q + dc], yl[ty + RB][q + dc])};
    };
    D2 ux, uxx, uyy;
    {
      const D2 c30 = d2_mul_f(T(0, 0), pk(30.0f, 30.0f));
      const D2 xp1 = T(0, 1), xm1 = T(0, -1), xp2 = T(0, 2), xm2 = T(0, -2);
      ux = d2_mul(d2_sub(d2_scale2(d2_sub(xp1, xm1), 8.0f), d2_sub(xp2, xm2)), bc(K.Mh));
      uxx = d2_mul(d2_sub(d2_sub(d2_scale2(d2_add(xp1, xm1), 16.0f), d2_add(xp2, xm2)), c30),
                   bc(K.Mh2));
      uyy = d2_mul(d2_sub(d2_sub(d2_scale2(d2_add(T(1, 0), T(-1, 0)), 16.0f),
                                 d2_add(T(2, 0), T(-2, 0))),
                          c30),
                   bc(K.Nh2));
    }
    const D2 uy = d2_mul(Y(0), bc(K.Nh));
    const D2 uxy =
        d2_mul(d2_sub(d2_scale2(d2_sub(Y(1), Y(-1)), 8.0f), d2_sub(Y(2), Y(-2))), bc(K.MNh));
    // the displaced points in grid units: cells and fractions (dd_floor per lane)
    int fa, fb;
    auto split = [&](D2 p, D2* t) {
      float pa, pb, ra, rb;
      upk(p.h, pa, pb);
      pa = floorf(pa);
      pb = floorf(pb);
      D2 f = d2_sub(p, D2{pk(pa, pb), 0ull});
      upk(f.h, ra, rb);
      if (ra < 0.f || ra >= 1.f || rb < 0.f || rb >= 1.f) {
        const float da = ra < 0.f ? 1.f : (ra >= 1.f ? -1.f : 0.f);
        const float db = rb < 0.f ? 1.f : (rb >= 1.f ? -1.f : 0.f);
        pa -= da;
        pb -= db;
        f = d2_add_f(f, pk(da, db));
      }
      *t = f;
      fa = (int)pa;
      fb = (int)pb;
    };
    D2 tX, tY;
    split(d2_add_f(d2_mul_f(ux, pk(K.M, K.M)), pk((float)j, (float)j)), &tX);
    auto wrap = [](int a, int L) { return (unsigned)a < (unsigned)L ? a : wrapi(a, L); };
    int ja[4], jb[4];
    ja[1] = wrap(fa, M);
    jb[1] = wrap(fb, M);
    split(d2_add_f(d2_mul_f(uy, pk(K.N, K.N)), pk((float)i, (float)(i + RB))), &tY);
    int ia[4], ib[4];
    ia[1] = wrap(fa, N);
    ib[1] = wrap(fb, N);
    auto taps = [](int (&k)[4], int L) {
      k[0] = k[1] == 0 ? L - 1 : k[1] - 1;
      k[2] = wrap_near(k[1] + 1, L);
      k[3] = wrap_near(k[1] + 2, L);
    };
    taps(ja, M);
    taps(jb, M);
    taps(ia, N);
    taps(ib, N);
    // the 16-tap gather, rows 0, 1 and rows 2, 3 summed apart; value weights in double-float, the gradient's in FP32 (Jacobian only)
    D2 wv[4];
    bspline6_dd2(tX, wv);
    u64 nw[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) nw[a] = neg2(wv[a].h);
    u64 wxf[4], dwx[4];
    bspline_w2(tX.h, wxf, dwx);
    D2 wy[4];
    bspline6_dd2(tY, wy);
    u64 wyf[4], dwy[4];
    bspline_w2(tY.h, wyf, dwy);
    D2 Gr[2];
    u64 gx = 0ull, gy = 0ull;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float2* ra = cdd + (size_t)ia[b] * M;
      const float2* rb = cdd + (size_t)ib[b] * M;
      D2 sv;
      u64 svf = 0ull, sdf = 0ull;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2 ca = __ldg(ra + ja[a]), cb = __ldg(rb + jb[a]);
        const D2 cv{pk(ca.x, cb.x), pk(ca.y, cb.y)};
        const D2 m = d2_mul_n(cv, wv[a], nw[a]);
        sv = a == 0 ? m : d2_add(m, sv);
        svf = a == 0 ? mul2(cv.h, wxf[0]) : fma2(cv.h, wxf[a], svf);
        sdf = a == 0 ? mul2(cv.h, dwx[0]) : fma2(cv.h, dwx[a], sdf);
      }
      const D2 m = d2_mul(sv, wy[b]);
      Gr[b / 2] = b % 2 == 0 ? m : d2_add(m, Gr[b / 2]);
      gx = b == 0 ? mul2(sdf, wyf[0]) : fma2(sdf, wyf[b], gx);
      gy = b == 0 ? mul2(svf, dwy[0]) : fma2(svf, dwy[b], gy);
    }
    const D2 G = d2_mul(d2_add(Gr[0], Gr[1]), bc(K.inv36));
    const D2 det = d2_sub(d2_mul(d2_add_f(uxx, one), d2_add_f(uyy, one)), d2_mul(uxy, uxy));
    const D2 fn = d2_mul(G, det);
    const size_t p = (size_t)i * M + j, pb = two ? p + (size_t)RB * M : p;
    const float2 f0 = __ldg(fdd + p), f1 = __ldg(fdd + pb);
    const D2 fr = d2_sub(D2{pk(f0.x, f1.x), pk(f0.y, f1.y)}, fn);
    dd ra, rb, na, nb, da, db;
    upk(fr.h, ra.hi, rb.hi);
    upk(fr.l, ra.lo, rb.lo);
    upk(fn.h, na.hi, nb.hi);
    upk(fn.l, na.lo, nb.lo);
    upk(det.h, da.hi, db.hi);
    upk(det.l, da.lo, db.lo);
    // coefficients of the linearisation (Jacobian only), FP32
    u64 cf[5];
    cf[0] = mul2(G.h, add2(one, uyy.h));
    cf[1] = neg2(mul2(G.h, uxy.h));
    cf[2] = mul2(G.h, add2(one, uxx.h));
    cf[3] = K.nob ? 0ull : mul2(det.h, mul2(gx, pk(K.M, K.M)));
    cf[4] = K.nob ? 0ull : mul2(det.h, mul2(gy, pk(K.N, K.N)));
    Fraw[p] = (double)ra.hi + (double)ra.lo;
    if (two) Fraw[pb] = (double)rb.hi + (double)rb.lo;
    const float w = ((i & 1) ? 4.0f : 2.0f) * K.w3N * wx;  // (rows i and i + RB alike)
#pragma unroll
    for (int a = 0; a < 5; ++a) {
      float x, y;
      upk(cf[a], x, y);
      coef[a * P + p] = x;
      simp[a] = fmaf(w, x, simp[a]);
      if (two) {
        coef[a * P + pb] = y;
        simp[a] = fmaf(w, y, simp[a]);
      }
    }
    auto finite = [](dd v) { return fabsf(v.hi) < INFINITY && fabsf(v.lo) < INFINITY; };
    if (finite(na)) {
      if (dd_gt(ra, acc.fmax)) acc.fmax = ra;
      if (dd_gt(acc.fmin, ra)) acc.fmin = ra;
    } else {
      na = dd{0.f, 0.f};
      ++acc.bad;
    }
    if (dd_gt(acc.dmin, da)) acc.dmin = da;
    if (two) {
      if (finite(nb)) {
        if (dd_gt(rb, acc.fmax)) acc.fmax = rb;
        if (dd_gt(acc.fmin, rb)) acc.fmin = rb;
      } else {
        nb = dd{0.f, 0.f};
        ++acc.bad;
      }
      if (dd_gt(acc.dmin, db)) acc.dmin = db;
    } else {
      nb = dd{0.f, 0.f};
    }
    sfn = d2_add(sfn, D2{pk(na.hi, nb.hi), pk(na.lo, nb.lo)});
  }
  {
    dd a, b;
    upk(sfn.h, a.hi, b.hi);
    upk(sfn.l, a.lo, b.lo);
    acc.s[0] = dd_add(a, b);
#pragma unroll
    for (int k = 0; k < 5; ++k) acc.s[1 + k] = dd{simp[k], 0.f};
  }
  // grid reductions: a block's ten values, then those of all blocks in the last one
  __shared__ bool last;
  __shared__ float2 tot[10];
  float2* pf = reinterpret_cast<float2*>(partials);
  const unsigned int nblk = gridDim.x * gridDim.y;
  resid_block_sums<RB>(acc, pf + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 10);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&sc->ticket[TK_RESID], 1u) == nblk - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  acc.fmax = dd{-INFINITY, 0.f};
  acc.fmin = acc.dmin = dd{INFINITY, 0.f};
  acc.bad = 0;
#pragma unroll
  for (int a = 0; a < 6; ++a) acc.s[a] = dd{0.f, 0.f};
  for (unsigned int b = tid; b < nblk; b += RB * RTX) {
    dd v[10];
#pragma unroll
    for (int a = 0; a < 10; ++a) {
      const float2 t = __ldcg(pf + (size_t)b * 10 + a);
      v[a] = dd{t.x, t.y};
    }
#pragma unroll
    for (int a = 0; a < 6; ++a) acc.s[a] = dd_add(acc.s[a], v[a]);
    if (dd_gt(v[6], acc.fmax)) acc.fmax = v[6];
    if (dd_gt(acc.fmin, v[7])) acc.fmin = v[7];
    if (dd_gt(acc.dmin, v[8])) acc.dmin = v[8];
    acc.bad += (int)v[9].hi;
  }
  resid_block_sums<RB>(acc, tot);
  __syncthreads();
  if (tid == 0) {
    double v[10];
    for (int a = 0; a < 10; ++a) v[a] = (double)tot[a].x + (double)tot[a].y;
    residual_close(sc, v, N, M);
  }
}

// split FP64 values into (hi, lo) float pairs
__global__ void k_split_dd(const double* __restrict__ in, float2* __restrict__ out, long n,
                           Bat bat) {
  in = badv(in, bat);
  out = badv(out, bat);
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n;
       k += (long)gridDim.x * blockDim.x) {
    const dd v = dd_from_double(in[k]);
    out[k] = make_float2(v.hi, v.lo);
  }
}

cudaError_t launch_split_dd(const double* in, float2* out, long n, cudaStream_t st, Bat bat) {
  long nb = (n + 255) / 256;
  if (nb > 4096) nb = 4096;
  if (nb < 1) nb = 1;
  k_split_dd<<<bgrid(dim3((int)nb), bat), 256, 0, st>>>(in, out, n, bat);
  return cudaGetLastError();
}

static dd host_dd(double v) {
  dd r;
  r.hi = (float)v;
  r.lo = (float)(v - (double)r.hi);
  return r;
}

cudaError_t launch_residual_dd(const float2* fdd, const float2* cdd, const double* ua, int N,
                               int M, double* Fraw, float* coef, double* partials,
                               DevScalars* sc, cudaStream_t st, const double* ub, int sel,
                               int simplified, Bat bat, Interp ip) {
  ResidConstsDD K;
  K.Mh = host_dd((double)M / 12.0);
  K.Nh = host_dd((double)N / 12.0);
  K.Mh2 = host_dd((double)M * (double)M / 12.0);
  K.Nh2 = host_dd((double)N * (double)N / 12.0);
  K.MNh = host_dd((double)M * (double)N / 144.0);
  K.inv36 = host_dd(1.0 / 36.0);
  K.M = (float)M;
  K.N = (float)N;
  K.w3M = (float)(1.0 / (3.0 * (double)M));
  K.w3N = (float)(1.0 / (3.0 * (double)N));
  K.nob = simplified ? 1 : 0;
  K.interp = ip.mode;
  K.gx = ip.gx32;
  K.gy = ip.gy32;
  if (ip.mode && !(ip.gx32 && ip.gy32)) return cudaErrorInvalidValue;
  const int mx = (M + RTX - 1) / RTX;
  const long tiles = (long)mx * ((N + 31) / 32) * (bat.on ? bat.n : 1);
  if (ip.mode) {
    // 32-row tiles (four points per thread), 8-row tiles on the smallest grids, where a thread's
    // four points in a row are the time.  8 / 32 rows, us, one GB300, bilinear: 10.4 / 16.3 at 128^2,
    // 13.2 / 16.6 at 256^2, 15.9 / 17.4 at 384 x 256 (96 tiles), 19.2 / 17.8 at 384^2 (144), 94 / 57 at
    // 1024^2; nearest node 15.3 / 16.3 and 18.4 / 16.6 at 96 and 144 tiles
    if (tiles > 96)
      k_residual_dd<4><<<bgrid(dim3(mx, (N + 31) / 32), bat), 8 * RTX, 0, st>>>(
          fdd, cdd, ua, ub, sel, N, M, K, Fraw, coef, partials, sc, bat);
    else
      k_residual_dd<1><<<bgrid(dim3(mx, (N + 7) / 8), bat), 8 * RTX, 0, st>>>(
          fdd, cdd, ua, ub, sel, N, M, K, Fraw, coef, partials, sc, bat);
    return cudaGetLastError();
  }
  // 16-row tiles by 256 threads (a pair of points each) while few blocks have to finish soon, by
  // 128 threads (two pairs) on middling grids, 32-row tiles by 128 (four pairs: least halo and
  // block sums) on large ones.  us, one GB300, in this order: 128^2 (16 tiles) 10.8 / 13.4 / 20.0,
  // 384^2 (144) 16.3 / 17.9 / 22.0, 512^2 (256) 24.2 / 24.4 / 25.5, five of 256^2 (320) 29.7 / 29.4 /
  // 31.8, five of 384^2 (720) 51.2 / 47.8 / 49.1, 1024^2 (1024) 71.1 / 67.0 / 63.6, 16 of 512^2
  // (4096) 268 / 238 / 226; one point per thread took 11.4, 22.2, 28.2, 37.6, 55.5, 75.5 and 258.
  if (tiles <= 256)
    k_residual_dd2<8, 1, 2><<<bgrid(dim3(mx, (N + 15) / 16), bat), 8 * RTX, 0, st>>>(
        fdd, cdd, ua, ub, sel, N, M, K, Fraw, coef, partials, sc, bat);
  else if (tiles < 1000)
    k_residual_dd2<4, 2, 4><<<bgrid(dim3(mx, (N + 15) / 16), bat), 4 * RTX, 0, st>>>(
        fdd, cdd, ua, ub, sel, N, M, K, Fraw, coef, partials, sc, bat);
  else
    k_residual_dd2<4, 4, 4><<<bgrid(dim3(mx, (N + 31) / 32), bat), 4 * RTX, 0, st>>>(
        fdd, cdd, ua, ub, sel, N, M, K, Fraw, coef, partials, sc, bat);
  return cudaGetLastError();
}

// mean-zero gauge: u <- u - mean(u) (two launches: sum, then subtract)
__global__ void k_sum(const double* __restrict__ u, long P, double* partials, DevScalars* sc,
                      double* mean_out) {
  double v[1] = {0.0};
  const int kind[1] = {0};
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    v[0] += u[p];
  block_reduce<1>(v, kind);
  if (!publish_partials<1>(v, partials, &sc->ticket[TK_NORM])) return;
  reduce_partials<1>(v, kind, partials, gridDim.x);
  if (threadIdx.x == 0) {
    *mean_out = v[0] / (double)P;
    sc->ticket[TK_NORM] = 0;
  }
}

__global__ void k_sub(double* __restrict__ u, long P, const double* __restrict__ mean) {
  const double m = *mean;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    u[p] -= m;
}

cudaError_t launch_subtract_mean(double* u, int N, int M, double* partials, DevScalars* sc,
                                 double* mean_out, cudaStream_t st) {
  const int nb = reduce_blocks((long)N * M);
  k_sum<<<nb, 256, 0, st>>>(u, (long)N * M, partials, sc, mean_out);
  k_sub<<<nb, 256, 0, st>>>(u, (long)N * M, mean_out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// GMRES(m) (Sec. 4.2).  The basis V_i is stored unnormalised with v_i = scale[i] V_i so
// that no kernel pass is spent on normalisation.  Arnoldi uses classical Gram-Schmidt: a
// multi-dot pass (V_i.w and w.w) and an update pass, whose first block also closes the step: the
// norm of the new vector by Pythagoras, the Givens rotation.  A plan set's large classes close it in
// the multi-dot's last block, and with reorthogonalisation (two such rounds) the second
// update's last block does, from the new vector's own norm.
// Every kernel returns at once when the current cycle is finished (cycle_done), so a fixed
// sequence of launches can be queued without host round trips.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void k_gmres_init(const double* __restrict__ Fraw, const T* __restrict__ w,
                             T* __restrict__ V0, long P, int restart, double* partials,
                             DevScalars* sc, T* __restrict__ sigma, Bat bat) {
  Fraw = badv(Fraw, bat);
  w = badv(w, bat);
  V0 = badv(V0, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  sigma = badv(sigma, bat);
  if (bskip(sc, bat)) return;
  const double s = sc->shift, inv_tau = 1.0 / sc->tau;
  double v[1] = {0.0};
  const int kind[1] = {0};
  T acc = (T)0;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x) {
    if (sigma) sigma[p] = (T)0;
    T bt;
    if constexpr (sizeof(T) == 4) {
      // the shifted residual in FP64 (one add), the rest in the vector precision
      float b = dd_from_double(Fraw[p] + s).hi * (float)inv_tau;  // h = (f - f~_n) / tau
      if (restart) b -= w[p];
      bt = b;
    } else {
      double b = (Fraw[p] + s) * inv_tau;
      if (restart) b -= (double)w[p];
      bt = (T)b;
    }
    V0[p] = bt;
    acc += bt * bt;
  }
  if constexpr (sizeof(T) == 4) {
    float a[1] = {acc};
    if (!grid_sum_f<1>(a, partials, &sc->ticket[TK_INIT])) return;
    v[0] = (double)a[0];
  } else {
    v[0] = (double)acc;
    block_reduce<1>(v, kind);
    if (!publish_partials<1>(v, partials, &sc->ticket[TK_INIT])) return;
    reduce_partials<1>(v, kind, partials, gridDim.x);
  }
  if (threadIdx.x == 0) {
    const double beta = sqrt(v[0]);
    if (!restart) {
      // a new Newton step: the last residual evaluated was the current iterate's
      for (int a = 0; a < 5; ++a) sc->abar_n[a] = sc->abar[a];
      sc->bnorm = beta;
      sc->iters = 0;
      sc->cycles = 0;
      sc->converged = (beta == 0.0);
    } else {
      if (beta <= sc->eta * sc->bnorm) sc->converged = 1;
    }
    sc->beta = beta;
    sc->j = 0;
    sc->jend = 0;
    sc->cycle_done = sc->converged;
    if (!sc->converged) sc->cycles += 1;
    for (int k = 0; k <= OTGB_MAXM; ++k) sc->gv[k] = 0.0;
    sc->gv[0] = beta;
    sc->scale[0] = beta > 0.0 ? 1.0 / beta : 0.0;
    sc->ticket[TK_INIT] = 0;
  }
}

// 16-byte vector access to the Krylov vectors (float4 / double2): when P is a multiple of
// the width every vector V_i = V + i P stays 16-byte aligned and the loops run over whole
// vectors (the loop over q below), else element by element (the tail loop covers all).
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  using type = float4;
  static constexpr int W = 4;
};
template <> struct Vec16<double> {
  using type = double2;
  static constexpr int W = 2;
};
template <typename T>
__device__ __forceinline__ void vld(const T* __restrict__ base, long q, T (&x)[Vec16<T>::W]) {
  const typename Vec16<T>::type v = reinterpret_cast<const typename Vec16<T>::type*>(base)[q];
  memcpy(x, &v, sizeof(v));
}
template <typename T>
__device__ __forceinline__ void vst(T* __restrict__ base, long q, const T (&x)[Vec16<T>::W]) {
  typename Vec16<T>::type v;
  memcpy(&v, x, sizeof(v));
  reinterpret_cast<typename Vec16<T>::type*>(base)[q] = v;
}
// number of whole vectors of the 16-byte loops (0: element loop only)
__device__ __forceinline__ long nvec(long P, int W) { return P % W == 0 ? P / W : 0; }

// Close Arnoldi step j (one thread): H(j+1, j) = hn, the previous Givens rotations and a new
// one on column j, the residual estimate |g_(j+1)|, convergence / end of cycle, v_(j+1) =
// w / hn, and the conditional handle of step j + 1.  weak: hn came out below the resolution
// of the Pythagorean norm; the cycle ends without a convergence claim (the restart
// recomputes the residual explicitly).
__device__ void arnoldi_close(DevScalars* sc, int j, double hn, bool weak) {
  double* H = sc->H;
  const int m = sc->m;
  H[(j + 1) * m + j] = hn;
  for (int i = 0; i < j; ++i) {  // previous rotations on column j
    const double t0 = H[i * m + j], t1 = H[(i + 1) * m + j];
    H[i * m + j] = sc->cs[i] * t0 + sc->sn[i] * t1;
    H[(i + 1) * m + j] = -sc->sn[i] * t0 + sc->cs[i] * t1;
  }
  const double a = H[j * m + j], b = H[(j + 1) * m + j];
  const double r = sqrt(a * a + b * b);
  sc->cs[j] = (r == 0.0) ? 1.0 : a / r;
  sc->sn[j] = (r == 0.0) ? 0.0 : b / r;
  H[j * m + j] = r;
  H[(j + 1) * m + j] = 0.0;
  sc->gv[j + 1] = -sc->sn[j] * sc->gv[j];
  sc->gv[j] = sc->cs[j] * sc->gv[j];
  sc->iters += 1;
  sc->jend = j + 1;
  if (weak) {
    sc->cycle_done = 1;
  } else if (fabs(sc->gv[j + 1]) <= sc->eta * sc->bnorm || hn == 0.0) {
    sc->converged = 1;
    sc->cycle_done = 1;
  } else {
    sc->scale[j + 1] = 1.0 / hn;
    if (j + 1 == m) sc->cycle_done = 1;
  }
  sc->j = j + 1;
  // the handle of step j + 1 (the tail WHILE of the captured cycle for j + 1 >= its plain
  // steps, including j + 1 = m, where the cycle is done and the loop ends)
  if (sc->graph && j + 1 < OTGB_MAXM && sc->h_step[j + 1])
    cudaGraphSetConditional(sc->h_step[j + 1], sc->cycle_done ? 0u : 1u);
}

// Per-thread partial sums are kept in the vector precision T (a thread covers a few vectors
// of 16 bytes); partials are combined across threads and blocks in FP64.
template <typename T, int J>
__device__ __forceinline__ void dots_j(const T* __restrict__ V, const T* __restrict__ w, long P,
                                       double* partials, DevScalars* sc, int pass,
                                       bool split) {
  constexpr int W = Vec16<T>::W;
  T acc[J + 1];  // V_i . w (i < J) and w . w
#pragma unroll
  for (int i = 0; i <= J; ++i) acc[i] = (T)0;
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long nth = (long)gridDim.x * blockDim.x, PV = nvec(P, W);
  for (long q = tid; q < PV; q += nth) {
    T wv[W];
    vld<T>(w, q, wv);
#pragma unroll
    for (int i = 0; i < J; ++i) {
      T x[W];
      vld<T>(V + (size_t)i * P, q, x);
#pragma unroll
      for (int k = 0; k < W; ++k) acc[i] += x[k] * wv[k];
    }
#pragma unroll
    for (int k = 0; k < W; ++k) acc[J] += wv[k] * wv[k];
  }
  for (long p = PV * W + tid; p < P; p += nth) {
    const T wp = w[p];
#pragma unroll
    for (int i = 0; i < J; ++i) acc[i] += V[(size_t)i * P + p] * wp;
    acc[J] += wp * wp;
  }
  double v[J + 1];
  if constexpr (sizeof(T) == 4) {
    if (split && pass == 0 && !sc->reorth) {
      // single-reduction step (split): the block's sums go to its partials and the
      // update kernel finishes the step (every block of it sums the partials in the same
      // order; its block 0 closes the step) -- no last-block pass and no serial close here
      block_sum_f<J + 1>(acc);
      if (threadIdx.x == 0) {
        float* pf = reinterpret_cast<float*>(partials);
#pragma unroll
        for (int a = 0; a <= J; ++a) pf[(size_t)blockIdx.x * (J + 1) + a] = acc[a];
        if (blockIdx.x == 0) sc->jd = J - 1;
      }
      return;
    }
    if (!grid_sum_f<J + 1>(acc, partials, &sc->ticket[TK_DOTS])) return;
#pragma unroll
    for (int i = 0; i <= J; ++i) v[i] = (double)acc[i];
  } else {
    if (split && pass == 0 && !sc->reorth) {
      // the same split in FP64, the sums value by value
      double s;
      if (block_fold<J + 1>(acc, s))
        partials[(size_t)(threadIdx.x >> 3) * gridDim.x + blockIdx.x] = s;
      if (blockIdx.x == 0 && threadIdx.x == 0) sc->jd = J - 1;
      return;
    }
    int kind[J + 1];
#pragma unroll
    for (int i = 0; i <= J; ++i) {
      v[i] = (double)acc[i];
      kind[i] = 0;
    }
    block_reduce<J + 1>(v, kind);
    if (!publish_partials<J + 1>(v, partials, &sc->ticket[TK_DOTS])) return;
    reduce_partials<J + 1>(v, kind, partials, gridDim.x);
  }
  if (threadIdx.x == 0) {
    const int m = sc->m, j = J - 1;
    if (pass == 0 && !sc->reorth) {
      // one reduction per Arnoldi step: with v_i orthonormal, ||w - sum h_i v_i||^2 =
      // ||w||^2 - sum h_i^2 (Pythagoras), so the norm and the Givens rotation finish here
      // and the update of w is a plain elementwise pass (mode 3) that ends no reduction.
      // The difference loses accuracy when w lies almost in span(v_0..v_j); below 1e-6
      // ||w||^2 (the FP32 sums' resolution) the cycle ends and the restart's explicit
      // residual decides.
      double h[J], hs = 0.0;
#pragma unroll
      for (int i = 0; i < J; ++i) h[i] = sc->scale[i] * v[i];
#pragma unroll
      for (int i = 0; i < J; ++i) {
        sc->hcol[i] = h[i];
        hs += h[i] * h[i];
      }
      const double ww = v[J], hn2 = ww - hs;
      const bool weak = !(hn2 > 1e-6 * ww);
      const double inv_hn = weak ? 0.0 : rsqrt(hn2);
      arnoldi_close_j<J>(sc, h, hn2 * inv_hn, weak, inv_hn);
    } else if (pass == 0) {
#pragma unroll
      for (int i = 0; i < J; ++i) sc->H[i * m + j] = sc->scale[i] * v[i];
    } else {
#pragma unroll
      for (int i = 0; i < J; ++i) {
        sc->h2[i] = sc->scale[i] * v[i];
        sc->H[i * m + j] += sc->h2[i];
      }
    }
    sc->ticket[TK_DOTS] = 0;
  }
}

template <typename T>
__global__ void k_gmres_dots(const T* __restrict__ V, const T* __restrict__ w, long P,
                             double* partials, DevScalars* sc, int pass, Bat bat) {
  V = badv(V, bat);
  w = badv(w, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat) || sc->cycle_done) return;
  if (pass) w = V + (size_t)(sc->j + 1) * P;
  // the split step (close in the update) serves single problems and small classes of a plan
  // set; large classes close in the multi-dot's last block
  const bool split = !bat.on || bat.split;
  switch (sc->j) {
#define OTGB_DOTS_CASE(k) \
  case k:                 \
    dots_j<T, k + 1>(V, w, P, partials, sc, pass, split); break;
    OTGB_DOTS_CASE(0) OTGB_DOTS_CASE(1) OTGB_DOTS_CASE(2) OTGB_DOTS_CASE(3)
    OTGB_DOTS_CASE(4) OTGB_DOTS_CASE(5) OTGB_DOTS_CASE(6) OTGB_DOTS_CASE(7)
    OTGB_DOTS_CASE(8) OTGB_DOTS_CASE(9) OTGB_DOTS_CASE(10) OTGB_DOTS_CASE(11)
    OTGB_DOTS_CASE(12) OTGB_DOTS_CASE(13) OTGB_DOTS_CASE(14)
#undef OTGB_DOTS_CASE
  }
}

template <typename T, int J>
__device__ __forceinline__ void update_j(T* __restrict__ V, const T* __restrict__ w, long P,
                                         double* partials, DevScalars* sc, int mode,
                                         bool split) {
  const int j = J - 1, m = sc->m;
  T coefs[J];
  double hv[J], hn = 0.0, inv_hn = 0.0;
  bool weak = false;
  if (mode == 3 && split) {
    finish_multidot<T, J>(partials, gridDim.x, sc, hv, hn, inv_hn, weak, coefs);
  } else {
#pragma unroll
    for (int i = 0; i < J; ++i)
      coefs[i] = (T)((mode == 2 ? sc->h2[i] : (mode == 3 ? sc->hcol[i] : sc->H[i * m + j])) *
                     sc->scale[i]);
  }
  T* Vn = V + (size_t)(j + 1) * P;
  const T* src = (mode == 2) ? Vn : w;
  T acc = (T)0;
  constexpr int W = Vec16<T>::W;
  // split mode 3: block 0 closes the step (one thread's serial FP64 work and round trips)
  // while the other blocks form v_(j+1); otherwise every block takes part
  const bool closer = mode == 3 && split && gridDim.x > 1;
  if (closer && blockIdx.x == 0) {
    if (threadIdx.x == 0) {
#pragma unroll
      for (int i = 0; i < J; ++i) sc->hcol[i] = hv[i];
      arnoldi_close_j<J>(sc, hv, hn, weak, inv_hn);
    }
    return;
  }
  const long bid = closer ? blockIdx.x - 1 : blockIdx.x, nbk = closer ? gridDim.x - 1 : gridDim.x;
  const long tid = bid * (long)blockDim.x + threadIdx.x;
  const long nth = nbk * blockDim.x, PV = nvec(P, W);
  for (long q = tid; q < PV; q += nth) {
    T x[W];
    vld<T>(src, q, x);
#pragma unroll
    for (int i = 0; i < J; ++i) {
      T y[W];
      vld<T>(V + (size_t)i * P, q, y);
#pragma unroll
      for (int k = 0; k < W; ++k) x[k] -= coefs[i] * y[k];
    }
    vst<T>(Vn, q, x);
#pragma unroll
    for (int k = 0; k < W; ++k) acc += x[k] * x[k];
  }
  for (long p = PV * W + tid; p < P; p += nth) {
    T x = src[p];
#pragma unroll
    for (int i = 0; i < J; ++i) x -= coefs[i] * V[(size_t)i * P + p];
    Vn[p] = x;
    acc += x * x;
  }
  // mode 1: first of two passes, the norm follows the second; mode 3: the step was closed
  // by block 0 above or by the multi-dot (a plan set's large classes)
  if (mode == 1 || mode == 3) {
    if (mode == 3 && split && !closer && blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
      for (int i = 0; i < J; ++i) sc->hcol[i] = hv[i];
      arnoldi_close_j<J>(sc, hv, hn, weak, inv_hn);
    }
    return;
  }
  double v[1] = {(double)acc};
  if constexpr (sizeof(T) == 4) {
    float a[1] = {acc};
    if (!grid_sum_f<1>(a, partials, &sc->ticket[TK_UPDATE])) return;
    v[0] = (double)a[0];
  } else {
    const int kind[1] = {0};
    block_reduce<1>(v, kind);
    if (!publish_partials<1>(v, partials, &sc->ticket[TK_UPDATE])) return;
    reduce_partials<1>(v, kind, partials, gridDim.x);
  }
  if (threadIdx.x == 0) {
    arnoldi_close(sc, j, sqrt(v[0]), false);
    sc->ticket[TK_UPDATE] = 0;
  }
}

template <typename T>
__global__ void k_gmres_update(T* __restrict__ V, const T* __restrict__ w, long P,
                               double* partials, DevScalars* sc, int mode, Bat bat) {
  V = badv(V, bat);
  w = badv(w, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat) || sc->cycle_done) return;
  // mode 3 follows the multi-dot of step jd (split: the update closes the step itself and
  // advances sc->j, so it reads the step from jd; else the multi-dot closed it and advanced
  // sc->j)
  const bool split = !bat.on || bat.split;
  switch (mode == 3 ? (split ? sc->jd : sc->j - 1) : sc->j) {
#define OTGB_UPD_CASE(k) \
  case k:                \
    update_j<T, k + 1>(V, w, P, partials, sc, mode, split); break;
    OTGB_UPD_CASE(0) OTGB_UPD_CASE(1) OTGB_UPD_CASE(2) OTGB_UPD_CASE(3)
    OTGB_UPD_CASE(4) OTGB_UPD_CASE(5) OTGB_UPD_CASE(6) OTGB_UPD_CASE(7)
    OTGB_UPD_CASE(8) OTGB_UPD_CASE(9) OTGB_UPD_CASE(10) OTGB_UPD_CASE(11)
    OTGB_UPD_CASE(12) OTGB_UPD_CASE(13) OTGB_UPD_CASE(14)
#undef OTGB_UPD_CASE
  }
}

// y = R^{-1} g by back substitution: the 32 threads stage R and g in shared memory (one
// round of independent loads), thread 0 solves there
__global__ void k_gmres_finish(DevScalars* sc, Bat bat) {
  __shared__ double R[OTGB_MAXM * OTGB_MAXM], g[OTGB_MAXM], y[OTGB_MAXM];
  sc = badv(sc, bat);
  if (blockIdx.x != 0 || bskip(sc, bat)) return;
  const int n = sc->jend, m = sc->m;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) R[e] = sc->H[(e / n) * m + e % n];
  for (int e = threadIdx.x; e < n; e += blockDim.x) g[e] = sc->gv[e];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = n - 1; i >= 0; --i) {
      double s = g[i];
      for (int k = i + 1; k < n; ++k) s -= R[i * n + k] * y[k];
      y[i] = s / R[i * n + i];
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += blockDim.x) sc->y[e] = y[e];
}

cudaError_t launch_gmres_finish(DevScalars* sc, cudaStream_t st, Bat bat) {
  k_gmres_finish<<<bgrid(dim3(1), bat), 32, 0, st>>>(sc, bat);
  return cudaGetLastError();
}

// sigma += sum_i y_i scale_i V_i
template <typename T, int J>
__device__ __forceinline__ void combine_j(const T* __restrict__ V, T* __restrict__ sigma, long P,
                                          const DevScalars* __restrict__ sc) {
  T coefs[J];
#pragma unroll
  for (int i = 0; i < J; ++i) coefs[i] = (T)(sc->y[i] * sc->scale[i]);
  constexpr int W = Vec16<T>::W;
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long nth = (long)gridDim.x * blockDim.x, PV = nvec(P, W);
  for (long q = tid; q < PV; q += nth) {
    T x[W];
    vld<T>(sigma, q, x);
#pragma unroll
    for (int i = 0; i < J; ++i) {
      T y[W];
      vld<T>(V + (size_t)i * P, q, y);
#pragma unroll
      for (int k = 0; k < W; ++k) x[k] += coefs[i] * y[k];
    }
    vst<T>(sigma, q, x);
  }
  for (long p = PV * W + tid; p < P; p += nth) {
    T x = sigma[p];
#pragma unroll
    for (int i = 0; i < J; ++i) x += coefs[i] * V[(size_t)i * P + p];
    sigma[p] = x;
  }
}

template <typename T>
__global__ void k_gmres_combine(const T* __restrict__ V, T* __restrict__ sigma, long P,
                                const DevScalars* __restrict__ sc, Bat bat) {
  V = badv(V, bat);
  sigma = badv(sigma, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  switch (sc->jend) {
#define OTGB_CMB_CASE(k) \
  case k:                \
    combine_j<T, k>(V, sigma, P, sc); break;
    OTGB_CMB_CASE(1) OTGB_CMB_CASE(2) OTGB_CMB_CASE(3) OTGB_CMB_CASE(4)
    OTGB_CMB_CASE(5) OTGB_CMB_CASE(6) OTGB_CMB_CASE(7) OTGB_CMB_CASE(8)
    OTGB_CMB_CASE(9) OTGB_CMB_CASE(10) OTGB_CMB_CASE(11) OTGB_CMB_CASE(12)
    OTGB_CMB_CASE(13) OTGB_CMB_CASE(14) OTGB_CMB_CASE(15)
#undef OTGB_CMB_CASE
    default: break;
  }
}

template <typename T>
cudaError_t launch_gmres_init(const double* Fraw, const T* w, T* V0, long P, int restart,
                              double* partials, DevScalars* sc, int nblocks, cudaStream_t st,
                              T* sigma, Bat bat) {
  k_gmres_init<T><<<bgrid(dim3(nblocks), bat), 256, 0, st>>>(Fraw, w, V0, P, restart, partials,
                                                             sc, sigma, bat);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_gmres_dots(const T* V, const T* w, long P, double* partials, DevScalars* sc,
                              int nblocks, cudaStream_t st, int pass, Bat bat) {
  k_gmres_dots<T><<<bgrid(dim3(nblocks), bat), 256, 0, st>>>(V, w, P, partials, sc, pass, bat);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_gmres_update(T* V, const T* w, long P, double* partials, DevScalars* sc,
                                int nblocks, cudaStream_t st, int mode, Bat bat) {
  k_gmres_update<T><<<bgrid(dim3(nblocks), bat), 256, 0, st>>>(V, w, P, partials, sc, mode,
                                                               bat);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_gmres_combine(const T* V, T* sigma, long P, const DevScalars* sc,
                                 int nblocks, cudaStream_t st, Bat bat) {
  k_gmres_combine<T><<<bgrid(dim3(nblocks), bat), 256, 0, st>>>(V, sigma, P, sc, bat);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Device-resident Newton control (Eq. linma with the convexity safeguard), one thread.
// Mirrors the host loop: stop tests before each solve, step halving on an inadmissible
// candidate, s doubled (capped at 1) after an accepted step.
// ---------------------------------------------------------------------------------------
#define OT_STATUS_OK 0
#define OT_STATUS_EINVAL (-1)
#define OT_STATUS_ENOCONV (-2)
#define OT_STATUS_EDIVERGED (-3)

__device__ __forceinline__ void set_cond(const DevScalars* sc, unsigned long long h,
                                         unsigned int v) {
  if (sc->graph && h) cudaGraphSetConditional(h, v);
}

// One control operation on one problem's scalars.  handles = 0: a batched solve, whose
// conditional handles are set once for all pairs by k_ctl_batch (and whose Arnoldi steps are
// not conditional); the return value is what the operation's handle would receive.
__device__ int ctl_apply(int op, DevScalars* sc, int add, bool handles) {
  sc->kcount += add;
  int cont = 0;
  switch (op) {
    case CTL_NEWTON: {
      // tau schedule: the damping drops to 1 for good once max|F| < tau_switch
      if (sc->tau_switch > 0.0 && sc->res_inf < sc->tau_switch) sc->tau = 1.0;
      if (sc->in_bad) {
        sc->status = OT_STATUS_EINVAL;
      } else if (!sc->admissible) {
        sc->status = OT_STATUS_EDIVERGED;
      } else if (sc->res_inf < sc->tol) {
        sc->status = OT_STATUS_OK;
      } else if (sc->newton_n >= sc->max_newton) {
        sc->status = OT_STATUS_ENOCONV;
      } else {
        sc->status = OT_STATUS_OK;
        cont = 1;
      }
      sc->active = cont;
      if (handles) set_cond(sc, sc->h_newton, cont);
      break;
    }
    case CTL_ACCEPT: {
      const double s = sc->step_s;
      if (!sc->safeguard || sc->admissible || s < 0x1p-30) {
        sc->upar ^= 1;
        sc->newton_n += 1;
        sc->step_s = (2.0 * s < 1.0) ? 2.0 * s : 1.0;
      } else {
        sc->step_s = 0.5 * s;
        sc->halvings += 1;
        cont = 1;
      }
      sc->halve = cont;
      if (handles) set_cond(sc, sc->h_halve, cont);
      break;
    }
    case CTL_PRE_CYCLE:
      cont = sc->converged ? 0 : 1;
      sc->in_cycle = cont;
      if (handles) set_cond(sc, sc->h_cycle, cont);
      break;
    case CTL_CYCLE_BEGIN:
      if (handles) {
        for (int k = 1; k < sc->m; ++k) set_cond(sc, sc->h_step[k], 0);
        set_cond(sc, sc->h_step[0], sc->converged ? 0u : 1u);
      }
      break;
    case CTL_CYCLE_END: {
      // the unconditional Arnoldi steps a short cycle left also launched (and skipped)
      if (handles && sc->jend < sc->steps_uncond)
        sc->kcount += (long long)sc->step_kernels * (sc->steps_uncond - sc->jend);
      cont = (!sc->converged && sc->cycles < sc->max_restarts) ? 1 : 0;
      sc->in_cycle = cont;
      if (handles) {
        set_cond(sc, sc->h_cycle, cont);
        set_cond(sc, sc->h_restart, cont);
        if (cont) sc->kcount += 4;  // restart residual: 3 matvec passes + init
      }
      break;
    }
    case CTL_FORCING:
      // Eisenstat & Walker (1996), choice 2 with gamma = 0.9, alpha = 2: eta = gamma
      // (|F_k| / |F_k-1|)^2, kept >= gamma eta_prev^2 when that exceeds 0.1, at most eta_max;
      // and no tighter than needed to reach the Newton tolerance (0.5 tol / |F_k|)
      if (sc->forcing) {
        const double r = sc->res_inf, rp = sc->res_prev;
        double e = sc->eta_max;
        if (rp > 0.0) {
          const double q = r / rp;
          e = 0.9 * q * q;
          const double sg = 0.9 * sc->eta * sc->eta;
          if (sg > 0.1) e = fmax(e, sg);
          e = fmin(e, sc->eta_max);
        }
        e = fmax(e, fmin(sc->eta_max, 0.5 * sc->tol / r));
        e = fmax(e, 1e-6);
        sc->eta = e;
        sc->res_prev = r;
      }
      break;
    case CTL_GMRES_DONE:
      // Arnoldi steps: 3 matvec passes + dots + update (+ dots + update when reorthogonal.;
      // the fused update carries the next step's first matvec pass)
      if (handles) sc->kcount += (long long)sc->step_kernels * sc->iters;
      sc->gmres_iters_total += sc->iters;
      sc->gmres_cycles_total += sc->cycles;
      break;
  }
  return cont;
}

__global__ void k_ctl(int op, DevScalars* sc, int add) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  ctl_apply(op, sc, add, true);
}

// The same operation for every pair of a batched solve the mask selects (one thread per
// pair), then the operation's conditional handle set to "any pair continues".  Kernel
// launches are counted on pair 0 (the launches are shared by the pairs).
__global__ void k_ctl_batch(int op, DevScalars* sc, int add, Bat bat) {
  int cont = 0;
  const int b = threadIdx.x;
  if (b < bat.n) {
    DevScalars* s = reinterpret_cast<DevScalars*>(reinterpret_cast<uintptr_t>(sc) +
                                                  (size_t)b * bat.slab);
    if (!bskip(s, bat)) cont = ctl_apply(op, s, b == 0 ? add : 0, false);
  }
  const int any = __syncthreads_or(cont);
  if (threadIdx.x == 0) {
    switch (op) {
      case CTL_NEWTON: set_cond(sc, sc->h_newton, any); break;
      case CTL_ACCEPT: set_cond(sc, sc->h_halve, any); break;
      case CTL_PRE_CYCLE: set_cond(sc, sc->h_cycle, any); break;
      case CTL_CYCLE_END:
        set_cond(sc, sc->h_cycle, any);
        set_cond(sc, sc->h_restart, any);
        if (any) sc->kcount += 4;
        break;
    }
  }
}

cudaError_t launch_ctl(int op, DevScalars* sc, cudaStream_t st, int add, Bat bat) {
  if (bat.on) {
    if (bat.n > 1024) return cudaErrorInvalidValue;
    k_ctl_batch<<<1, (bat.n + 31) / 32 * 32, 0, st>>>(op, sc, add, bat);
  } else {
    k_ctl<<<1, 32, 0, st>>>(op, sc, add);
  }
  return cudaGetLastError();
}

__global__ void k_sum_sel(UPair up, long P, double* partials, DevScalars* sc, double* mean_out,
                          Bat bat) {
  up.a = badv(up.a, bat);
  up.b = badv(up.b, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  mean_out = badv(mean_out, bat);
  if (bskip(sc, bat)) return;
  const double* __restrict__ u = (sc->upar & 1) ? up.b : up.a;
  double v[1] = {0.0};
  const int kind[1] = {0};
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    v[0] += u[p];
  block_reduce<1>(v, kind);
  if (!publish_partials<1>(v, partials, &sc->ticket[TK_NORM])) return;
  reduce_partials<1>(v, kind, partials, gridDim.x);
  if (threadIdx.x == 0) {
    *mean_out = v[0] / (double)P;
    sc->ticket[TK_NORM] = 0;
  }
}

__global__ void k_sub_sel(UPair up, double* __restrict__ out, long P,
                          const DevScalars* __restrict__ sc, const double* __restrict__ mean,
                          Bat bat) {
  up.a = badv(up.a, bat);
  up.b = badv(up.b, bat);
  out = badv(out, bat);
  sc = badv(sc, bat);
  mean = badv(mean, bat);
  if (bskip(sc, bat)) return;
  const double* __restrict__ u = (sc->upar & 1) ? up.b : up.a;
  const double m = *mean;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    out[p] = u[p] - m;
}

cudaError_t launch_final_gauge(UPair u, double* out, int N, int M, double* partials,
                               DevScalars* sc, double* mean_out, cudaStream_t st, Bat bat) {
  const dim3 nb = bgrid(dim3(reduce_blocks((long)N * M)), bat);
  k_sum_sel<<<nb, 256, 0, st>>>(u, (long)N * M, partials, sc, mean_out, bat);
  k_sub_sel<<<nb, 256, 0, st>>>(u, out, (long)N * M, sc, mean_out, bat);
  return cudaGetLastError();
}

// grid gradient of g by the 4th-order centred differences (periodic), FP64 and FP32 copies:
// the nearest-node and bilinear interpolation modes interpolate it at the displaced points
__global__ void k_grad4(const double* __restrict__ g, int N, int M, double* __restrict__ gx,
                        double* __restrict__ gy, float* __restrict__ gx32,
                        float* __restrict__ gy32) {
  const long P = (long)N * M;
  const double sx = (double)M / 12.0, sy = (double)N / 12.0;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x) {
    const int i = (int)(p / M), j = (int)(p - (long)i * M);
    const double* row = g + (size_t)i * M;
    const int jm1 = wrapi(j - 1, M), jm2 = wrapi(j - 2, M), jp1 = wrapi(j + 1, M),
              jp2 = wrapi(j + 2, M);
    const int im1 = wrapi(i - 1, N), im2 = wrapi(i - 2, N), ip1 = wrapi(i + 1, N),
              ip2 = wrapi(i + 2, N);
    const double a = (-row[jp2] + 8.0 * row[jp1] - 8.0 * row[jm1] + row[jm2]) * sx;
    const double b = (-g[(size_t)ip2 * M + j] + 8.0 * g[(size_t)ip1 * M + j] -
                      8.0 * g[(size_t)im1 * M + j] + g[(size_t)im2 * M + j]) * sy;
    gx[p] = a;
    gy[p] = b;
    gx32[p] = (float)a;
    gy32[p] = (float)b;
  }
}

cudaError_t launch_grad4(const double* g, int N, int M, double* gx, double* gy, float* gx32,
                         float* gy32, cudaStream_t st) {
  k_grad4<<<reduce_blocks((long)N * M), 256, 0, st>>>(g, N, M, gx, gy, gx32, gy32);
  return cudaGetLastError();
}

// 2-norm and normalisation of a vector (the power iteration of the inverse operator)
__global__ void k_norm2(const double* __restrict__ x, long P, double* partials, DevScalars* sc) {
  double v[1] = {0.0};
  const int kind[1] = {0};
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    v[0] += x[p] * x[p];
  block_reduce<1>(v, kind);
  if (!publish_partials<1>(v, partials, &sc->ticket[TK_NORM])) return;
  reduce_partials<1>(v, kind, partials, gridDim.x);
  if (threadIdx.x == 0) {
    sc->pw_norm = sqrt(v[0]);
    sc->ticket[TK_NORM] = 0;
  }
}

__global__ void k_scale_by_norm(double* __restrict__ x, long P, const DevScalars* __restrict__ sc) {
  const double n = sc->pw_norm;
  const double s = n > 0.0 ? 1.0 / n : 0.0;
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    x[p] *= s;
}

// kernel timing: put an Arnoldi step back to step j of an open cycle, outside any graph
// (the step's close must not touch the conditional handles of the plan's solve graph, which
// may have been destroyed since)
__global__ void k_set_step(DevScalars* sc, int j) {
  sc->j = j;
  sc->jd = j;
  sc->cycle_done = 0;
  sc->graph = 0;
  sc->ticket[TK_DOTS] = 0;
}

cudaError_t launch_set_step(DevScalars* sc, int j, cudaStream_t st) {
  k_set_step<<<1, 1, 0, st>>>(sc, j);
  return cudaGetLastError();
}

cudaError_t launch_normalize(double* x, long P, double* partials, DevScalars* sc,
                             cudaStream_t st) {
  const int nb = reduce_blocks(P);
  k_norm2<<<nb, 256, 0, st>>>(x, P, partials, sc);
  k_scale_by_norm<<<nb, 256, 0, st>>>(x, P, sc);
  return cudaGetLastError();
}

// batched solve: copies between the pairs' slabs and the caller's per-pair planes
__global__ void k_gather(const double* const* __restrict__ tab, double* __restrict__ dst, long P,
                         Bat bat) {
  const double* __restrict__ src = tab[blockIdx.z];
  dst = badv(dst, bat);
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    dst[p] = src[p];
}

__global__ void k_scatter(const double* __restrict__ src, double* const* __restrict__ tab,
                          long P, const DevScalars* __restrict__ sc, Bat bat) {
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  double* __restrict__ dst = tab[blockIdx.z];
  src = badv(src, bat);
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < P;
       p += (long)gridDim.x * blockDim.x)
    dst[p] = src[p];
}

cudaError_t launch_gather(const double* const* tab, double* dst, long P, Bat bat,
                          cudaStream_t st) {
  k_gather<<<bgrid(dim3(reduce_blocks(P)), bat), 256, 0, st>>>(tab, dst, P, bat);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const double* src, double* const* tab, long P, const DevScalars* sc,
                           Bat bat, cudaStream_t st) {
  k_scatter<<<bgrid(dim3(reduce_blocks(P)), bat), 256, 0, st>>>(src, tab, P, sc, bat);
  return cudaGetLastError();
}

template <typename TI, typename TO>
__global__ void k_convert(const TI* __restrict__ in, TO* __restrict__ out, long n) {
  for (long p = blockIdx.x * (long)blockDim.x + threadIdx.x; p < n;
       p += (long)gridDim.x * blockDim.x)
    out[p] = (TO)in[p];
}

template <typename T>
cudaError_t launch_convert(const void* in, int in_d, void* out, int out_d, long n,
                           cudaStream_t st) {
  const int nb = reduce_blocks(n);
  if (in_d && out_d)
    k_convert<double, double><<<nb, 256, 0, st>>>((const double*)in, (double*)out, n);
  else if (in_d)
    k_convert<double, float><<<nb, 256, 0, st>>>((const double*)in, (float*)out, n);
  else if (out_d)
    k_convert<float, double><<<nb, 256, 0, st>>>((const float*)in, (double*)out, n);
  else
    k_convert<float, float><<<nb, 256, 0, st>>>((const float*)in, (float*)out, n);
  return cudaGetLastError();
}

#define OTGB_INST_NEWTON(T)                                                                   \
  template cudaError_t launch_gmres_init<T>(const double*, const T*, T*, long, int, double*,  \
                                            DevScalars*, int, cudaStream_t, T*, Bat);         \
  template cudaError_t launch_gmres_dots<T>(const T*, const T*, long, double*, DevScalars*,   \
                                            int, cudaStream_t, int, Bat);                     \
  template cudaError_t launch_gmres_update<T>(T*, const T*, long, double*, DevScalars*, int,  \
                                              cudaStream_t, int, Bat);                        \
  template cudaError_t launch_gmres_combine<T>(const T*, T*, long, const DevScalars*, int,    \
                                               cudaStream_t, Bat);                            \
  template cudaError_t launch_convert<T>(const void*, int, void*, int, long, cudaStream_t);

OTGB_INST_NEWTON(float)
OTGB_INST_NEWTON(double)

}  // namespace otgb

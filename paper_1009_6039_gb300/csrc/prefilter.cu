// Cubic B-spline prefilter (Sec. 4, interpolation of g: the coefficients c, with
// (c[k-1] + 4 c[k] + c[k+1]) / 6 = g[k] along each axis, periodic) as recursive filters.
// The periodic inverse of the stencil (1, 4, 1) / 6 is 6 h * with h[k] = z z^|k| / (z^2 - 1),
// z = sqrt(3) - 2 the root of z^2 + 4 z + 1 inside the unit circle (its DTFT is
// 1 / (4 + 2 cos t)), and sum_k z^|k| s[i - k] = cp[i] + ca[i] - s[i] with the first-order
// recursions cp[i] = s[i] + z cp[i - 1] (causal) and ca[i] = s[i] + z ca[i + 1] (anticausal).
//
// What bounds it: the recursions' serial chains, not their few multiply-adds per point.  So a
// thread runs them over chunks of 8 points only: first from zero, for the chunk's contribution
// to its neighbours (e+ = sum z^(7-i) s_i, e- = sum z^i s_i), then from the carry that four
// neighbouring chunks leave, sum_q z^(8 (q - 1)) e+[c - q] (|z|^32 = 5e-19, below FP64
// round-off): chains of 8 + 4 + 8 steps, where one chunk of 32 points and 40 of warm-up took 72
// each way.  A block stages 16 lines x (64 points + 32 on each side, periodic) in shared memory
// with coalesced loads.
//
// The mixed mode runs the same passes in double-float arithmetic (FP64 runs at a small fraction
// of the FP32 rate on this GPU); its column pass leaves the (hi, lo) result in the scratch plane.
// Both double-float passes, us, one GB300 (before: chunks of 32 points in tiles of 32 lines x 256
// points -> now): 128^2 47.7 -> 11.8, 512^2 79 -> 16.2, five problems of 512^2 115 -> 48.
#include <math.h>

#include "dd.cuh"
#include "otgb_internal.cuh"

namespace otgb {
namespace {

constexpr int CH = 8, NQ = 4, HALO = CH * NQ;   // chunk, carried chunks, points beyond the tile
constexpr int TP = 64, LN = 16, SW = LN + 1;    // tile points, lines, shared-memory row stride
constexpr int EP = TP + 2 * HALO, NC = EP / CH;  // staged points and chunks
static_assert(NC * LN == 256, "one thread per staged chunk");

// arithmetic of the two forms: the value in registers, in shared memory, a z + s
template <typename T> struct Ops;
template <> struct Ops<double> {
  using S = double;
  static __device__ __forceinline__ double load(const double* s, const float2*, long o) {
    return s[o];
  }
  static __device__ __forceinline__ double val(double s) { return s; }
  static __device__ __forceinline__ double mem(double v) { return v; }
  static __device__ __forceinline__ void store(long o, double r, float2*, double* out, float*) {
    out[o] = r;
  }
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double step(double z, double a, double s) { return fma(z, a, s); }
  static __device__ __forceinline__ double close(double A, double p, double a, double s) {
    return A * (p + a - s);
  }
};
template <> struct Ops<dd> {
  using S = float2;
  static __device__ __forceinline__ float2 load(const double* s, const float2* q, long o) {
    return s ? mem(dd_from_double(s[o])) : q[o];
  }
  static __device__ __forceinline__ dd val(float2 s) { return dd{s.x, s.y}; }
  static __device__ __forceinline__ float2 mem(dd v) { return make_float2(v.hi, v.lo); }
  static __device__ __forceinline__ void store(long o, float2 r, float2* odd, double* out,
                                               float* o32) {
    odd[o] = r;
    if (o32) o32[o] = r.x;
    if (out) out[o] = dd_to_double(dd{r.x, r.y});
  }
  static __device__ __forceinline__ dd zero() { return dd{0.f, 0.f}; }
  static __device__ __forceinline__ dd step(dd z, dd a, dd s) { return dd_add(dd_mul(z, a), s); }
  static __device__ __forceinline__ dd close(dd A, dd p, dd a, dd s) {
    return dd_mul(A, dd_sub(dd_add(p, a), s));
  }
};

// One axis.  XPASS: lines are rows (points along x), else columns.  Input: s64, or sdd when it is
// null; output: out64 and / or odd, and with odd (without a batch) its high parts in out32.
template <typename T, bool XPASS>
__global__ void __launch_bounds__(256)
    k_prefilter(const double* __restrict__ s64, const float2* __restrict__ sdd,
                float2* __restrict__ odd, double* __restrict__ out64, float* __restrict__ out32,
                int N, int M, double z64, double z8, double A64, Bat bat) {
  using O = Ops<T>;
  __shared__ typename O::S x[EP][SW];  // [staged point][line]
  __shared__ typename O::S ep[NC][LN], ea[NC][LN];
  s64 = badv(s64, bat);
  sdd = badv(sdd, bat);
  odd = badv(odd, bat);
  out64 = badv(out64, bat);
  const int tid = threadIdx.x;
  const int L = XPASS ? M : N, nlines = XPASS ? N : M;
  const long ls = XPASS ? M : 1, ps = XPASS ? 1 : M;
  const int line0 = blockIdx.x * LN, p0 = blockIdx.y * TP;
  const int first = (p0 + HALO * (L - 1)) % L;  // p0 - HALO modulo L
  // stage (lines fastest for columns, points fastest for rows: both coalesced)
#pragma unroll
  for (int i = 0; i < EP * LN / 256; ++i) {
    const int e = tid + 256 * i;
    const int k = XPASS ? e % EP : e / LN, ln = XPASS ? e / EP : e % LN;
    typename O::S v = O::mem(O::zero());
    if (line0 + ln < nlines)
      v = O::load(s64, sdd, (line0 + ln) * ls + (long)((first + k) % L) * ps);
    x[k][ln] = v;
  }
  __syncthreads();
  const T z(z64), zc(z8), A(A64);
  const int ln = tid % LN, c = tid / LN;
  {
    T p = O::zero(), a = O::zero();
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      p = O::step(z, p, O::val(x[c * CH + i][ln]));
      a = O::step(z, a, O::val(x[c * CH + CH - 1 - i][ln]));
    }
    ep[c][ln] = O::mem(p);
    ea[c][ln] = O::mem(a);
  }
  __syncthreads();
  if (c >= NQ && c < NC - NQ) {
    T p = O::zero(), a = O::zero();
#pragma unroll
    for (int q = NQ; q > 0; --q) {
      p = O::step(zc, p, O::val(ep[c - q][ln]));
      a = O::step(zc, a, O::val(ea[c + q][ln]));
    }
    T v[CH];
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      p = O::step(z, p, O::val(x[c * CH + i][ln]));
      v[i] = p;
    }
#pragma unroll
    for (int i = CH - 1; i >= 0; --i) {  // (only this thread reads or writes these points now)
      const T s = O::val(x[c * CH + i][ln]);
      a = O::step(z, a, s);
      x[c * CH + i][ln] = O::mem(O::close(A, v[i], a, s));
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TP * LN / 256; ++i) {
    const int e = tid + 256 * i;
    const int k = XPASS ? e % TP : e / LN, l2 = XPASS ? e / TP : e % LN;
    if (line0 + l2 >= nlines || p0 + k >= L) continue;
    const typename O::S r = x[HALO + k][l2];
    O::store((line0 + l2) * ls + (long)(p0 + k) * ps, r, odd, out64, out32);
  }
}

}  // namespace

cudaError_t launch_prefilter(const double* g, double* scratch, double* c, float2* cdd, int N,
                             int M, cudaStream_t st, Bat bat, float* c32) {
  const double z = sqrt(3.0) - 2.0, z2 = z * z, z4 = z2 * z2, z8 = z4 * z4;
  const double A = 6.0 * z / (z2 - 1.0);
  // columns (along y), then rows (along x)
  const dim3 gy = bgrid(dim3((M + LN - 1) / LN, (N + TP - 1) / TP), bat);
  const dim3 gx = bgrid(dim3((N + LN - 1) / LN, (M + TP - 1) / TP), bat);
  if (cdd) {
    float2* mid = reinterpret_cast<float2*>(scratch);
    k_prefilter<dd, false><<<gy, 256, 0, st>>>(g, nullptr, mid, nullptr, nullptr, N, M, z, z8, A,
                                               bat);
    k_prefilter<dd, true><<<gx, 256, 0, st>>>(nullptr, mid, cdd, c, c32, N, M, z, z8, A, bat);
  } else {
    k_prefilter<double, false><<<gy, 256, 0, st>>>(g, nullptr, nullptr, scratch, nullptr, N, M, z, z8,
                                                   A, bat);
    k_prefilter<double, true><<<gx, 256, 0, st>>>(scratch, nullptr, nullptr, c, nullptr, N, M, z, z8,
                                                  A, bat);
  }
  return cudaGetLastError();
}

}  // namespace otgb

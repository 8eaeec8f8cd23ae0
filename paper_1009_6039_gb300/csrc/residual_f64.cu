// The FP64 residual and linearised coefficients (Eq. ma2, linearmaeq, translation), and the pass
// that shifts the residual by the mass translation and sums its squares.
//
// What bounds the residual: FP64 instructions (two per clock and SM on GB300, see
// spectral_f64.cu).  A point takes about 119: stencils 22, displaced position 6, spline weights
// 26, 16-tap gather of the value and the gradient 44, determinant, f_n, F and coefficients 12,
// sums 6, and the tile's halo, so 198 us at 1024^2 with every SM busy.  What keeps the count down:
//   - 1 + u_xx and 1 + u_yy in one FMA each, M u_x and N u_y straight from the differences (u_x
//     itself is not needed), the floor and the fraction by FMAs with a constant (cell);
//   - the weights as 6 w and 2 w' (13 instructions per axis), their factors in G's and in the
//     determinant's scale;
//   - maxima, minima and finiteness on the integer pipe (doubles as ordered integers), the
//     Simpson weight of a thread's points (all of one parity) taken once at the end;
//   - block sums of six values folded over a warp (9 additions instead of 30).
// A block covers 32 columns x TH rows: 32 where that gives four blocks per SM, else 8 or 4, so
// that small grids reach every SM.  Measured (us per launch under ncu, one GB300; before: 160
// instructions per point, 32-row tiles): 1024^2 349 -> 256 (FP64 pipe 85 % busy), 250 x 333 65 -> 35.
// Graph-replayed, with the floor from the nearest integer -> rounded down, with the test for far
// displacements: 1024^2 251.7 -> 248.9, 256^2 27.2 -> 26.9.
#include <math.h>

#include "otgb_internal.cuh"
#include "reduce.cuh"

namespace otgb {
namespace {

constexpr int TWX = 32;  // tile columns

struct ResidK {
  double MM, NN, MNh;  // M^2/12, N^2/12, M N / 144
  double Mg, Ng;       // M/12, N/12 (of the 6 w, 2 w' weights)
  double w3;           // 1/(9 M N): Simpson weights (2 or 4 per axis) x this
  double Md, Nd, iM, iN;  // M, N, 1/M, 1/N
  int nob;             // 1: the simplified operator (b = 0, Sec. 3.3 remark)
  // interpolation of g (Sec. 4 intro; Sec. 5.2, 5.3): 0 cubic B-spline of the coefficients c;
  // 1 bilinear, 2 nearest node of the grid values (then c = g) and of the grid gradient gx, gy
  int interp;
  const double* gx;
  const double* gy;
};

__device__ __forceinline__ int wrap_any(int a, int L) {
  const int r = a % L;
  return r < 0 ? r + L : r;
}

// 1.5 x 2^52 + 2^31: a sum with it, rounded down, holds the floor k as k + 2^31 in its low word, and its
// high word is kNear for -2^31 <= k < 2^31 alone
constexpr double kMagic = 6755399441055744.0 + 2147483648.0;
constexpr int kNear = 0x43380000;
// 2^30 or more in size, or not finite
__device__ __forceinline__ bool far(double x) {
  return (__double2hiint(x) & 0x7fffffff) >= 0x41d00000;
}
// Cell of the position n + d s, in [0, L), and the fraction t in [0, 1], for any displacement d s (0 <=
// n < L, iL = 1 / L).  The product enters the floor and the fraction unrounded: two FMAs, and one
// test of the high word for displacements beyond an int (a diverging iterate's).  Those positions are
// reduced first: each x - floor(x / L) L is exact, two leave less than 2^30 of any |x| < 2^100, and
// beyond, where neighbouring doubles are 2^47 cells apart, node 0 is taken.
__device__ __forceinline__ int cell(int n, double d, double s, int L, double Ld, double iL,
                                    double* t) {
  double m = __fma_rd(d, s, kMagic);
  if (__double2hiint(m) == kNear) {
    *t = fma(d, s, -(m - kMagic));
  } else {
    double x = __dadd_rn((double)n, __dmul_rn(d, s));
    n = 0;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) x = fma(-floor(x * iL), Ld, x);
    if (far(x)) x *= 0.0;  // (NaN stays NaN, infinity becomes NaN)
    m = __dadd_rd(x, kMagic);
    *t = x - (m - kMagic);
  }
  const int j = wrap_any((int)((unsigned)__double2loint(m) ^ 0x80000000u), L) + n;
  return j >= L ? j - L : j;
}

// the result of an operation is NaN (a quiet one: its high word tells)
__device__ __forceinline__ bool nan_result(double x) {
  return (__double2hiint(x) & 0x7fffffff) > 0x7ff00000;
}

// sums of six values, a maximum, two minima and a count over the block; the block's results are
// in the first lanes of warp 0: lane v < 6 holds sum v in s[0], lane 0 the others
struct Red {
  double s[6];
  long long kmax, kmin, kdet;
  int bad;
};
template <int NW>
__device__ __forceinline__ void block_reduce_res(Red& r) {
  __shared__ double rs[NW][8];
  __shared__ long long rk[NW][3];
  __shared__ int rb[NW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // fold: lanes exchange halves of the values, so that lane 4 v + . ends with value v
  double v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double hi = i < 2 ? r.s[i + 4] : 0.0;
    const bool up = lane & 16;
    v[i] = (up ? hi : r.s[i]) + __shfl_xor_sync(0xffffffffu, up ? r.s[i] : hi, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool up = lane & 8;
    v[i] = (up ? v[i + 2] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + 2], 8);
  }
  {
    const bool up = lane & 4;
    v[0] = (up ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], 4);
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    r.kmax = max(r.kmax, __shfl_xor_sync(0xffffffffu, r.kmax, o));
    r.kmin = min(r.kmin, __shfl_xor_sync(0xffffffffu, r.kmin, o));
    r.kdet = min(r.kdet, __shfl_xor_sync(0xffffffffu, r.kdet, o));
  }
  r.bad = __reduce_add_sync(0xffffffffu, r.bad);
  if ((lane & 3) == 0) rs[wid][lane >> 2] = v[0];
  if (lane == 0) {
    rk[wid][0] = r.kmax;
    rk[wid][1] = r.kmin;
    rk[wid][2] = r.kdet;
    rb[wid] = r.bad;
  }
  __syncthreads();
  if (wid == 0) {
    double x = 0.0;
#pragma unroll
    for (int w = 0; w < NW; w += 4) x += rs[w + (lane >> 3)][lane & 7];
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 16);
    r.s[0] = x;
    r.kmax = rk[0][0];
    r.kmin = rk[0][1];
    r.kdet = rk[0][2];
    r.bad = rb[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      r.kmax = max(r.kmax, rk[w][0]);
      r.kmin = min(r.kmin, rk[w][1]);
      r.kdet = min(r.kdet, rk[w][2]);
      r.bad += rb[w];
    }
  }
  __syncthreads();
}

template <int TH>
__global__ void __launch_bounds__(TWX * (TH < 8 ? TH : 8), TH == 32 ? 3 : 4)
    k64_residual(const double* __restrict__ f, const double* __restrict__ c,
                 const double* __restrict__ ua, const double* __restrict__ ub, int sel, int N,
                 int M, ResidK K, double* __restrict__ Fraw, double* __restrict__ coef,
                 double* partials, DevScalars* sc) {
  constexpr int NW = TH < 8 ? TH : 8, NT = 32 * NW;
  __shared__ double tile[TH + 4][TWX + 4];
  __shared__ double dyt[TH][TWX + 4];  // unscaled y-difference of u (halo 2 in x)
  __shared__ bool last;
  const double* __restrict__ u = (ub && ((sc->upar ^ sel) & 1)) ? ub : ua;
  const int bx = blockIdx.x * TWX, by = blockIdx.y * TH;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < (TH + 4) * (TWX + 4); idx += NT) {
    const int r = idx / (TWX + 4), cc = idx - r * (TWX + 4);
    int gi = by + r - 2, gj = bx + cc - 2;
    while (gi < 0) gi += N;
    while (gi >= N) gi -= N;
    while (gj < 0) gj += M;
    while (gj >= M) gj -= M;
    tile[r][cc] = u[(size_t)gi * M + gj];
  }
  __syncthreads();
  for (int idx = tid; idx < TH * (TWX + 4); idx += NT) {
    const int r = idx / (TWX + 4), cc = idx - r * (TWX + 4);
    dyt[r][cc] = fma(-8.0, tile[r + 1][cc], fma(8.0, tile[r + 3][cc], -tile[r + 4][cc])) + tile[r][cc];
  }
  __syncthreads();
  Red red;
#pragma unroll
  for (int a = 0; a < 6; ++a) red.s[a] = 0.0;
  red.kmax = ordered_key(-INFINITY);
  red.kmin = red.kdet = ordered_key(INFINITY);
  red.bad = 0;
  const int tx = tid & 31, ty0 = tid >> 5;
  const int j = bx + tx;
  const size_t P = (size_t)N * M;
#pragma unroll 1
  for (int ty = ty0; ty < TH; ty += NW) {
    const int i = by + ty;
    if (i >= N || j >= M) continue;
    const size_t p = (size_t)i * M + j;
    const double fv = f[p];
    const int r = ty + 2, q = tx + 2;
    const double u0 = tile[r][q], xm2 = tile[r][q - 2], xm1 = tile[r][q - 1],
                 xp1 = tile[r][q + 1], xp2 = tile[r][q + 2];
    // M u_x, N u_y (grid cells) over MM, NN; 1 + u_xx, 1 + u_yy; u_xy
    const double dx = fma(-8.0, xm1, fma(8.0, xp1, -xp2)) + xm2, dy = dyt[ty][q];
    const double axx = fma(fma(16.0, xm1, fma(-30.0, u0, fma(16.0, xp1, -xp2))) - xm2, K.MM, 1.0);
    const double ayy = fma(fma(16.0, tile[r - 1][q],
                               fma(-30.0, u0, fma(16.0, tile[r + 1][q], -tile[r + 2][q]))) -
                               tile[r - 2][q], K.NN, 1.0);
    const double uxy = (fma(-8.0, dyt[ty][q - 1], fma(8.0, dyt[ty][q + 1], -dyt[ty][q + 2])) +
                        dyt[ty][q - 2]) * K.MNh;
    const double det = fma(axx, ayy, -(uxy * uxy));
    // g at the displaced point x + grad u, in grid units, periodic cubic B-spline
    double t, s;
    const int j0 = cell(j, dx, K.MM, M, K.Md, K.iM, &t), i0 = cell(i, dy, K.NN, N, K.Nd, K.iN, &s);
    int jj[4], ii[4];
    jj[0] = j0 == 0 ? M - 1 : j0 - 1;
    jj[1] = j0;
    jj[2] = j0 + 1 == M ? 0 : j0 + 1;
    jj[3] = jj[2] + 1 == M ? 0 : jj[2] + 1;
    ii[0] = i0 == 0 ? N - 1 : i0 - 1;
    ii[1] = i0;
    ii[2] = i0 + 1 == N ? 0 : i0 + 1;
    ii[3] = ii[2] + 1 == N ? 0 : ii[2] + 1;
    double G, b1, b2;
    if (K.interp == 0) {
      double wx[4], dwx[4], wy[4], dwy[4];
      auto weights = [](double a, double w[4], double d[4]) {  // 6 w, 2 w' at a
        const double b = 1.0 - a, a2 = a * a, c2 = b * b;
        w[0] = c2 * b;
        w[1] = fma(a2, fma(3.0, a, -6.0), 4.0);
        w[2] = fma(c2, fma(3.0, b, -6.0), 4.0);
        w[3] = a2 * a;
        d[0] = -c2;
        d[1] = a * fma(3.0, a, -4.0);
        d[2] = -(b * fma(3.0, b, -4.0));
        d[3] = a2;
      };
      weights(t, wx, dwx);
      weights(s, wy, dwy);
      double g = 0.0, gx = 0.0, gy = 0.0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const double* crow = c + (size_t)ii[b] * M;
        const double c0 = __ldg(crow + jj[0]), c1 = __ldg(crow + jj[1]), c2 = __ldg(crow + jj[2]),
                     c3 = __ldg(crow + jj[3]);
        const double sv = fma(c3, wx[3], fma(c2, wx[2], fma(c1, wx[1], c0 * wx[0])));
        const double sd = fma(c3, dwx[3], fma(c2, dwx[2], fma(c1, dwx[1], c0 * dwx[0])));
        g = b ? fma(sv, wy[b], g) : sv * wy[0];
        gx = b ? fma(sd, wy[b], gx) : sd * wy[0];
        gy = b ? fma(sv, dwy[b], gy) : sv * dwy[0];
      }
      G = g * (1.0 / 36.0);
      b1 = (det * K.Mg) * gx;
      b2 = (det * K.Ng) * gy;
    } else if (K.interp == 2) {  // nearest node (round half up)
      const size_t n = (size_t)(s >= 0.5 ? ii[2] : i0) * M + (t >= 0.5 ? jj[2] : j0);
      G = __ldg(c + n);
      b1 = det * __ldg(K.gx + n);
      b2 = det * __ldg(K.gy + n);
    } else {  // bilinear on the cell (i0, j0) .. (i0 + 1, j0 + 1)
      const double w[4] = {(1.0 - t) * (1.0 - s), t * (1.0 - s), (1.0 - t) * s, t * s};
      const size_t n[4] = {(size_t)ii[1] * M + jj[1], (size_t)ii[1] * M + jj[2],
                           (size_t)ii[2] * M + jj[1], (size_t)ii[2] * M + jj[2]};
      double gx = 0.0, gy = 0.0;
      G = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        G += w[k] * __ldg(c + n[k]);
        gx += w[k] * __ldg(K.gx + n[k]);
        gy += w[k] * __ldg(K.gy + n[k]);
      }
      b1 = det * gx;
      b2 = det * gy;
    }
    const double fn = G * det;
    const double fr = fv - fn;
    if (K.nob) b1 = b2 = 0.0;
    const double a11 = G * ayy, a12 = -(G * uxy), a22 = G * axx;
    Fraw[p] = fr;
    coef[p] = a11;
    coef[P + p] = a12;
    coef[2 * P + p] = a22;
    coef[3 * P + p] = b1;
    coef[4 * P + p] = b2;
    red.s[1] += a11;
    red.s[2] += a12;
    red.s[3] += a22;
    red.s[4] += b1;
    red.s[5] += b2;
    if (finite_key(fn)) {
      red.s[0] += fn;
      if (!nan_result(fr)) {  // (a NaN in f: the other points' extremes stand)
        red.kmax = max(red.kmax, ordered_key(fr));
        red.kmin = min(red.kmin, ordered_key(fr));
      }
    } else {
      red.bad += 1;
    }
    if (!nan_key(det)) red.kdet = min(red.kdet, ordered_key(det));
  }
  // composite Simpson: weights 2 / 4 by the parity of i and j, both fixed per thread
  const double w = (((by + ty0) & 1) ? 4.0 : 2.0) * ((j & 1) ? 4.0 : 2.0) * K.w3;
#pragma unroll
  for (int a = 1; a < 6; ++a) red.s[a] *= w;
  block_reduce_res<NW>(red);
  const unsigned int nb = gridDim.x * gridDim.y;
  const size_t bid = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
  // per block: six sums, then the ordered integers of max F, min F, min det, and the count
  if (tid < 32) {
    if (tid < 6) partials[bid * 10 + tid] = red.s[0];
    if (tid == 0) {
      partials[bid * 10 + 6] = __longlong_as_double(red.kmax);
      partials[bid * 10 + 7] = __longlong_as_double(red.kmin);
      partials[bid * 10 + 8] = __longlong_as_double(red.kdet);
      partials[bid * 10 + 9] = __longlong_as_double(red.bad);
    }
    __syncwarp();
    if (tid == 0) {
      __threadfence();
      last = atomicAdd(&sc->ticket[TK_RESID], 1u) == nb - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int a = 0; a < 6; ++a) red.s[a] = 0.0;
  red.kmax = ordered_key(-INFINITY);
  red.kmin = red.kdet = ordered_key(INFINITY);
  red.bad = 0;
  for (unsigned int b = tid; b < nb; b += NT) {
    const double* q = partials + (size_t)b * 10;
#pragma unroll
    for (int a = 0; a < 6; ++a) red.s[a] += __ldcg(q + a);
    red.kmax = max(red.kmax, __double_as_longlong(__ldcg(q + 6)));
    red.kmin = min(red.kmin, __double_as_longlong(__ldcg(q + 7)));
    red.kdet = min(red.kdet, __double_as_longlong(__ldcg(q + 8)));
    red.bad += (int)__double_as_longlong(__ldcg(q + 9));
  }
  block_reduce_res<NW>(red);
  if (tid >= 32) return;
  double tot[6];
#pragma unroll
  for (int a = 0; a < 6; ++a) tot[a] = __shfl_sync(0xffffffffu, red.s[0], a);
  if (tid == 0) {
    const double mean_fn = tot[0] / ((double)N * (double)M);
    const double shift = mean_fn - 1.0, dmin = key_value(red.kdet);
    sc->mean_fn = mean_fn;
    sc->shift = shift;
    sc->res_inf = fmax(fabs(key_value(red.kmax) + shift), fabs(key_value(red.kmin) + shift));
    for (int a = 0; a < 5; ++a) sc->abar[a] = tot[1 + a];
    sc->min_det = dmin;
    sc->k1_nonfinite = red.bad;
    sc->admissible = (red.bad == 0 && isfinite(sc->res_inf) && dmin > 0.0) ? 1 : 0;
    sc->ticket[TK_RESID] = 0;
  }
}

// sum of (Fraw + shift)^2 -> res_l2sum; F (optional, may be Fraw) = Fraw + shift
__global__ void __launch_bounds__(256)
    k_residual_l2(const double* Fraw, double* F, long P, double* partials, DevScalars* sc,
                  Bat bat) {
  Fraw = badv(Fraw, bat);
  partials = badv(partials, bat);
  sc = badv(sc, bat);
  if (bskip(sc, bat)) return;
  const double s = sc->shift;
  double v[1] = {0.0};
  const int kind[1] = {0};
  // four loads in flight per thread
  const long p0 = blockIdx.x * (long)blockDim.x + threadIdx.x, nth = (long)gridDim.x * blockDim.x;
  for (long p = p0; p < P; p += 4 * nth) {
    double x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = p + k * nth < P ? Fraw[p + k * nth] : 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (p + k * nth >= P) break;
      const double r = x[k] + s;
      if (F) F[p + k * nth] = r;
      v[0] = fma(r, r, v[0]);
    }
  }
  block_reduce<1>(v, kind);
  if (!publish_partials<1>(v, partials, &sc->ticket[TK_NORM])) return;
  reduce_partials<1>(v, kind, partials, gridDim.x);
  if (threadIdx.x == 0) {
    sc->res_l2sum = v[0];
    sc->ticket[TK_NORM] = 0;
  }
}

inline int tiles(int N, int M, int th) { return ((M + TWX - 1) / TWX) * ((N + th - 1) / th); }

// tile rows: the largest form with four blocks per SM, else the smallest.  (A grid of fewer
// blocks leaves SMs idle: 64^2 in 32-row tiles ran on 4 of 152 SMs.)
inline int tile_rows(int N, int M) {
  for (int th : {32, 8})
    if (tiles(N, M, th) >= 4 * 152) return th;
  return 4;
}

}  // namespace

int residual_partial_blocks(int N, int M) { return tiles(N, M, tile_rows(N, M)); }

cudaError_t launch_residual(const double* f, const double* c, const double* ua, int N, int M,
                            double* Fraw, double* coef, double* partials, DevScalars* sc,
                            cudaStream_t st, const double* ub, int sel, int simplified,
                            Interp ip) {
  ResidK K;
  K.Md = (double)M;
  K.Nd = (double)N;
  K.iM = 1.0 / K.Md;
  K.iN = 1.0 / K.Nd;
  K.MM = (double)M * (double)M / 12.0;
  K.NN = (double)N * (double)N / 12.0;
  K.MNh = (double)M * (double)N / 144.0;
  K.Mg = (double)M / 12.0;
  K.Ng = (double)N / 12.0;
  K.w3 = 1.0 / (9.0 * (double)M * (double)N);
  K.nob = simplified ? 1 : 0;
  K.interp = ip.mode;
  K.gx = ip.gx;
  K.gy = ip.gy;
  if (ip.mode && !(ip.gx && ip.gy)) return cudaErrorInvalidValue;
  const int th = tile_rows(N, M);
  const dim3 grid((M + TWX - 1) / TWX, (N + th - 1) / th);
  if (th == 32)
    k64_residual<32><<<grid, 256, 0, st>>>(f, c, ua, ub, sel, N, M, K, Fraw, coef, partials, sc);
  else if (th == 8)
    k64_residual<8><<<grid, 256, 0, st>>>(f, c, ua, ub, sel, N, M, K, Fraw, coef, partials, sc);
  else
    k64_residual<4><<<grid, 128, 0, st>>>(f, c, ua, ub, sel, N, M, K, Fraw, coef, partials, sc);
  return cudaGetLastError();
}

cudaError_t launch_residual_l2(const double* Fraw, int N, int M, double* partials,
                               DevScalars* sc, cudaStream_t st, Bat bat, double* F) {
  const long P = (long)N * M;
  if (bat.on && F) return cudaErrorInvalidValue;
  // 1024 points per block, at most two blocks per SM
  const long nb = (P + 1023) / 1024;
  k_residual_l2<<<bgrid(dim3((unsigned)(nb < 2 * 152 ? nb : 2 * 152)), bat), 256, 0, st>>>(
      Fraw, F, P, partials, sc, bat);
  return cudaGetLastError();
}

}  // namespace otgb

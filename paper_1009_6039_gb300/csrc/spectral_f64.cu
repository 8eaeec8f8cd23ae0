// FP64 spectral passes of Strain's method (Sec. 4.2): the three passes of the matvec, of
// theta = Lbar^{-1} sigma and of the plain transforms, in the data layout of spectral.cuh.
//
// What bounds them: GB300 starts two FP64 instructions per clock and SM (a warp instruction
// takes 16 clocks; an FMA, an addition and a product cost the same), 32 times fewer than FP32,
// while everything else (addresses, shared memory, L2) has 64 issue slots per FP64 warp
// instruction.  So a pass costs its FP64 instruction count over the SMs that take part, and
//   - every butterfly is in FMA form: with the twiddle as w = g (1 + i r) or i g (1 + i r), |r| <= 1,
//     u = b + i r b takes two FMAs and a +- g u four, 6 instructions with the twiddle included (a
//     product, a sum and a difference take 8), 3 per point and level whatever the radix, and the real
//     split and its inverse take 5 per frequency (8 and 6); radix 4, whose 56 to 80 registers leave
//     room for many warps; the exchange of parts and signs that i g asks for is on the integer pipe (as
//     negations in FP64 it cost 13 %);
//   - a block holds one row or column (more rows only where the blocks would be tiny), so that
//     all SMs get work and the last wave is a single row's;
//   - the independent transforms of a row (five) or column (three) run side by side in thread
//     groups, not one after the other, which is what small grids wait for.
// Measured on one GB300 (us per launch, graph-replayed; before: radix 8, one thread group per
// row or column with its terms in sequence, product-and-sum butterflies) ->
//             64^2           384 x 768        1024^2          2048^2
//   row r2c   11.1 ->  5.8   23.5 -> 13.1     46.9 ->  35.0   188 -> 142
//   column    62.0 -> 12.0    102 -> 49        202 -> 160     801 -> 674
//   combine   48.4 ->  9.1    114 -> 65        230 -> 189     987 -> 771
//   theta col 49.6 -> 15.9   64.3 -> 32        118 ->  91     442 -> 369
// The FP64 pipe is 82 to 89 % busy in the 2048^2 passes (issue-bound), 10 to 20 % at 64^2
// (latency: one row or column per SM).
//
// Rounding: a + w b and a - w b are each rounded once at their own size.  (As s = a + w b in four FMAs and
// 2 a - s in two, the sum's rounding enters the difference: an image-like density's low frequencies
// leave theirs in the high ones.)  Relative rms error of a transform against long double, in 1e-16,
// radix 8 with separate products and sums / 2 a - s / this form: forward 2.32 / 2.86 / 2.33 and inverse 2.24 /
// 3.16 / 2.30 on smoothed noise and blobs at 512^2, 1.79 / 2.23 / 1.88 and 1.85 / 2.37 / 1.90 at 64^2, 3.87 /
// 4.15 / 4.03 on white noise at 512^2.  Radix 4 with separate products and sums is no closer and takes 683 us for
// the two 2048^2 transforms, 2 a - s 585, this form 562 (and 0.2 us a column pass more at 64^2, latency).
#include "spectral.cuh"

namespace otgb {
namespace {

constexpr int kMaxThreads = 768;  // launch bound: 80 registers, for two to ten blocks per SM

// the butterflies' table of length L behind its base table (fill_butterflies of api.cu)
__device__ __forceinline__ const double2* stage_table(const double2* tw, int L) {
  return tw + (size_t)stage_table_slot<4>() * L;
}

// ---------------------------------------------------------------------------------------
// Butterflies.  SIGN -1 forward, +1 inverse (the twiddles are conjugated).
// ---------------------------------------------------------------------------------------
// A twiddle w = exp(-i t) as its larger part and the ratio of the two (the scaled butterflies of Linzer and
// Feig's FMA transforms), so that a +- w b take three
// FMAs a part and each is rounded once at its own size: not turned (|cos t| >= |sin t|), w = g (1 +
// i r) with g = cos t; turned, w = i g (1 + i r) with g = -sin t; |r| <= 1.
struct Tw {
  double2 gr;
  bool turned;
};
// (a, b) <- (a + w b, a - w b); QUARTER: with -i w for w (conjugated for the inverse)
template <int SIGN, bool QUARTER = false>
__device__ __forceinline__ void bf(double2& a, double2& b, const Tw& w) {
  const double g = w.gr.x, r = SIGN < 0 ? w.gr.y : -w.gr.y;
  // i b (forward) or -i b, and back by a quarter: on the integer pipe (a negation can become an
  // FP64 addition)
  const bool take = w.turned != QUARTER;
  const unsigned flip = take ? 0x80000000u : 0u;
  constexpr bool up = (SIGN < 0) != QUARTER;  // (-b.y, b.x), else (b.y, -b.x)
  const double2 c = make_double2(
      __hiloint2double((take ? __double2hiint(b.y) : __double2hiint(b.x)) ^ (up ? flip : 0u),
                       take ? __double2loint(b.y) : __double2loint(b.x)),
      __hiloint2double((take ? __double2hiint(b.x) : __double2hiint(b.y)) ^ (up ? 0u : flip),
                       take ? __double2loint(b.x) : __double2loint(b.y)));
  const double2 u = make_double2(fma(-r, c.y, c.x), fma(r, c.x, c.y));
  b = make_double2(fma(-g, u.x, a.x), fma(-g, u.y, a.y));
  a = make_double2(fma(g, u.x, a.x), fma(g, u.y, a.y));
}
// (a, b) <- (a + b, a - b)
__device__ __forceinline__ void bf1(double2& a, double2& b) {
  const double2 d = make_double2(a.x - b.x, a.y - b.y);
  a = make_double2(a.x + b.x, a.y + b.y);
  b = d;
}
// (a, b) <- (a + SIGN i b, a - SIGN i b)
template <int SIGN>
__device__ __forceinline__ void bfi(double2& a, double2& b) {
  const double2 t = SIGN > 0 ? make_double2(-b.y, b.x) : make_double2(b.y, -b.x);
  b = make_double2(a.x - t.x, a.y - t.y);
  a = make_double2(a.x + t.x, a.y + t.y);
}

// DFT of size R of v[r] w^r, w = w1 the stage twiddle (TW 0: w = 1) and w2 = w^2, by decimation
// in the bits of r, most significant first; results in natural order.
template <int R, int SIGN, bool TW> struct Dft;
template <int SIGN, bool TW> struct Dft<2, SIGN, TW> {
  __device__ __forceinline__ static void run(double2* v, const Tw& w1, const Tw&) {
    if (TW) bf<SIGN>(v[0], v[1], w1);
    else bf1(v[0], v[1]);
  }
};
template <int SIGN, bool TW> struct Dft<4, SIGN, TW> {
  __device__ __forceinline__ static void run(double2* v, const Tw& w1, const Tw& w2) {
    if (TW) {
      bf<SIGN>(v[0], v[2], w2);
      bf<SIGN>(v[1], v[3], w2);
      bf<SIGN>(v[0], v[1], w1);
      bf<SIGN, true>(v[2], v[3], w1);
    } else {
      bf1(v[0], v[2]);
      bf1(v[1], v[3]);
      bf1(v[0], v[1]);
      bfi<SIGN>(v[2], v[3]);
    }
    const double2 x1 = v[2], x2 = v[1];  // (v0, v1) = (X0, X2), (v2, v3) = (X1, X3)
    v[1] = x1;
    v[2] = x2;
  }
};
// radix 3 (the first stage of a length 3 2^a, no twiddles)
template <int SIGN>
__device__ __forceinline__ void dft3(double2* v) {
  const double c = SIGN * OTGB_SQRT3_HALF;
  const double2 a = v[0], s = make_double2(v[1].x + v[2].x, v[1].y + v[2].y),
                d = make_double2(v[1].x - v[2].x, v[1].y - v[2].y);
  const double2 t = make_double2(fma(-0.5, s.x, a.x), fma(-0.5, s.y, a.y));
  v[0] = make_double2(a.x + s.x, a.y + s.y);
  v[1] = make_double2(fma(-c, d.y, t.x), fma(c, d.x, t.y));  // t + SIGN i sqrt(3)/2 d
  v[2] = make_double2(fma(c, d.y, t.x), fma(-c, d.x, t.y));
}

// One Stockham stage in place on buf, as stockham_stage of spectral.cuh with these butterflies,
// by the L / 4 threads of a transform: a butterfly each (radix 4), two (radix 2), or one or two
// (radix 3).  st: the stage table of this length.
template <int R, int SIGN>
__device__ __forceinline__ void stage(double2* buf, int L, int Ns, int t, bool active,
                                      const double2* __restrict__ st, bool pin, bool pout) {
  constexpr int NB = R == 4 ? 1 : 2;
  const int T = L / 4, LR = L / R;
  double2 v[NB * R];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int j = t + b * T;
    if (active && (R != 3 || j < LR))
#pragma unroll
      for (int r = 0; r < R; ++r) v[b * R + r] = buf[spad(j + r * LR, pin)];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int j = t + b * T;
    if (!active || (R == 3 && j >= LR)) continue;
    const int a = __ffs(Ns) - 1;
    const int qd = (Ns >> a) == 1 ? (j >> a) : ((j >> a) / 3);
    const int k = j - qd * Ns;
    double2* x = &v[b * R];
    if constexpr (R == 3) {
      dft3<SIGN>(x);
    } else if (Ns == 1) {
      const Tw one{make_double2(1.0, 0.0), false};
      Dft<R, SIGN, false>::run(x, one, one);
    } else {
      // w's angle is 2 pi k / (R Ns): turned between an eighth and three eighths of a circle
      const double2* s = st + (Ns - 1) + k;
      const bool mid = 4 * k > Ns && 4 * k < 3 * Ns;
      const Tw w1{s[0], R == 2 ? mid : 2 * k > Ns}, w2{R == 2 ? s[0] : s[Ns], mid};
      Dft<R, SIGN, true>::run(x, w1, w2);
    }
    const int d = qd * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) buf[spad(d + r * Ns, pout)] = x[r];
  }
  __syncthreads();
}

// Full unnormalised transform in place (plain layout in and out) by L / 4 threads; the radices
// are [3,] then 4 while it divides, then 2.
template <int SIGN>
__device__ __forceinline__ void fft64(double2* buf, int L, int t, bool active,
                                      const double2* __restrict__ tw) {
  const double2* __restrict__ st = stage_table(tw, L);
  int Ns = 1, rem = L;
  if (L % 3 == 0) {
    stage<3, SIGN>(buf, L, 1, t, active, st, false, rem > 3);
    Ns = 3;
    rem /= 3;
  }
#pragma unroll 1
  while (rem > 1) {
    const bool pin = Ns > 1;
    if (rem % 4 == 0) {
      stage<4, SIGN>(buf, L, Ns, t, active, st, pin, rem > 4);
      Ns *= 4;
      rem /= 4;
    } else {
      stage<2, SIGN>(buf, L, Ns, t, active, st, pin, rem > 2);
      Ns *= 2;
      rem /= 2;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Row real-to-complex transform: RB rows per block, TPT = M / 2 / E threads each.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kMaxThreads)
    k64_row_r2c(const double* __restrict__ xbase, size_t x_stride, const int* __restrict__ jptr,
                const double* __restrict__ scale, double2* __restrict__ spec, int N, int M,
                const double2* __restrict__ twL, const double2* __restrict__ twM,
                const int* __restrict__ skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int L = M / 2, TPT = L / 4;
  const int q = threadIdx.x / TPT, t = threadIdx.x - q * TPT;
  const int row = blockIdx.x * (blockDim.x / TPT) + q;
  const bool active = row < N;
  double2* buf = reinterpret_cast<double2*>(smem_raw) + q * FB(L);
  const int jv = jptr ? *jptr : 0;
  // the split's factors 1/2 are taken here, with the vector's scale (exact)
  const double sc = 0.5 * (scale ? scale[jv] : 1.0);
  if (active) {
    const double2* xr =
        reinterpret_cast<const double2*>(xbase + (size_t)jv * x_stride + (size_t)row * M);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int n = t + e * TPT;
      const double2 z = xr[n];
      buf[n] = make_double2(z.x * sc, z.y * sc);
    }
  }
  __syncthreads();
  fft64<-1>(buf, L, t, active, twL);
  if (!active) return;
  // with Z of the halved row: Ev = Zk + conj Zm, Ov = -i (Zk - conj Zm), X_k = Ev + W_M^k Ov,
  // X_(L-k) = conj(2 Ev - X_k)
  double2* out = spec + (size_t)row * L;
  for (int k = t; k <= L / 2; k += TPT) {
    if (k == 0) {
      const double2 z = buf[0];
      out[0] = make_double2(2.0 * (z.x + z.y), 2.0 * (z.x - z.y));
    } else {
      const double2 zk = buf[k], zm = buf[L - k], w = twM[k];
      const double2 ev = make_double2(zk.x + zm.x, zk.y - zm.y),
                    ov = make_double2(zk.y + zm.y, zm.x - zk.x);
      const double2 s = make_double2(fma(-w.x, ov.x, fma(w.y, ov.y, ev.x)),
                                     fma(w.x, ov.y, fma(w.y, ov.x, -ev.y)));
      out[k] = make_double2(fma(2.0, ev.x, -s.x), fma(2.0, ev.y, s.y));
      if (2 * k != L) out[L - k] = s;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Column transforms with the spectral multiplies, one column per block.  G = 3 (matvec): three
// thread groups and buffers per column, one per inverse transform (group 0 also runs the
// forward one); G = 1: one group, the matvec's inverse transforms one after the other.
// ---------------------------------------------------------------------------------------
// inv rho-bar(k), rho-bar as in spectral.cuh: one division for both parts
__device__ __forceinline__ double2 rho_bar64(const double* ab, double2 sx, double2 sy, double inv) {
  const double dr = fma(ab[2], sy.y, fma(-2.0 * (ab[1] * sx.x), sy.x, ab[0] * sx.y));
  const double di = fma(ab[4], sy.x, ab[3] * sx.x);
  const double den = fma(dr, dr, di * di);
  const double r = den == 0.0 ? 0.0 : inv / den;
  return make_double2(dr * r, -di * r);
}
__device__ __forceinline__ double2 cmul64(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

// the column's G buffers to planes p0 .. p0 + G - 1
template <int G>
__device__ __forceinline__ void col_out(int p0, const double2* sm, double2* out0, double2* out1,
                                        double2* out2, int N, int Lc, int col, int F) {
#pragma unroll
  for (int p = 0; p < G; ++p) {
    double2* dst = p0 + p == 0 ? out0 : (p0 + p == 1 ? out1 : out2);
    for (int n = threadIdx.x; n < N; n += blockDim.x) dst[(size_t)n * Lc + col] = sm[p * F + n];
  }
}

template <int MODE, int G>
__global__ void __launch_bounds__(kMaxThreads)
    k64_col(const double2* __restrict__ spec, double2* __restrict__ out0,
            double2* __restrict__ out1, double2* __restrict__ out2, int N, int M, double inv_nm, const double2* __restrict__ twN, const double2* __restrict__ twM,
            const DevScalars* __restrict__ sc, const int* __restrict__ skip,
            const double2* __restrict__ symx, const double2* __restrict__ symy) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf0 = reinterpret_cast<double2*>(smem_raw);
  const int Lc = M / 2, TPT = N / 4, F = FB(N);
  const int r = threadIdx.x, g = G == 1 ? 0 : r / TPT, t = r - g * TPT;
  const int col = blockIdx.x;
  double2* buf = buf0 + g * F;
  for (int n = r; n < N; n += blockDim.x) buf0[n] = spec[(size_t)n * Lc + col];
  __syncthreads();
  if constexpr (MODE == COL_INV) {
    fft64<+1>(buf, N, t, true, twN);
  } else {
    fft64<-1>(buf0, N, t, g == 0, twN);
  }
  if constexpr (MODE != COL_INV && MODE != COL_FWD) {
    double ab[5];
#pragma unroll
    for (int a = 0; a < 5; ++a)
      ab[a] = sc ? (MODE == COL_LBARINV ? sc->abar_n[a] : sc->abar[a]) : 0.0;
    // the column's points over all its threads: S = rho-bar sigma-hat / (N M), held until
    // every thread has read (column 0 pairs k with N - k)
    constexpr int PT = (4 + G - 1) / G;
    double2 s[PT], s0[PT];
#pragma unroll
    for (int e = 0; e < PT; ++e) {
      const int k = r + e * G * TPT;
      if (k >= N) continue;
      const double2 z = buf0[k];
      if (col == 0) {
        // unpack the two real columns k1 = 0 and k1 = M/2 carried as X0 + i XL
        const double2 p = buf0[k ? N - k : 0];
        double2 A = make_double2(0.5 * (z.x + p.x), 0.5 * (z.y - p.y));
        double2 B = make_double2(0.5 * (z.y + p.y), -0.5 * (z.x - p.x));
        double2 Bn = make_double2(0.0, 0.0);
        if constexpr (MODE == COL_POISSON || MODE == COL_POISSON_LP) {
          bool nyq2;
          const int k2 = sfreq(k, N, &nyq2);
          const double ly = fd_lap<double>(twN[k].x, N);
          A = cscale<double>(A, inv_nm * (inv_or_zero<double>(ly) *
                                          lowpass<double, MODE>(0, k2, M, N)));
          B = cscale<double>(B, inv_nm * (inv_or_zero<double>(fd_lap<double>(-1.0, M) + ly) *
                                          lowpass<double, MODE>(M / 2, k2, M, N)));
        } else {
          A = cmul64(rho_bar64(ab, symx[0], symy[k], inv_nm), A);
          B = cmul64(rho_bar64(ab, symx[M / 2], symy[k], inv_nm), B);
          // Q0's Nyquist channel is premultiplied by d11(M/2) (see k_col in spectral.cuh)
          if (MODE == COL_MATVEC) Bn = cscale<double>(B, symx[M / 2].y);
        }
        s[e] = make_double2(A.x - B.y, A.y + B.x);  // A + i B
        s0[e] = make_double2(A.x - Bn.y, A.y + Bn.x);
      } else {
        if constexpr (MODE == COL_POISSON || MODE == COL_POISSON_LP) {
          bool nyq2;
          const int k2 = sfreq(k, N, &nyq2);
          s[e] = cscale<double>(
              z, inv_nm * (inv_or_zero<double>(fd_lap<double>(twM[col].x, M) +
                                               fd_lap<double>(twN[k].x, N)) *
                           lowpass<double, MODE>(col, k2, M, N)));
        } else {
          s[e] = cmul64(rho_bar64(ab, symx[col], symy[k], inv_nm), z);
        }
        s0[e] = s[e];
      }
    }
    __syncthreads();
    // Q0 = S, Q1 = (i s1(k2)) S, Q2 = s2(k2) S (the other modes: S), G at a time
    constexpr int OUT = MODE == COL_MATVEC ? 3 : 1;
#pragma unroll 1
    for (int p0 = 0; p0 < OUT; p0 += G) {
#pragma unroll
      for (int e = 0; e < PT; ++e) {
        const int k = r + e * G * TPT;
        if (k >= N) continue;
        if constexpr (MODE == COL_MATVEC) {
          const double2 sy = symy[k];
          if (G == 3 || p0 == 0) buf0[k] = s0[e];
          if (G == 3 || p0 == 1) buf0[(G == 3) * F + k] = make_double2(-sy.x * s[e].y, sy.x * s[e].x);
          if (G == 3 || p0 == 2) buf0[(G == 3) * 2 * F + k] = cscale<double>(s[e], sy.y);
        } else {
          buf0[k] = s[e];
        }
      }
      __syncthreads();
      fft64<+1>(buf, N, t, true, twN);
      col_out<G>(p0, buf0, out0, out1, out2, N, Lc, col, F);
      if (p0 + G < OUT) __syncthreads();
    }
    return;
  }
  col_out<1>(0, buf0, out0, out1, out2, N, Lc, col, F);
}

// ---------------------------------------------------------------------------------------
// Row complex-to-real transforms.  RB rows per block.  G = 5 (combine): five thread groups and
// buffers per row, one per term; G = 1: one group, the combine's terms one after the other.
// ---------------------------------------------------------------------------------------
template <int MODE, int G>
__global__ void __launch_bounds__(kMaxThreads)
    k64_row_c2r(const double2* __restrict__ q0, const double2* __restrict__ q1,
                const double2* __restrict__ q2, const double* __restrict__ coef,
                double* __restrict__ out, const double* __restrict__ u_in,
                double* __restrict__ u_out, double step, double out_scale, int N, int M,
                const double2* __restrict__ twL, const double2* __restrict__ twM,
                const int* __restrict__ skip, const DevScalars* __restrict__ sc,
                const double2* __restrict__ symx) {
  if (skip && *skip) return;
  if (MODE == ROWINV_UPDATE && sc) {
    // device-resident control: step s and the current / candidate buffers come from sc
    step = sc->step_s;
    if (sc->upar & 1) {
      double* x = const_cast<double*>(u_in);
      u_in = u_out;
      u_out = x;
    }
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int L = M / 2, TPT = L / 4, F = FB(L);
  const int q = threadIdx.x / (G * TPT), r = threadIdx.x - q * (G * TPT);
  const int g = G == 1 ? 0 : r / TPT, t = r - g * TPT;
  const int row = blockIdx.x * (blockDim.x / (G * TPT)) + q;
  const bool active = row < N;
  double2* rows = reinterpret_cast<double2*>(smem_raw) + q * G * F;
  double2* buf = rows + g * F;
  const size_t P2 = (size_t)N * L;
  const double2* c = reinterpret_cast<const double2*>(coef + (size_t)row * M);
  constexpr int TERMS = MODE == ROWINV_COMBINE ? 5 : 1;
  double2 acc[MODE == ROWINV_COMBINE && G == 1 ? 4 : 1];
#pragma unroll 1
  for (int p = g; p < TERMS; p += G) {
    if (active) {
      // term p: d_xx Q0, d_x Q0, d_x Q1, Q1, Q2 (row symbols 2, 1, 1, 0, 0).  The symbol and
      // the complex-to-real pre-processing on the way in: Z_k = Ev + i conj(W_M^k) dv,
      // Z_(L-k) = conj(2 Ev - Z_k), Ev = X_k + conj X_(L-k), dv = X_k - conj X_(L-k)
      const double2* src = (p < 2 ? q0 : (p < 4 ? q1 : q2)) + (size_t)row * L;
      const int kind = TERMS == 1 ? 0 : (p == 0 ? 2 : (p < 3 ? 1 : 0));
      for (int k = t; k <= L / 2; k += TPT) {
        const double2 xk = row_symbol_apply<double>(src[k], k, kind, symx);
        if (k == 0) {
          buf[0] = make_double2(xk.x + xk.y, xk.x - xk.y);
        } else {
          const double2 xm = row_symbol_apply<double>(src[L - k], L - k, kind, symx);
          const double2 w = twM[k];
          const double2 ev = make_double2(xk.x + xm.x, xk.y - xm.y),
                        dv = make_double2(xk.x - xm.x, xk.y + xm.y);
          // i conj(w) = (w.y, w.x)
          const double2 s = make_double2(fma(w.y, dv.x, fma(-w.x, dv.y, ev.x)),
                                         fma(w.y, dv.y, fma(w.x, dv.x, ev.y)));
          buf[k] = s;
          if (2 * k != L)
            buf[L - k] = make_double2(fma(2.0, ev.x, -s.x), -fma(2.0, ev.y, -s.y));
        }
      }
    }
    __syncthreads();
    fft64<+1>(buf, L, t, active, twL);
    if constexpr (MODE == ROWINV_COMBINE && G == 1) {
      // coefficient planes a11, b1, 2 a12, b2, a22 of the five terms
      const double2* cp = c + (p == 0 ? 0 : (p == 1 ? 3 : (p == 2 ? 1 : (p == 3 ? 4 : 2)))) * P2;
      const double mult = p == 2 ? 2.0 : 1.0;
      if (active) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const double2 a = cp[t + e * TPT], y = buf[t + e * TPT];
          if (p == 0) acc[e] = make_double2(0.0, 0.0);
          acc[e].x = fma(mult * a.x, y.x, acc[e].x);
          acc[e].y = fma(mult * a.y, y.y, acc[e].y);
        }
      }
      if (p + 1 < TERMS) __syncthreads();
    }
  }
  if (!active) return;
  if constexpr (MODE == ROWINV_COMBINE && G == 1) {
    double2* o = reinterpret_cast<double2*>(out + (size_t)row * M);
#pragma unroll
    for (int e = 0; e < 4; ++e) o[t + e * TPT] = acc[e];
  } else if constexpr (MODE == ROWINV_COMBINE) {
    double2* o = reinterpret_cast<double2*>(out + (size_t)row * M);
    for (int n = r; n < L; n += G * TPT) {
      const double2 a11 = c[n], a12 = c[P2 + n], a22 = c[2 * P2 + n], b1 = c[3 * P2 + n],
                    b2 = c[4 * P2 + n];
      const double2 y0 = rows[n], y1 = rows[F + n], y2 = rows[2 * F + n], y3 = rows[3 * F + n],
                    y4 = rows[4 * F + n];
      // a11 y0 + b1 y1 + 2 a12 y2 + b2 y3 + a22 y4
      o[n] = make_double2(
          fma(a22.x, y4.x, fma(b2.x, y3.x, fma(2.0 * a12.x, y2.x, fma(b1.x, y1.x, a11.x * y0.x)))),
          fma(a22.y, y4.y, fma(b2.y, y3.y, fma(2.0 * a12.y, y2.y, fma(b1.y, y1.y, a11.y * y0.y)))));
    }
  } else if constexpr (MODE == ROWINV_UPDATE) {
    const double2* ui = reinterpret_cast<const double2*>(u_in + (size_t)row * M);
    double2* uo = reinterpret_cast<double2*>(u_out + (size_t)row * M);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int n = t + e * TPT;
      const double2 a = ui[n], y = buf[n];
      uo[n] = make_double2(fma(step, y.x, a.x), fma(step, y.y, a.y));
    }
  } else {
    double2* o = reinterpret_cast<double2*>(out + (size_t)row * M);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int n = t + e * TPT;
      o[n] = cscale<double>(buf[n], out_scale);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------------------
// Whether a multi-transform pass runs its `terms` transforms side by side: while the grid has
// fewer than eight lines per SM and the block fits in 512 threads (larger ones leave no second
// block on the SM); else one after the other, whose lines overlap each other instead.
// Side by side / in sequence, us: combine 9.2 / 30.5 at 64^2, 14.3 / 35.6 at 256^2, 51.6 / 54.4
// at 512^2, 89.5 / 95.4 at 1024 x 512; column pass 12.5 / 24.0, 17.7 / 28.4, 46.0 / 47.9 at
// 64^2, 256^2, 512^2, and 186 / 166 at 1024^2 (768 threads).
bool side_by_side(int terms, int L, int lines) {
  return lines < 8 * 152 && terms * (L / 4) <= 512;
}

// rows per block: one, or as many as keep a block within 128 threads while the
// grid still has four blocks per SM
int per_block(int threads, int lines) {
  int n = 1;
  while (2 * n * threads <= 128 && lines / (2 * n) >= 4 * 152) n *= 2;
  return n;
}

cudaError_t r2c64(const double* x, size_t xs, const int* jptr, const double* scale,
                  double2* spec, int N, int M, const SpecTables& tb, const int* skip,
                  cudaStream_t st) {
  const int L = M / 2, TPT = L / 4, RB = per_block(TPT, N);
  const size_t sm = (size_t)RB * FB(L) * sizeof(double2);
  const cudaError_t e = prepare_launch(k64_row_r2c, RB * TPT, sm);
  if (e != cudaSuccess) return e;
  k64_row_r2c<<<(N + RB - 1) / RB, RB * TPT, sm, st>>>(
      x, xs, jptr, scale, spec, N, M, (const double2*)tb.twL, (const double2*)tb.twM, skip);
  return cudaGetLastError();
}

template <int MODE, int G>
cudaError_t col64(const double2* spec, double2* o0, double2* o1, double2* o2, int N, int M,
                    const SpecTables& tb, const DevScalars* sc, const int* skip,
                    cudaStream_t st) {
  const int T = G * (N / 4);
  const size_t sm = (size_t)G * FB(N) * sizeof(double2);
  const cudaError_t e = prepare_launch(k64_col<MODE, G>, T, sm);
  if (e != cudaSuccess) return e;
  k64_col<MODE, G><<<M / 2, T, sm, st>>>(
      spec, o0, o1, o2, N, M, 1.0 / ((double)N * (double)M), (const double2*)tb.twN,
      (const double2*)tb.twM, sc, skip, (const double2*)tb.symx, (const double2*)tb.symy);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t col_mode64(const double2* spec, double2* o0, double2* o1, double2* o2, int N, int M,
                       const SpecTables& tb, const DevScalars* sc, const int* skip,
                       cudaStream_t st) {
  constexpr int G = MODE == COL_MATVEC ? 3 : 1;
  if (G > 1 && side_by_side(G, N, M / 2))
    return col64<MODE, G>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
  return col64<MODE, 1>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
}

template <int MODE, int G>
cudaError_t c2r64(const double2* q0, const double2* q1, const double2* q2, const double* coef,
                  double* out, const double* u_in, double* u_out, double step, double os, int N,
                  int M, const SpecTables& tb, const int* skip, cudaStream_t st,
                  const DevScalars* sc) {
  const int L = M / 2, T = G * (L / 4), RB = per_block(T, N);
  const size_t sm = (size_t)RB * G * FB(L) * sizeof(double2);
  const cudaError_t e = prepare_launch(k64_row_c2r<MODE, G>, RB * T, sm);
  if (e != cudaSuccess) return e;
  k64_row_c2r<MODE, G><<<(N + RB - 1) / RB, RB * T, sm, st>>>(
      q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, (const double2*)tb.twL,
      (const double2*)tb.twM, skip, sc, (const double2*)tb.symx);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t c2r_mode(const double2* q0, const double2* q1, const double2* q2,
                     const double* coef, double* out, const double* u_in, double* u_out,
                     double step, double os, int N, int M, const SpecTables& tb,
                     const int* skip, cudaStream_t st, const DevScalars* sc) {
  constexpr int G = MODE == ROWINV_COMBINE ? 5 : 1;
  if (G > 1 && side_by_side(G, M / 2, N))
    return c2r64<MODE, G>(q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, tb, skip, st,
                             sc);
  return c2r64<MODE, 1>(q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, tb, skip, st,
                           sc);
}

}  // namespace

// (plan sets are mixed precision: no batched FP64 pass)
template <>
cudaError_t launch_row_r2c<double>(const double* x, size_t xs, const int* jptr,
                                   const double* scale, double2* spec, int N, int M,
                                   const SpecTables& tb, const int* skip, cudaStream_t st,
                                   Bat bat, const DevScalars*) {
  if (bat.on) return cudaErrorInvalidValue;
  return r2c64(x, xs, jptr, scale, spec, N, M, tb, skip, st);
}

template <>
cudaError_t launch_col<double>(int mode, const double2* spec, double2* o0, double2* o1,
                               double2* o2, int N, int M, const SpecTables& tb,
                               const DevScalars* sc, const int* skip, cudaStream_t st, Bat bat) {
  if (bat.on) return cudaErrorInvalidValue;
  switch (mode) {
    case COL_FWD: return col_mode64<COL_FWD>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
    case COL_INV: return col_mode64<COL_INV>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
    case COL_MATVEC: return col_mode64<COL_MATVEC>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
    case COL_LBARINV: return col_mode64<COL_LBARINV>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
    case COL_POISSON: return col_mode64<COL_POISSON>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
    case COL_POISSON_LP:
      return col_mode64<COL_POISSON_LP>(spec, o0, o1, o2, N, M, tb, sc, skip, st);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_row_c2r<double>(int mode, const double2* q0, const double2* q1,
                                   const double2* q2, const double* coef, double* out,
                                   const double* u_in, double* u_out, double step, double os,
                                   int N, int M, const SpecTables& tb, const int* skip,
                                   cudaStream_t st, const DevScalars* sc, Bat bat) {
  if (bat.on) return cudaErrorInvalidValue;
  switch (mode) {
    case ROWINV_PLAIN:
      return c2r_mode<ROWINV_PLAIN>(q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, tb,
                                    skip, st, sc);
    case ROWINV_COMBINE:
      return c2r_mode<ROWINV_COMBINE>(q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, tb,
                                      skip, st, sc);
    case ROWINV_UPDATE:
      return c2r_mode<ROWINV_UPDATE>(q0, q1, q2, coef, out, u_in, u_out, step, os, N, M, tb,
                                     skip, st, sc);
  }
  return cudaErrorInvalidValue;
}

}  // namespace otgb

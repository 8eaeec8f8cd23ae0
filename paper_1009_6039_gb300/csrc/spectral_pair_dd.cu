// theta = Lbar^{-1} sigma (Sec. 4.2) and the warm start's Poisson solves on column and row
// pairs, with the double-float inverse transforms in packed FP32 arithmetic.
//
// These compute what k_col_lbarinv_dd and k_row_c2r_update_dd compute, but hold two
// columns (rows) side by side: a double-float value is the pair (hi, lo) of FP32 numbers,
// and the two columns' values share register pairs, (hi_a, hi_b) and (lo_a, lo_b).  Every
// step of the error-free transformations (TwoSum, FastTwoSum, the FMA TwoProduct of dd.cuh)
// then runs once for both columns as a packed instruction (add/sub/mul/fma.rn.f32x2, per
// lane the scalar round-to-nearest operation), in the scalar kernels' order of operations,
// so a lane computes bit for bit the scalar double-float result from the same inputs.  The
// column pass's forward transform and symbol step are FP32 (the forward on packed pairs as in
// k_col_pair).  Double-float elements live in two shared-memory planes, the high words
// (re, im) and the low words, 16 bytes per element each, under the swizzle of pair.cuh.
#include "dd2.cuh"
#include "pair.cuh"

namespace otgb {
namespace {

using namespace pair;

// two double-float complex numbers
struct DC {
  D2 re, im;
};
__device__ __forceinline__ DC dc_add(DC a, DC b) {
  return DC{d2_add(a.re, b.re), d2_add(a.im, b.im)};
}
__device__ __forceinline__ DC dc_sub(DC a, DC b) {
  return DC{d2_sub(a.re, b.re), d2_sub(a.im, b.im)};
}
// a * w, w = (wx, wy) broadcast to both lanes (the scalar complex product's order)
__device__ __forceinline__ DC dc_mul(DC a, D2 wx, D2 wy) {
  return DC{d2_sub(d2_mul(a.re, wx), d2_mul(a.im, wy)),
            d2_add(d2_mul(a.re, wy), d2_mul(a.im, wx))};
}
// SIGN i a
template <int SIGN>
__device__ __forceinline__ DC dc_mul_si(DC a) {
  return SIGN > 0 ? DC{d2_neg(a.im), a.re} : DC{a.im, d2_neg(a.re)};
}

template <int R, int SIGN> struct BflyDC;
template <int SIGN> struct BflyDC<2, SIGN> {
  __device__ __forceinline__ static void run(DC* v) {
    const DC a = v[0], b = v[1];
    v[0] = dc_add(a, b);
    v[1] = dc_sub(a, b);
  }
};
template <int SIGN> struct BflyDC<3, SIGN> {  // the scalar butterfly's operations
  __device__ __forceinline__ static void run(DC* v) {
    const DC a = v[0], s = dc_add(v[1], v[2]), d = dc_sub(v[1], v[2]);
    const D2 half{pk(0.5f, 0.5f), 0ull};
    const dd c = dd(OTGB_SQRT3_HALF);
    const D2 cc{pk(c.hi, c.hi), pk(c.lo, c.lo)};
    const DC t{d2_sub(a.re, d2_mul(half, s.re)), d2_sub(a.im, d2_mul(half, s.im))};
    const DC e = dc_mul_si<SIGN>(d);
    const DC u{d2_mul(e.re, cc), d2_mul(e.im, cc)};
    v[0] = dc_add(a, s);
    v[1] = dc_add(t, u);
    v[2] = dc_sub(t, u);
  }
};
template <int SIGN> struct BflyDC<4, SIGN> {
  __device__ __forceinline__ static void run(DC* v) {
    const DC t0 = dc_add(v[0], v[2]), t1 = dc_sub(v[0], v[2]);
    const DC t2 = dc_add(v[1], v[3]), t3 = dc_mul_si<SIGN>(dc_sub(v[1], v[3]));
    v[0] = dc_add(t0, t2);
    v[2] = dc_sub(t0, t2);
    v[1] = dc_add(t1, t3);
    v[3] = dc_sub(t1, t3);
  }
};

// a double-float complex pair buffer: high words (re, im) and low words, L elements each
struct DBuf {
  ulonglong2* h;
  ulonglong2* l;
};
__device__ __forceinline__ DC dld(DBuf b, int i) {
  const ulonglong2 x = b.h[i], y = b.l[i];
  return DC{D2{x.x, y.x}, D2{x.y, y.y}};
}
__device__ __forceinline__ void dst(DBuf b, int i, DC v) {
  b.h[i] = make_ulonglong2(v.re.h, v.im.h);
  b.l[i] = make_ulonglong2(v.re.l, v.im.l);
}
__device__ __forceinline__ DC dc_from(ddc a, ddc b) {
  return DC{D2{pk(a.x.hi, b.x.hi), pk(a.x.lo, b.x.lo)},
            D2{pk(a.y.hi, b.y.hi), pk(a.y.lo, b.y.lo)}};
}
__device__ __forceinline__ void dc_to(DC v, ddc& a, ddc& b) {
  upk(v.re.h, a.x.hi, b.x.hi);
  upk(v.re.l, a.x.lo, b.x.lo);
  upk(v.im.h, a.y.hi, b.y.hi);
  upk(v.im.l, a.y.lo, b.y.lo);
}

// the stage twiddles of the double-float transforms of length L, broadcast to both
// lanes: high words (x, y) in th, low words in tl
template <int L>
__device__ __forceinline__ void load_twdd(ulonglong2* th, ulonglong2* tl,
                                          const ddc* __restrict__ twb, int t, int nthreads) {
  const ddc* __restrict__ st = pstage_table<L>(twb);
  for (int i = t; i < L; i += nthreads) {
    const ddc w = st[i];
    th[i] = make_ulonglong2(pk(w.x.hi, w.x.hi), pk(w.y.hi, w.y.hi));
    tl[i] = make_ulonglong2(pk(w.x.lo, w.x.lo), pk(w.y.lo, w.y.lo));
  }
}

// a double-float stage of radix R (span Ns), in pload, pbfly and pstore's three steps and with their
// slots
template <int R, int L>
__device__ __forceinline__ void dload(DBuf in, DC (&v)[pslots<R>()], int t, int sx = 0) {
  constexpr int T = R == 3 ? L / 3 : L / 4, LR = L / R;
#pragma unroll
  for (int s = 0; s < pslots<R>(); ++s) v[s] = dld(in, swz(t + (s / R) * T + (s % R) * LR) ^ sx);
}
template <int R, int SIGN, int L, int Ns>
__device__ __forceinline__ void dbfly(DC (&v)[pslots<R>()], int t,
                                      const ulonglong2* __restrict__ th,
                                      const ulonglong2* __restrict__ tl) {
  constexpr int T = R == 3 ? L / 3 : L / 4;
#pragma unroll
  for (int b = 0; b < pslots<R>() / R; ++b) {
    if (Ns > 1) {
      const int k = (int)((unsigned)(t + b * T) % (unsigned)Ns);
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const int ti = (Ns - 1) + (r - 1) * Ns + k;
        const ulonglong2 wh = th[ti], wl = tl[ti];
        const D2 wx{wh.x, wl.x};
        D2 wy{wh.y, wl.y};
        if (SIGN > 0) wy = d2_neg(wy);
        v[b * R + r] = dc_mul(v[b * R + r], wx, wy);
      }
    }
    BflyDC<R, SIGN>::run(&v[b * R]);
  }
}
template <int R, int L, int Ns>
__device__ __forceinline__ void dstore(DBuf out, const DC (&v)[pslots<R>()], int t, int sx = 0) {
  constexpr int T = R == 3 ? L / 3 : L / 4;
#pragma unroll
  for (int s = 0; s < pslots<R>(); ++s) {
    const int j = t + (s / R) * T;
    const int qd = (int)((unsigned)j / (unsigned)Ns);
    dst(out, swz(qd * (Ns * R) + (j - qd * Ns) + (s % R) * Ns) ^ sx, v[s]);
  }
}
// in -> out (in place: the stores wait for every thread's loads)
template <int R, int SIGN, int L, int Ns, bool INPLACE>
__device__ __forceinline__ void dstage(DBuf in, DBuf out, int t,
                                       const ulonglong2* __restrict__ th,
                                       const ulonglong2* __restrict__ tl, int sx = 0) {
  const bool active = pactive<R, L>(t);
  DC v[pslots<R>()];
  if (active) dload<R, L>(in, v, t, sx);
  if (INPLACE) __syncthreads();
  if (active) {
    dbfly<R, SIGN, L, Ns>(v, t, th, tl);
    dstore<R, L, Ns>(out, v, t, sx);
  }
  __syncthreads();
}

// the inverse transform's stages from span Ns on, without the last one: in place (INPLACE), or
// alternating between a and b from a
template <int SIGN, int L, int Ns, int REM, bool INPLACE, bool FROM_A>
__device__ __forceinline__ void dfft(DBuf a, DBuf b, int t, const ulonglong2* __restrict__ th,
                                     const ulonglong2* __restrict__ tl, int sx = 0) {
  constexpr int R = pradix<REM>();
  if constexpr (REM > R) {
    if constexpr (INPLACE)
      dstage<R, SIGN, L, Ns, true>(a, a, t, th, tl, sx);
    else if constexpr (FROM_A)
      dstage<R, SIGN, L, Ns, false>(a, b, t, th, tl, sx);
    else
      dstage<R, SIGN, L, Ns, false>(b, a, t, th, tl, sx);
    dfft<SIGN, L, Ns * R, REM / R, INPLACE, !FROM_A>(a, b, t, th, tl, sx);
  }
}

__device__ __forceinline__ float lowpass_of(int mode, int k1, int k2, int M, int N) {
  return mode == COL_POISSON_LP ? lowpass_f<COL_POISSON_LP>(k1, k2, M, N) : 1.f;
}

// theta's column pass (mode COL_LBARINV: S = rho-bar(abar_n) sigma-hat / (N M)) or, POISSON, the
// Poisson solves' (modes COL_POISSON, COL_POISSON_LP: division by the 4th-order FD Laplacian's
// eigenvalues, zero mode -> 0, _LP with the Gaussian low-pass) on column pairs: the FP32
// forward column transform, the scalar symbol step of k_col_lbarinv_dd per column, the
// double-float inverse column transform (out of place), ddc output
template <int N, bool POISSON, int G>
__global__ void __launch_bounds__(pthreads<N>() * G, N * G <= 1024 ? 2 : 1)
    k_col_lbarinv_pair(const float2* __restrict__ spec, ddc* __restrict__ out, int M, int mode,
                       float inv, const float2* __restrict__ twN32,
                       const float2* __restrict__ twM32, const ddc* __restrict__ twNdd,
                       const DevScalars* __restrict__ sc, const float2* __restrict__ symx,
                       const float2* __restrict__ symy, Bat bat) {
  spec = badv(spec, bat);
  out = badv(out, bat);
  sc = badv(sc, bat);
  if (bat.on && bskip(sc, bat)) return;
  constexpr int TPT = pthreads<N>(), E = pelems<N>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* tw4 = reinterpret_cast<ulonglong2*>(smem_raw);
  ulonglong2* th = tw4 + N;
  ulonglong2* tl = th + N;
  const int grp = G == 1 ? 0 : threadIdx.x % G, sx = 8 / G * grp;  // as in k_col_pair
  ulonglong2* base = tl + N + (size_t)grp * 4 * N;
  // double-float buffers A (h, l) and B (h, l); the FP32 forward ping-pongs inside A
  const DBuf A{base, base + N}, B{base + 2 * N, base + 3 * N};
  PC* const F0 = reinterpret_cast<PC*>(A.h);
  PC* const F1 = reinterpret_cast<PC*>(A.l);
  const int Lc = M / 2;
  const int c0 = 2 * (G * blockIdx.x + grp);
  const int t = threadIdx.x / G;
  // the column pair's loads first, so that they are in flight with the twiddle tables' loads
  float4 xs[E];
#pragma unroll
  for (int e = 0; e < E; ++e)
    xs[e] = *reinterpret_cast<const float4*>(spec + (size_t)(t + e * TPT) * Lc + c0);
  load_tw4<N>(tw4, twN32, threadIdx.x, TPT * G);
  load_twdd<N>(th, tl, twNdd, threadIdx.x, TPT * G);
  constexpr int R0 = pradix<N>(), RL = plast<N>();
  constexpr bool FLIP = pstage_count<N>() % 2 == 1;  // the stages between end in the second buffer
  const bool last = pactive<RL, N>(t);
  PC zf[1][E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    zf[0][e].re = pk(xs[e].x, xs[e].z);
    zf[0][e].im = pk(xs[e].y, xs[e].w);
  }
  {
    PC* const a[1] = {F0};
    PC* const b[1] = {F1};
    pfirst_regs<-1, N, 1>(zf, a, t, sx);
    pfft_rec<-1, N, R0, N / R0, 1, true, false>(a, b, t, tw4, sx);
  }
  PC* const F[1] = {FLIP ? F1 : F0};
  PC* const X = FLIP ? F0 : F1;  // the exchange, as in k_col_pair
  PC f[1][4];
  if (last) plast_regs<-1, N, 1>(F, f, t, tw4, sx);
  if (N % 3 == 0 || blockIdx.x == 0) {
    if (last) {
#pragma unroll
      for (int q = 0; q < 4; ++q) X[swz(pout<RL, N>(t, q)) ^ sx] = f[0][q];
    }
    __syncthreads();
  }

  float ab[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) ab[q] = !POISSON ? (float)sc->abar_n[q] : 0.f;
  DC v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int k = t + e * TPT;
    PC z2;
    if constexpr (N % 3 == 0)
      z2 = X[swz(k) ^ sx];
    else
      z2 = f[0][RL == 4 ? e : (e & 1) * 2 + (e >> 1)];
    float2 zc[2];
    upk(z2.re, zc[0].x, zc[1].x);
    upk(z2.im, zc[0].y, zc[1].y);
    float2 s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int col = c0 + h;
      const float2 z = zc[h];
      float2 r;
      if (col == 0) {
        const PC p2 = X[swz((N - k) % N) ^ sx];
        float2 pz, pother;
        upk(p2.re, pz.x, pother.x);
        upk(p2.im, pz.y, pother.y);
        float2 Av = mk2<float>(0.5f * (z.x + pz.x), 0.5f * (z.y - pz.y));
        float2 Bv = mk2<float>(0.5f * (z.y + pz.y), -0.5f * (z.x - pz.x));
        if (!POISSON) {
          Av = cmul<float>(rho_bar<float>(ab, symx[0], symy[k]), Av);
          Bv = cmul<float>(rho_bar<float>(ab, symx[M / 2], symy[k]), Bv);
        } else {
          bool nyq2;
          const int k2 = sfreq(k, N, &nyq2);
          const float ly = fd_lap_w(twN32[k], N);
          const float lxn = -16.f / 3.f * (float)M * (float)M;  // k1 = M/2 (cos t = -1)
          Av = cscale<float>(Av, inv_or_zero<float>(ly) * lowpass_of(mode, 0, k2, M, N));
          Bv = cscale<float>(Bv,
                             inv_or_zero<float>(lxn + ly) * lowpass_of(mode, M / 2, k2, M, N));
        }
        r = mk2<float>(Av.x - Bv.y, Av.y + Bv.x);
      } else if (!POISSON) {
        r = cmul<float>(rho_bar<float>(ab, symx[col], symy[k]), z);
      } else {
        bool nyq2;
        const int k2 = sfreq(k, N, &nyq2);
        r = cscale<float>(z, inv_or_zero<float>(fd_lap_w(twM32[col], M) +
                                                fd_lap_w(twN32[k], N)) *
                                 lowpass_of(mode, col, k2, M, N));
      }
      s[h] = mk2<float>(r.x * inv, r.y * inv);
    }
    v[e].re = D2{pk(s[0].x, s[1].x), 0ull};
    v[e].im = D2{pk(s[0].y, s[1].y), 0ull};
  }
  // inverse in double-float from B (scratch A, behind the first stage's barrier)
  dbfly<R0, +1, N, 1>(v, t, th, tl);
  dstore<R0, N, 1>(B, v, t, sx);
  __syncthreads();
  dfft<+1, N, R0, N / R0, false, true>(B, A, t, th, tl, sx);
  if (!last) return;
  DC r[4];
  dload<RL, N>(FLIP ? A : B, r, t, sx);
  dbfly<RL, +1, N, N / RL>(r, t, th, tl);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    ddc a, b;
    dc_to(r[q], a, b);
    ddc* o = out + (size_t)pout<RL, N>(t, q) * Lc + c0;
    o[0] = a;
    o[1] = b;
  }
}

// theta's rows (complex-to-real, double-float) on row pairs, then u_out = u_in + step theta
// in FP64 (u_in == nullptr: u_out = step theta; with sc the step and the current / candidate
// buffers come from the device scalars, as in k_row_c2r_update_dd); in-place stages
template <int L>
__global__ void __launch_bounds__(pthreads<L>(), L <= 512 ? 4 : 2)
    k_row_update_pair(const ddc* __restrict__ q, const double* __restrict__ u_in,
                      double* __restrict__ u_out, double step, int N,
                      const ddc* __restrict__ twL, const ddc* __restrict__ twM,
                      const DevScalars* __restrict__ sc, Bat bat) {
  q = badv(q, bat);
  u_in = badv(u_in, bat);
  u_out = badv(u_out, bat);
  sc = badv(sc, bat);
  if (bat.on && bskip(sc, bat)) return;
  if (sc) {
    step = sc->step_s;
    if (sc->upar & 1) {
      double* tmp = const_cast<double*>(u_in);
      u_in = u_out;
      u_out = tmp;
    }
  }
  constexpr int TPT = pthreads<L>(), E = pelems<L>();
  constexpr int M = 2 * L;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* th = reinterpret_cast<ulonglong2*>(smem_raw);
  ulonglong2* tl = th + L;
  const DBuf A{tl + L, tl + 2 * L};
  const int r0 = 2 * blockIdx.x;
  const int t = threadIdx.x;
  // the rows' loads first, so that they are in flight with the twiddle table's loads
  const ddc* qa = q + (size_t)r0 * L;
  const ddc* qb = qa + L;
  ddc ra[E], rb[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    ra[e] = qa[t + e * TPT];
    rb[e] = qb[t + e * TPT];
  }
  load_twdd<L>(th, tl, twL, t, TPT);
#pragma unroll
  for (int e = 0; e < E; ++e) dst(A, swz(t + e * TPT), dc_from(ra[e], rb[e]));
  __syncthreads();
  // complex-to-real pre-processing (as c2r_preprocess on dd): each pair (k, L - k) by one
  // thread
  for (int k = t; k <= L / 2; k += TPT) {
    if (k == 0) {
      const int d = swz(0);
      const DC x = dld(A, d);
      dst(A, d, DC{d2_add(x.re, x.im), d2_sub(x.re, x.im)});
    } else {
      const ddc w = twM[k];
      const D2 wx{pk(w.x.hi, w.x.hi), pk(w.x.lo, w.x.lo)};
      // conj(W_M^k)
      const D2 wy = d2_neg(D2{pk(w.y.hi, w.y.hi), pk(w.y.lo, w.y.lo)});
      const int dk = swz(k), dm = swz(L - k);
      const DC xk = dld(A, dk), xm = dld(A, dm);
      const DC Ev{d2_add(xk.re, xm.re), d2_sub(xk.im, xm.im)};
      const DC dv{d2_sub(xk.re, xm.re), d2_add(xk.im, xm.im)};
      const DC Ov = dc_mul(dv, wx, wy);
      dst(A, dk, DC{d2_sub(Ev.re, Ov.im), d2_add(Ev.im, Ov.re)});
      if (2 * k != L) dst(A, dm, DC{d2_add(Ev.re, Ov.im), d2_add(d2_neg(Ev.im), Ov.re)});
    }
  }
  __syncthreads();
  constexpr int R0 = pradix<L>(), RL = plast<L>();
  dstage<R0, +1, L, 1, true>(A, A, t, th, tl);
  dfft<+1, L, R0, L / R0, true, true>(A, A, t, th, tl);
  if (!pactive<RL, L>(t)) return;
  DC r[4];
  dload<RL, L>(A, r, t);
  dbfly<RL, +1, L, L / RL>(r, t, th, tl);
  const double2* uia = u_in ? reinterpret_cast<const double2*>(u_in + (size_t)r0 * M) : nullptr;
  const double2* uib = u_in ? uia + L : nullptr;
  double2* uoa = reinterpret_cast<double2*>(u_out + (size_t)r0 * M);
  double2* uob = uoa + L;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int n = pout<RL, L>(t, e);
    ddc za, zb;
    dc_to(r[e], za, zb);
    double2 a = uia ? uia[n] : make_double2(0.0, 0.0);
    double2 b = uib ? uib[n] : make_double2(0.0, 0.0);
    a.x = fma(step, dd_to_double(za.x), a.x);
    a.y = fma(step, dd_to_double(za.y), a.y);
    b.x = fma(step, dd_to_double(zb.x), b.x);
    b.y = fma(step, dd_to_double(zb.y), b.y);
    uoa[n] = a;
    uob[n] = b;
  }
}

template <int N, bool POISSON, int G>
cudaError_t col_lbarinv_pair_launch(const float2* spec, ddc* out, int M, const SpecTables& tb32,
                               const SpecTables& tbdd, const DevScalars* sc, cudaStream_t st,
                               int mode, Bat bat) {
  const size_t sm = (3 + 4 * G) * (size_t)N * sizeof(ulonglong2);
  cudaError_t e = prepare_launch(k_col_lbarinv_pair<N, POISSON, G>, pthreads<N>() * G, sm);
  if (e != cudaSuccess) return e;
  k_col_lbarinv_pair<N, POISSON, G><<<bgrid(dim3(M / 4 / G), bat), pthreads<N>() * G, sm, st>>>(
      spec, out, M, mode, (float)(1.0 / ((double)N * (double)M)), (const float2*)tb32.twN,
      (const float2*)tb32.twM, (const ddc*)tbdd.twN, sc, (const float2*)tb32.symx,
      (const float2*)tb32.symy, bat);
  return cudaGetLastError();
}

template <int N>
cudaError_t col_lbarinv_pair_N(const float2* spec, ddc* out, int M, const SpecTables& tb32,
                               const SpecTables& tbdd, const DevScalars* sc, cudaStream_t st,
                               int mode, Bat bat) {
  if constexpr (N <= 1024) {
    if (two_pairs(M, bat)) {
      if (mode == COL_LBARINV)
        return col_lbarinv_pair_launch<N, false, 2>(spec, out, M, tb32, tbdd, sc, st, mode, bat);
      return col_lbarinv_pair_launch<N, true, 2>(spec, out, M, tb32, tbdd, sc, st, mode, bat);
    }
  }
  if (mode == COL_LBARINV)
    return col_lbarinv_pair_launch<N, false, 1>(spec, out, M, tb32, tbdd, sc, st, mode, bat);
  return col_lbarinv_pair_launch<N, true, 1>(spec, out, M, tb32, tbdd, sc, st, mode, bat);
}

template <int L>
cudaError_t row_update_pair_L(const ddc* q, const double* u_in, double* u_out, double step,
                              int N, const SpecTables& tbdd, const DevScalars* sc,
                              cudaStream_t st, Bat bat) {
  const size_t sm = 4 * (size_t)L * sizeof(ulonglong2);
  cudaError_t e = prepare_launch(k_row_update_pair<L>, pthreads<L>(), sm);
  if (e != cudaSuccess) return e;
  k_row_update_pair<L><<<bgrid(dim3(N / 2), bat), pthreads<L>(), sm, st>>>(
      q, u_in, u_out, step, N, (const ddc*)tbdd.twL, (const ddc*)tbdd.twM, sc, bat);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_col_lbarinv_pair(const float2* spec, ddc* out, int N, int M,
                                    const SpecTables& tb32, const SpecTables& tbdd,
                                    const DevScalars* sc, cudaStream_t st, int mode, Bat bat) {
  if (!col_pair_supported(N, M)) return cudaErrorInvalidValue;
  if (mode != COL_LBARINV && mode != COL_POISSON && mode != COL_POISSON_LP)
    return cudaErrorInvalidValue;
  if ((mode == COL_LBARINV || bat.on) && !sc) return cudaErrorInvalidValue;
  if (((uintptr_t)spec | bat.slab) & 15) return cudaErrorMisalignedAddress;
#define OTGB_CALL(n) col_lbarinv_pair_N<n>(spec, out, M, tb32, tbdd, sc, st, mode, bat)
  OTGB_COL_LENGTHS(N, OTGB_CALL)
#undef OTGB_CALL
  return cudaErrorInvalidValue;
}

cudaError_t launch_row_update_pair(const ddc* q, const double* u_in, double* u_out,
                                   double step, int N, int M, const SpecTables& tbdd,
                                   const DevScalars* sc, cudaStream_t st, Bat bat) {
  if (!comb_pair_supported(N, M) || (bat.on && !sc)) return cudaErrorInvalidValue;
#define OTGB_CALL(n) row_update_pair_L<n>(q, u_in, u_out, step, N, tbdd, sc, st, bat)
  OTGB_ROW_LENGTHS(M / 2, OTGB_CALL)
#undef OTGB_CALL
  return cudaErrorInvalidValue;
}

}  // namespace otgb

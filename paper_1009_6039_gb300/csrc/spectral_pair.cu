// Column pass of the FP32 matvec (Sec. 4.2) on column pairs with packed FP32 arithmetic.
//
// The pass computes what k_col<float, E, COL_MATVEC> computes -- per column of the packed
// N x M/2 half spectrum: the forward column FFT, S = rho-bar sigma-hat / (N M), and the
// inverse column FFTs of S (its Nyquist channel premultiplied), (i s1(k2)) S and s2(k2) S --
// but one block takes two neighbouring columns c0 = 2b and c0 + 1 and holds them side by
// side: the element n of a transform pair is the 16-byte word (a.x, b.x, a.y, b.y) of the
// two columns' values a and b.  The real parts and the imaginary parts of the pair are then
// register pairs, so every complex addition of a butterfly is one packed instruction
// (add/sub.rn.f32x2) for both columns, and every twiddle multiplication two packed
// multiply-adds per part, with the twiddle broadcast to both lanes; the multiplication by
// +-i exchanges the parts and costs nothing.  A thread holds 4 elements (radix-4 stages,
// one radix-2 stage for odd powers of two), the length is fixed at compile time
// (96 ... 2048), and the stages run out of place between two buffer sets (one barrier a
// stage).  The loaded column enters the first stage in registers, the last forward stage's
// results take the symbols and enter the first inverse stage there (a factor 3 exchanges them
// once, and columns 0 and M/2 their mirrored entries), and the last stage stores to global
// memory: 8 passes through shared memory where there were 13.  Shared memory is addressed through an XOR swizzle of the 16-byte element index,
// i ^ ((i >> 2) & 7), under which every stage's reads and writes of a quarter warp fall in
// distinct bank groups.  The symbol multiplies are the scalar operations of k_col.
// (In place on three buffers -- 64 N instead of 112 N bytes, two barriers a stage -- measured the
// same within 3 % for plan sets' classes and single grids of 512^2 to 2048^2.)
#include "pair.cuh"

namespace otgb {
namespace {

using namespace pair;

// G column pairs per block, a pair per group of every G-th thread, so that a row's G pairs are read
// and written by neighbouring threads (G == 2: whole 32-byte sectors; one pair's 16 bytes are half
// of one, and the kernel waited for them: 1024^2 15.9 -> 12.9 us, 5 problems of 512^2 19.2 -> 16.0).
// The groups have their own buffers, the second one's swizzled by 4 elements more (sx): the four
// elements of either group that a quarter warp accesses then lie in distinct bank groups.
// (G == 4 is no better: 5 of 512^2 18.6 us, 16 of 384^2 24.0 against 25.3.)
template <int N, int G>
__global__ void __launch_bounds__(pthreads<N>() * G, N * G <= 1024 ? 2 : 1)
    k_col_pair(const float2* __restrict__ spec, float2* __restrict__ out0,
               float2* __restrict__ out1, float2* __restrict__ out2, int M, float inv,
               const float2* __restrict__ twN, const DevScalars* __restrict__ sc,
               const int* __restrict__ skip, const float2* __restrict__ symx,
               const float2* __restrict__ symy, Bat bat) {
  spec = badv(spec, bat);
  out0 = badv(out0, bat);
  out1 = badv(out1, bat);
  out2 = badv(out2, bat);
  sc = badv(sc, bat);
  skip = badv(skip, bat);
  if ((skip && *skip) || (bat.on && bskip(sc, bat))) return;
  constexpr int TPT = pthreads<N>(), E = pelems<N>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* tw4 = reinterpret_cast<ulonglong2*>(smem_raw);
  const int grp = G == 1 ? 0 : threadIdx.x % G, sx = 8 / G * grp;
  PC* pb = reinterpret_cast<PC*>(smem_raw + (size_t)N * sizeof(ulonglong2)) + (size_t)grp * 6 * N;
  PC* const P[6] = {pb, pb + N, pb + 2 * N, pb + 3 * N, pb + 4 * N, pb + 5 * N};
  const int Lc = M / 2;
  const int c0 = 2 * (G * blockIdx.x + grp);
  const int t = threadIdx.x / G;

  // the column pair: one 16-byte load per row, issued before the twiddle table is built so
  // that both sets of loads are in flight together, then regrouped into (re, im) pairs
  float4 xs[E];
#pragma unroll
  for (int e = 0; e < E; ++e)
    xs[e] = *reinterpret_cast<const float4*>(spec + (size_t)(t + e * TPT) * Lc + c0);
  float2 sy[E];
#pragma unroll
  for (int e = 0; e < E; ++e) sy[e] = symy[t + e * TPT];
  const float2 sxa = symx[c0], sxb = symx[c0 + 1];
  float ab[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) ab[q] = sc ? (float)sc->abar[q] : 0.f;
  load_tw4<N>(tw4, twN, threadIdx.x, TPT * G);

  // forward column transforms of both columns (in P0 and P3)
  constexpr int R0 = pradix<N>(), RL = plast<N>();
  constexpr bool FLIP = pstage_count<N>() % 2 == 1;  // the stages between end in P3
  const bool last = pactive<RL, N>(t);
  PC z[1][E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    z[0][e].re = pk(xs[e].x, xs[e].z);
    z[0][e].im = pk(xs[e].y, xs[e].w);
  }
  {
    PC* const a[1] = {P[0]};
    PC* const b[1] = {P[3]};
    pfirst_regs<-1, N, 1>(z, a, t, sx);
    pfft_rec<-1, N, R0, N / R0, 1, true, false>(a, b, t, tw4, sx);
  }
  PC* const F[1] = {FLIP ? P[3] : P[0]};
  // the exchange of the transformed columns (a set apart from F and from the inverse
  // transforms' first one): where a thread's slots of the last stage are not those of the first
  // (a factor 3), and for the mirrored entries of columns 0 and M / 2
  PC* const X = FLIP ? P[4] : P[1];
  PC f[1][4];
  if (last) plast_regs<-1, N, 1>(F, f, t, tw4, sx);
  if (N % 3 == 0 || blockIdx.x == 0) {
    if (last) {
#pragma unroll
      for (int s = 0; s < 4; ++s) X[swz(pout<RL, N>(t, s)) ^ sx] = f[0][s];
    }
    __syncthreads();
  }

  PC v[3][E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int k = t + e * TPT;
    PC zk;
    if constexpr (N % 3 == 0)
      zk = X[swz(k) ^ sx];
    else  // slot s = b RL + r is element t + (b + r 4 / RL) N / 4
      zk = f[0][RL == 4 ? e : (e & 1) * 2 + (e >> 1)];
    float2 za, zb;
    upk(zk.re, za.x, zb.x);
    upk(zk.im, za.y, zb.y);
    float2 sa, s0a;
    if (c0 == 0) {
      // the two real columns k1 = 0 and k1 = M/2 carried as X0 + i XL (as in k_col)
      const PC pz = X[swz((N - k) % N) ^ sx];
      float2 p, pbv;
      upk(pz.re, p.x, pbv.x);
      upk(pz.im, p.y, pbv.y);
      float2 A = mk2<float>(0.5f * (za.x + p.x), 0.5f * (za.y - p.y));
      float2 B = mk2<float>(0.5f * (za.y + p.y), -0.5f * (za.x - p.x));
      A = cmul<float>(rho_bar<float>(ab, symx[0], sy[e]), A);
      B = cmul<float>(rho_bar<float>(ab, symx[M / 2], sy[e]), B);
      const float2 Bn = cscale<float>(B, symx[M / 2].y);
      s0a = cscale<float>(mk2<float>(A.x - Bn.y, A.y + Bn.x), inv);
      sa = cscale<float>(mk2<float>(A.x - B.y, A.y + B.x), inv);
    } else {
      sa = cscale<float>(cmul<float>(rho_bar<float>(ab, sxa, sy[e]), za), inv);
      s0a = sa;
    }
    const float2 sb = cscale<float>(cmul<float>(rho_bar<float>(ab, sxb, sy[e]), zb), inv);
    v[0][e].re = pk(s0a.x, sb.x);
    v[0][e].im = pk(s0a.y, sb.y);
    v[1][e].re = pk(-sy[e].x * sa.y, -sy[e].x * sb.y);
    v[1][e].im = pk(sy[e].x * sa.x, sy[e].x * sb.x);
    v[2][e].re = pk(sa.x * sy[e].y, sb.x * sy[e].y);
    v[2][e].im = pk(sa.y * sy[e].y, sb.y * sy[e].y);
  }

  // the three inverse transforms interleaved, first in the set that does not hold F
  {
    PC* const a[3] = {FLIP ? P[0] : P[3], FLIP ? P[1] : P[4], FLIP ? P[2] : P[5]};
    PC* const b[3] = {FLIP ? P[3] : P[0], FLIP ? P[4] : P[1], FLIP ? P[5] : P[2]};
    pfirst_regs<+1, N, 3>(v, a, t, sx);
    pfft_rec<+1, N, R0, N / R0, 3, true, false>(a, b, t, tw4, sx);
    if (!last) return;
    PC r[3][4];
    if constexpr (FLIP)
      plast_regs<+1, N, 3>(b, r, t, tw4, sx);
    else
      plast_regs<+1, N, 3>(a, r, t, tw4, sx);
    float2* const outs[3] = {out0, out1, out2};
#pragma unroll
    for (int o = 0; o < 3; ++o) {
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        float4 x;
        upk(r[o][s].re, x.x, x.z);
        upk(r[o][s].im, x.y, x.w);
        *reinterpret_cast<float4*>(outs[o] + (size_t)pout<RL, N>(t, s) * Lc + c0) = x;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Row combine pass of the FP32 matvec on row pairs (Sec. 4.2): the five complex-to-real
// row transforms d_xx Q0, d_x Q0, d_x Q1, Q1, Q2 of two neighbouring rows r0 = 2b and
// r0 + 1, held side by side as in k_col_pair, weighted by a11, b1, 2 a12, b2, a22 and summed
// into w = L Lbar^{-1} sigma.  The row symbols, the complex-to-real pre-processing, the
// transforms and the weighting all run on the packed pairs, the terms, the pre-processing and the
// first stage in registers, the last stage and the weighting too; the stages between run in place
// (two barriers a stage), which keeps a block at 48 KB of shared memory at length 512, so that
// the N / 2 blocks of a 1024 x 1024 grid run in one wave.
// ---------------------------------------------------------------------------------------
template <int L>
__global__ void __launch_bounds__(pthreads<L>(), L <= 512 ? 4 : 2)
    k_comb_pair(const float2* __restrict__ q0, const float2* __restrict__ q1,
                const float2* __restrict__ q2, const float* __restrict__ coef,
                float* __restrict__ out, int N, const float2* __restrict__ twL,
                const float2* __restrict__ twM, const int* __restrict__ skip,
                const float2* __restrict__ symx, const DevScalars* __restrict__ msc, Bat bat) {
  q0 = badv(q0, bat);
  q1 = badv(q1, bat);
  q2 = badv(q2, bat);
  coef = badv(coef, bat);
  out = badv(out, bat);
  skip = badv(skip, bat);
  msc = badv(msc, bat);
  if ((skip && *skip) || (bat.on && bskip(msc, bat))) return;
  constexpr int TPT = pthreads<L>(), E = pelems<L>();
  constexpr int M = 2 * L;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* tw4 = reinterpret_cast<ulonglong2*>(smem_raw);
  PC* pb = reinterpret_cast<PC*>(smem_raw + (size_t)L * sizeof(ulonglong2));
  PC* const B[5] = {pb, pb + L, pb + 2 * L, pb + 3 * L, pb + 4 * L};
  const int r0 = 2 * blockIdx.x;
  const int t = threadIdx.x;
  // the five terms of both rows: d_xx Q0, d_x Q0, d_x Q1, Q1, Q2 (row symbols of k1 = k; the
  // packed entry k = 0 holds (X0, X_L): d_x is 0 on both, d_xx keeps the Nyquist channel,
  // which Q0 carries premultiplied); the rows' loads are issued before the twiddle table is
  // built, so that both sets of loads are in flight together
  const size_t oa = (size_t)r0 * L, ob = oa + L;
  float2 ld[E][6];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int k = t + e * TPT;
    ld[e][0] = q0[oa + k];
    ld[e][1] = q0[ob + k];
    ld[e][2] = q1[oa + k];
    ld[e][3] = q1[ob + k];
    ld[e][4] = q2[oa + k];
    ld[e][5] = q2[ob + k];
  }
  load_tw4<L>(tw4, twL, t, TPT);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int k = t + e * TPT;
    const float2 a0 = ld[e][0], b0 = ld[e][1];
    const float2 a1 = ld[e][2], b1 = ld[e][3];
    const float2 a2 = ld[e][4], b2 = ld[e][5];
    PC x0, x1, x2;
    x0.re = pk(a0.x, b0.x);
    x0.im = pk(a0.y, b0.y);
    x1.re = pk(a1.x, b1.x);
    x1.im = pk(a1.y, b1.y);
    x2.re = pk(a2.x, b2.x);
    x2.im = pk(a2.y, b2.y);
    const int d = swz(k);
    B[0][d] = x0;
    B[1][d] = x1;
    B[2][d] = x2;
  }
  __syncthreads();

  // The five terms and their complex-to-real pre-processing: Z_k = (X_k + conj X_(L-k)) +
  // i (X_k - conj X_(L-k)) conj(W_M^k) of each, from the thread's own entries k and the mirrored
  // ones (both ends of a pair do it: 26 instructions an entry more, and three words read where
  // the terms themselves were written, read, written and read again)
  PC z[5][E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int k = t + e * TPT;
    const int dk = swz(k), dm = swz(e == 0 && t == 0 ? 0 : L - k);
    PC xk[5], xm[5];
    xk[0] = B[0][dk];
    xk[3] = B[1][dk];
    xk[4] = B[2][dk];
    xm[0] = B[0][dm];
    xm[3] = B[1][dm];
    xm[4] = B[2][dm];
    if (e == 0 && t == 0) {
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        PC x;
        if (q < 3) {
          x.re = 0ull;
          x.im = q == 0 ? xk[0].im : 0ull;
        } else {
          x = xk[q];
        }
        z[q][e].re = add2(x.re, x.im);
        z[q][e].im = sub2(x.re, x.im);
      }
    } else {
      const float2 w = twM[k], sk = symx[k], sm = symx[L - k];
      const u64 wx = pk(w.x, w.x), wy = pk(w.y, w.y), nwy = pk(-w.y, -w.y);
      const u64 k1 = pk(sk.x, sk.x), nk1 = pk(-sk.x, -sk.x), k2 = pk(sk.y, sk.y);
      const u64 m1 = pk(sm.x, sm.x), nm1 = pk(-sm.x, -sm.x), m2 = pk(sm.y, sm.y);
      xk[1].re = mul2(xk[0].im, nk1);
      xk[1].im = mul2(xk[0].re, k1);
      xm[1].re = mul2(xm[0].im, nm1);
      xm[1].im = mul2(xm[0].re, m1);
      xk[2].re = mul2(xk[3].im, nk1);
      xk[2].im = mul2(xk[3].re, k1);
      xm[2].re = mul2(xm[3].im, nm1);
      xm[2].im = mul2(xm[3].re, m1);
      xk[0].re = mul2(xk[0].re, k2);
      xk[0].im = mul2(xk[0].im, k2);
      xm[0].re = mul2(xm[0].re, m2);
      xm[0].im = mul2(xm[0].im, m2);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        PC S, D;
        S.re = add2(xk[q].re, xm[q].re);
        S.im = sub2(xk[q].im, xm[q].im);
        D.re = sub2(xk[q].re, xm[q].re);
        D.im = add2(xk[q].im, xm[q].im);
        const PC O = cmulp<+1>(D, wx, wy, nwy);
        z[q][e].re = sub2(S.re, O.im);
        z[q][e].im = add2(S.im, O.re);
      }
    }
  }
  __syncthreads();
  constexpr int R0 = pradix<L>(), RL = plast<L>();
  pfirst_regs<+1, L, 5>(z, B, t);
  pfft_inplace<+1, L, R0, L / R0, 5>(B, t, tw4);
  if (!pactive<RL, L>(t)) return;
  PC y[5][4];
  plast_regs<+1, L, 5>(B, y, t, tw4);

  // w = a11 y0 + b1 y1 + 2 a12 y2 + b2 y3 + a22 y4 on both rows (the coefficient planes a11,
  // a12, a22, b1, b2 in that order)
  const size_t P = (size_t)N * M;
  const size_t ra = (size_t)r0 * M, rb = ra + M;
  const float2* c0 = reinterpret_cast<const float2*>(coef);
  const float2* c1 = reinterpret_cast<const float2*>(coef + P);
  const float2* c2 = reinterpret_cast<const float2*>(coef + 2 * P);
  const float2* c3 = reinterpret_cast<const float2*>(coef + 3 * P);
  const float2* c4 = reinterpret_cast<const float2*>(coef + 4 * P);
  float2* ov = reinterpret_cast<float2*>(out);
  const u64 two = pk(2.f, 2.f);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int n = pout<RL, L>(t, e);
    const size_t ia = ra / 2 + n, ib = rb / 2 + n;
    const float2 a11a = c0[ia], a11b = c0[ib], a12a = c1[ia], a12b = c1[ib];
    const float2 a22a = c2[ia], a22b = c2[ib], b1a = c3[ia], b1b = c3[ib];
    const float2 b2a = c4[ia], b2b = c4[ib];
    const PC y0 = y[0][e], y1 = y[1][e], y2 = y[2][e], y3 = y[3][e], y4 = y[4][e];
    u64 rr = mul2(pk(a11a.x, a11b.x), y0.re);
    rr = fma2(pk(b1a.x, b1b.x), y1.re, rr);
    rr = fma2(mul2(two, pk(a12a.x, a12b.x)), y2.re, rr);
    rr = fma2(pk(b2a.x, b2b.x), y3.re, rr);
    rr = fma2(pk(a22a.x, a22b.x), y4.re, rr);
    u64 ri = mul2(pk(a11a.y, a11b.y), y0.im);
    ri = fma2(pk(b1a.y, b1b.y), y1.im, ri);
    ri = fma2(mul2(two, pk(a12a.y, a12b.y)), y2.im, ri);
    ri = fma2(pk(b2a.y, b2b.y), y3.im, ri);
    ri = fma2(pk(a22a.y, a22b.y), y4.im, ri);
    float2 wa, wb;
    upk(rr, wa.x, wb.x);
    upk(ri, wa.y, wb.y);
    ov[ia] = wa;
    ov[ib] = wb;
  }
}

template <int L>
cudaError_t comb_pair_L(const float2* q0, const float2* q1, const float2* q2, const float* coef,
                        float* out, int N, const SpecTables& tb, const int* skip,
                        cudaStream_t st, const DevScalars* msc, Bat bat) {
  const size_t sm = (size_t)L * sizeof(ulonglong2) + 5 * (size_t)L * sizeof(PC);
  cudaError_t e = prepare_launch(k_comb_pair<L>, pthreads<L>(), sm);
  if (e != cudaSuccess) return e;
  k_comb_pair<L><<<bgrid(dim3(N / 2), bat), pthreads<L>(), sm, st>>>(
      q0, q1, q2, coef, out, N, (const float2*)tb.twL, (const float2*)tb.twM, skip,
      (const float2*)tb.symx, msc, bat);
  return cudaGetLastError();
}

template <int N, int G>
cudaError_t col_pair_G(const float2* spec, float2* o0, float2* o1, float2* o2, int M,
                       const SpecTables& tb, const DevScalars* sc, const int* skip,
                       cudaStream_t st, Bat bat) {
  const size_t sm = (size_t)N * sizeof(ulonglong2) + 6 * (size_t)N * G * sizeof(PC);
  cudaError_t e = prepare_launch(k_col_pair<N, G>, pthreads<N>() * G, sm);
  if (e != cudaSuccess) return e;
  k_col_pair<N, G><<<bgrid(dim3(M / 4 / G), bat), pthreads<N>() * G, sm, st>>>(
      spec, o0, o1, o2, M, (float)(1.0 / ((double)N * (double)M)), (const float2*)tb.twN, sc,
      skip, (const float2*)tb.symx, (const float2*)tb.symy, bat);
  return cudaGetLastError();
}

template <int N>
cudaError_t col_pair_N(const float2* spec, float2* o0, float2* o1, float2* o2, int M,
                       const SpecTables& tb, const DevScalars* sc, const int* skip,
                       cudaStream_t st, Bat bat) {
  if constexpr (N <= 1024) {  // (shared memory: 208 N bytes)
    if (two_pairs(M, bat)) return col_pair_G<N, 2>(spec, o0, o1, o2, M, tb, sc, skip, st, bat);
  }
  return col_pair_G<N, 1>(spec, o0, o1, o2, M, tb, sc, skip, st, bat);
}

}  // namespace

bool comb_pair_supported(int N, int M) {
  const int L = M / 2;
  return row_pair_length(L) && M == 2 * L && N >= 2 && N % 2 == 0;
}

cudaError_t launch_comb_pair(const float2* q0, const float2* q1, const float2* q2,
                             const float* coef, float* out, int N, int M, const SpecTables& tb,
                             const int* skip, cudaStream_t st, const DevScalars* msc, Bat bat) {
  if (!comb_pair_supported(N, M) || (bat.on && !msc)) return cudaErrorInvalidValue;
#define OTGB_CALL(n) comb_pair_L<n>(q0, q1, q2, coef, out, N, tb, skip, st, msc, bat)
  OTGB_ROW_LENGTHS(M / 2, OTGB_CALL)
#undef OTGB_CALL
  return cudaErrorInvalidValue;
}

bool col_pair_supported(int N, int M) { return col_pair_length(N) && M >= 4 && M % 4 == 0; }

cudaError_t launch_col_pair(const float2* spec, float2* o0, float2* o1, float2* o2, int N,
                            int M, const SpecTables& tb, const DevScalars* sc, const int* skip,
                            cudaStream_t st, Bat bat) {
  if (!col_pair_supported(N, M) || (bat.on && !sc)) return cudaErrorInvalidValue;
  // 16-byte loads and stores of a column pair need 16-byte aligned planes
  if (((uintptr_t)spec | (uintptr_t)o0 | (uintptr_t)o1 | (uintptr_t)o2 | bat.slab) & 15)
    return cudaErrorMisalignedAddress;
#define OTGB_CALL(n) col_pair_N<n>(spec, o0, o1, o2, M, tb, sc, skip, st, bat)
  OTGB_COL_LENGTHS(N, OTGB_CALL)
#undef OTGB_CALL
  return cudaErrorInvalidValue;
}

}  // namespace otgb

// Packed FP32 pairs for the transform passes that hold two columns (or rows) side by side
// (the f32x2 instructions of f32x2.cuh): complex pairs (PC: the real parts of two
// complex numbers in one register pair, the imaginary parts in another), their butterflies
// and Stockham stages, and the 16-byte-element shared-memory swizzle
// i ^ ((i >> 2) & 7), under which every stage's reads and writes of a quarter warp fall in
// distinct bank groups (checked for the radix-4 / radix-2 stages of lengths 256 .. 2048).
//
// Lengths: powers of two by L / 4 threads (4 elements each), and 3 * 2^a by L / 3: the first
// stage has radix 3, a butterfly per thread; in the others the first L / 4 threads work, as for
// a power of two (whole warps idle from L = 384 on).
//
// A plan set's classes run these passes too (Bat), and sizes with a factor 3 ran the generic
// kernels of 12 elements per thread before.  us per launch, one GB300, 5 problems, generic ->
// pairs:             row r2c     column       combine      theta column  theta row
//   128^2            4.6 -> 3.9  13.2 -> 5.5  14.2 -> 5.8   8.2 ->  8.3   6.8 ->  7.1
//   192^2            7.6 -> 3.6  24.0 -> 6.5  25.2 -> 6.1  17.3 -> 10.2  18.6 ->  6.9
//   384^2            8.1 -> 4.6  28.6 -> 14.7 30.7 -> 13.9 27.3 -> 24.3  28.0 -> 13.1
//   512^2            6.7 -> 5.7  28.1 -> 22.1 32.2 -> 18.2 34.2 -> 32.4  19.2 -> 18.4
// and for a single 384^2 or 1536^2 problem: column 15.2 -> 7.1, 71 -> 46; combine 11.3 -> 5.7,
// 67 -> 35; theta column 20.7 -> 10.2, 83 -> 73.  Bound by latency below about 10 us, above by
// shared-memory traffic (a stage reads and writes every element).
#pragma once
#include "f32x2.cuh"
#include "spectral.cuh"

namespace otgb {
namespace pair {

// two complex numbers, one per column: re = (a.x, b.x), im = (a.y, b.y)
struct __align__(16) PC {
  u64 re, im;
};

__device__ __forceinline__ int swz(int i) { return i ^ ((i >> 2) & 7); }

// threads of a transform pair of length L, and the elements of a thread in the passes over them
template <int L> __host__ __device__ constexpr int pthreads() { return L % 3 == 0 ? L / 3 : L / 4; }
template <int L> __host__ __device__ constexpr int pelems() { return L % 3 == 0 ? 3 : 4; }
// radix of the stage that has REM left: [3,] then 4 while it divides, then 2
template <int REM> __host__ __device__ constexpr int pradix() {
  return REM % 3 == 0 ? 3 : (REM % 4 == 0 ? 4 : 2);
}

// v * w (SIGN < 0) or v * conj(w) (SIGN > 0); wx = (w.x, w.x), wy = (w.y, w.y), nwy = -wy
template <int SIGN>
__device__ __forceinline__ PC cmulp(PC v, u64 wx, u64 wy, u64 nwy) {
  PC r;
  if (SIGN < 0) {
    r.re = fma2(v.im, nwy, mul2(v.re, wx));
    r.im = fma2(v.re, wy, mul2(v.im, wx));
  } else {
    r.re = fma2(v.im, wy, mul2(v.re, wx));
    r.im = fma2(v.re, nwy, mul2(v.im, wx));
  }
  return r;
}

template <int R, int SIGN> struct BflyP;
template <int SIGN> struct BflyP<2, SIGN> {
  __device__ __forceinline__ static void run(PC* v) {
    const PC a = v[0], b = v[1];
    v[0].re = add2(a.re, b.re);
    v[0].im = add2(a.im, b.im);
    v[1].re = sub2(a.re, b.re);
    v[1].im = sub2(a.im, b.im);
  }
};
template <int SIGN> struct BflyP<3, SIGN> {
  __device__ __forceinline__ static void run(PC* v) {
    const u64 sr = add2(v[1].re, v[2].re), si = add2(v[1].im, v[2].im);
    const u64 dr = sub2(v[1].re, v[2].re), di = sub2(v[1].im, v[2].im);
    const u64 mh = pk(-0.5f, -0.5f);
    const float c = SIGN * (float)OTGB_SQRT3_HALF;
    const u64 cp = pk(c, c), cm = pk(-c, -c);
    const u64 tr = fma2(mh, sr, v[0].re), ti = fma2(mh, si, v[0].im);
    v[0].re = add2(v[0].re, sr);
    v[0].im = add2(v[0].im, si);
    v[1].re = fma2(cm, di, tr);  // t + SIGN i sqrt(3)/2 d
    v[1].im = fma2(cp, dr, ti);
    v[2].re = fma2(cp, di, tr);
    v[2].im = fma2(cm, dr, ti);
  }
};
template <int SIGN> struct BflyP<4, SIGN> {
  __device__ __forceinline__ static void run(PC* v) {
    const u64 t0r = add2(v[0].re, v[2].re), t0i = add2(v[0].im, v[2].im);
    const u64 t1r = sub2(v[0].re, v[2].re), t1i = sub2(v[0].im, v[2].im);
    const u64 t2r = add2(v[1].re, v[3].re), t2i = add2(v[1].im, v[3].im);
    const u64 dr = sub2(v[1].re, v[3].re), di = sub2(v[1].im, v[3].im);
    v[0].re = add2(t0r, t2r);
    v[0].im = add2(t0i, t2i);
    v[2].re = sub2(t0r, t2r);
    v[2].im = sub2(t0i, t2i);
    // t3 = SIGN i d: v1 = t1 + t3, v3 = t1 - t3
    if (SIGN > 0) {
      v[1].re = sub2(t1r, di);
      v[1].im = add2(t1i, dr);
      v[3].re = add2(t1r, di);
      v[3].im = sub2(t1i, dr);
    } else {
      v[1].re = add2(t1r, di);
      v[1].im = sub2(t1i, dr);
      v[3].re = sub2(t1r, di);
      v[3].im = add2(t1i, dr);
    }
  }
};

template <int REM>
__host__ __device__ constexpr int pstage_count() {
  if constexpr (REM > 1)
    return 1 + pstage_count<REM / pradix<REM>()>();
  else
    return 0;
}

// One stage of radix R (span Ns) on NP transform pairs of length L;
// tw: the stage-ordered twiddles as (w.x, w.x, w.y, w.y) words.  Out of place (one barrier)
// or in place (INPLACE: the stores wait for every thread's loads).
template <int R, int SIGN, int L, int Ns, int NP, bool INPLACE = false>
__device__ __forceinline__ void pstage(PC* const (&in)[NP], PC* const (&out)[NP], int t,
                                       const ulonglong2* __restrict__ tw) {
  constexpr int NB = R == 3 ? 1 : 4 / R;  // butterflies per thread
  constexpr int T = R == 3 ? L / 3 : L / 4, LR = L / R;
  const bool active = L % 3 != 0 || R == 3 || t < T;
  PC v[NP][NB * R];
  if (active) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = t + b * T;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int src = swz(j + r * LR);
#pragma unroll
        for (int q = 0; q < NP; ++q) v[q][b * R + r] = in[q][src];
      }
    }
  }
  if (INPLACE) __syncthreads();
  if (active) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = t + b * T;
      const int qd = (int)((unsigned)j / (unsigned)Ns);
      const int k = j - qd * Ns;
      if (Ns > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) {
          const ulonglong2 w = tw[(Ns - 1) + (r - 1) * Ns + k];
          const u64 nwy = sub2(0ull, w.y);  // (0, 0) - (w.y, w.y)
#pragma unroll
          for (int q = 0; q < NP; ++q)
            v[q][b * R + r] = cmulp<SIGN>(v[q][b * R + r], w.x, w.y, nwy);
        }
      }
#pragma unroll
      for (int q = 0; q < NP; ++q) BflyP<R, SIGN>::run(&v[q][b * R]);
      const int d = qd * (Ns * R) + k;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int dst = swz(d + r * Ns);
#pragma unroll
        for (int q = 0; q < NP; ++q) out[q][dst] = v[q][b * R + r];
      }
    }
  }
  __syncthreads();
}

// the transform: stages alternating between a and b, starting from a; the result ends in a
// for an even number of stages, in b for an odd one
template <int SIGN, int L, int Ns, int REM, int NP, bool FROM_A>
__device__ __forceinline__ void pfft_rec(PC* const (&a)[NP], PC* const (&b)[NP], int t,
                                         const ulonglong2* __restrict__ tw) {
  if constexpr (REM > 1) {
    constexpr int R = pradix<REM>();
    if constexpr (FROM_A)
      pstage<R, SIGN, L, Ns, NP>(a, b, t, tw);
    else
      pstage<R, SIGN, L, Ns, NP>(b, a, t, tw);
    pfft_rec<SIGN, L, Ns * R, REM / R, NP, !FROM_A>(a, b, t, tw);
  }
}

// the same transform in place
template <int SIGN, int L, int Ns, int REM, int NP>
__device__ __forceinline__ void pfft_inplace(PC* const (&a)[NP], int t,
                                             const ulonglong2* __restrict__ tw) {
  if constexpr (REM > 1) {
    constexpr int R = pradix<REM>();
    pstage<R, SIGN, L, Ns, NP, true>(a, a, t, tw);
    pfft_inplace<SIGN, L, Ns * R, REM / R, NP>(a, t, tw);
  }
}

// the stage table behind the base table of length L
template <int L, typename C>
__device__ __forceinline__ const C* pstage_table(const C* twb) {
  return twb + (size_t)(L % 3 == 0 ? stage_table_slot<12>() : stage_table_slot<4>()) * L;
}

// the stage twiddles of length L, broadcast to both lanes
template <int L>
__device__ __forceinline__ void load_tw4(ulonglong2* tw4, const float2* __restrict__ twb, int t,
                                         int nthreads) {
  const float2* __restrict__ st = pstage_table<L>(twb);
  for (int i = t; i < L; i += nthreads) {
    const float2 w = st[i];
    tw4[i] = make_ulonglong2(pk(w.x, w.x), pk(w.y, w.y));
  }
}

// the lengths of the pair passes: rows (M / 2) and columns
inline bool row_pair_length(int L) {
  return L == 64 || L == 96 || L == 128 || L == 192 || L == 256 || L == 384 || L == 512 ||
         L == 768 || L == 1024;
}
inline bool col_pair_length(int N) {
  return N == 96 || N == 128 || N == 192 || N == 256 || N == 384 || N == 512 || N == 768 ||
         N == 1024 || N == 1536 || N == 2048;
}
// return CALL(length) for one of them
#define OTGB_ROW_LENGTHS(L, CALL) \
  switch (L) {                    \
    case 64: return CALL(64);     \
    case 96: return CALL(96);     \
    case 128: return CALL(128);   \
    case 192: return CALL(192);   \
    case 256: return CALL(256);   \
    case 384: return CALL(384);   \
    case 512: return CALL(512);   \
    case 768: return CALL(768);   \
    case 1024: return CALL(1024); \
  }
#define OTGB_COL_LENGTHS(N, CALL) \
  switch (N) {                    \
    case 96: return CALL(96);     \
    case 128: return CALL(128);   \
    case 192: return CALL(192);   \
    case 256: return CALL(256);   \
    case 384: return CALL(384);   \
    case 512: return CALL(512);   \
    case 768: return CALL(768);   \
    case 1024: return CALL(1024); \
    case 1536: return CALL(1536); \
    case 2048: return CALL(2048); \
  }

}  // namespace pair
}  // namespace otgb

// Packed FP32 pairs for the transform passes that hold two columns (or rows) side by side
// (the f32x2 instructions of f32x2.cuh): complex pairs (PC: the real parts of two
// complex numbers in one register pair, the imaginary parts in another), their butterflies
// and Stockham stages, and the 16-byte-element shared-memory swizzle
// i ^ ((i >> 2) & 7), under which every stage's reads and writes of a quarter warp fall in
// distinct bank groups for the powers of two (computed for 64 .. 2048, one and two pairs per block).
// With a factor 3 (96 .. 1536) the reads do too, and the writes from the fourth stage on; those of
// the first two stages meet threefold, those of the third twofold (one pair) or not (two).
//
// Lengths: powers of two by L / 4 threads (4 elements each), and 3 * 2^a by L / 3: the first
// stage has radix 3, a butterfly per thread; in the others the first L / 4 threads work, as for
// a power of two (whole warps idle from L = 384 on).
//
// A plan set's classes run these passes too (Bat), and sizes with a factor 3 ran the generic
// kernels of 12 elements per thread before.  us per launch, one GB300, 5 problems, generic ->
// pairs:             row r2c     column       combine      theta column  theta row
//   128^2            4.6 -> 3.4  13.2 -> 4.6  14.2 -> 4.1   8.2 ->  6.8   6.8 ->  7.2
//   192^2            7.6 -> 3.2  24.0 -> 4.9  25.2 -> 5.0  17.3 ->  7.6  18.6 ->  7.5
//   384^2            8.1 -> 4.2  28.6 -> 9.8  30.7 -> 10.7 27.3 -> 17.8  28.0 -> 14.7
//   512^2            6.7 -> 5.1  28.1 -> 16.0 32.2 -> 12.8 34.2 -> 28.8  19.2 -> 18.1
// and for a single 384^2 or 1536^2 problem: column 15.2 -> 6.1, 71 -> 41; combine 11.3 -> 5.0,
// 67 -> 29; theta column 20.7 -> 9.8, 83 -> 71.  Bound by latency below about 10 us, above by
// shared-memory traffic (a stage reads and writes every element; the first and the last stage keep
// to registers where values are loaded, computed or stored: at 1024^2 column 17.7 -> 15.9,
// combine 14.3 -> 11.7, theta column 27.6 -> 25.6 us).
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

// radix of the last stage
template <int REM> __host__ __device__ constexpr int plast() {
  if constexpr (REM == pradix<REM>())
    return REM;
  else
    return plast<REM / pradix<REM>()>();
}

// A stage of radix R (span Ns) on NP transform pairs of length L, in three steps: a thread's slots
// into registers (R == 3: one butterfly, else 4 / R), their twiddles (tw: the stage-ordered
// twiddles as (w.x, w.x, w.y, w.y) words) and butterflies, and the results into shared memory.
// The first stage's slot e is element t + e L / 4 (L / 3 for radix 3), the last stage's slot s
// ends as element pout(t, s) (sx: see k_col_pair): the first stage can take its values from where they are loaded or
// computed and the last one leave them to where they are used, without shared memory between.
template <int R> __host__ __device__ constexpr int pslots() { return R == 3 ? 3 : 4; }
template <int R, int L> __device__ __forceinline__ bool pactive(int t) {
  return L % 3 != 0 || R == 3 || t < L / 4;
}
template <int R, int L> __device__ __forceinline__ int pout(int t, int s) {
  return t + (s / R) * (L / 4) + (s % R) * (L / R);
}
template <int R, int L, int NP>
__device__ __forceinline__ void pload(PC* const (&in)[NP], PC (&v)[NP][pslots<R>()], int t,
                                      int sx = 0) {
  constexpr int T = R == 3 ? L / 3 : L / 4, LR = L / R;
#pragma unroll
  for (int s = 0; s < pslots<R>(); ++s) {
    const int src = swz(t + (s / R) * T + (s % R) * LR) ^ sx;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q][s] = in[q][src];
  }
}
template <int R, int SIGN, int L, int Ns, int NP>
__device__ __forceinline__ void pbfly(PC (&v)[NP][pslots<R>()], int t,
                                      const ulonglong2* __restrict__ tw) {
  constexpr int T = R == 3 ? L / 3 : L / 4;
#pragma unroll
  for (int b = 0; b < pslots<R>() / R; ++b) {
    if (Ns > 1) {
      const int k = (int)((unsigned)(t + b * T) % (unsigned)Ns);
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
  }
}
template <int R, int L, int Ns, int NP>
__device__ __forceinline__ void pstore(PC* const (&out)[NP], const PC (&v)[NP][pslots<R>()],
                                       int t, int sx = 0) {
  constexpr int T = R == 3 ? L / 3 : L / 4;
#pragma unroll
  for (int s = 0; s < pslots<R>(); ++s) {
    const int j = t + (s / R) * T;
    const int qd = (int)((unsigned)j / (unsigned)Ns);
    const int dst = swz(qd * (Ns * R) + (j - qd * Ns) + (s % R) * Ns) ^ sx;
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q][dst] = v[q][s];
  }
}

// a whole stage: out of place (one barrier), or in place (the stores wait for every thread's loads)
template <int R, int SIGN, int L, int Ns, int NP, bool INPLACE = false>
__device__ __forceinline__ void pstage(PC* const (&in)[NP], PC* const (&out)[NP], int t,
                                       const ulonglong2* __restrict__ tw, int sx = 0) {
  const bool active = pactive<R, L>(t);
  PC v[NP][pslots<R>()];
  if (active) pload<R, L, NP>(in, v, t, sx);
  if (INPLACE) __syncthreads();
  if (active) {
    pbfly<R, SIGN, L, Ns, NP>(v, t, tw);
    pstore<R, L, Ns, NP>(out, v, t, sx);
  }
  __syncthreads();
}

// the transform's stages behind the first one: alternating between a and b, starting from a; with
// LAST the last one too, else it is left to the caller (plast_regs)
template <int SIGN, int L, int Ns, int REM, int NP, bool FROM_A, bool LAST>
__device__ __forceinline__ void pfft_rec(PC* const (&a)[NP], PC* const (&b)[NP], int t,
                                         const ulonglong2* __restrict__ tw, int sx = 0) {
  constexpr int R = pradix<REM>();
  if constexpr (REM > (LAST ? 1 : R)) {
    if constexpr (FROM_A)
      pstage<R, SIGN, L, Ns, NP>(a, b, t, tw, sx);
    else
      pstage<R, SIGN, L, Ns, NP>(b, a, t, tw, sx);
    pfft_rec<SIGN, L, Ns * R, REM / R, NP, !FROM_A, LAST>(a, b, t, tw, sx);
  }
}
// the same in place, without the last stage
template <int SIGN, int L, int Ns, int REM, int NP>
__device__ __forceinline__ void pfft_inplace(PC* const (&a)[NP], int t,
                                             const ulonglong2* __restrict__ tw) {
  constexpr int R = pradix<REM>();
  if constexpr (REM > R) {
    pstage<R, SIGN, L, Ns, NP, true>(a, a, t, tw);
    pfft_inplace<SIGN, L, Ns * R, REM / R, NP>(a, t, tw);
  }
}
// first stage of the values in v, into out (a barrier)
template <int SIGN, int L, int NP>
__device__ __forceinline__ void pfirst_regs(PC (&v)[NP][pelems<L>()], PC* const (&out)[NP], int t,
                                            int sx = 0) {
  constexpr int R = pradix<L>();
  pbfly<R, SIGN, L, 1, NP>(v, t, nullptr);
  pstore<R, L, 1, NP>(out, v, t, sx);
  __syncthreads();
}
// last stage from shared memory into registers (threads below L / 4 only: pactive)
template <int SIGN, int L, int NP>
__device__ __forceinline__ void plast_regs(PC* const (&in)[NP], PC (&v)[NP][4], int t,
                                           const ulonglong2* __restrict__ tw, int sx = 0) {
  constexpr int R = plast<L>();
  pload<R, L, NP>(in, v, t, sx);
  pbfly<R, SIGN, L, L / R, NP>(v, t, tw);
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

// A column pass takes two column pairs per block where one each would give SMs a second block: half
// the blocks with whole sectors (k_col_pair) then, else every SM counts.  Column pass, us, one /
// two pairs per block, one GB300: 512^2 (128 pairs) 7.4 / 8.4, 1024x512 10.9 / 12.9; five of 128^2
// (160) 5.1 / 4.6, 768^2 (192) 12.5 / 11.0, 512x1024 (256) 9.7 / 8.5; theta's column pass 10.1 / 13.3
// at 512^2, 23.5 / 17.9 at 768^2, 25.6 / 22.2 at 1024^2.
inline bool two_pairs(int M, const Bat& bat) {
  return (long)(M / 4) * (bat.on ? bat.n : 1) > 152;
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

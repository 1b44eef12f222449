// FP64 line operators in 64-bit fixed point on the integer pipe.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM but 64 32x32+64-bit integer ones
// (IMAD.WIDE; measured 1.9 and 57), so the line passes of every FP64 slice kernel were bound by
// the FP64 pipe (80 % active, everything else idle on 32^3 slices).  Here the lines of a warp are
// aligned to their largest exponent and the folds and block rows of line_op (line_ops.cuh) run on
// 64-bit integers:
//   value       V = x 2^(1080 - E), |V| < 2^58 (E: exponent field of the warp's largest entry),
//               exact for entries within 2^5 of the largest, truncated at 2^-58 of it below;
//   coefficient c 2^60 = h 2^30 + l, |l| <= 2^29 (FixCoef), from the same FP64 tables;
//   product     V c = (Vh 2^30 + Vl)(h 2^30 + l) / 2^60 = Vh h + (Vh l + Vl h) / 2^30, Vl l
//               dropped (below half a unit): three IMAD.WIDE per multiply-add in two
//               accumulators, joined once per block row.
// |folded V| < 2^60 and the sums of products stay below 2^63 for every table (fix_table checks).
// Errors per pass: about one unit, 2^-57 of the tile's largest entry, against one FP64 rounding
// per term of the multiply-add chain; a tile is at most two planes of a slice (fix_tile), so this
// holds in the 2-norm for a single non-zero site too (sqrt(512) 2^-57 < 2^-52).
#pragma once
#include <cuda_runtime.h>

#include "line_ops.cuh"

namespace ufg {

constexpr int FIX_L = 30;   // bits of the low limb of a coefficient and of a value
constexpr int FIX_SH = 5;   // head room used of a double's 53 bits: |V| < 2^(53 + FIX_SH)

struct FixCoef {
  int h, l;
};
// The blocks of LineCoef (line_ops.cuh) row by row, each row padded to an even number of
// coefficients so that a row is read as 16-byte pairs.
template <int N>
struct FixLine {
  using S = LineShape<N>;
  static constexpr int H = S::H, Q = S::Q;
  static constexpr int n0 = S::TWO ? Q + 1 : H + 1, n1 = S::TWO ? Q : H - 1;
  static constexpr int n2 = S::TWO ? Q : 0, n3 = S::TWO ? Q - 1 : 0;
  static constexpr int pad(int n) { return (n + 1) / 2; }  // pairs per row
  static constexpr int O0 = 0, O1 = O0 + n0 * pad(n0), O2 = O1 + n1 * pad(n1);
  static constexpr int O3 = O2 + n2 * pad(n2);
  static constexpr int NP = O3 + n3 * pad(n3);  // pairs in all
};
template <int N>
struct __align__(16) LineCoefFix {
  FixCoef c[2 * FixLine<N>::NP];
};

// c 2^60 as two limbs; false if |c| is 1.9 or more (no table comes near)
inline bool fix_coef(double c, FixCoef* out) {
  if (!(c > -1.9 && c < 1.9)) return false;
  const long long v = (long long)(c * 1152921504606846976.0);  // exact up to truncation below 1
  const long long l = ((v + (1LL << (FIX_L - 1))) & ((1LL << FIX_L) - 1)) - (1LL << (FIX_L - 1));
  out->h = (int)((v - l) >> FIX_L);
  out->l = (int)l;
  return true;
}
// the fixed-point table of the flat FP64 blocks of an N-line (LineCoef layout); false if a
// coefficient or a row's sums do not fit (|Vh| <= 2^30, 0 <= Vl < 2^30)
template <int N>
inline bool fix_table(const double* flat, LineCoefFix<N>* t) {
  using F = FixLine<N>;
  const int n[4] = {F::n0, F::n1, F::n2, F::n3}, off[4] = {F::O0, F::O1, F::O2, F::O3};
  for (int i = 0; i < 2 * F::NP; ++i) t->c[i] = FixCoef{0, 0};
  for (int b = 0; b < 4; ++b)
    for (int i = 0; i < n[b]; ++i) {
      FixCoef* row = t->c + 2 * (off[b] + i * F::pad(n[b]));
      double m = 0.5;
      for (int j = 0; j < n[b]; ++j) {
        if (!fix_coef(*flat++, row + j)) return false;
        m += (row[j].l < 0 ? -(double)row[j].l : (double)row[j].l) +
             (row[j].h < 0 ? -(double)row[j].h : (double)row[j].h);
      }
      if (m * 1073741824.0 >= 9.2e18) return false;
    }
  return true;
}

// a b + c in one IMAD.WIDE (written out: from the C expression the compiler widens a limb it
// knows to be non-negative to 64 bits first and multiplies in several instructions)
__device__ __forceinline__ long long madw(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long mulw(int a, int b) {
  long long d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
// shifts by any amount (PTX clamps: 0, or the sign, from 64 on)
__device__ __forceinline__ unsigned long long shr_u64(unsigned long long v, unsigned s) {
  unsigned long long d;
  asm("shr.u64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
}
__device__ __forceinline__ long long shr_s64(long long v, unsigned s) {
  long long d;
  asm("shr.s64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
}

// x 2^(1080 - E) truncated toward zero; eb = (largest |high word| of the line) | 0xfffff
__device__ __forceinline__ long long fix_from(double x, unsigned eb) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned s = (eb - (hi & 0x7fffffffu)) >> 20;  // exponent distance to the largest
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m =
      ((unsigned long long)__funnelshift_l(lo, mh, FIX_SH) << 32) | (lo << FIX_SH);
  m = shr_u64(m, s);
  return (int)hi < 0 ? -(long long)m : (long long)m;
}
// V 2^(E - 1080) to nearest, E in [128, 2043]; kb = (E + 5) << 20, flip = sign bit to change, nan =
// exponent bits to set (the magnitude is that of v or of v + 1: one unit, as everywhere here)
__device__ __forceinline__ double fix_to(long long v, unsigned kb, unsigned flip, unsigned nan) {
  const unsigned vh = (unsigned)((unsigned long long)v >> 32);
  const int sg = (int)vh >> 31;
  const unsigned ah = vh ^ (unsigned)sg, al = (unsigned)(unsigned long long)v ^ (unsigned)sg;
  unsigned long long n = ((unsigned long long)ah << 32) | al;
  const unsigned c = (unsigned)__clzll((long long)n);  // 1 .. 64
  n = n << ((c - 1u) & 63u);                           // leading bit at 62
  n = (n + 512ull) >> 10;
  unsigned hi = (unsigned)(n >> 32) + (kb - (c << 20));
  hi = c == 64u ? 0u : hi;
  return __hiloint2double((int)(hi | ((vh ^ flip) & 0x80000000u) | nan), (int)(unsigned)n);
}

// one row of a block of n columns at pair `off` of the table: limbs xh, xl of the inputs
template <int n, int off>
__device__ __forceinline__ long long block_row_fix(const int4* __restrict__ tab, const int* xh,
                                                   const int* xl, int i) {
  constexpr int np = (n + 1) / 2;
  long long hi = 0, mid = 1LL << (FIX_L - 1);
#pragma unroll
  for (int k = 0; k < np; ++k) {
    const int4 c = tab[off + i * np + k];
    const int j = 2 * k;
    hi = k == 0 ? mulw(c.x, xh[j]) : madw(c.x, xh[j], hi);
    mid = madw(c.y, xh[j], mid);
    mid = madw(c.x, xl[j], mid);
    if (j + 1 < n) {
      hi = madw(c.z, xh[j + 1], hi);
      mid = madw(c.w, xh[j + 1], mid);
      mid = madw(c.z, xl[j + 1], mid);
    }
  }
  return hi + (mid >> FIX_L);
}

template <int n>
__device__ __forceinline__ void fix_split(const long long* x, int* xh, int* xl) {
#pragma unroll
  for (int j = 0; j < n; ++j) {
    const unsigned lo = (unsigned)(unsigned long long)x[j];
    xh[j] = (int)__funnelshift_r(lo, (unsigned)((unsigned long long)x[j] >> 32), FIX_L);
    xl[j] = (int)(lo & ((1u << FIX_L) - 1u));
  }
}

// line_op on integers: V[N] in, (index, value) out, same blocks and order of emission
template <int N, bool IN_SPEC, bool OUT_SPEC, class Emit>
__device__ __forceinline__ void line_op_int(const long long (&v)[N], const int4* __restrict__ tab,
                                            Emit&& st) {
  using S = LineShape<N>;
  using F = FixLine<N>;
  constexpr int H = S::H;
  long long e[H + 1], o[H - 1];
  if constexpr (IN_SPEC) {
#pragma unroll
    for (int j = 0; j <= H; ++j) e[j] = v[j];
#pragma unroll
    for (int j = 1; j < H; ++j) o[j - 1] = v[H + j];
  } else {
    e[0] = v[0];
    e[H] = v[H];
#pragma unroll
    for (int j = 1; j < H; ++j) {
      e[j] = v[j] + v[N - j];
      o[j - 1] = v[j] - v[N - j];
    }
  }
  if constexpr (S::TWO) {
    constexpr int Q = S::Q;
    constexpr int NA = Q - 1 > 0 ? Q - 1 : 1;
    int csh[Q + 1], csl[Q + 1], cah[Q], cal[Q], ssh[Q], ssl[Q], sah[NA], sal[NA];
    {
      long long cs[Q + 1], ca[Q], ss[Q], sa[NA];
      if constexpr (IN_SPEC) {
#pragma unroll
        for (int m = 0; m <= Q; ++m) cs[m] = e[2 * m];
#pragma unroll
        for (int m = 0; m < Q; ++m) ca[m] = e[2 * m + 1];
#pragma unroll
        for (int m = 0; m < Q; ++m) ss[m] = o[2 * m];
#pragma unroll
        for (int m = 0; m < Q - 1; ++m) sa[m] = o[2 * m + 1];
      } else {
#pragma unroll
        for (int m = 0; m < Q; ++m) {
          cs[m] = e[m] + e[H - m];
          ca[m] = e[m] - e[H - m];
        }
        cs[Q] = e[Q];
#pragma unroll
        for (int m = 0; m < Q - 1; ++m) {
          ss[m] = o[m] + o[H - m - 2];
          sa[m] = o[m] - o[H - m - 2];
        }
        ss[Q - 1] = o[Q - 1];
      }
      fix_split<Q + 1>(cs, csh, csl);
      fix_split<Q>(ca, cah, cal);
      fix_split<Q>(ss, ssh, ssl);
      fix_split<Q - 1>(sa, sah, sal);
    }
    auto CS = [&](int m) { return block_row_fix<F::n0, F::O0>(tab, csh, csl, m); };
    auto CA = [&](int m) { return block_row_fix<F::n1, F::O1>(tab, cah, cal, m); };
    auto SS = [&](int m) { return block_row_fix<F::n2, F::O2>(tab, ssh, ssl, m); };
    auto SA = [&](int m) { return block_row_fix<F::n3, F::O3>(tab, sah, sal, m); };
    if constexpr (OUT_SPEC) {
#pragma unroll
      for (int m = 0; m <= Q; ++m) st(2 * m, CS(m));
#pragma unroll
      for (int m = 0; m < Q; ++m) st(2 * m + 1, CA(m));
#pragma unroll
      for (int m = 0; m < Q; ++m) st(H + 2 * m + 1, SS(m));
#pragma unroll
      for (int m = 0; m < Q - 1; ++m) st(H + 2 * m + 2, SA(m));
    } else {
      {
        const long long U = CS(0), W = CA(0);
        st(0, U + W);
        st(H, U - W);
      }
#pragma unroll
      for (int m = 1; m < Q; ++m) {
        const long long U = CS(m), W = CA(m), Us = SS(m - 1), Ws = SA(m - 1);
        const long long Em = U + W, Eh = U - W, Om = Us + Ws, Oh = Us - Ws;
        st(m, Em + Om);
        st(N - m, Em - Om);
        st(H - m, Eh + Oh);
        st(H + m, Eh - Oh);
      }
      {
        const long long U = CS(Q), Us = SS(Q - 1);
        st(Q, U + Us);
        st(N - Q, U - Us);
      }
    }
  } else {
    int eh[H + 1], el[H + 1], oh[H - 1], ol[H - 1];
    fix_split<H + 1>(e, eh, el);
    fix_split<H - 1>(o, oh, ol);
#pragma unroll
    for (int i = 0; i <= H; ++i) {
      const long long E = block_row_fix<F::n0, F::O0>(tab, eh, el, i);
      if (i == 0 || i == H) {
        st(i, E);
      } else {
        const long long O = block_row_fix<F::n1, F::O1>(tab, oh, ol, i - 1);
        if constexpr (OUT_SPEC) {
          st(i, E);
          st(H + i, O);
        } else {
          st(i, E + O);
          st(N - i, E - O);
        }
      }
    }
  }
}

// ---- tiles: the lines one warp holds, with one exponent --------------------------------------
// A tile's values are V 2^(E - 1080).  E is the exponent field of its largest entry at first and
// moves with the shifts below; FIX_ZERO and FIX_NAN stand for an all-zero tile and one with an
// infinity or a NaN.
constexpr int FIX_ZERO = -100000;
constexpr int FIX_NAN = 100000;
constexpr int FIX_TOP = 58;  // |V| < 2^58 between passes

// doubles of one warp to a tile; lanes without a line pass zeros.  All 32 lanes take part.
template <int N>
__device__ __forceinline__ int fix_tile(double (&v)[N], long long (&V)[N]) {
  unsigned eb = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) eb = max(eb, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
  eb = __reduce_max_sync(0xffffffffu, eb);
  int shift = 0;
  if (eb < (128u << 20)) {  // zeros, denormals and the lowest range, through a power of two
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] *= 0x1p600;
    eb = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) eb = max(eb, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
    eb = __reduce_max_sync(0xffffffffu, eb);
    shift = 600;
  }
  const int e = (int)(eb >> 20);
  eb |= 0xfffffu;
#pragma unroll
  for (int i = 0; i < N; ++i) V[i] = fix_from(v[i], eb);
  return e == 0 ? FIX_ZERO : (e == 2047 ? FIX_NAN : e - shift);
}

// bits that any |V| of the line uses above 2^32 (the high words' magnitudes, or-ed)
__device__ __forceinline__ unsigned fix_mag(unsigned m, long long v) {
  const int h = (int)(v >> 32);
  return m | (unsigned)(h ^ (h >> 31));
}
// left shift (right if negative) that brings a tile whose magnitudes are m back to 2^57 <= max
// |V| < 2^58; 0 while it is within a factor of 4 of that
__device__ __forceinline__ int fix_renorm(unsigned m) {
  m = __reduce_or_sync(0xffffffffu, m);
  const int lz = __clz((int)m);
  return (lz < 64 - FIX_TOP || (lz > 66 - FIX_TOP && m != 0u)) ? lz - (64 - FIX_TOP) : 0;
}
__device__ __forceinline__ long long fix_shift(long long v, int left) {
  return left >= 0 ? (long long)((unsigned long long)v << left) : v >> -left;
}
// right shift of a value by d >= 0 units of its tile's exponent
__device__ __forceinline__ long long fix_align(long long v, int d) { return shr_s64(v, (unsigned)d); }

// Conversion of a tile of exponent E back to doubles (`neg`: with the opposite sign).  A tile whose
// largest entry is below 2^-895 is shifted down to the exponent range of fix_to (its results lose
// relative precision there and end at zero below 2^-953); one with an infinity, a NaN or an entry
// of 2^1021 or more becomes NaN throughout.
struct FixOut {
  unsigned kb, flip, nan;
};
template <int N>
__device__ __forceinline__ FixOut fix_out(long long (&V)[N], int E, bool neg = false) {
  FixOut f;
  f.flip = neg ? 0x80000000u : 0u;
  f.nan = 0u;
  if ((unsigned)(E - 128) > 2043u - 128u) {  // rare
    if (E < 128) {
#pragma unroll
      for (int i = 0; i < N; ++i) V[i] = fix_align(V[i], 128 - E);
    } else {
      f.nan = 0x7ff80000u;
    }
    E = 128;
  }
  f.kb = (unsigned)(E + 5) << 20;
  return f;
}
__device__ __forceinline__ double fix_get(const FixOut& f, long long v) {
  return fix_to(v, f.kb, f.flip, f.nan);
}

}  // namespace ufg

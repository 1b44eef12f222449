// FP64 line operators in 64-bit fixed point on the integer pipe.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM but 64 32x32+64-bit integer ones
// (IMAD.WIDE; measured 1.9 and 57), so line passes on the FP64 pipe are bound by it (80 % active,
// everything else idle on 32^3 slices).  Here each line is aligned to its own largest exponent and
// the folds and block rows of line_op (line_ops.cuh) run on 64-bit integers:
//   value       V = x 2^(1080 - E), |V| < 2^58 (E: exponent field of the line's largest entry),
//               exact for entries within 2^5 of the largest, rounded at 2^-58 of it below;
//   coefficient c 2^(60 + g) = h 2^30 + l, |l| <= 2^29 (FixCoef), from the same FP64 tables;
//   product     V c 2^g = (Vh 2^30 + Vl)(h 2^30 + l) / 2^60 = Vh h + (Vh l + Vl h) / 2^30, Vl l
//               dropped (below half a unit): three IMAD.WIDE per multiply-add in two
//               accumulators, joined once per block row.
// |folded V| < 2^60, the sums of products stay below 2^63 and g (2 at N = 32, 3 or 4 below for most
// tables) is what both the coefficients and the results leave free (fix_table).
//
// Precision: a result is off by about a unit, 2^-58 of its line's largest entry, so a pass has the
// accuracy of FP64 multiply-adds along the line entry by entry, whatever the sizes of the lines
// (emulated against long double for N = 4 .. 32, tau = 0.05 .. 20, both dispersions and points,
// normal, graded and log-uniform vectors: median, 99th percentile and largest relative error of the
// entries and the 2-norm as those of line_op, where the tables' rounding dominates).  One exponent
// per warp (one to four planes) was 8 % faster at N = 16 and 32 and 1.3x at 10 and 12 (M 16^3 x 1024
// 41 against 45 us, 12^3 x 1024 30 against 39), but left the far entries of a point source 8e-11 off
// instead of 5e-13 at N = 16.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "line_ops.cuh"

namespace ufg {

constexpr int FIX_L = 30;   // bits of the low limb of a coefficient and of a value
constexpr int FIX_TOP = 58;           // |V| < 2^58 into a pass
constexpr int FIX_LZ = 64 - FIX_TOP;  // leading zeros of such a value's magnitude, at least
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
  int g;  // results are values times 2^g
};

// c 2^k as two limbs; false if the high one would not fit
inline bool fix_coef(double c, int k, FixCoef* out) {
  const double s = std::ldexp(c, k);
  if (!(s > -2305843008139952128.0 && s < 2305843008139952128.0)) return false;  // 2^61 - 2^30
  const long long v = std::llrint(s);
  const long long l = ((v + (1LL << (FIX_L - 1))) & ((1LL << FIX_L) - 1)) - (1LL << (FIX_L - 1));
  out->h = (int)((v - l) >> FIX_L);
  out->l = (int)l;
  return true;
}
// the fixed-point table of the flat FP64 blocks of an N-line (LineCoef layout) with coefficients
// c 2^k; false if a coefficient or a row's sums do not fit (|Vh| <= 2^30, 0 <= Vl < 2^30)
template <int N>
inline bool fix_table_at(const double* flat, int k, LineCoefFix<N>* t) {
  using F = FixLine<N>;
  const int n[4] = {F::n0, F::n1, F::n2, F::n3}, off[4] = {F::O0, F::O1, F::O2, F::O3};
  for (int i = 0; i < 2 * F::NP; ++i) t->c[i] = FixCoef{0, 0};
  for (int b = 0; b < 4; ++b)
    for (int i = 0; i < n[b]; ++i) {
      FixCoef* row = t->c + 2 * (off[b] + i * F::pad(n[b]));
      double m = 0.5;
      for (int j = 0; j < n[b]; ++j) {
        if (!fix_coef(*flat++, k, row + j)) return false;
        m += (row[j].l < 0 ? -(double)row[j].l : (double)row[j].l) +
             (row[j].h < 0 ? -(double)row[j].h : (double)row[j].h);
      }
      if (m * 1073741824.0 >= 9.2e18) return false;
    }
  return true;
}
// The largest k that the table allows and for which results, of up to norm 2^58 (the operator's
// largest row sum of magnitudes), fit: the more bits of a coefficient, the more a result keeps
// below the inputs' unit.
template <int N>
inline bool fix_table(const double* flat, double norm, LineCoefFix<N>* t) {
  for (int g = FIX_LZ - 1; g >= 0; --g)
    if (norm * std::ldexp(1.0, FIX_TOP + g) < 9.2e18 && fix_table_at<N>(flat, 2 * FIX_L + g, t)) {
      t->g = g;
      return true;
    }
  return false;
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
__device__ __forceinline__ unsigned long long shl_u64(unsigned long long v, unsigned s) {
  unsigned long long d;
  asm("shl.b64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
}
__device__ __forceinline__ long long shr_s64(long long v, unsigned s) {
  long long d;
  asm("shr.s64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
}

// x 2^(1080 - E) to nearest; eb = (largest |high word| of the line) | 0xfffff
__device__ __forceinline__ long long fix_from(double x, unsigned eb) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned s = (eb - (hi & 0x7fffffffu)) >> 20;  // exponent distance to the largest
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m =
      ((unsigned long long)__funnelshift_l(lo, mh, FIX_SH) << 32) | (lo << FIX_SH);
  m = shr_u64(m + (shl_u64(1, s) >> 1), s);
  return (int)hi < 0 ? -(long long)m : (long long)m;
}
// V 2^(E - 1080) to nearest, E in [128, 2040]; kb = (E + 5) << 20, flip = sign bit to change (the
// magnitude is that of v or of v + 1: one unit, as everywhere here)
__device__ __forceinline__ double fix_to(long long v, unsigned kb, unsigned flip) {
  const unsigned vh = (unsigned)((unsigned long long)v >> 32);
  const int sg = (int)vh >> 31;
  const unsigned ah = vh ^ (unsigned)sg, al = (unsigned)(unsigned long long)v ^ (unsigned)sg;
  unsigned long long n = ((unsigned long long)ah << 32) | al;
  const unsigned c = (unsigned)__clzll((long long)n);  // 1 .. 64
  n = n << ((c - 1u) & 63u);                           // leading bit at 62
  n = (n + 512ull) >> 10;
  unsigned hi = (unsigned)(n >> 32) + (kb - (c << 20));
  hi = c == 64u ? 0u : hi;
  return __hiloint2double((int)(hi | ((vh ^ flip) & 0x80000000u)), (int)(unsigned)n);
}

// one row of a block of n columns at pair `off` of the table: limbs xh, xl of the inputs
template <int n, int off, int N>
__device__ __forceinline__ long long block_row_fix(const LineCoefFix<N>& cf, const int* xh,
                                                   const int* xl, int i) {
  constexpr int np = (n + 1) / 2;
  const int4* tab = reinterpret_cast<const int4*>(cf.c);
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

// line_op on integers: V[N] in, (index, value 2^g) out, same blocks and order of emission
template <int N, bool IN_SPEC, bool OUT_SPEC, class Emit>
__device__ __forceinline__ void line_op_int(const long long (&v)[N], const LineCoefFix<N>& cf,
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
    auto CS = [&](int m) { return block_row_fix<F::n0, F::O0>(cf, csh, csl, m); };
    auto CA = [&](int m) { return block_row_fix<F::n1, F::O1>(cf, cah, cal, m); };
    auto SS = [&](int m) { return block_row_fix<F::n2, F::O2>(cf, ssh, ssl, m); };
    auto SA = [&](int m) { return block_row_fix<F::n3, F::O3>(cf, sah, sal, m); };
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
      const long long E = block_row_fix<F::n0, F::O0>(cf, eh, el, i);
      if (i == 0 || i == H) {
        st(i, E);
      } else {
        const long long O = block_row_fix<F::n1, F::O1>(cf, oh, ol, i - 1);
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

// ---- lines with an exponent -------------------------------------------------------------------
// The values of a line are V 2^(E - 1080).  E is the exponent field of its largest entry at first
// and moves with the shifts below; FIX_ZERO and FIX_NAN stand for an all-zero line and one with an
// infinity or a NaN.
constexpr int FIX_ZERO = -100000;
constexpr int FIX_NAN = 100000;

// a thread's line of doubles to fixed point; E returned
template <int N>
__device__ __forceinline__ int fix_line(double (&v)[N], long long (&V)[N]) {
  unsigned eb = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) eb = max(eb, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
  int shift = 0;
  if (eb < (128u << 20)) {  // zeros, denormals and the lowest range, through a power of two
    eb = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i] *= 0x1p600;
      eb = max(eb, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
    }
    shift = 600;
  }
  const int e = (int)(eb >> 20);
  eb |= 0xfffffu;
#pragma unroll
  for (int i = 0; i < N; ++i) V[i] = fix_from(v[i], eb);
  return e == 0 ? FIX_ZERO : (e == 2047 ? FIX_NAN : e - shift);
}

// bits that any |V| of a line uses above 2^32 (the high words' magnitudes, or-ed)
__device__ __forceinline__ unsigned fix_mag(unsigned m, long long v) {
  const int h = (int)(v >> 32);
  return m | (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned long long fix_abs(long long v) {
  return (unsigned long long)(v ^ (v >> 63));  // |v|, or one less
}
__device__ __forceinline__ long long fix_shl(long long v, int s) {
  return (long long)((unsigned long long)v << s);
}

// The lines of one pass are read by those of the next across each other, so each leaves two
// exponents beside its values W 2^(raw - 1080): `raw`, and `top`, the one at which its largest entry
// would stand at the top of a pass's range (2^57 to 2^58).
// Exponents of a line just left at dst[i STEP], `m` its or-ed high words.  A line below 2^57 is
// shifted up there first, so that its values keep all their bits when they are aligned to others.
template <int N, int STEP>
__device__ __forceinline__ void fix_publish(long long* dst, unsigned m, int e, int* top, int* raw) {
  const int lz = __clz((int)m);
  if (lz > FIX_LZ) {
    unsigned long long a = 0;
#pragma unroll 4
    for (int i = 0; i < N; ++i) a |= fix_abs(dst[i * STEP]);
    const int sh = a == 0 ? FIX_TOP : __clzll((long long)a) - FIX_LZ;  // (0 and -1 alike)
#pragma unroll 4
    for (int i = 0; i < N; ++i) dst[i * STEP] = fix_shl(dst[i * STEP], sh);
    *top = *raw = e - sh;
  } else {
    *top = e + FIX_LZ - lz;
    *raw = e;
  }
}

// Exponents are read in groups of Q, one vector load from an aligned address.
template <int N>
constexpr int fix_group() {
  return N % 4 == 0 ? 4 : 2;
}
template <int Q>
struct FixWords {
  int w[Q];
  __device__ __forceinline__ explicit FixWords(const int* src) {
    if constexpr (Q == 4) {
      const int4 v = *reinterpret_cast<const int4*>(src);
      w[0] = v.x;
      w[1] = v.y;
      w[2] = v.z;
      w[3] = v.w;
    } else {
      const int2 v = *reinterpret_cast<const int2*>(src);
      w[0] = v.x;
      w[1] = v.y;
    }
  }
};
// A line from entry i of N published lines, at(i) with exponents top(i) and raw(i), that no other
// thread with `on` reads: aligned to the largest of them or, where its own largest entry is 8 or more times
// below that, to that entry (in place first: unrolled on registers this spilled at N = 16 and 32).
// E returned.
template <int N, class Top, class Raw, class At>
__device__ __forceinline__ int fix_gather(Top&& top, Raw&& raw, At&& at, bool on,
                                          long long (&V)[N]) {
  constexpr int Q = fix_group<N>();
  int E = -0x7fffffff - 1;
#pragma unroll
  for (int i = 0; i < N; i += Q) {
    const FixWords<Q> q(&top(i));
#pragma unroll
    for (int j = 0; j < Q; ++j) E = max(E, q.w[j]);
  }
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < N; i += Q) {
    const FixWords<Q> q(&raw(i));
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      V[i + j] = shr_s64(at(i + j), (unsigned)(E - q.w[j]));
      m = fix_mag(m, V[i + j]);
    }
  }
  if (on && __clz((int)m) > FIX_LZ + 2) {
    unsigned long long a = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) a |= fix_abs(V[i]);
    E -= a == 0 ? FIX_TOP : __clzll((long long)a) - FIX_LZ;
#pragma unroll(N <= 8 ? N : 1)
    for (int i = 0; i < N; ++i) {
      const int s = E - raw(i);
      at(i) = s >= 0 ? shr_s64(at(i), (unsigned)s) : fix_shl(at(i), -s);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) V[i] = at(i);
  }
  return E;
}

// Conversion of the results of a line of exponent E back to doubles (`neg`: with the opposite
// sign).  Outside the exponents that fix_to covers, fix_get's values are short of a factor of
// post = 2^shift, which the caller puts into an operation that it does anyway (a multiply-add with
// 1, an exponent; by itself it cost 12 % at N = 10 and 12 on the FP64 pipe): subnormal results are
// rounded, those past the range become infinite, and a line with an infinity or a NaN is NaN
// throughout.
struct FixOut {
  unsigned kb, flip;
  int shift;
  double post;
};
__device__ __forceinline__ FixOut fix_out(int E, int g, bool neg = false) {
  FixOut f;
  f.flip = neg ? 0x80000000u : 0u;
  f.shift = 0;
  f.post = 1.0;
  E -= g;
  if ((unsigned)(E - 128) > 2040u - 128u) {  // rare
    const int Ec = E < 128 ? 128 : 1900;
    f.shift = E - Ec;
    f.post = E > 4000 ? __hiloint2double(0x7ff80000, 0)
                      : __hiloint2double((max(f.shift, -1022) + 1023) << 20, 0);
    E = Ec;
  }
  f.kb = (unsigned)(E + 5) << 20;
  return f;
}
__device__ __forceinline__ double fix_get(const FixOut& f, long long v) {
  return fix_to(v, f.kb, f.flip);
}

}  // namespace ufg

// FP64 contractions on the integer pipes.
//
// GB300 issues two FP64 operations per clock and multiprocessor against 32
// 32 x 32 + 64 bit integer multiply-adds and 64 operations of the integer ALU,
// so an n-term dot product of doubles is cheaper as an exact fixed-point one.
// A line of doubles is written as integers on the common scale of its largest
// magnitude (59 bits and a sign, so 6 bits more than a double's 53 stay below
// the largest element's last place), the operator's rows as 62-bit integers on
// the scale of the largest row sum; the products of the high words with both
// accumulate exactly, the low 64 bits of the sum are cut, and the result is
// rounded to a double once.  Lines for which that scale does not do, steep ones
// and those near the ends of the FP64 range, take the FP64 pipe (fx_apply).
//
// Largest error of the derivative's rows on lines whose elements differ by
// 2^4 and more, in units of the largest row sum times the line's largest element
// (tests/test_gpu_fixed_products.py prints it; the FMA chain on the same lines):
// n = 2 8.2e-17 (9.8e-17), n = 3 7.8e-17 (9.6e-17), n = 4 6.8e-17 (1.5e-16), n = 6
// 4.1e-17 (1.1e-16), n = 8 4.2e-17 (1.4e-16), n = 10 2.9e-17 (9.1e-17).  What the
// kernels gained stands at each of them.
#pragma once

#include <stdint.h>

#include "adg_internal.h"

namespace adg {

// A data element on its line's scale, f = h 2^32 + l with l signed, |f| < 2^59.
struct FxVal {
  int h, l;
};

// Exponent fields (of doubles) between which a line is worked on in integers;
// lines below 2^-959, from 2^977 on, or with an infinity or a NaN take the
// FP64 pipe.
constexpr unsigned FX_E_MIN = 64, FX_E_MAX = 2000;
// ... and those of results (fx_double)
constexpr int FX_B_MIN = 70, FX_B_MAX = 2040;

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// Scale exponent g of an operator whose largest row sum of magnitudes is s
// (positive): s < 2^(g - 1), so every entry is below 2^62.  (An overflown s:
// out of every range, so that the FP64 pipe takes the lines.)
__device__ __forceinline__ int fx_scale(double s) {
  const int e = (__double2hiint(s) >> 20) & 0x7ff;
  return e == 0x7ff ? 1 << 16 : e - 1023 + 2;
}

// Entry m of an operator with scale exponent g.
__device__ __forceinline__ FxOp fx_op(double m, int g) {
  const long long v = __double2ll_rn(scalbn(m, 63 - g));
  FxOp o;
  o.l = (int)v;
  o.h = (int)((v - o.l) >> 32);
  return o;
}

// Sort key of a double's magnitude (its exponent field is key >> 21).
__device__ __forceinline__ unsigned fx_key(double x) { return (unsigned)__double2hiint(x) * 2u; }

// x on the scale of exponent field e (that of the line's largest magnitude, at
// least FX_E_MIN), cut toward zero at 2^-58 of the scale.
__device__ __forceinline__ FxVal fx_val(double x, unsigned e) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned s = e + 5u - (((unsigned)hi * 2u) >> 21);
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  // the mantissa at the top of 64 bits, then down to its place (the shift is
  // clamped: far smaller elements, zeros and subnormals among them, become 0)
  unsigned long long f;
  asm("{.reg .b64 a; mov.b64 a, {%1, %2}; shr.u64 %0, a, %3;}"
      : "=l"(f)
      : "r"(lo << 11), "r"(__funnelshift_l(lo, mh, 11)), "r"(s));
  const unsigned sg = (unsigned)(hi >> 31);          // all ones: negative
  unsigned fl, fh;
  asm("{sub.cc.u32 %0, %2, %4; subc.u32 %1, %3, %4;}"
      : "=r"(fl), "=r"(fh)
      : "r"((unsigned)f ^ sg), "r"((unsigned)(f >> 32) ^ sg), "r"(sg));
  FxVal o;
  o.l = (int)fl;
  o.h = (int)(fh + (fl >> 31));
  return o;
}

// A dot product in units of 2^64: (r 2^32 + f) 2^-32, |r| < 2^58.
struct FxSum {
  long long r;
  unsigned f;
};

// Accumulator of a dot product: entries times values, without the low x low
// products (below 2^-57 of the row sum times the largest element).
struct FxAcc {
  long long hh, hl;
  __device__ __forceinline__ FxAcc() : hh(0), hl(0) {}
  __device__ __forceinline__ void add(FxVal x, FxOp m) {
    hh = fx_mad(x.h, m.h, hh);
    hl = fx_mad(x.h, m.l, hl);
    hl = fx_mad(x.l, m.h, hl);
  }
  __device__ __forceinline__ FxSum sum() const { return {fx_mad((int)(hl >> 32), 1, hh), (unsigned)hl}; }
};

// The sum R, cut toward zero to whole units, times 2^(b - 1085) as a double,
// rounded to nearest (b: an exponent field in FX_B_MIN .. FX_B_MAX).
// Odd in R, and zero where the whole units are.  A dot product of a line with
// exponent field e by an operator with scale exponent g has b = e + g + 5.
__device__ __forceinline__ double fx_double(FxSum R, int b) {
  int rl, rh;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(rl), "=r"(rh) : "l"(R.r));
  const unsigned s = (unsigned)(rh >> 31);
  // whole units of |R|: of a negative one the complement of r, one more if f = 0
  unsigned al, ah;
  asm("{.reg .u32 d; add.cc.u32 d, %4, 0xffffffff; addc.cc.u32 %0, %2, 0; addc.u32 %1, %3, 0;}"
      : "=r"(al), "=r"(ah)
      : "r"((unsigned)rl ^ s), "r"((unsigned)rh ^ s), "r"(R.f == 0u ? s : 0u));
  const bool z = ah == 0;
  const unsigned x = z ? al : ah, y = z ? 0u : al;
  const int lz = __clz((int)x);
  const unsigned nh = __funnelshift_l(y, x, lz), nl = y << (lz & 31);
  const unsigned bl = __funnelshift_r(nl, nh, 11), bh = nh >> 11;     // leading one in bit 52
  const unsigned eb = (unsigned)((z ? b - 32 : b) - lz) << 20;        // the one adds to the field
  unsigned ol, oh;
  // round half up: bit 10 of the cut part, as the carry of doubling it
  asm("{.reg .u32 d; add.cc.u32 d, %2, %2; addc.cc.u32 %0, %3, 0; addc.u32 %1, %4, %5;}"
      : "=r"(ol), "=r"(oh)
      : "r"(nl << 21), "r"(bl), "r"(bh), "r"(eb));
  return __hiloint2double(x == 0u ? 0 : (int)(oh | (s & 0x80000000u)), (int)ol);
}

// Rows of doubles, times c: y(a) = c sum_j m[a n + j] x[j] on the FP64 pipe.
// Out of line: the lines that take it are few, and its code would cost the
// others registers.
template <int n>
__device__ __noinline__ void fx_rows(const double* m, double c, int rows, const double* x, double* y) {
  double v[n];
#pragma unroll
  for (int j = 0; j < n; ++j) v[j] = x[j];
#pragma unroll 1
  for (int a = 0; a < rows; ++a) {
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < n; ++j) acc = fma(m[a * n + j], v[j], acc);
    y[a] = c * acc;
  }
}
struct FxRows {
  const double* m;
  double c;
  template <int n, int ROWS>
  __device__ __forceinline__ void apply(const double* x, double* y) const {
    fx_rows<n>(m, c, ROWS, x, y);
  }
};

// Rows that are the row sums of an operator of L columns, on "lines" of one.
template <int L>
struct FxSums {
  const double* m;
  template <int n, int ROWS>
  __device__ __forceinline__ void apply(const double* x, double* y) const {
    const double x0 = x[0];                             // (y may lie over x)
#pragma unroll 1
    for (int a = 0; a < ROWS; ++a) {
      double s = 0.0;
#pragma unroll 1
      for (int j = 0; j < L; ++j) s += m[a * L + j];
      y[a] = s * x0;
    }
  }
};

// ROWS outputs of an operator on the line x: out(a, sum_j m[a n + j] x[j]) for
// a < ROWS, m of scale exponent g, `rows` its rows in FP64.
//
// Two kinds of lines take the FP64 pipe: those out of the range, and steep ones.
// The integers hold every element to 2^-58 of the largest, and a row may give the
// largest next to no weight: the far side of a jump, or a spike in the middle of a
// differentiated line.  Its result then has only the small elements' bits.  Each
// row's large weights are those of the nodes around its own, so with one of every
// two neighbours (of three, one of the outer ones too) within 2^-5 of the largest
// the error stays that of the FMA chain; other lines (the cells a shock runs
// through) are left to it.  EVEN: no need to look (every weight of the operator is
// at least 1/32 of its row, or as its caller says).
template <int n, int ROWS, bool EVEN, typename Rows, typename Out>
__device__ __forceinline__ void fx_apply(const double* x, const FxOp* __restrict__ m, int g, Rows rows,
                                         Out out) {
  unsigned key = fx_key(x[0]), low = ~0u;
#pragma unroll
  for (int j = 1; j < n; ++j) {
    if (!EVEN && n > 2) low = min(low, max(fx_key(x[j - 1]), fx_key(x[j])));
    key = max(key, fx_key(x[j]));
  }
  if (!EVEN && n == 3) low = min(low, max(fx_key(x[0]), fx_key(x[n - 1])));
  const unsigned e = key >> 21;
  const int b = (int)e + g + 5;
  const bool steep = !EVEN && n > 2 && (low >> 21) + 5u < e;
  if (e >= FX_E_MIN && e < FX_E_MAX && b >= FX_B_MIN && b <= FX_B_MAX && !steep) {
    FxVal f[n];
#pragma unroll
    for (int j = 0; j < n; ++j) f[j] = fx_val(x[j], e);
    constexpr int U = ROWS < 2 ? 1 : 2;
#pragma unroll U
    for (int a = 0; a < ROWS; ++a) {
      FxAcc acc;
#pragma unroll
      for (int j = 0; j < n; ++j) acc.add(f[j], m[a * n + j]);
      out(a, fx_double(acc.sum(), b));
    }
  } else {
    unsigned any = key;                                 // (a line of zeros, a flow at rest, has no sums)
#pragma unroll
    for (int j = 0; j < n; ++j) any |= (unsigned)__double2loint(x[j]);
    // (in place where there are more results than elements: the projection's
    // kernels then keep their registers, the predictor's do not)
    double y[ROWS], w[n];
    double* v = ROWS > n ? y : w;
#pragma unroll
    for (int j = 0; j < n; ++j) v[j] = x[j];
    if (any) rows.template apply<n, ROWS>(v, y);
#pragma unroll 1
    for (int a = 0; a < ROWS; ++a) out(a, any ? y[a] : 0.0);
  }
}

}  // namespace adg

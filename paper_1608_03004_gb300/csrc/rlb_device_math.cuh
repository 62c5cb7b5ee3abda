// Device arithmetic of the stage kernel that is worth testing on its own: the reciprocal and the two halves
// of the WENO5 interface value. Included by rlb.cu and by the GPU unit test of these functions.
#pragma once

namespace rlbdev {

// 1/d for positive, normal d: the hardware approximation of rcp.approx.ftz.f64 (relative error ~1e-6,
// measured) refined by one cubically convergent Newton-Raphson step, x1 = x0 (1 + e + e^2) with
// e = 1 - d x0 (the truncated geometric series of 1/(1 - e)); the result is within 2 ulp of the
// correctly rounded quotient. Costs three FP64 FMAs instead of the ~8 FP64-pipe slots of an IEEE division.
__device__ __forceinline__ double rcp_nr(double d) {
  double x0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x0) : "d"(d));
  const double e = fma(-d, x0, 1.0);
  return fma(x0, fma(e, e, e), x0);
}

// The same with 1 in a register that the compiler does not know, for loops bound by the FP64 pipe (an immediate operand
// costs three of its cycles).
__device__ __forceinline__ double rcp_nr(double d, double one) {
  double x0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x0) : "d"(d));
  const double e = fma(-d, x0, one);
  return fma(x0, fma(e, e, e), x0);
}

// 1/sqrt(x) for positive, normal x: the hardware approximation of rsqrt.approx.ftz.f64 refined by one step of
// third order, y1 = y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 (the binomial series of (1 - e)^(-1/2)): five FP64
// operations and no branch, where 1.0 / sqrt(x) takes about 35.
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// rsqrt_nr for subnormal x too, which the hardware approximation would take as zero: scaled by 2^106.
__device__ __forceinline__ double rsqrt_any(double x) {
  if ((unsigned)__double2hiint(x) >= 0x100000u) return rsqrt_nr(x);
  return rsqrt_nr(x * 0x1p106) * 0x1p53;
}

// sqrt(x) for x >= 0 (0 gives 0): x rsqrt(x) and one Newton-Raphson correction from the remainder x - s^2.
__device__ __forceinline__ double sqrt_nr(double x) {
  const double y = rsqrt_any(x), s = x * y;
  const double r = fma(fma(-s, s, x), 0.5 * y, s);
  return x == 0.0 ? 0.0 : r;
}

// a/d for positive, normal d: a times the reciprocal, corrected once from the remainder a - q d.
__device__ __forceinline__ double div_nr(double a, double d) {
  const double r = rcp_nr(d), q = a * r;
  return fma(fma(-q, d, a), r, q);
}

constexpr double WENO_EPS = 1e-6;

// Products and sums that are rounded exactly as written. The compiler may contract a product into a following
// addition (an FMA), and may do so differently in different inlined copies of the same expression. The
// reduced-precision kernel forms the indicator squares at a lane's edges twice (once in each lane that uses them), and
// its compensated sums are error-free only if every addition is rounded as written, so its FP32 arithmetic goes through
// these (mul.rn / add.rn / sub.rn are never contracted). The double forms of these and of the functions up to
// weno5_interface serve the unit test of the formulas only: the FP64 kernels take the packed limiter (weno5_pair_df2,
// weno5_combine6_df2) and its gradient (weno5_grad) below.
__device__ __forceinline__ float mul_x(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_x(double a, double b) { return a * b; }
__device__ __forceinline__ float add_x(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_x(double a, double b) { return a + b; }
__device__ __forceinline__ float sub_x(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_x(double a, double b) { return a - b; }

// Fifth-order WENO (Jiang & Shu) written on first differences d_l = v_l - v_{l-1} of five samples
// v0..v4 ordered along the wind (v2 is the upwind cell next to the interface, whose value is v2 + G):
//   candidates (2,-7,11)/6, (-1,5,2)/6, (2,5,-1)/6  =  v2 + r_k/6,  r0 = 5 d2 - 2 d1, r1 = d2 + 2 d3,
//   r2 = 4 d3 - d4;
//   smoothness indicators (weights 13/12 and 1/4): 3 beta_k = SL(d1,d2), SC(d2,d3), SR(d3,d4) with
//   SL(x,y) = 4x^2 - 11xy + 10y^2, SC = 4x^2 - 5xy + 4y^2, SR = 10x^2 - 11xy + 4y^2;
//   alpha_k = d_k / (eps + beta_k)^2 with d = (1, 6, 3)/10 equals 9 / s_k, s_k = u_k^2,
//   u_k = (3 eps + 3 beta_k) / sqrt(d_k); the normalised weights are w_k = prod_{l!=k} s_l / sum_m prod_{l!=m} s_l.
// Each indicator depends on one pair of adjacent differences, and each pair serves three interfaces, so
// a kernel evaluates the three scaled squares once per pair (weno5_pair) and combines three pairs per
// interface (weno5_combine6). For a wind toward decreasing index the stencil is mirrored: the differences
// change sign and order, which swaps the roles of SL and SR.
constexpr double C0 = 3.1622776601683795;  // sqrt(10)
constexpr double C1 = 1.2909944487358056;  // sqrt(10/6)
constexpr double C2 = 1.8257418583505538;  // sqrt(10/3)
// epsilon terms 3 eps (C0, C1, C2) of indicators taken on weight-normalised values
constexpr float EPS_A = (float)(3.0 * WENO_EPS * C0);
constexpr float EPS_B = (float)(3.0 * WENO_EPS * C1);
constexpr float EPS_C = (float)(3.0 * WENO_EPS * C2);

// Reciprocal of weno5_combine6: in FP32 the hardware approximation alone (about 1 ulp of FP32, below the rounding of
// the FP32 state it serves).
__device__ __forceinline__ double rcp_fast(double d) { return rcp_nr(d); }
__device__ __forceinline__ float rcp_fast(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}

// Scaled indicator squares of the pair (x, y) = (d_j, d_{j+1}) in memory order. fwd: wind toward increasing
// index; then sA = (C0 (SL + 3eps))^2, sB = (C1 (SC + 3eps))^2, sC = (C2 (SR + 3eps))^2; otherwise SL and SR
// trade places. (eA, eB, eC) = 3 eps (C0, C1, C2): the velocity's epsilon term, which scales with the square
// of its quadrature weight.
template <typename T>
__device__ __forceinline__ void weno5_pair(T x, T y, bool fwd, T eA, T eB, T eC, T& sA, T& sB, T& sC) {
  const T qx = mul_x(x, x), pxy = mul_x(x, y), qy = mul_x(y, y);
  const T ax = fwd ? T(4.0 * C0) : T(10.0 * C0), ay = fwd ? T(10.0 * C0) : T(4.0 * C0);
  const T cx = fwd ? T(10.0 * C2) : T(4.0 * C2), cy = fwd ? T(4.0 * C2) : T(10.0 * C2);
  const T uA = fma(ax, qx, fma(T(-11.0 * C0), pxy, fma(ay, qy, eA)));
  const T uB = fma(T(4.0 * C1), qx, fma(T(-5.0 * C1), pxy, fma(T(4.0 * C1), qy, eB)));
  const T uC = fma(cx, qx, fma(T(-11.0 * C2), pxy, fma(cy, qy, eC)));
  sA = mul_x(uA, uA);
  sB = mul_x(uB, uB);
  sC = mul_x(uC, uC);
}

// 6 G of the interface from the three scaled squares (s0, s1, s2) of its stencils and the differences
// d1..d4 in wind order (the kernels apply the 1/6 in the flux difference, where it costs nothing).
template <typename T>
__device__ __forceinline__ T weno5_combine6(T s0, T s1, T s2, T d1, T d2, T d3, T d4) {
  const T r0 = fma(T(5.0), d2, mul_x(T(-2.0), d1)), r1 = fma(T(2.0), d3, d2), r2 = fma(T(4.0), d3, -d4);
  const T a0 = mul_x(s1, s2);
  const T num = fma(s0, fma(s2, r1, mul_x(s1, r2)), mul_x(a0, r0));
  const T den = fma(s0, add_x(s1, s2), a0);
  return mul_x(num, rcp_fast(den));
}

// G of the interface.
template <typename T>
__device__ __forceinline__ T weno5_combine(T s0, T s1, T s2, T d1, T d2, T d3, T d4) {
  return weno5_combine6(s0, s1, s2, d1, d2, d3, d4) * T(1.0 / 6.0);
}

// Interface value v2 + G of five samples in memory order m0..m4 around the interface between m2 and m3
// (wind toward increasing index, fwd) or between m1 and m2 (wind toward decreasing index): pairs first, then the
// combination, as the reduced-precision kernel forms it. eps: the limiter's epsilon.
template <typename T>
__device__ __forceinline__ T weno5_interface(T m0, T m1, T m2, T m3, T m4, bool fwd, double eps = WENO_EPS) {
  const T D1 = m1 - m0, D2 = m2 - m1, D3 = m3 - m2, D4 = m4 - m3;
  const T eA = T(3.0 * eps * C0), eB = T(3.0 * eps * C1), eC = T(3.0 * eps * C2);
  T a[3], b[3], c[3];
  weno5_pair(D1, D2, fwd, eA, eB, eC, a[0], b[0], c[0]);
  weno5_pair(D2, D3, fwd, eA, eB, eC, a[1], b[1], c[1]);
  weno5_pair(D3, D4, fwd, eA, eB, eC, a[2], b[2], c[2]);
  if (fwd) return m2 + weno5_combine(a[0], b[1], c[2], D1, D2, D3, D4);
  return m2 + weno5_combine(a[2], b[1], c[0], -D4, -D3, -D2, -D1);
}

// Compensated (double-float) accumulation in FP32 for the moment sums of the reduced-precision path: an
// unevaluated sum hi + lo, the error of each addition recovered with Knuth's TwoSum and of each product with
// an FMA (the error-free transformations of Ogita, Rump and Oishi's accurate dot product). Weights are
// themselves given as hi + lo float pairs, so the sums reach about 1e-13 relative before they are reduced
// in FP64.
struct DF {
  float hi, lo;
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// d rounded to the nearest float, ties to even, by integer operations on its bits: a conversion instruction occupies
// the FP64 pipe. Values outside FP32's normal range (a thin gas has coefficients among FP32's subnormals) are converted
// by that instruction, in a volatile statement, which the compiler leaves in its branch. With the rounding to subnormals
// written out in the branch, the FP32 steps of 128 moving tubes took 7 % longer.
__device__ __forceinline__ float round_f32(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  if (((hi >> 20) & 0x7FFu) - 897u >= 254u) {
    float f;
    asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(d));
    return f;
  }
  const unsigned m = (((hi & 0x7FFFFFFFu) - (896u << 20)) << 3) | (lo >> 29), rest = lo << 3;
  const unsigned up = rest > 0x80000000u || (rest == 0x80000000u && (m & 1u)) ? 1u : 0u;
  return __uint_as_float((hi & 0x80000000u) | (m + up));  // a carry into the exponent is the right value, up to infinity
}

// acc += a (xhi + xlo)
__device__ __forceinline__ void df_add_dfprod(DF& acc, DF a, float xhi, float xlo) {
  const float p = __fmul_rn(a.hi, xhi);
  float e = fmaf(a.hi, xhi, -p);
  e = fmaf(a.hi, xlo, e);
  e = fmaf(a.lo, xhi, e);
  float s, t;
  two_sum(acc.hi, p, s, t);
  acc.hi = s;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t, e));
}

// acc += a
__device__ __forceinline__ void df_add(DF& acc, DF a) {
  float s, t;
  two_sum(acc.hi, a.hi, s, t);
  acc.hi = s;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t, a.lo));
}


// ---------------------------------------------------------------------------------------------------------
// Packed FP32 arithmetic: two floats in a 64-bit register pair, one instruction per operation on both
// (fma/add/sub/mul.rn.f32x2: each half rounded as the scalar operation rounds it). On GB300 a
// packed operation occupies the FP32 pipe like two scalar ones (1.94 of them per SM and clock, measured, against 3.9
// scalar) but takes one issue slot instead of two.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ F2 f2(float x) { return f2(x, x); }
__device__ __forceinline__ float lo_of(F2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi_of(F2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 neg2(F2 a) { return {a.v ^ 0x8000000080000000ull}; }

// ptxas fuses a packed product into a following packed sum (measured, with .rn written and with contraction switched
// off), which would round an interface value differently in different inlined copies and break the error-free
// transformations. A product that feeds a sum is therefore taken as a b + (-0) with a -0 that the compiler does not
// know: minus_zero2() reads it from memory once per kernel.
static __device__ unsigned long long g_minus_zero2 = 0x8000000080000000ull;
__device__ __forceinline__ F2 minus_zero2() { return {*const_cast<const volatile unsigned long long*>(&g_minus_zero2)}; }
__device__ __forceinline__ F2 mulx2(F2 a, F2 b, F2 nz) { return fma2(a, b, nz); }

// Two double-floats, one in each half.
struct DF2 {
  F2 hi, lo;
};

// ---------------------------------------------------------------------------------------------------------
// WENO5 limiter of the FP64 stage kernel in double-float arithmetic, two interfaces at a time.
//
// GB300 executes FP32 at 64 times its FP64 rate, and the FP64 stage kernel is bound by the FP64 pipe. The limiter
// (indicators, nonlinear weights, the weighted candidate sum) is about two thirds of the method's FP64 operations,
// so the kernel evaluates it in double-float: a value is an unevaluated sum hi + lo of two floats (about 47
// significant bits), combined with the error-free transformations TwoSum (Knuth), FastTwoSum (Dekker) and the
// FMA-based TwoProduct. The two halves of every packed operand belong to the two rows of a mirror pair of
// directions: the row with the wind toward -x is held in reversed order, so that both rows take the same operations.
// The differences entering the limiter come from the FP64 state; the 6 G returned per interface carries an
// absolute error of a few 1e-14 of the differences around it (the error of the limiter's FP64 form is ~1e-16 of
// them), well inside the FP64 path's 1e-12 parity.
//
// Indicators: with the linear weights d = (1, 6, 3)/10 taken out of the squares, the three indicators of a
// pair of adjacent differences (x, y) are v = S + e with S the integer quadratic forms
//   SL(x, y) = 4x^2 - 11xy + 10y^2, SC = 4x^2 - 5xy + 4y^2, SR = 10x^2 - 11xy + 4y^2  (= 3 beta_k)
// and e = 3 eps ws^2 (the velocity's epsilon term). With t_k = v_k^2 the interface value is
//   6 G = [t1 t2 r0 + 3 t0 (2 t2 r1 + t1 r2)] / [t1 t2 + 3 t0 (2 t2 + t1)],
// the weights d_k / t_k multiplied through by t0 t1 t2 / 10 (r_k as in weno5_combine6). The v_k of one
// interface are first scaled by a common power of two so that the largest lies in [1, 2): the weights are
// homogeneous in t, and the scaling keeps the products of the t's inside the FP32 exponent range.
//
// A packed operation has no free sign change, so a product is formed negated where its rounding error needs it
// (-p from (-a) b, then a b + (-p)) and the sums of such products run on the negated values: negation is exact, so
// nothing else changes.

// s + e = a + b exactly, for the high parts of sums
__device__ __forceinline__ void two_sum2(F2 a, F2 b, F2& s, F2& e) {
  s = add2(a, b);
  const F2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// a + b = s + e exactly, |a| >= |b|, with a given negated (na = -a)
__device__ __forceinline__ DF2 fast_two_sum_n(F2 na, F2 b) {
  const F2 s = sub2(b, na);
  return {s, sub2(b, add2(s, na))};
}

// a + b of two double-floats whose high parts are summed as s + t, t completed with the low parts: the last TwoSum
// (robust to cancellation of the high parts)
__device__ __forceinline__ DF2 renorm2(F2 s, F2 t) {
  DF2 r;
  two_sum2(s, t, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ DF2 df2_plus(DF2 a, DF2 b) {
  F2 s, t;
  two_sum2(a.hi, b.hi, s, t);
  return renorm2(s, add2(t, add2(a.lo, b.lo)));
}
__device__ __forceinline__ DF2 df2_minus(DF2 a, DF2 b) {
  const F2 s = sub2(a.hi, b.hi), bb = sub2(s, a.hi);
  const F2 t = sub2(sub2(a.hi, sub2(s, bb)), add2(b.hi, bb));
  return renorm2(s, add2(t, sub2(a.lo, b.lo)));
}

// a + b for a, b >= 0 (no cancellation)
__device__ __forceinline__ DF2 df2_plus_pos(DF2 a, DF2 b) {
  F2 s, t;
  two_sum2(a.hi, b.hi, s, t);
  t = add2(t, add2(a.lo, b.lo));
  const F2 u = add2(s, t);
  return {u, sub2(t, sub2(u, s))};
}

__device__ __forceinline__ DF2 df2_pow2(DF2 a, F2 p) { return {mul2(a.hi, p), mul2(a.lo, p)}; }

// a * b, with -a.hi given
__device__ __forceinline__ DF2 df2_times(DF2 a, F2 na, DF2 b, F2 nz) {
  const F2 np = mulx2(na, b.hi, nz);
  return fast_two_sum_n(np, fma2(a.hi, b.lo, fma2(a.lo, b.hi, fma2(a.hi, b.hi, np))));
}

// d = hi + lo with hi the top 24 significant bits of d (truncated) and lo the next 23 (|lo| < ulp(hi)); by
// integer operations on d's bits, so that the split costs no FP64 instruction. |d| < 2^-126 gives 0 (such a
// difference is far below the epsilon term and the values around it); |d| >= 2^128 gives FP32's overflow.
__device__ __forceinline__ DF df_split(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const int e = (int)((hi >> 20) & 0x7FFu);
  if (e <= 896) return {0.0f, 0.0f};
  const unsigned sgn = hi & 0x80000000u;
  // (integer operations here too: a conversion would be taken out of the branch and occupy the FP64 pipe)
  if (e >= 1151) return {__uint_as_float(sgn | 0x7F800000u | (e == 2047 && ((hi & 0xFFFFFu) | lo) ? 1u : 0u)), 0.0f};
  const float h = __uint_as_float(sgn | ((unsigned)(e - 896) << 23) | (__funnelshift_l(lo, hi, 3) & 0x7FFFFFu));
  float l = 0.0f;
  if (e >= 920) {  // x 2^(E - 46) with x the next 23 bits, E = e - 1023: (2^23 + x) 2^(E - 23) - 2^(E - 23)
    const unsigned k = sgn | ((unsigned)(e - 919) << 23);
    l = __fsub_rn(__uint_as_float(k | ((lo & 0x1FFFFFFFu) >> 6)), __uint_as_float(k));
  }
  return {h, l};
}

// The double equal to the float f (0 for zero and subnormal f), by integer operations on f's bits (unit test of df_split).
__device__ __forceinline__ double df_widen(float f) {
  const unsigned b = __float_as_uint(f), ef = (b >> 23) & 0xFFu;
  const unsigned hi = (b & 0x80000000u) | ((ef + 896u) << 20) | ((b >> 3) & 0xFFFFFu);
  const double w = __hiloint2double((int)hi, (int)(b << 29));
  return ef == 0u ? 0.0 : w;
}

// The double equal to any float (subnormals, infinities and NaN too), by integer operations.
__device__ __forceinline__ double widen_f32(float f) {
  const unsigned b = __float_as_uint(f), sgn = b & 0x80000000u;
  unsigned ef = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
  if (ef == 255u) {
    ef = 1151u;  // the double's exponent field is 2047
  } else if (ef == 0u) {
    if (m == 0u) return __hiloint2double((int)sgn, 0);
    const int s = __clz(m) - 8;  // normalise: the leading bit to bit 23
    return __hiloint2double((int)(sgn | ((unsigned)(897 - s) << 20) | (((m << s) >> 3) & 0xFFFFFu)), (int)((m << s) << 29));
  }
  return __hiloint2double((int)(sgn | ((ef + 896u) << 20) | (m >> 3)), (int)(m << 29));
}

// hi + lo of a normalised double-float (|lo| <= ulp(hi)/2) as one double, rounded at its 53rd bit: an addition on the
// bits of hi widened, in place of an FP64 operation that widens lo on its own. Where lo points toward zero, the float
// next to hi is widened and lo is added to 2^29 units of that double's last place, so that the sum never leaves the
// binade whose units it counts. Zero and subnormal hi give 0; infinities and NaN pass through.
__device__ __forceinline__ double df_join(float hi, float lo) {
  const unsigned b = __float_as_uint(hi), ef = (b >> 23) & 0xFFu;
  if (ef == 0u) return 0.0;
  // (no conversion instruction here: it would be taken out of the branch and occupy the FP64 pipe for every value)
  if (ef == 255u) return __hiloint2double((int)((b & 0x80000000u) | 0x7FF00000u | ((b >> 3) & 0xFFFFFu)), (int)(b << 29));
  const unsigned bl = __float_as_uint(lo), down = (b ^ bl) >> 31, p = b - down, ep = (p >> 23) & 0xFFu;
  // lo, with hi's sign taken out, in units of 2^(ep - 127 - 52): scale 2^(179 - ep), in two factors where it exceeds
  // FP32's range
  float l = __uint_as_float(bl ^ (b & 0x80000000u));
  unsigned top = 306u;
  if (ef < 64u) {
    l = __fmul_rn(l, 0x1p64f);
    top = 242u;
  }
  const unsigned add = (unsigned)__float2int_rn(__fmul_rn(l, __uint_as_float((top - ep) << 23))) + (down << 29);
  const unsigned wh = (p & 0x80000000u) | (((p & 0x7FFFFFFFu) >> 3) + (896u << 20)), wl = (p << 29) + add;
  return __hiloint2double((int)(wh + (wl < add ? 1u : 0u)), (int)wl);
}

// hi + lo of any double-float, as one double: normalised first (TwoSum), then joined. Outside FP32's normal range the
// high part is converted as it is (below 2^-126 it is the exact sum, which df_join would drop; the volatile statement
// stays in its branch).
__device__ __forceinline__ double df_sum(float hi, float lo) {
  float s, t;
  two_sum(hi, lo, s, t);
  if (((__float_as_uint(s) >> 23) & 0xFFu) - 1u >= 254u) {
    double w;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(w) : "f"(s));
    return w;
  }
  return df_join(s, t);
}

// Indicators v_A, v_B, v_C of the pairs (x, y) = (d_j, d_{j+1}) in wind order, e the epsilon term:
// (v_A, v_B, v_C) = (SL, SC, SR)(x, y) + e.
__device__ __forceinline__ void weno5_pair_df2(DF2 x, DF2 y, F2 ne_hi, F2 e_lo, F2 nz, DF2& vA,
                                               DF2& vB, DF2& vC) {
  // -x^2, -x y, -y^2 rounded (the high parts), their errors plus the cross terms (the low parts)
  const F2 nx = neg2(x.hi), ny = neg2(y.hi);
  const F2 X = mul2(nx, x.hi), Y = mul2(ny, y.hi), Z = mul2(nx, y.hi);
  const F2 Xl = fma2(add2(x.hi, x.hi), x.lo, fma2(x.hi, x.hi, X));
  const F2 Yl = fma2(add2(y.hi, y.hi), y.lo, fma2(y.hi, y.hi, Y));
  const F2 Zl = fma2(x.hi, y.lo, fma2(x.lo, y.hi, fma2(x.hi, y.hi, Z)));
  const F2 c4 = f2(4.0f), c5 = f2(5.0f), c10 = f2(10.0f), c11 = f2(11.0f);
  const F2 m5 = f2(-5.0f), m10 = f2(-10.0f), m11 = f2(-11.0f);
  // the integer multiples, high parts negated (those by 4 are exact, fused or not)
  const F2 X4 = mul2(X, c4), Y4 = mul2(Y, c4), X4l = mul2(Xl, c4), Y4l = mul2(Yl, c4);
  const F2 X10 = mulx2(X, c10, nz), X10l = fma2(Xl, c10, fma2(X, m10, X10));
  const F2 Y10 = mulx2(Y, c10, nz), Y10l = fma2(Yl, c10, fma2(Y, m10, Y10));
  const F2 Z11 = mulx2(Z, m11, nz), Z11l = fma2(Zl, m11, fma2(Z, c11, Z11));
  const F2 Z5 = mulx2(Z, m5, nz), Z5l = fma2(Zl, m5, fma2(Z, c5, Z5));
  // (a, b, c) + e: exact sums of the (negated) high parts, then the low parts and the errors; v > 0 is a positive
  // definite form plus e, so the final FastTwoSum's ordering holds
  auto sum3 = [&](F2 a, F2 al, F2 b, F2 bl, F2 c, F2 cl) {
    F2 s, t1, t2, t3;
    two_sum2(a, b, s, t1);
    two_sum2(s, c, s, t2);
    two_sum2(s, ne_hi, s, t3);
    const F2 lo = sub2(add2(add2(al, bl), add2(cl, e_lo)), add2(add2(t1, t2), t3));
    return fast_two_sum_n(s, lo);
  };
  vA = sum3(X4, X4l, Z11, Z11l, Y10, Y10l);
  vB = sum3(X4, X4l, Z5, Z5l, Y4, Y4l);
  vC = sum3(X10, X10l, Z11, Z11l, Y4, Y4l);
}

// 1 / 2^(exponent of the largest v): the scale that brings it into [1, 2)
__device__ __forceinline__ float weno5_scale(float v0, float v1, float v2) {
  return __uint_as_float((254u - (__float_as_uint(fmaxf(fmaxf(v0, v1), v2)) >> 23)) << 23);
}

// 6 G of two interfaces from the indicators (v0, v1, v2) of their stencils and the differences d1..d4 in wind order.
__device__ __forceinline__ DF2 weno5_combine6_df2(DF2 v0, DF2 v1, DF2 v2, DF2 d1, DF2 d2, DF2 d3, DF2 d4,
                                                   F2 nz) {
  const F2 sc = f2(weno5_scale(lo_of(v0.hi), lo_of(v1.hi), lo_of(v2.hi)),
                   weno5_scale(hi_of(v0.hi), hi_of(v1.hi), hi_of(v2.hi)));
  const F2 nsc = neg2(sc);
  auto square = [&](DF2 v) {
    const F2 h = mul2(v.hi, sc), nh = mul2(v.hi, nsc), l = mul2(v.lo, sc), np = mulx2(nh, h, nz);
    return fast_two_sum_n(np, fma2(add2(h, h), l, fma2(h, h, np)));
  };
  const DF2 t0 = square(v0), t1 = square(v1), t2 = square(v2);
  // r0 = 5 d2 - 2 d1, r1 = d2 + 2 d3, r2 = 4 d3 - d4 (6 times the candidates' corrections)
  const F2 c2 = f2(2.0f), c3 = f2(3.0f), c4 = f2(4.0f), c5 = f2(5.0f), m5 = f2(-5.0f);
  const F2 n5 = mulx2(d2.hi, m5, nz);
  const DF2 r0 = df2_minus({neg2(n5), fma2(d2.lo, c5, fma2(d2.hi, c5, n5))}, df2_pow2(d1, c2));
  const DF2 r1 = df2_plus(d2, df2_pow2(d3, c2));
  const DF2 r2 = df2_minus(df2_pow2(d3, c4), d4);
  const F2 nt1 = neg2(t1.hi), nt2 = neg2(t2.hi);
  const DF2 a0 = df2_times(t1, nt1, t2, nz);
  const F2 n3 = mulx2(t0.hi, f2(-3.0f), nz);
  const DF2 t03 = fast_two_sum_n(n3, fma2(t0.lo, c3, fma2(t0.hi, c3, n3)));
  const F2 nt03 = neg2(t03.hi);
  const DF2 p0 = df2_times(a0, neg2(a0.hi), r0, nz), p1 = df2_times(t2, nt2, r1, nz), p2 = df2_times(t1, nt1, r2, nz);
  const DF2 num = df2_plus(p0, df2_times(t03, nt03, df2_plus(df2_pow2(p1, c2), p2), nz));
  const DF2 den = df2_plus_pos(a0, df2_times(t03, nt03, df2_plus_pos(df2_pow2(t2, c2), t1), nz));
  // num / den: a quotient from FP32's reciprocal (approximation refined by one Newton-Raphson step to about
  // half an ulp), then one correction from the remainder
  float ra, rb;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ra) : "f"(lo_of(den.hi)));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rb) : "f"(hi_of(den.hi)));
  F2 rc = f2(ra, rb);
  const F2 nden = neg2(den.hi);
  rc = fma2(rc, fma2(nden, rc, f2(1.0f)), rc);
  const F2 q1 = mulx2(num.hi, rc, nz), np = mulx2(q1, nden, nz);
  const F2 pe = fma2(q1, den.lo, fma2(q1, den.hi, np));
  const F2 rem = add2(add2(num.hi, np), sub2(num.lo, pe));
  DF2 G;
  two_sum2(q1, mulx2(rem, rc, nz), G.hi, G.lo);
  // all but one t below FP32's range (indicator ratios beyond ~1e19): that stencil's value
  const float da = lo_of(den.hi), db = hi_of(den.hi);
  if (da == 0.0f || db == 0.0f) {
    auto pick = [&](float a0_, float a1_, float a2_, float x0, float x1, float x2) {
      const bool k0 = a0_ <= a1_ && a0_ <= a2_, k1 = !k0 && a1_ <= a2_;
      return k0 ? x0 : (k1 ? x1 : x2);
    };
    float gh[2] = {lo_of(G.hi), hi_of(G.hi)}, gl[2] = {lo_of(G.lo), hi_of(G.lo)};
    if (da == 0.0f) {
      gh[0] = pick(lo_of(v0.hi), lo_of(v1.hi), lo_of(v2.hi), lo_of(r0.hi), lo_of(r1.hi), lo_of(r2.hi));
      gl[0] = pick(lo_of(v0.hi), lo_of(v1.hi), lo_of(v2.hi), lo_of(r0.lo), lo_of(r1.lo), lo_of(r2.lo));
    }
    if (db == 0.0f) {
      gh[1] = pick(hi_of(v0.hi), hi_of(v1.hi), hi_of(v2.hi), hi_of(r0.hi), hi_of(r1.hi), hi_of(r2.hi));
      gl[1] = pick(hi_of(v0.hi), hi_of(v1.hi), hi_of(v2.hi), hi_of(r0.lo), hi_of(r1.lo), hi_of(r2.lo));
    }
    G = {f2(gh[0], gh[1]), f2(gl[0], gl[1])};
  }
  return G;
}

// Interface value v2 + G computed as the FP64 stage kernel does with the double-float limiter (differences in
// FP64, split, pairs, combination, 6 G widened and divided by 6 in FP64); eps: the limiter's epsilon. A wind
// toward decreasing index takes the samples in reversed order. Both halves of the packed operands hold the interface.
__device__ __forceinline__ double weno5_interface_df(double m0, double m1, double m2, double m3, double m4, bool fwd,
                                                     double eps = WENO_EPS) {
  const double v0 = fwd ? m0 : m4, v1 = fwd ? m1 : m3, v3 = fwd ? m3 : m1, v4 = fwd ? m4 : m0;
  auto both = [](DF q) { return DF2{f2(q.hi), f2(q.lo)}; };
  const DF2 D1 = both(df_split(v1 - v0)), D2 = both(df_split(m2 - v1)), D3 = both(df_split(v3 - m2)),
            D4 = both(df_split(v4 - v3));
  const DF2 e = both(df_split(3.0 * eps));
  const F2 ne = neg2(e.hi), nz = minus_zero2();
  DF2 a[3], b[3], c[3];
  weno5_pair_df2(D1, D2, ne, e.lo, nz, a[0], b[0], c[0]);
  weno5_pair_df2(D2, D3, ne, e.lo, nz, a[1], b[1], c[1]);
  weno5_pair_df2(D3, D4, ne, e.lo, nz, a[2], b[2], c[2]);
  const DF2 G = weno5_combine6_df2(a[0], b[1], c[2], D1, D2, D3, D4, nz);
  return fma(df_join(lo_of(G.hi), lo_of(G.lo)), 1.0 / 6.0, m2);
}

// ---------------------------------------------------------------------------------------------------------
// Gradient of the WENO5 interface value with respect to its five samples, from the differences d1..d4 in wind order
// (their common sign does not matter): with Phi = v2 + G(d), dPhi/dv_m = g_m - g_{m+1} + [m = 2], g_l = dG/dd_l, g_0 =
// g_5 = 0. Returns 1.5 g_l (1.5 = 6/4): 6 G = sum_k w_k r_k, w_k = (c_k / v_k^2) / sum, (c_k) = (1, 6, 3), and
//   d(6G)/dv_k = 2 w_k (6G - r_k) / v_k,  v_k = x a + y b + e with a, b half the partials of the quadratic form,
// so that g_l collects -2 w_0, 5 w_0 + w_1, 2 w_1 + 4 w_2, -w_2 and 4 z_k a_k, z_k = w_k (6G - r_k) / v_k, over 6. 66 FP64
// operations; written on samples with every partial formed on its own it took about 130.
// k: the constants, in registers (ADJ_CST from shared memory: FP64 operations with an immediate operand, additions and
// multiplications issue every 19 cycles instead of 16; all-immediate, the row kernel took 11 % longer).
enum { C_ONE, C_NZ, C_55, C_25, C_4, C_10, C_6, C_3, C_2, C_H, C_Q, C_125, C_15, ADJ_CST };
__device__ __forceinline__ double grad_constant(int i) {
  constexpr double v[ADJ_CST] = {1.0, -0.0, 5.5, 2.5, 4.0, 10.0, 6.0, 3.0, 2.0, 0.5, 0.25, 1.25, 1.5};
  return v[i];
}
__device__ __forceinline__ void weno5_grad(double d1, double d2, double d3, double d4, double e,
                                           const volatile double* k, double (&g)[4]) {
  const double one = k[C_ONE], nz = k[C_NZ], c55 = k[C_55], c25 = k[C_25], c4 = k[C_4], c10 = k[C_10];
  const double t1 = fma(c55, d1, nz), t2 = fma(c55, d2, nz), t3 = fma(c55, d3, nz), t4 = fma(c55, d4, nz);
  const double s2 = fma(c25, d2, nz), s3 = fma(c25, d3, nz);
  const double ax0 = fma(c4, d1, -t2), ay0 = fma(c10, d2, -t1);  // 4x^2 - 11xy + 10y^2 of (d1, d2)
  const double ax1 = fma(c4, d2, -s3), ay1 = fma(c4, d3, -s2);   // 4x^2 - 5xy + 4y^2 of (d2, d3)
  const double ax2 = fma(c10, d3, -t4), ay2 = fma(c4, d4, -t3);  // 10x^2 - 11xy + 4y^2 of (d3, d4)
  const double i0 = rcp_nr(fma(d1, ax0, fma(d2, ay0, e)), one);
  const double i1 = rcp_nr(fma(d2, ax1, fma(d3, ay1, e)), one);
  const double i2 = rcp_nr(fma(d3, ax2, fma(d4, ay2, e)), one);
  const double q0 = fma(i0, i0, nz), q1 = fma(k[C_6], fma(i1, i1, nz), nz), q2 = fma(k[C_3], fma(i2, i2, nz), nz);
  const double is = rcp_nr(fma(fma(q0, one, q1), one, q2), one);
  const double w0 = fma(q0, is, nz), w1 = fma(q1, is, nz), w2 = fma(q2, is, nz);
  const double c2 = k[C_2];
  const double r0 = fma(c2, s2, -fma(c2, d1, nz)), r1 = fma(c2, d3, d2), r2 = fma(c4, d3, -d4);
  const double G = fma(w0, r0, fma(w1, r1, fma(w2, r2, nz)));
  const double z0 = fma(fma(w0, i0, nz), fma(-r0, one, G), nz), z1 = fma(fma(w1, i1, nz), fma(-r1, one, G), nz),
               z2 = fma(fma(w2, i2, nz), fma(-r2, one, G), nz);
  const double ch = k[C_H], cq = k[C_Q];
  g[0] = fma(z0, ax0, -fma(ch, w0, nz));
  g[1] = fma(z0, ay0, fma(z1, ax1, fma(cq, w1, fma(k[C_125], w0, nz))));
  g[2] = fma(z1, ay1, fma(z2, ax2, fma(ch, w1, w2)));
  g[3] = fma(z2, ay2, -fma(cq, w2, nz));
}

}  // namespace rlbdev

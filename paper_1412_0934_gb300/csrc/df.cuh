// Double-float numbers: a value hi + lo held in two floats with |lo| <= ulp(hi)/2, about 48
// significant bits, computed on the FP32 pipes (GB300 runs FP64 at 1/73 of its FP32 rate).
// Built from the error-free transformations of Dekker (1971) and Knuth (TwoSum) and the
// double-word algorithms analysed by Joldes, Muller & Popescu (ACM TOMS 2017), u = 2^-24:
//   add  the "sloppy" double-word sum (TwoSum of the high words, the low words added in float,
//        Fast2Sum): 11 operations, absolute error below about 3u^2 (|x| + |y|) -- as accurate as
//        the "accurate" 20-operation sum except under cancellation, where its error is relative to
//        the operands rather than to the result: the same backward-stable behaviour as a double
//        add at 2^-48 in place of 2^-53.  add_acc is the accurate sum (relative error < 3u^2 +
//        13u^3), kept for the pressure recovery E - |m|^2/(2 rho), where cancellation in cold,
//        fast gas is the reason for extra precision;
//   mul  double-word x double-word with FMA, the low-by-low product dropped: 8 operations,
//        relative error below about 6u^2; mulf_ (double-word x float) 6 operations;
//   rcp, div, sqrt: one Newton correction of an SFU approximation, relative error ~2^-45.
// Comparisons are exact (lexicographic on (hi, lo) of normalised values).  The exponent range is
// that of float: the hydro state here stays far inside it.
#pragma once
#include <cuda_runtime.h>

namespace hydro {

struct df {
  float h, l;
  df() = default;
  __host__ __device__ constexpr df(float hi, float lo) : h(hi), l(lo) {}
  __host__ __device__ df(double x) : h((float)x), l((float)(x - (double)(float)x)) {}
  __host__ __device__ df(float x) : h(x), l(0.f) {}
  __host__ __device__ df(int x) : h((float)x), l(0.f) {}
  __host__ __device__ explicit operator double() const { return (double)h + (double)l; }
};

__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = a + b;
  const float bp = s - a;
  return df(s, (a - (s - bp)) + (b - bp));
}
__device__ __forceinline__ df fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
  const float s = a + b;
  return df(s, b - (s - a));
}
__device__ __forceinline__ df two_prod(float a, float b) {
  const float p = a * b;
  return df(p, fmaf(a, b, -p));
}

__device__ __forceinline__ df operator-(const df& x) { return df(-x.h, -x.l); }

__device__ __forceinline__ df operator+(const df& x, const df& y) {
  const df s = two_sum(x.h, y.h);
  return fast_two_sum(s.h, s.l + (x.l + y.l));
}
__device__ __forceinline__ df operator-(const df& x, const df& y) { return x + (-y); }
__device__ __forceinline__ df add_acc(const df& x, const df& y) {
  const df s = two_sum(x.h, y.h);
  const df t = two_sum(x.l, y.l);
  const df v = fast_two_sum(s.h, s.l + t.h);
  return fast_two_sum(v.h, v.l + t.l);
}

__device__ __forceinline__ df operator*(const df& x, const df& y) {
  const df c = two_prod(x.h, y.h);
  const float t = fmaf(x.l, y.h, x.h * y.l);
  return fast_two_sum(c.h, c.l + t);
}

// Exact scaling by a power of two, and double-word x float (TwoProd + one FMA + Fast2Sum).
__device__ __forceinline__ df half_(const df& x) { return df(0.5f * x.h, 0.5f * x.l); }
__device__ __forceinline__ df twice_(const df& x) { return df(2.f * x.h, 2.f * x.l); }
__device__ __forceinline__ df mulf_(const df& x, float f) {
  const df c = two_prod(x.h, f);
  return fast_two_sum(c.h, fmaf(x.l, f, c.l));
}
__device__ __forceinline__ df rabs(const df& x) { return x.h < 0.f ? -x : x; }

// Reciprocal: r0 from the SFU, then r = r0 + r0 (1 - y r0) with the residual formed exactly.
__device__ __forceinline__ df rcp_(const df& y) {
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(y.h));
  const df p = two_prod(y.h, r0);          // y.h r0 exactly
  const float e = (1.f - p.h) - p.l;        // 1 - y.h r0 (1 - p.h is exact near 1)
  const float res = fmaf(-y.l, r0, e);      // 1 - y r0
  return fast_two_sum(r0, r0 * res);
}
__device__ __forceinline__ df div_(const df& x, const df& y) {
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(y.h));
  const float q1 = x.h * r0;
  const df r = x - mulf_(y, q1);  // remainder x - y q1
  const float q2 = r.h * r0;
  return fast_two_sum(q1, q2);
}
__device__ __forceinline__ df rsqrt_(const df& x) {  // the square root (named like the float one)
  if (!(x.h > 0.f)) return df(0.f, 0.f);
  float s0;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s0) : "f"(x.h));
  const df p = two_prod(s0, s0);
  const float r = ((x.h - p.h) - p.l) + x.l;  // x - s0^2
  float i0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(i0) : "f"(s0));
  return fast_two_sum(s0, 0.5f * r * i0);
}

// ------------------------------------------------------------------ unnormalised forms
// Inside a formula a value may stay an unnormalised pair, |l| up to a few ulp(h) (or, after
// cancellation, up to a few 2^-24 of the operands): the Fast2Sum that closes each operator above
// then happens once per result instead of once per operation.  prod_ drops only l*l and rounds its
// low word three times, sum_ rounds its low word twice: the same absolute bounds (a few u^2 of the
// operands) as the normalising operators.
__device__ __forceinline__ df prod_(const df& x, const df& y) {  // 4 operations (mul: 8)
  const float p = x.h * y.h;
  return df(p, fmaf(x.h, y.l, fmaf(x.l, y.h, fmaf(x.h, y.h, -p))));
}
__device__ __forceinline__ df sum_(const df& x, const df& y) {  // 8 operations (add: 11)
  const df s = two_sum(x.h, y.h);
  return df(s.h, s.l + (x.l + y.l));
}
__device__ __forceinline__ df norm_(const df& x) { return fast_two_sum(x.h, x.l); }

// Reciprocal, quotient and square root of (possibly unnormalised) pairs, unnormalised results.  The
// reciprocal r0 (1 + e + e^2), e = 1 - y r0, keeps e^2: the approximation's e is up to 2^-23, so e^2 is
// the largest error of a step whose reciprocals stop at r0 (1 + e).  The
// quotient's remainder num.h - den.h q is exact in its leading difference (q is the float quotient to
// a few ulp); the root is one Newton correction, s = s0 + (x - s0^2) / (2 s0).  Relative errors below 2^-45
// (sqrt(t/r), further down: 2^-43) where operands, results and t/r lie between 2^-100 and 2^100.
__device__ __forceinline__ df rcpu_(const df& y) {
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(y.h));
  const float p = y.h * r0;
  const float e = fmaf(-y.l, r0, (1.f - p) - fmaf(y.h, r0, -p));  // 1 - y r0
  return df(r0, r0 * fmaf(e, e, e));
}
__device__ __forceinline__ df quot_(const df& x, const df& y) {
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(y.h));
  const float q = x.h * r0, p = y.h * q;
  const float r = ((x.h - p) - fmaf(y.h, q, -p)) + fmaf(-y.l, q, x.l);
  return df(q, r * fmaf(fmaf(-y.h, r0, 1.f), r0, r0));
}
__device__ __forceinline__ df rootu_(const df& x) {
  float s0, i0;  // independent approximations: the root's own error is squared, 1/root's only scales it
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s0) : "f"(x.h));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(i0) : "f"(x.h));
  i0 = x.h > 1.2e-38f ? i0 : 0.f;  // zero (and what .ftz reads as zero) has root zero
  const float p = s0 * s0;
  const float r = ((x.h - p) - fmaf(s0, s0, -p)) + x.l;
  return df(s0, 0.5f * r * i0);
}

// ------------------------------------------------------------------ two values side by side
// sm_103a's packed FP32 instructions do two lanes' add, multiply or FMA in one issue slot (at the
// scalar rate of the pipe: 119 results per clock per SM either way).  A df2 holds two double-float
// values as pairs of high and of low words; its operations are the ones above, lane by lane, bit for
// bit.  Operand negation is folded into the instruction.  The double-float step was bound by issue slots
// (64% of them, ~5730 thread instructions per cell): with the packed and the unnormalised forms a cell
// takes ~4100, and a 512^3 step went from 32.2 to 24.7 ms (22.5 with the comparisons below), its error
// against 64-bit arithmetic from 1.49e-15 to 1.41e-15 (2-norm, density, Mach 5).
struct df2 {
  float2 h, l;
};
__device__ __forceinline__ df2 pair_(const df& a, const df& b) { return df2{make_float2(a.h, b.h), make_float2(a.l, b.l)}; }
__device__ __forceinline__ df2 both_(const df& a) { return pair_(a, a); }
__device__ __forceinline__ df first_(const df2& x) { return df(x.h.x, x.l.x); }
__device__ __forceinline__ df second_(const df2& x) { return df(x.h.y, x.l.y); }
__device__ __forceinline__ float2 neg_(const float2& a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2_(const float2& a, const float2& b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2_(const float2& a, const float2& b) { return __fadd2_rn(a, neg_(b)); }
__device__ __forceinline__ float2 mul2_(const float2& a, const float2& b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2_(const float2& a, const float2& b, const float2& c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ df2 neg_(const df2& x) { return df2{neg_(x.h), neg_(x.l)}; }
__device__ __forceinline__ df2 half_(const df2& x) {
  const float2 c = make_float2(0.5f, 0.5f);
  return df2{mul2_(x.h, c), mul2_(x.l, c)};
}
__device__ __forceinline__ df2 norm_(const df2& x) {
  const float2 s = add2_(x.h, x.l);
  return df2{s, sub2_(x.l, sub2_(s, x.h))};
}
__device__ __forceinline__ df2 two_sum2_(const float2& a, const float2& b) {
  const float2 s = add2_(a, b), t = sub2_(s, a);
  return df2{s, add2_(sub2_(a, sub2_(s, t)), sub2_(b, t))};
}
__device__ __forceinline__ df2 sum_(const df2& x, const df2& y) {
  const df2 s = two_sum2_(x.h, y.h);
  return df2{s.h, add2_(s.l, add2_(x.l, y.l))};
}
__device__ __forceinline__ df2 operator+(const df2& x, const df2& y) { return norm_(sum_(x, y)); }
__device__ __forceinline__ df2 operator-(const df2& x, const df2& y) { return norm_(sum_(x, neg_(y))); }
__device__ __forceinline__ df2 prod_(const df2& x, const df2& y) {
  const float2 p = mul2_(x.h, y.h);
  return df2{p, fma2_(x.h, y.l, fma2_(x.l, y.h, fma2_(x.h, y.h, neg_(p))))};
}
__device__ __forceinline__ df2 add_acc(const df2& x, const df2& y) {  // the accurate sum
  const df2 s = two_sum2_(x.h, y.h), t = two_sum2_(x.l, y.l);
  const df2 v = norm_(df2{s.h, add2_(s.l, t.h)});
  return norm_(df2{v.h, add2_(v.l, t.l)});
}
__device__ __forceinline__ df2 rcpu_(const df2& y) {
  float2 r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0.x) : "f"(y.h.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0.y) : "f"(y.h.y));
  const float2 p = mul2_(y.h, r0);
  const float2 e = fma2_(neg_(y.l), r0, sub2_(sub2_(make_float2(1.f, 1.f), p), fma2_(y.h, r0, neg_(p))));
  return df2{r0, mul2_(r0, fma2_(e, e, e))};
}
__device__ __forceinline__ df2 rootu_(const df2& x) {
  float2 s0, i0;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s0.x) : "f"(x.h.x));
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(s0.y) : "f"(x.h.y));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(i0.x) : "f"(x.h.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(i0.y) : "f"(x.h.y));
  i0.x = x.h.x > 1.2e-38f ? i0.x : 0.f;
  i0.y = x.h.y > 1.2e-38f ? i0.y : 0.f;
  const float2 p = mul2_(s0, s0);
  const float2 r = add2_(sub2_(sub2_(x.h, p), fma2_(s0, s0, neg_(p))), x.l);
  return df2{s0, mul2_(mul2_(r, make_float2(0.5f, 0.5f)), i0)};
}

// sqrt(t/r), as a third-order correction of s0 = t y0, y0 = rsqrt(t) rsqrt(r): two SFU approximations per
// value where the reciprocal and the root took three, and no quotient.  (One rsqrt(t r) would do, but the
// product of a pressure and a density leaves the float range long before either does, and the speed would
// come out as zero.)  With d = 1 - s0^2 r / t the root is s0 (1 + d/2 + 3 d^2/8 ...); d is up to 2^-20 (the
// approximations and four roundings), so a Newton step's missing 3 d^2/8, 2^-42, would be the largest error
// of the wave speeds.
__device__ __forceinline__ df2 rootq_(const df2& t, const df2& r) {
  float2 yt, yr;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yt.x) : "f"(t.h.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yt.y) : "f"(t.h.y));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yr.x) : "f"(r.h.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yr.y) : "f"(r.h.y));
  yt.x = t.h.x > 1.2e-38f ? yt.x : 0.f;  // zero (and what .ftz reads as zero) has root zero
  yt.y = t.h.y > 1.2e-38f ? yt.y : 0.f;
  const float2 y0 = mul2_(yt, yr), s0 = mul2_(t.h, y0), p = mul2_(s0, s0);
  const df2 w = prod_(df2{p, fma2_(s0, s0, neg_(p))}, r);  // s0^2 r
  const float2 e = add2_(sub2_(sub2_(t.h, w.h), w.l), t.l);  // t - s0^2 r
  const float2 c = mul2_(e, y0);                   // s0 d
  const float2 d = mul2_(c, mul2_(y0, r.h));       // d
  return df2{s0, mul2_(c, fma2_(d, make_float2(0.375f, 0.375f), make_float2(0.5f, 0.5f)))};
}

// Comparisons of normalised values.
// (Evaluated in full: a short circuit is a branch, and the warps waited on those: 512^3 step 24.7 -> 22.7
// ms, 191x203x187 PPM step 4.0 -> 2.9 ms.)
__device__ __forceinline__ bool operator<(const df& a, const df& b) {
  return (a.h < b.h) | ((a.h == b.h) & (a.l < b.l));
}
__device__ __forceinline__ bool operator>(const df& a, const df& b) { return b < a; }
__device__ __forceinline__ bool operator<=(const df& a, const df& b) { return !(b < a); }
__device__ __forceinline__ bool operator>=(const df& a, const df& b) { return !(a < b); }
__device__ __forceinline__ df dabs(const df& x) { return x.h < 0.f ? -x : x; }

__device__ __forceinline__ bool cmp_lt_floor(const df& x, const df& f) { return x < f; }
__device__ __forceinline__ bool cmp_neg(const df& x) { return x.h < 0.f; }
__device__ __forceinline__ bool cmp_pos(const df& x) { return x.h > 0.f; }
__device__ __forceinline__ bool abs_le(const df& a, const df& b) { return dabs(a) <= dabs(b); }
__device__ __forceinline__ bool abs_lt(const df& a, const df& b) { return dabs(a) < dabs(b); }
__device__ __forceinline__ bool prod_nonpos(const df& a, const df& b) {
  return (a.h == 0.f) | (b.h == 0.f) | ((a.h > 0.f) != (b.h > 0.f));
}
__device__ __forceinline__ bool isfinite_(const df& x) { return isfinite(x.h); }

__device__ __forceinline__ df shfl_xor_(const df& v, int o) {
  return df(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
}

}  // namespace hydro

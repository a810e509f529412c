// Double-float ("df64") arithmetic on the FP32 pipe, and the mat-vec pair
// in that arithmetic.
//
// A value is an unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// about 48 significant bits.  The operations are built from error-free
// transformations: Knuth's TwoSum, Dekker's FastTwoSum (|a| >= |b|) and the
// FMA-based TwoProduct (see Dekker 1971; Shewchuk 1997; Hida, Li and Bailey
// 2001 for the double-double analogue).  The __f*_rn intrinsics keep the
// compiler from contracting or reassociating them.
//
// GB300 executes FP64 at 2 lanes per SM per cycle against 128 for FP32, so
// a mat-vec pair in df64 (several hundred FP32 instructions) is several
// times faster than the same pair in native FP64 while keeping a relative
// accuracy near 1e-13; it serves as the high-precision residual of the mixed
// solve.
//
// exp(-kappa r) follows Tang's table-driven method (ACM TOMS 15, 1989) with
// a table of 1024 values: x = k L + f, L = ln2/1024, |f| <= L/2, exp(x) =
// 2^(k>>10) 2^((k&1023)/1024) exp(f).  The table values 2^(j/1024) are df64
// (computed on the host, copied into shared memory by every CTA).  The
// reduction takes L = l1 + l2 with l1 = fl(L): x.hi - k l1 is exact in one
// FMA (a multiple of 2^-35 below 2^-11.5), and x.lo - k l2 rounds far below
// the result.  With |f| <= 3.4e-4 the polynomial is short: exp(f) = 1 + f +
// (f^2/2 + f^3/6), the bracket in FP32 (it is below 5.8e-8, so its FP32
// rounding is below 2^-46), and the truncation f^4/24 is below 6e-16.
// 1/sqrt(r2) is one third-order step in df64 from the MUFU estimate (error
// cubed: below 2^-65, so only the rounding of the correction remains).
//
// What bounds the kernels built on this header is the FP32 pipe: every sum
// of a df64 value costs the additions that recover its rounding error.  So
// a product is added to a sum in one FMA whose error is recovered with the
// unrounded product (prod_sum below: no separate TwoProduct and TwoSum), and
// renormalising FastTwoSums are left out wherever the trailing part is taken
// by an FP32 multiply-add anyway.  FP32 operations of one unordered pair of the
// symmetric mat-vec: 21 differences, 20 r2, 13 1/r and r, 18 exp, 24 the
// radial factors, 56 the dots n.d, 18 n_i.n_j, 91 coefficients, 96 the eight
// accumulations; N = 20480, kappa = 0.1257: 3.03 -> 2.59 ms, error against
// 64 bits 1.5e-14 -> 1.5e-15 (the second-order 1/sqrt of before was its
// largest part).  Reaction and source passes, 40961 elements x 4 x 2000
// charges: 4.11 -> 3.40 ms.
#pragma once
#include <cuda_runtime.h>

namespace bipb {

struct df {
  float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return df{s, e};
}
__device__ __forceinline__ df fast_two_sum(float a, float b) {  // |a| >= |b|
  float s = __fadd_rn(a, b);
  float e = __fsub_rn(b, __fsub_rn(s, a));
  return df{s, e};
}
__device__ __forceinline__ df two_prod(float a, float b) {
  float p = __fmul_rn(a, b);
  float e = __fmaf_rn(a, b, -p);
  return df{p, e};
}
// x + y: exact TwoSum of the leading parts, the trailing parts added in FP32.
// Absolute error about 2^-47 max(|x|, |y|).
__device__ __forceinline__ df df_add(df x, df y) {
  df s = two_sum(x.hi, y.hi);
  s.lo = __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo));
  return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ df df_neg(df x) { return df{-x.hi, -x.lo}; }
__device__ __forceinline__ df df_sub(df x, df y) { return df_add(x, df_neg(y)); }
// Products are left unnormalised: the trailing part (the exact error of the
// leading product plus the cross terms) is below a few ulp of the leading
// part, so the next product or sum takes it as it is at no loss of accuracy
// (a chain of d products has a relative error of about d 2^-46), and the
// renormalising FastTwoSum is paid only in sums, where cancellation can
// shrink the leading part.
__device__ __forceinline__ df df_mul(df x, df y) {
  float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return df{p, e};
}
__device__ __forceinline__ df df_sqr(df x) {
  float p = __fmul_rn(x.hi, x.hi);
  float e = __fmaf_rn(x.hi, x.hi, -p);
  e = __fmaf_rn(__fadd_rn(x.hi, x.hi), x.lo, e);
  return df{p, e};
}
__device__ __forceinline__ df df_norm(df x) { return fast_two_sum(x.hi, x.lo); }
// x^3, the square normalised in between
__device__ __forceinline__ df df_cube(df x) { return df_mul(df_norm(df_sqr(x)), x); }
__device__ __forceinline__ df df_scale(df x, float pow2) { return df{__fmul_rn(x.hi, pow2), __fmul_rn(x.lo, pow2)}; }
__device__ __forceinline__ double df_to_double(df x) { return (double)x.hi + (double)x.lo; }
__device__ __forceinline__ df df_from_double(double v) {
  float hi = __double2float_rn(v);
  return df{hi, __double2float_rn(v - (double)hi)};
}
// (h, lo) += x y for floats with h and x y of one sign, the product unrounded:
// the sum in one FMA, its error by the steps of TwoSum with the product in
// place of the second term (7 operations; TwoProduct and TwoSum take 10).
// With opposite signs h + x y may cancel to a result on a finer grid than h,
// whose difference from h is then not exact.
__device__ __forceinline__ void prod_sum_pos(float& h, float& lo, float x, float y) {
  const float s = __fmaf_rn(x, y, h);
  const float b = __fsub_rn(s, h);
  const float d = __fsub_rn(h, __fsub_rn(s, b));
  lo = __fadd_rn(lo, __fadd_rn(__fmaf_rn(x, y, -b), d));
  h = s;
}
// x + a b for df64 values, left unnormalised (12 operations).
__device__ __forceinline__ df df_fma(df a, df b, df x) {
  const df p = two_prod(a.hi, b.hi);
  const float plo = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
  const df s = two_sum(x.hi, p.hi);
  return df{s.hi, __fadd_rn(x.lo, __fadd_rn(s.lo, plo))};
}
// The same for a float x (11 operations), and normalised (14).
__device__ __forceinline__ df df_fma_lazy(df a, df b, float x) {
  const df p = two_prod(a.hi, b.hi);
  const float plo = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
  const df s = two_sum(x, p.hi);
  return df{s.hi, __fadd_rn(s.lo, plo)};
}
__device__ __forceinline__ df df_fma_f(df a, df b, float x) {
  const df r = df_fma_lazy(a, b, x);
  return fast_two_sum(r.hi, r.lo);
}
// x + 3 a (11 operations).
__device__ __forceinline__ df df_add_3(df a, df x) {
  const df p = two_prod(3.0f, a.hi);
  const df s = two_sum(x.hi, p.hi);
  return df{s.hi, __fadd_rn(__fadd_rn(s.lo, p.lo), __fmaf_rn(3.0f, a.lo, x.lo))};
}
// a b - x y, left unnormalised (17 operations).
__device__ __forceinline__ df df_det(df a, df b, df x, df y) {
  const df p = two_prod(a.hi, b.hi), q = two_prod(-x.hi, y.hi);
  const float plo = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
  const float qlo = __fmaf_rn(-x.hi, y.lo, __fmaf_rn(-x.lo, y.hi, q.lo));
  const df s = two_sum(p.hi, q.hi);
  return df{s.hi, __fadd_rn(s.lo, __fadd_rn(plo, qlo))};
}
// Dot product of two df 3-vectors of any size, left unnormalised (28 operations).
__device__ __forceinline__ df df_dot(const df* a, const df* b) {
  return df_fma(a[2], b[2], df_fma(a[1], b[1], df_mul(a[0], b[0])));
}
// Dot product of two unit vectors (18 operations, unnormalised): added to 6,
// every product is rounded to the grid of the floats in [4, 8), so that each
// sum's difference from the one before is exact and an FMA gives the
// product's rest.  Absolute error about 2^-46 (relative to the vectors'
// lengths; df_dot's is a quarter of that, which n.d needs -- it cancels for
// near pairs -- and n_i.n_j does not).
__device__ __forceinline__ df df_dot_unit(const df* a, const df* b) {
  const float s0 = __fmaf_rn(a[0].hi, b[0].hi, 6.0f);
  const float s1 = __fmaf_rn(a[1].hi, b[1].hi, s0);
  const float s2 = __fmaf_rn(a[2].hi, b[2].hi, s1);
  float e0 = __fmaf_rn(a[0].hi, b[0].hi, -__fsub_rn(s0, 6.0f));
  float e1 = __fmaf_rn(a[1].hi, b[1].hi, -__fsub_rn(s1, s0));
  float e2 = __fmaf_rn(a[2].hi, b[2].hi, -__fsub_rn(s2, s1));
  e0 = __fmaf_rn(a[0].hi, b[0].lo, __fmaf_rn(a[0].lo, b[0].hi, e0));
  e1 = __fmaf_rn(a[1].hi, b[1].lo, __fmaf_rn(a[1].lo, b[1].hi, e1));
  e2 = __fmaf_rn(a[2].hi, b[2].lo, __fmaf_rn(a[2].lo, b[2].hi, e2));
  return df{__fsub_rn(s2, 6.0f), __fadd_rn(__fadd_rn(e0, e1), e2)};
}
// Squared length of a df 3-vector, left unnormalised (20 operations).
__device__ __forceinline__ df df_norm2(const df* a) {
  float h = __fmul_rn(a[0].hi, a[0].hi);
  float lo = __fmaf_rn(a[0].hi, a[0].hi, -h);
  prod_sum_pos(h, lo, a[1].hi, a[1].hi);
  prod_sum_pos(h, lo, a[2].hi, a[2].hi);
  const float c = __fmaf_rn(a[0].hi, a[0].lo, __fmaf_rn(a[1].hi, a[1].lo, __fmul_rn(a[2].hi, a[2].lo)));
  return df{h, __fmaf_rn(2.0f, c, lo)};
}
// A coordinate as h + l + m: h a multiple of g = 2^(c-23) and l a multiple of
// 2^-24 g, where every coordinate of the pass lies below 2^c in magnitude, so
// that |h| <= 2^23 g, |l| <= g / 2 and |m| <= 2^-25 g (the value to about
// 2^(c-72)).  Leading and middle differences are then exact, and the leading
// one is zero or at least as large as the middle one: a difference takes 7
// operations (11 with a TwoSum of df64 values) and keeps more digits of
// nearby points than df64 values hold (up to a spread of 2^23 between the
// pass's largest coordinate and the points' own).
struct df_pos {
  float h, l, m;
};
// x on the grid g (a power of two): h and l by adding and taking away 1.5 2^52 grid units
// (of a product x the compiler's multiply-adds take the unrounded one: no branch on g here)
__device__ __forceinline__ df_pos df_split_grid(double x, double g) {
  const double M = 0x1.8p52 * g, M2 = 0x1.8p28 * g;
  const double h = (x + M) - M;
  const double r = x - h;
  const double l = (r + M2) - M2;
  return df_pos{__double2float_rn(h), __double2float_rn(l), __double2float_rn(r - l)};
}
// x on the grid g, or in three floats on no grid (WIDE, below)
template <bool WIDE>
__device__ __forceinline__ df_pos df_split_point(double x, double g) {
  if constexpr (!WIDE) return df_split_grid(x, g);
  const float h = __double2float_rn(x);
  const float l = __double2float_rn(x - (double)h);
  return df_pos{h, l, __double2float_rn(x - (double)h - (double)l)};
}
// WIDE: of three floats on no grid, for passes whose points spread further than a
// grid resolves; every sum recovers its error.
template <bool WIDE = false>
__device__ __forceinline__ df df_diff(df_pos x, df_pos y) {
  if constexpr (WIDE) {
    const df s = two_sum(x.h, -y.h), t = two_sum(x.l, -y.l), u = two_sum(s.hi, t.hi);
    return fast_two_sum(u.hi, __fadd_rn(u.lo, __fadd_rn(s.lo, __fadd_rn(t.lo, __fsub_rn(x.m, y.m)))));
  }
  df d = fast_two_sum(__fsub_rn(x.h, y.h), __fsub_rn(x.l, y.l));
  d.lo = __fadd_rn(d.lo, __fsub_rn(x.m, y.m));
  return d;
}

constexpr int kExpTab = 1024;  // entries of the exp table, 2^(j/1024) for j < 1024 (k >> 10 below)

struct DFConst {
  df eps, inveps, kappa;  // eps_out/eps_in, its inverse, kappa
  float l1, l2, l3;       // ln2/1024 = l1 + l2 + l3, l1 and l1 + l2 rounded to their digits
  float inv_l;            // 1024/ln2
  const float4* tab;      // device copy of the exp table, two df64 entries per float4
};

// Every thread of the CTA copies its share of the exp table into sh (16-byte
// aligned, kExpTab entries); the caller's next barrier makes it visible.
__device__ __forceinline__ void df_load_exp_table(df* sh, const DFConst& c) {
  float4* s4 = reinterpret_cast<float4*>(sh);
  for (int i = threadIdx.x; i < kExpTab / 2; i += blockDim.x) s4[i] = c.tab[i];
}

// s = 1/sqrt(r2) and r = r2 s for r2 > 0 (any normalisation): MUFU estimate
// s0, e = 1 - r2 s0^2 with exact leading steps, and s = s0 (1 + e/2 + 3 e^2/8).
__device__ __forceinline__ void df_rsqrt_r(df r2, df& s, df& r) {
  float s0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s0) : "f"(r2.hi));
  const float t = __fmul_rn(r2.hi, s0);
  const float tl = __fmaf_rn(r2.lo, s0, __fmaf_rn(r2.hi, s0, -t));
  const float e = __fmaf_rn(-tl, s0, __fmaf_rn(-t, s0, 1.0f));
  const float g = __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f));
  s = fast_two_sum(s0, __fmul_rn(s0, g));
  r = df{t, __fmaf_rn(t, g, tl)};
}

// exp(-x) for x >= 0 (x.hi clamped at 80), tab[j] = 2^(j/1024) as df64.  The absolute error
// is below 2^-47; relative to the value it grows as the square of the reduction's
// trailing part (2e-13 at x = 8, 2e-12 at 32).  REL: the reduction in double-float with
// L in three parts, 1e-14 of the value at any x (15 more operations), for sums in which
// every term is proportional to it.
template <bool REL = false>
__device__ __forceinline__ df df_exp_minus(df x, const DFConst& c, const df* tab) {
  const float xh = fmaxf(-x.hi, -80.0f);
  // k = rint(x / L): adding 1.5 * 2^23 leaves the integer in the low mantissa bits
  const float km = __fmaf_rn(xh, c.inv_l, 12582912.0f);
  const int k = __float_as_int(km) - 0x4B400000;
  const float kf = __fsub_rn(km, 12582912.0f);
  float f = __fmaf_rn(-kf, c.l1, xh);       // exact
  float fl;
  if constexpr (REL) {
    const df p = two_prod(kf, c.l2), a = two_sum(-x.lo, -p.hi), g = two_sum(f, a.hi);
    f = g.hi;
    fl = __fadd_rn(g.lo, __fmaf_rn(-kf, c.l3, __fsub_rn(a.lo, p.lo)));
  } else {
    fl = __fmaf_rn(-kf, c.l2, -x.lo);
  }
  // exp(f + fl) = 1 + f + q, q = f^2/2 + f^3/6 + fl (1 + f)
  const float q = __fmaf_rn(__fmul_rn(f, f), __fmaf_rn(f, 1.0f / 6.0f, 0.5f), __fmaf_rn(f, fl, fl));
  df ef = fast_two_sum(1.0f, f);  // |f| < 1
  ef.lo = __fadd_rn(ef.lo, q);
  const df r = df_mul(ef, tab[k & (kExpTab - 1)]);
  return df_scale(r, __int_as_float((127 + (k >> 10)) << 23));  // 2^floor(k / 1024)
}

// The radial factors of a pair from d (kappa-scaled when SCALED: kappa r = r
// then), with x = kappa r: s = 1/r, e = exp(-x), e1 = e - 1, t = e (1 + x) and
// t1 = t - 1.  e1 + e x = t1 is ordered (1 - e >= e x), as is 1 + t1, so
// neither needs a TwoSum.  t1 is normalised: for small x it is x^2 / 2 beside a trailing
// part of e's size (2^-25), and every product below would round that anew (K4, which has s^3,
// was off by 1.4e-14 s^3 below x = 0.3 where 2e-15 s^3 is e's rounding).
// self (MASK): s = 0, every other factor finite.
struct DfRadial {
  df s, kr, e, e1, t1, t;
};
template <bool MASK, bool SCALED, bool REL = false>
__device__ __forceinline__ DfRadial df_radial(const df* d, bool self, const DFConst& c, const df* tab) {
  DfRadial R;
  df r2 = df_norm2(d), r;
  if (MASK && self) r2 = df{1.0f, 0.0f};
  df_rsqrt_r(r2, R.s, r);
  if (MASK && self) R.s = df{0.0f, 0.0f};
  R.kr = SCALED ? r : df_mul(r, c.kappa);
  R.e = df_exp_minus<REL>(R.kr, c, tab);
  const df o = fast_two_sum(-1.0f, R.e.hi);
  R.e1 = df{o.hi, __fadd_rn(o.lo, R.e.lo)};
  const df p = df_mul(R.e, R.kr);
  const df v = fast_two_sum(R.e1.hi, p.hi);
  const float vl = __fadd_rn(v.lo, __fadd_rn(R.e1.lo, p.lo));
  R.t1 = fast_two_sum(v.hi, vl);  // exact enough below |vl| too: its error is 2^-24 of vl
  const df u = fast_two_sum(1.0f, v.hi);
  R.t = df{u.hi, __fadd_rn(u.lo, vl)};
  return R;
}

// acc += a b, left unnormalised (renormalise with two_sum before the trailing
// part has gathered more than a few dozen terms).
__device__ __forceinline__ void df_mac(df& acc, df a, df b) { acc = df_fma(a, b, acc); }
// acc += x for an unnormalised x, left unnormalised.
__device__ __forceinline__ void df_acc(df& acc, df x) {
  const df s = two_sum(acc.hi, x.hi);
  acc = df{s.hi, __fadd_rn(acc.lo, __fadd_rn(s.lo, x.lo))};
}

// (w - 3) s^2 = 3 (t - 1) s^2 + e kappa^2, e kappa^2 = e in kappa-scaled units
template <bool SCALED>
__device__ __forceinline__ df df_wm3s2(const DfRadial& R, df s2, const DFConst& c) {
  return df_add_3(df_mul(R.t1, s2), SCALED ? R.e : df_mul(R.e, df_mul(c.kappa, c.kappa)));
}

// Forward pair (the formula of pair_forward in pair.cuh) in df64.
// MASK/self: see pair.cuh (s = 0 for the self pair).
template <bool MASK>
__device__ __forceinline__ void df_pair_forward(const df* xi, const df* ni, const df* xj, df a, const df* m, bool self,
                                                const DFConst& c, const df* tab, df& accP, df& accQ) {
  const df d[3] = {df_sub(xi[0], xj[0]), df_sub(xi[1], xj[1]), df_sub(xi[2], xj[2])};
  const DfRadial R = df_radial<MASK, false>(d, self, c, tab);
  const df s2 = df_sqr(R.s), s3 = df_mul(s2, R.s);
  const df ci = df_dot(ni, d), cm = df_dot(m, d), cim = df_dot(ni, m);
  // P = s (1 - e) a + s^3 (eps t - 1) cm
  df_mac(accP, df_neg(df_mul(R.e1, R.s)), a);
  df_mac(accP, df_mul(df_fma_f(c.eps, R.t, -1.0f), s3), cm);
  // Q = s^3 [ ci ((t/eps - 1) a - (w - 3) s^2 cm) + (t - 1) cim ]
  const df x = df_fma(df_neg(df_wm3s2<false>(R, s2, c)), cm, df_mul(df_fma_f(R.t, c.inveps, -1.0f), a));
  df_mac(accQ, df_fma(x, ci, df_mul(R.t1, cim)), s3);
}

// Transposed pair (the formula of pair_transpose in pair.cuh) in df64:
// output element j (x, n) gathers element i (xs, wphi, p = wpsi n_i).
template <bool MASK>
__device__ __forceinline__ void df_pair_transpose(const df* xj, const df* nj, const df* xi, df wphi, const df* pv,
                                                  bool self, const DFConst& c, const df* tab, df& accP, df& accQ) {
  const df d[3] = {df_sub(xi[0], xj[0]), df_sub(xi[1], xj[1]), df_sub(xi[2], xj[2])};
  const DfRadial R = df_radial<MASK, false>(d, self, c, tab);
  const df s2 = df_sqr(R.s), s3 = df_mul(s2, R.s);
  const df cj = df_dot(nj, d), cp = df_dot(pv, d), cnp = df_dot(nj, pv);
  // Zphi = s^3 [ c_j ((eps t - 1) wphi - (w - 3) s^2 (p.d)) + (t - 1)(n_j.p) ]
  const df x = df_fma(df_neg(df_wm3s2<false>(R, s2, c)), cp, df_mul(df_fma_f(c.eps, R.t, -1.0f), wphi));
  df_mac(accP, df_fma(x, cj, df_mul(R.t1, cnp)), s3);
  // Zpsi = s (1 - e) wphi + s^3 (t/eps - 1)(p.d)
  df_mac(accQ, df_neg(df_mul(R.e1, R.s)), wphi);
  df_mac(accQ, df_mul(df_fma_f(R.t, c.inveps, -1.0f), s3), cp);
}

// The four kernel values of pair (target i, source j) times ds_j (times 4 pi)
// in df64: k[0] = K2 ds, k[1] = K1 ds, k[2] = K4 ds, k[3] = K3 ds (the 2 x 2
// block that maps (phi_j, psi_j) to the (phi_i, psi_i) rows).  s = 0 for the
// self pair when MASK and self.  TRANS: the block of A^T instead, output
// element i gathering input element j (the transposed pair of pair.cuh, d =
// x_i - x_j): k[0] = K2_ji, k[1] = K4_ji (the phi row), k[2] = K1_ji, k[3] =
// K3_ji (the psi row), i.e. ((1 - eps t) c_i s^3, K4, (1 - e) s,
// (1 - t/eps) c_j s^3), without an area (the output's goes on the sums).
// SCALED: kappa-scaled coordinates; the phi (A^T: psi) column is multiplied by
// kappa here, the sums by (kappa, kappa^2) (A^T: (kappa^2, kappa)) elsewhere.
// r0, r1: factors of the phi and psi row (powers of two).
// The values are normalised: where a factor has cancelled, its trailing part
// is far above an ulp of its leading one, which the digits of the exact
// tensor-core form could not hold.
template <bool MASK, bool TRANS, bool SCALED>
__device__ __forceinline__ void df_kernel_block(const df_pos* xi, const df* ni, const df_pos* xj, const df* nj,
                                                df area, bool self, const DFConst& c, const df* tab, float r0,
                                                float r1, df* k) {
  const df d[3] = {df_diff(xi[0], xj[0]), df_diff(xi[1], xj[1]), df_diff(xi[2], xj[2])};
  const DfRadial R = df_radial<MASK, SCALED>(d, self, c, tab);
  const df s2 = df_sqr(R.s), sa = TRANS ? R.s : df_mul(R.s, area), s3 = df_mul(s2, sa);
  const df s3k = SCALED ? df_mul(s3, c.kappa) : s3;  // of the phi (A^T: psi) column
  const df ci = df_dot(ni, d), cj = df_dot(nj, d), cij = df_dot_unit(ni, nj);
  const df k1 = df_neg(df_mul(R.e1, df_scale(sa, TRANS ? r1 : r0)));
  const df k4 = df_mul(df_det(R.t1, cij, df_wm3s2<SCALED>(R, s2, c), df_mul(ci, cj)), df_scale(s3k, TRANS ? r0 : r1));
  const df et1 = df_fma_lazy(c.eps, R.t, -1.0f), te1 = df_fma_lazy(R.t, c.inveps, -1.0f);
  if (!TRANS) {
    k[0] = df_mul(df_mul(et1, cj), df_scale(s3k, r0));         // K2 ds
    k[1] = k1;                                    // K1 ds
    k[2] = k4;                                    // K4 ds
    k[3] = df_mul(df_mul(te1, ci), df_scale(s3, r1));          // K3 ds
  } else {
    k[0] = df_neg(df_mul(df_mul(et1, ci), df_scale(s3, r0)));  // K2_ji
    k[1] = k4;                                    // K4_ji
    k[2] = k1;                                    // K1_ji
    k[3] = df_neg(df_mul(df_mul(te1, cj), df_scale(s3k, r1)));  // K3_ji
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) k[v] = df_norm(k[v]);
}

// The symmetric pair of pair.cuh in df64.  The four accumulators
// are updated lazily (df_mac): renormalise them before use.  SCALED: the
// records are in kappa-scaled units as there (kappa r = r, (w - 3) s^2 =
// 3 (t - 1) s^2 + e; the caller rescales the sums); otherwise unscaled, for
// any kappa >= 0.
template <bool MASK, bool TRANS, bool SCALED>
__device__ __forceinline__ void df_sym_pair(const df* d, const df* nt, df at, df alt, const df* ns, df as, df als,
                                            bool self, const DFConst& c, const df* tab, df& Pt, df& Qt, df& Ps,
                                            df& Qs) {
  const DfRadial R = df_radial<MASK, SCALED>(d, self, c, tab);
  const df s2 = df_sqr(R.s), s3 = df_mul(s2, R.s);
  const df ci = df_dot(nt, d), cj = df_dot(ns, d), cij = df_dot_unit(nt, ns);
  const df U = df_det(R.t1, cij, df_wm3s2<SCALED>(R, s2, c), df_mul(ci, cj));
  // s and s^3 folded into the four coefficients every update uses
  const df ome_s = df_neg(df_mul(R.e1, R.s)), U_s3 = df_mul(U, s3);
  // t/eps - 1 left unnormalised: its trailing part is at most a few 2^-24, and the leading one is
  // of the order of 1 unless eps is close to 1 (360 -> 357 operations)
  const df et1_s3 = df_mul(df_fma_f(c.eps, R.t, -1.0f), s3), te1_s3 = df_mul(df_fma_lazy(R.t, c.inveps, -1.0f), s3);
  if (!TRANS) {
    df_mac(Pt, ome_s, as);
    df_mac(Pt, df_mul(et1_s3, cj), als);
    df_mac(Qt, df_mul(te1_s3, ci), as);
    df_mac(Qt, U_s3, als);
    df_mac(Ps, ome_s, at);
    df_mac(Ps, df_neg(df_mul(et1_s3, ci)), alt);
    df_mac(Qs, df_neg(df_mul(te1_s3, cj)), at);
    df_mac(Qs, U_s3, alt);
  } else {
    df_mac(Pt, U_s3, als);
    df_mac(Pt, df_neg(df_mul(et1_s3, ci)), as);
    df_mac(Qt, ome_s, as);
    df_mac(Qt, df_neg(df_mul(te1_s3, cj)), als);
    df_mac(Ps, U_s3, alt);
    df_mac(Ps, df_mul(et1_s3, cj), at);
    df_mac(Qs, ome_s, at);
    df_mac(Qs, df_mul(te1_s3, ci), alt);
  }
}

// Source term of one (element, charge) pair in df64: target element (x, n),
// charge (y, q), d = x - y:  S1 += q s,  S2 += -q (n.d) s^3  (times 4 pi eps_in).
template <bool WIDE>
__device__ __forceinline__ void df_source_pair(const df_pos* x, const df* nv, const df_pos* y, df q, df& s1, df& s2) {
  const df d[3] = {df_diff<WIDE>(x[0], y[0]), df_diff<WIDE>(x[1], y[1]), df_diff<WIDE>(x[2], y[2])};
  df s, r;
  df_rsqrt_r(df_norm2(d), s, r);
  const df qs = df_mul(q, s);
  df_acc(s1, qs);
  df_mac(s2, df_neg(df_mul(qs, df_sqr(s))), df_dot(nv, d));
}

// Reaction potential at a point y from one element (record: x, a = ds psi,
// normal n, alpha = ds phi), d = y - x (the K1, K2 terms with n_j only):
//   4 pi phi += s (1 - e) a + s^3 (eps t - 1) alpha (n.d)
template <bool WIDE>
__device__ __forceinline__ void df_reaction_pair(const df_pos* y, const df_pos* x, df a, const df* nv, df al,
                                                 const DFConst& c, const df* tab, df& acc) {
  const df d[3] = {df_diff<WIDE>(y[0], x[0]), df_diff<WIDE>(y[1], x[1]), df_diff<WIDE>(y[2], x[2])};
  const DfRadial R = df_radial<false, false>(d, false, c, tab);
  df_mac(acc, df_neg(df_mul(R.e1, R.s)), a);
  df_mac(acc, df_norm(df_mul(df_fma_f(c.eps, R.t, -1.0f), df_cube(R.s))), df_norm(df_mul(al, df_dot(nv, d))));
}

// Potential at a point y in the solvent from one element (the record of the
// reaction pair), d = y - x: the exterior representation (Eq.
// eqbim_2) with dphi2/dnu = psi / eps (flux continuity), times 4 pi:
//   4 pi phi += s^3 t alpha (n.d) - s (1/eps) e a   (-Gk dphi2/dnu + dGk/dnu_y phi)
template <bool WIDE>
__device__ __forceinline__ void df_exterior_pair(const df_pos* y, const df_pos* x, df a, const df* nv, df al,
                                                 const DFConst& c, const df* tab, df& acc) {
  const df d[3] = {df_diff<WIDE>(y[0], x[0]), df_diff<WIDE>(y[1], x[1]), df_diff<WIDE>(y[2], x[2])};
  const DfRadial R = df_radial<false, false, true>(d, false, c, tab);
  // every term is proportional to e: t = e (1 + kappa r) relative to its own size, and
  // no product smaller than the term (they come near the end of the FP32 range)
  float th = R.e.hi, tl = R.e.lo;
  prod_sum_pos(th, tl, R.e.hi, R.kr.hi);
  const df t = df{th, __fmaf_rn(R.e.hi, R.kr.lo, __fmaf_rn(R.e.lo, R.kr.hi, tl))};
  df_mac(acc, df_mul(t, R.s), df_mul(df_sqr(R.s), df_mul(al, df_dot(nv, d))));
  df_mac(acc, df_neg(df_mul(df_mul(c.inveps, R.e), R.s)), a);
}

// Energy row of one (element, charge) pair in df64: element j (x, n), charge
// (y, q), d = y - x (times 4 pi):  cphi += q (eps t - 1)(n.d) s^3,  cpsi += q (1 - e) s.
template <bool WIDE>
__device__ __forceinline__ void df_energy_row_pair(const df_pos* x, const df* nv, const df_pos* y, df q, const DFConst& c,
                                                   const df* tab, df& cphi, df& cpsi) {
  const df d[3] = {df_diff<WIDE>(y[0], x[0]), df_diff<WIDE>(y[1], x[1]), df_diff<WIDE>(y[2], x[2])};
  const DfRadial R = df_radial<false, false>(d, false, c, tab);
  const df qs = df_mul(q, R.s);
  df_mac(cphi, df_mul(df_fma_f(c.eps, R.t, -1.0f), df_mul(df_sqr(R.s), qs)), df_dot(nv, d));
  df_mac(cpsi, df_neg(R.e1), qs);
}

// Energy gradient at a charge y from one element in df64.  Element record:
// x, a = ds psi, normal n, alpha = ds phi (m = alpha n), l = lphi / eps_in and
// beta = lpsi / eps_in (p = beta n) from the adjoint lam = [lphi; lpsi];
// d = y - x, cn = n.d, H = (eps t - 1) alpha + beta (times 4 pi):
//   v   += s [ (1 - e) a + l ] + s^3 cn H
//   g_m += Cn n_m + Cd d_m, where  Cn = s^3 H
//   Cd = s^3 [ (t - 1) a - l - cn (3 H s^2 + eps kappa^2 e alpha) ]
// (the y-gradients of the energy row and of the adjoint-weighted source, with
// eps w - 3 = 3 (eps t - 1) + eps e kappa^2 r^2).
template <bool WIDE>
__device__ __forceinline__ void df_grad_pair(const df_pos* y, const df_pos* x, df a, const df* nv, df al, df l, df beta,
                                             const DFConst& c, const df* tab, df& v, df* g) {
  const df d[3] = {df_diff<WIDE>(y[0], x[0]), df_diff<WIDE>(y[1], x[1]), df_diff<WIDE>(y[2], x[2])};
  const DfRadial R = df_radial<false, false>(d, false, c, tab);
  const df s2 = df_sqr(R.s), s3 = df_mul(s2, R.s);
  const df cn = df_dot(nv, d);
  const df H = df_fma(df_fma_f(c.eps, R.t, -1.0f), al, beta);
  const df Cn = df_mul(H, s3);
  df_mac(v, df_fma(df_neg(R.e1), a, l), R.s);
  df_mac(v, Cn, cn);
  const df Z = df_add_3(df_mul(H, s2), df_mul(df_mul(df_mul(c.eps, df_mul(c.kappa, c.kappa)), R.e), al));
  const df Cd = df_mul(df_fma(df_neg(cn), Z, df_fma(R.t1, a, df_neg(l))), s3);
  for (int m = 0; m < 3; ++m) {
    df_mac(g[m], Cn, nv[m]);
    df_mac(g[m], Cd, d[m]);
  }
}

}  // namespace bipb

// The radial factors of an FP64 pair on the FP32 pipe, in triple-float
// arithmetic.
//
// GB300 executes FP64 at 2 lanes per SM per cycle against 128 for FP32: one
// FP64 instruction takes as long as 64 FP32 instructions, and 1/sqrt and exp
// in FP64 are some forty of them a pair.  A value here is an unevaluated sum of three
// floats a + b + c, |b| below a few ulp of a and |c| below a few ulp of b, built from
// the error-free transformations of df64.cuh (two of the components exact, the
// third by FP32 multiply-adds: about 2^-65 of the value; compare Hida, Li and
// Bailey 2001, who drop the terms below the last component alike).  The five
// coefficients of a pair come out within half an ulp and a few 2^-60 of FP64,
// i.e. rounded once, where the FP64 chain rounds some ten times.
//
//   r2 from differences of coordinates on a grid, exact to the third part.
//   1/sqrt(r2): the exponent of r2 is halved apart; of its mantissa one step of
//     third order from the MUFU estimate y (error 2^-22): y (1 + h/2 + 3 h^2/8 +
//     5 h^3/16), h = 1 - r2 y^2 to 2^-68.
//   exp(-x): Tang's table-driven method (ACM TOMS 15, 1989), x = k L + f with L =
//     ln2/1024 in three floats, exp(-f) = 1 - f + f^2/2 - ... to f^5, times
//     the table's 2^(j/1024) (FP64 values, as three floats).
//
// The differences of the coordinates and r2 are taken in the same arithmetic, and
// the differences assembled for the FP64 dot products: with r2 from FP64
// differences the error of a mat-vec was FP64's (4.7e-16 at N = 8000), now it
// is a quarter of it.  The product of the normals is an integer one.
//
// About 1000 FP32 and integer instructions a pair, which run beside the pair's 21
// FP64 operations (as long as 1344) and mostly hide behind them: 23.6 of the 27.7
// billion pairs a second that 2 lanes of 152 SMs allow.  N = 7001 3.65 -> 1.06
// ms, N = 33000 65.9 -> 23.1 ms a mat-vec, where CUDA's rsqrt and exp and the
// chain after them were 57 of 87 FP64 operations (1.36 and 29.6 ms with the
// differences, r2 and the normals' product, nine more operations, in FP64; 1.16
// and 25.0 ms with the last alone).
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "df64.cuh"
#include "pair.cuh"

namespace bipb {

struct tf {
  float a, b, c;
};

__device__ __forceinline__ tf tf_mul(tf x, tf y) {
  const df p = two_prod(x.a, y.a), q = two_prod(x.a, y.b), r = two_prod(x.b, y.a);
  const float c = __fmaf_rn(x.a, y.c, __fmaf_rn(x.c, y.a, __fmaf_rn(x.b, y.b, __fadd_rn(q.lo, r.lo))));
  const df s = two_sum(q.hi, r.hi), t = two_sum(p.lo, s.hi);
  return tf{p.hi, t.hi, __fadd_rn(c, __fadd_rn(s.lo, t.lo))};
}
__device__ __forceinline__ tf tf_sqr(tf x) {
  const float a2 = __fadd_rn(x.a, x.a);
  const df p = two_prod(x.a, x.a), q = two_prod(a2, x.b);
  const df t = two_sum(p.lo, q.hi);
  return tf{p.hi, t.hi, __fadd_rn(__fmaf_rn(a2, x.c, __fmaf_rn(x.b, x.b, q.lo)), t.lo)};
}
// times a float
__device__ __forceinline__ tf tf_mul_f(tf x, float f) {
  const df p = two_prod(x.a, f), q = two_prod(x.b, f);
  const df t = two_sum(p.lo, q.hi);
  return tf{p.hi, t.hi, __fmaf_rn(x.c, f, __fadd_rn(q.lo, t.lo))};
}
__device__ __forceinline__ tf tf_scale(tf x, float pow2) {
  return tf{__fmul_rn(x.a, pow2), __fmul_rn(x.b, pow2), __fmul_rn(x.c, pow2)};
}
// x - y, normalised where the leading parts cancel
__device__ __forceinline__ tf tf_sub(tf x, tf y) {
  const df s = two_sum(x.a, -y.a), t = two_sum(x.b, -y.b), u = two_sum(s.lo, t.hi);
  const df v = fast_two_sum(s.hi, u.hi);
  const df w = two_sum(v.lo, __fadd_rn(__fsub_rn(x.c, y.c), __fadd_rn(t.lo, u.lo)));
  return tf{v.hi, w.hi, w.lo};
}
// x - y of grid coordinates (exact but for the third part's rounding).  Each part
// is zero or at least as large as the next, but where the leading ones cancel (a
// component below 2^(c-23)) it can have so few digits that the next is above its ulp:
// normalised, as every product below expects.
__device__ __forceinline__ tf tf_diff(df_pos x, df_pos y) {
  const df d = fast_two_sum(__fsub_rn(x.h, y.h), __fsub_rn(x.l, y.l));
  const df e = fast_two_sum(d.lo, __fsub_rn(x.m, y.m)), u = fast_two_sum(d.hi, e.hi);
  return tf{u.hi, u.lo, e.lo};
}
// |d|^2
__device__ __forceinline__ tf tf_norm2(tf x, tf y, tf z) {
  const float x2 = __fadd_rn(x.a, x.a), y2 = __fadd_rn(y.a, y.a), z2 = __fadd_rn(z.a, z.a);
  const df px = two_prod(x.a, x.a), py = two_prod(y.a, y.a), pz = two_prod(z.a, z.a);
  const df qx = two_prod(x2, x.b), qy = two_prod(y2, y.b), qz = two_prod(z2, z.b);
  const float cx = __fmaf_rn(x2, x.c, __fmaf_rn(x.b, x.b, qx.lo)), cy = __fmaf_rn(y2, y.c, __fmaf_rn(y.b, y.b, qy.lo)),
              cz = __fmaf_rn(z2, z.c, __fmaf_rn(z.b, z.b, qz.lo));
  const df s = two_sum(px.hi, py.hi), t = two_sum(s.hi, pz.hi);
  // the eight terms of the second order
  const df a = two_sum(qx.hi, qy.hi), b = two_sum(a.hi, qz.hi), c = two_sum(px.lo, py.lo), d = two_sum(c.hi, pz.lo),
           e = two_sum(s.lo, t.lo), f = two_sum(b.hi, d.hi), g = two_sum(f.hi, e.hi);
  const float lo = __fadd_rn(__fadd_rn(__fadd_rn(cx, cy), __fadd_rn(cz, a.lo)),
                             __fadd_rn(__fadd_rn(__fadd_rn(b.lo, c.lo), __fadd_rn(d.lo, e.lo)), __fadd_rn(f.lo, g.lo)));
  const df n = fast_two_sum(t.hi, g.hi);
  return tf{n.hi, n.lo, lo};
}
// f - x for a float f, |f| >= |x|
__device__ __forceinline__ tf tf_rsub_f(float f, tf x) {
  const df s = fast_two_sum(f, -x.a), t = two_sum(s.lo, -x.b);
  const df v = fast_two_sum(s.hi, t.hi);
  return tf{v.hi, v.lo, __fsub_rn(t.lo, x.c)};
}

// x 2^shift in FP64, rounded once, by integer operations (an FP64 addition
// costs as much as 64 instructions): the leading float truncated towards zero,
// the rest, below its ulp, rounded to the 29 bits that follow.  NORMAL: |b| is at most
// half an ulp of a.  (c may be a few ulp of b: the integer takes it with its carry or borrow.)
template <bool NORMAL = false>
__device__ __forceinline__ double tf_to_double(tf x, int shift) {
  const df n = NORMAL ? df{x.a, x.b} : fast_two_sum(x.a, x.b);
  const int sgn = __float_as_int(n.hi) & 0x80000000;
  const float h = __int_as_float(__float_as_int(n.hi) ^ sgn), m = __int_as_float(__float_as_int(n.lo) ^ sgn),
              l = __int_as_float(__float_as_int(x.c) ^ sgn);
  const int hb = __float_as_int(h) - (m < 0.f ? 1 : 0);
  const df t = two_sum(__fsub_rn(h, __int_as_float(hb)), m);  // in [0, ulp)
  const float S = __int_as_float(min(306 - (hb >> 23), 254) << 23);  // 2^29 / ulp
  const int i = __float2int_rn(__fmul_rn(t.hi, S)) + __float2int_rn(__fmul_rn(__fadd_rn(t.lo, l), S));
  const unsigned lo0 = (unsigned)hb << 29, lo = lo0 + (unsigned)i;
  // i >= 0 (a carry), or below 0 by its parts' rounding or by c (a borrow)
  const int hi = (hb >> 3) + 0x38000000 + (int)((unsigned)shift << 20) + (i >= 0 ? (lo < lo0 ? 1 : 0) : (lo > lo0 ? -1 : 0));
  return hb == 0 ? 0.0 : __hiloint2double(hi | sgn, (int)lo);
}
// the three floats of an FP64 value (host and device: constants, table)
__host__ __device__ __forceinline__ tf tf_from_double(double v) {
  const float a = (float)v;
  const float b = (float)(v - (double)a);
  return tf{a, b, (float)(v - (double)a - (double)b)};
}

// A unit normal's component as two integers, n = h 2^-27 + l 2^-54 (|l| <= 2^26).
struct fix2 {
  int h, l;
};
__device__ __forceinline__ fix2 fix2_from_double(double n) {
  const int h = __double2int_rn(n * 0x1p27);
  return fix2{h, __double2int_rn((n - h * 0x1p-27) * 0x1p54)};
}
// n_i . n_j in FP64 by integer multiply-adds (three FP64 operations are as long
// as 192 instructions): exact products to 2^-54, the last rounded away (below 2^-55).
__device__ __forceinline__ double fix2_dot(const fix2* a, const fix2* b) {
  const long long s1 = (long long)a[0].h * b[0].h + (long long)a[1].h * b[1].h + (long long)a[2].h * b[2].h;
  const long long s2 = (long long)a[0].h * b[0].l + (long long)a[0].l * b[0].h + (long long)a[1].h * b[1].l +
                       (long long)a[1].l * b[1].h + (long long)a[2].h * b[2].l + (long long)a[2].l * b[2].h;
  const long long t = s1 + ((s2 + (1ll << 26)) >> 27);  // in units of 2^-54, |t| below 2^55
  const unsigned long long u = (unsigned long long)(t < 0 ? -t : t);
  const int z = __clzll((long long)u);
  const unsigned long long m = u << z;                          // bit 63 set
  unsigned long long v = (m >> 11) + ((m >> 10) & 1ull);        // rounded to 53 bits
  v += (unsigned long long)(1031 - z) << 52;                    // the implicit bit adds one to the exponent
  if (u == 0) v = 0;
  return __longlong_as_double((long long)(v | ((unsigned long long)t & 0x8000000000000000ull)));
}

constexpr int kTfTab = kExpTab;
// ln2/1024 in three floats and 1024/ln2
constexpr float kTfL1 = 0x1.62e43p-11f, kTfL2 = -0x1.05c61p-39f, kTfL3 = -0x1.950d88p-64f, kTfInvL = 0x1.715476p+10f;
// constants of one launch: eps - 1, eps, 1/eps - 1, 1/eps; the cap of 1/r (pair.cuh) in
// the records' units, cap 2^-qcap with cap in [0.5, 1), reached below r2 = rho_cap 4^qcap
struct TfConst {
  tf em1, eps, im1, inv, cap;
  int qcap;
  float rho_cap;
};
inline void tf_set_cap(TfConst& c, double smax) {
  int e = 0;
  double m = std::frexp(smax, &e);
  if (-e < -40 || -e > 40) m = 0.5, e = -e < 0 ? 40 : -40;  // kappa below 1e-6 or above 1e18: not met
  c.cap = tf_from_double(m);
  c.qcap = -e;
  c.rho_cap = (float)(1.0 / (m * m));
}

// exp(-x) for x >= 0 (0 above 87: below 2^-125); tab[j] = 2^(j/1024)
__device__ __forceinline__ tf tf_exp_minus(tf x, const float4* tab) {
  const bool big = x.a > 87.0f;
  if (big) x = tf{87.0f, 0.f, 0.f};
  const float mg = __fmaf_rn(x.a, kTfInvL, 12582912.0f);
  const float k = __fsub_rn(mg, 12582912.0f);
  const int kk = 0x4b400000 - __float_as_int(mg);  // -k
  const float4 T = tab[kk & (kTfTab - 1)];
  const df p = two_prod(k, kTfL1), q = two_prod(k, kTfL2);
  const df s = two_sum(x.b, -p.lo), u = two_sum(s.hi, -q.hi), r = two_sum(__fsub_rn(x.a, p.hi), u.hi);
  const float r2 = __fadd_rn(r.lo, __fadd_rn(__fadd_rn(s.lo, u.lo), __fmaf_rn(-k, kTfL3, __fsub_rn(x.c, q.lo))));
  // exp(-f) - 1 = -f + f^2/2 - f^3/6 + f^4/24 - f^5/120
  const float f = r.hi;
  const df Q = two_prod(f, f);
  const float ql = __fmaf_rn(__fadd_rn(f, f), r2, Q.lo);
  const float cub = __fmaf_rn(f, __fmaf_rn(f, -1.0f / 120.0f, 1.0f / 24.0f), -1.0f / 6.0f);
  const float tail = __fmaf_rn(__fmul_rn(f, Q.hi), cub, __fmaf_rn(0.5f, ql, -r2));
  const df e0 = fast_two_sum(-f, __fmul_rn(0.5f, Q.hi));
  const float p2 = __fadd_rn(e0.lo, tail);
  const df U = two_prod(T.x, e0.hi);
  const float v = __fmaf_rn(T.x, p2, __fmaf_rn(T.y, e0.hi, U.lo));
  const df w = fast_two_sum(T.x, U.hi), g = two_sum(T.y, w.lo), g2 = two_sum(g.hi, v);
  const float sc = big ? 0.f : __int_as_float((127 + (kk >> 10)) << 23);
  return tf_scale(tf{w.hi, g2.hi, __fadd_rn(T.z, __fadd_rn(g.lo, g2.lo))}, sc);
}

// The coefficients of the kappa-scaled pair (pair.cuh) of squared distance r2 >= 0
// (s = 1/r at most its cap, kappa r = r2 s: finite at r2 = 0 and where r2 leaves the FP32 range):
//   k1 = (1 - e) s, v = (t - 1) s^3, w = (w - 3) s^5, k2 = (eps t - 1) s^3, k3 = (t / eps - 1) s^3
// LAPLACE (e = t = 1, unscaled): k2 and k3 only.
struct TfRadial {
  double k1, v, w, k2, k3;
};
template <bool LAPLACE>
__device__ __forceinline__ TfRadial tf_radial(tf r2, const TfConst& c, const float4* tab) {
  // r2 = rho 4^q, rho in [1, 4), or below where q is that of the cap
  const int q = max(((__float_as_int(r2.a) >> 23) - 127) >> 1, c.qcap);
  const tf rho = tf_scale(r2, __int_as_float((127 - 2 * q) << 23));
  // sig = 1 / sqrt(rho)
  const float y = rsqrt_approx(rho.a);
  const df p = two_prod(y, y), A = two_prod(rho.a, p.hi), B = two_prod(rho.a, p.lo), C = two_prod(rho.b, p.hi);
  const float hl = __fmaf_rn(rho.b, p.lo, __fmaf_rn(rho.c, p.hi, __fadd_rn(B.lo, C.lo)));
  const df s1 = two_sum(B.hi, C.hi), s2 = two_sum(A.lo, s1.hi);
  const df h = two_sum(__fsub_rn(1.0f, A.hi), -s2.hi);
  const float h2 = __fsub_rn(h.lo, __fadd_rn(__fadd_rn(s1.lo, s2.lo), hl));
  const float cor = __fmaf_rn(__fmul_rn(h.hi, h.hi), __fmaf_rn(0.3125f, h.hi, 0.375f), __fmul_rn(0.5f, h2));
  const df g = two_prod(y, __fmul_rn(0.5f, h.hi));
  const bool capped = q == c.qcap && rho.a < c.rho_cap;
  const tf sig = capped ? c.cap : tf{y, g.hi, __fmaf_rn(y, cor, g.lo)};
  const tf sg2 = tf_sqr(sig), sg3 = tf_mul(sg2, sig);
  TfRadial R;
  if constexpr (LAPLACE) {
    R.k1 = R.v = R.w = 0.0;
    R.k2 = tf_to_double(tf_mul(c.em1, sg3), -3 * q);
    R.k3 = tf_to_double(tf_mul(c.im1, sg3), -3 * q);
  } else {
    const int qc = max(-60, min(60, q));
    const tf kr = tf_scale(tf_mul(rho, sig), __int_as_float((127 + qc) << 23));
    const tf e = tf_exp_minus(kr, tab);
    const tf ome = tf_rsub_f(1.0f, e);
    const tf omt = tf_sub(ome, tf_mul(e, kr));  // 1 - t
    const tf vs = tf_mul(omt, sg3);
    // (w - 3) s^2 = e - 3 (1 - t) s^2
    const tf ws = tf_sub(e, tf_mul_f(tf_scale(tf_mul(omt, sg2), __int_as_float((127 - 2 * qc) << 23)), 3.0f));
    R.k1 = tf_to_double(tf_mul(ome, sig), -q);
    R.v = -tf_to_double(vs, -3 * q);
    R.w = tf_to_double(tf_mul(ws, sg3), -3 * q);
    // eps t - 1 = (eps - 1) - eps (1 - t)
    R.k2 = tf_to_double(tf_mul(tf_sub(c.em1, tf_mul(c.eps, omt)), sg3), -3 * q);
    R.k3 = tf_to_double(tf_mul(tf_sub(c.im1, tf_mul(c.inv, omt)), sg3), -3 * q);
  }
  return R;
}

// Both directions of one unordered pair (pair.cuh) from its coefficients R (0
// for a masked pair) and c_ij, 21 FP64 operations: U = (t - 1) s^3 c_ij - (w - 3) s^5 c_i c_j.
template <bool TRANS, bool LAPLACE>
__device__ __forceinline__ void sym_pair64(double dx, double dy, double dz, double cij, const double* nt, double at,
                                           double alt, const double* ns, double as, double als, const TfRadial& R,
                                           double& Pt, double& Qt, double& Ps, double& Qs) {
  const double ci = nt[0] * dx + nt[1] * dy + nt[2] * dz;
  const double cj = ns[0] * dx + ns[1] * dy + ns[2] * dz;
  if constexpr (LAPLACE) {
    if (!TRANS) {
      Pt = (R.k2 * cj) * als + Pt;
      Qt = (R.k3 * ci) * as + Qt;
      Ps = Ps - (R.k2 * ci) * alt;
      Qs = Qs - (R.k3 * cj) * at;
    } else {
      Pt = Pt - (R.k2 * ci) * as;
      Qt = Qt - (R.k3 * cj) * als;
      Ps = (R.k2 * cj) * at + Ps;
      Qs = (R.k3 * ci) * alt + Qs;
    }
  } else {
    const double U = R.v * cij - R.w * (ci * cj);
    if (!TRANS) {
      Pt = (R.k2 * cj) * als + (R.k1 * as + Pt);
      Qt = U * als + ((R.k3 * ci) * as + Qt);
      Ps = R.k1 * at - ((R.k2 * ci) * alt - Ps);
      Qs = U * alt - ((R.k3 * cj) * at - Qs);
    } else {
      Pt = U * als - ((R.k2 * ci) * as - Pt);
      Qt = R.k1 * as - ((R.k3 * cj) * als - Qt);
      Ps = U * alt + ((R.k2 * cj) * at + Ps);
      Qs = R.k1 * at + ((R.k3 * ci) * alt + Qs);
    }
  }
}

}  // namespace bipb

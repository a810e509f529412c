// Pair interactions of the centroid-collocation boundary integral operator.
//
// For a target element i (centroid x_i, unit normal n_i) and a source element
// j (centroid x_j, unit normal n_j, area ds_j), with d = x_i - x_j, r = |d|,
// s = 1/r, e = exp(-kappa r), t = e (1 + kappa r),
// w = e (3 + 3 kappa r + kappa^2 r^2), c_i = n_i.d, c_j = n_j.d,
// c_ij = n_i.n_j and eps = eps_out / eps_in, the four kernels of Sec. 2.2.1
// (Eqs. for K1-K4, with the normal derivative in x taken as +n_x.grad_x)
// are, times 4 pi:
//   K1 = (1 - e) s                      K2 = (eps t - 1) c_j s^3
//   K3 = (t / eps - 1) c_i s^3          K4 = (t - 1) c_ij s^3 - (w - 3) c_i c_j s^5
// The mat-vec of Eqs. 5-6 needs, per pair,
//   K1 ds_j psi_j + K2 ds_j phi_j   and   K3 ds_j psi_j + K4 ds_j phi_j.
// Folding the source's area and values into its record,
//   a_j = ds_j psi_j,   m_j = ds_j phi_j n_j,
// these become
//   P = s [ (1 - e) a_j + (eps t - 1) (m_j.d) s^2 ]
//   Q = s^3 [ (t/eps - 1) c_i a_j + (t - 1) (n_i.m_j) - (w - 3) c_i (m_j.d) s^2 ]
// and w - 3 = 3 (t - 1) + (t - e) kappa r.  The 1/(4 pi) and the minus sign
// are applied once per output in the reduction kernel.
//
// The self pair j = i, omitted in Eqs. 5-6, is removed by setting s = 0 for
// it (the callers pass `self` only for source tiles that overlap the thread's
// own targets, so the common path carries no mask).  Every other factor is
// finite there, so both sums receive an exact zero.  Padding records carry
// zero values and m = 0 at a far-away position, and also add exact zeros.
// 1/r is clamped to its value at 1e-6 A in every FP32 and FP64 pair, so that closer
// centroids stay finite (surface creation refuses those whose FP32 copies coincide);
// the df64 pairs (df64.cuh) have no clamp.
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"

namespace bipb {

constexpr float kSMaxF = 1.0e6f;   // 1/r is capped at its value at 1e-6 A (an overflow guard, not a model)
constexpr double kSMaxD = 1.0e6;
constexpr double kPi = 3.14159265358979323846;
constexpr double kCoulomb = 332.0716;           // Sec. 2.1: phi * 332.0716 -> kcal/mol/e
constexpr double kKcal = 4.0 * kPi * 332.0716;  // internal units (G0 carries 1/(4 pi)) -> kcal

template <typename T>
struct PairConst {
  T eps;     // eps_out / eps_in
  T inveps;  // 1 / eps
  T kappa;   // inverse Debye length
  T nkl2e;   // -kappa * log2(e), the ex2 argument scale (FP32 path)
  T smax;    // clamp of 1/r in the units of the symmetric pair (1e6 / kappa when scaled by kappa)
};

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/r (clamped; 0 for the self pair) and exp(-kappa r) for both precisions.
template <bool MASK>
__device__ __forceinline__ void radial(float r2, bool self, const PairConst<float>& c, float& s,
                                       float& r, float& e) {
  s = fminf(rsqrt_approx(r2), kSMaxF);
  if (MASK) s = self ? 0.0f : s;
  r = r2 * s;
  e = ex2_approx(r * c.nkl2e);
}
template <bool MASK>
__device__ __forceinline__ void radial(double r2, bool self, const PairConst<double>& c, double& s,
                                       double& r, double& e) {
  s = fmin(rsqrt(r2), kSMaxD);
  if (MASK) s = self ? 0.0 : s;
  r = r2 * s;
  e = exp(-c.kappa * r);
}

// Forward pair: target (x, n) gathers source (xs, a = ds psi, m = ds phi n).
template <bool MASK, typename T>
__device__ __forceinline__ void pair_forward(T xi, T yi, T zi, T nxi, T nyi, T nzi, T xj, T yj, T zj,
                                             T a, T mx, T my, T mz, bool self, const PairConst<T>& c,
                                             T& accP, T& accQ) {
  T dx = xi - xj, dy = yi - yj, dz = zi - zj;
  T r2 = dx * dx + dy * dy + dz * dz;
  T s, r, e;
  radial<MASK>(r2, self, c, s, r, e);
  T kr = r * c.kappa;
  T ci = nxi * dx + nyi * dy + nzi * dz;
  T cm = mx * dx + my * dy + mz * dz;
  T cim = nxi * mx + nyi * my + nzi * mz;
  T t = e * kr + e;
  T tm1 = t - T(1);
  T wm3 = (t - e) * kr + T(3) * tm1;
  T s2 = s * s;
  // P = s [ (1 - e) a + (eps t - 1) cm s^2 ]
  T p = a - e * a;
  p = ((c.eps * t - T(1)) * cm) * s2 + p;
  accP = p * s + accP;
  // Q = s^3 [ (t/eps - 1) ci a + (t - 1) cim - (w - 3) ci cm s^2 ]
  T q = ((t * c.inveps - T(1)) * ci) * a;
  q = tm1 * cim + q;
  q = q - wm3 * ((ci * cm) * s2);
  accQ = q * (s2 * s) + accQ;
}

// Transposed pair: output element j (x, n) gathers element i (xs, wphi, p = wpsi n_i),
// d = x_i - x_j:
//   Zphi = s^3 [ (eps t - 1) c_j wphi + (t - 1) (n_j.p) - (w - 3) (p.d) c_j s^2 ]
//   Zpsi = s [ (1 - e) wphi + (t/eps - 1) (p.d) s^2 ]
// (K2 and K4 gathered into the phi output, K1 and K3 into the psi output; the
// output element's area ds_j is applied in the reduction.)
template <bool MASK, typename T>
__device__ __forceinline__ void pair_transpose(T xj, T yj, T zj, T nxj, T nyj, T nzj, T xi, T yi, T zi,
                                               T wphi, T px, T py, T pz, bool self,
                                               const PairConst<T>& c, T& accP, T& accQ) {
  T dx = xi - xj, dy = yi - yj, dz = zi - zj;
  T r2 = dx * dx + dy * dy + dz * dz;
  T s, r, e;
  radial<MASK>(r2, self, c, s, r, e);
  T kr = r * c.kappa;
  T cj = nxj * dx + nyj * dy + nzj * dz;
  T cp = px * dx + py * dy + pz * dz;
  T cnp = nxj * px + nyj * py + nzj * pz;
  T t = e * kr + e;
  T tm1 = t - T(1);
  T wm3 = (t - e) * kr + T(3) * tm1;
  T s2 = s * s;
  T q = ((c.eps * t - T(1)) * cj) * wphi;
  q = tm1 * cnp + q;
  q = q - wm3 * ((cp * cj) * s2);
  accP = q * (s2 * s) + accP;
  T p = wphi - e * wphi;
  p = ((t * c.inveps - T(1)) * cp) * s2 + p;
  accQ = p * s + accQ;
}

// ------------------------------------------------------------------ symmetric pairs
// The four kernels depend on the pair through r, e, t, w (symmetric in i and
// j) and through c_i = n_i.d, c_j = n_j.d, c_ij = n_i.n_j (d = x_i - x_j, so
// d_ji = -d).  A kernel that visits the unordered pair {i, j} once computes
// them once and applies them in both directions.  With each element's record
// holding its normal, write m = alpha n (alpha = ds phi for A u; for A^T w
// the record's second field p = beta n with beta = wpsi): then m_j.d =
// alpha_j c_j, n_i.m_j = alpha_j c_ij, and both directions share
//   U = (t - 1) c_ij - (w - 3) s^2 c_i c_j.
// A u (a = ds psi):
//   P_i += s [ (1 - e) a_j + (eps t - 1) s^2 alpha_j c_j ]
//   Q_i += s^3 [ (t/eps - 1) c_i a_j + alpha_j U ]
//   P_j += s [ (1 - e) a_i - (eps t - 1) s^2 alpha_i c_i ]
//   Q_j += s^3 [ -(t/eps - 1) c_j a_i + alpha_i U ]
// A^T w (a = wphi; the phi output gathers K2, K4, the psi output K1, K3):
//   Zphi_i += s^3 [ -(eps t - 1) c_i a_j + beta_j U ]
//   Zpsi_i += s [ (1 - e) a_j - (t/eps - 1) s^2 beta_j c_j ]
//   Zphi_j += s^3 [ (eps t - 1) c_j a_i + beta_i U ]
//   Zpsi_j += s [ (1 - e) a_i + (t/eps - 1) s^2 beta_i c_i ]
// (t = target i of the thread, s = source j; P/Q the two outputs of each.)
// Two forms, chosen per launch:
// - SCALED (kappa > 0): positions are multiplied by kappa when the records
//   are packed, so d, r and s are in units of the Debye length; then
//   kappa r = r2 s and (w - 3) s^2 = 3 (t - 1) s^2 + e (with r s = 1).  The
//   kernels scale as K1 ~ kappa, K2, K3 ~ kappa^2, K4 ~ kappa^3, a product of
//   a row factor and a column factor: the records' alpha is multiplied by
//   kappa as well, and the caller multiplies the sums (A u: P by kappa, Q by
//   kappa^2; A^T w: P by kappa^2, Q by kappa).
// - LAPLACE (kappa = 0, unscaled): e = t = 1, w = 3, so K1 = K4 = 0 and only
//   the double-layer terms (eps - 1) c_j s^3 and (1/eps - 1) c_i s^3 remain.

// The symmetric pair in FP32 for two targets t (packed) and one source s (every
// value in both halves), the formulas above with signs placed so that no
// packed operand needs a negation: 1 - t for t - 1, -U, -(eps t - 1) s^3 and
// -(t/eps - 1) s^3, and in scaled units (1 - e) s = (1 - t) s + e (kappa r s =
// 1).  ft: a, -alpha and alpha (A u) or -a (A^T w) of the targets; fs: a,
// -alpha and -a (A u) or alpha (A^T w) of the source.  A masked pair has s = e = 0.
template <bool MASK, bool TRANS, bool LAPLACE>
__device__ __forceinline__ void sym_pair2(const f2* xt, const f2* nt, const f2* ft, const f2* xs, const f2* ns,
                                          const f2* fs, bool m0, bool m1, const PairConst<float>& c, f2& Pt, f2& Qt,
                                          f2& Ps, f2& Qs) {
  const f2 dx = f2_sub(xt[0], xs[0]), dy = f2_sub(xt[1], xs[1]), dz = f2_sub(xt[2], xs[2]);
  const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
  float ra, rb;
  f2_get(r2, ra, rb);
  float sa = fminf(rsqrt_approx(ra), c.smax), sb = fminf(rsqrt_approx(rb), c.smax);
  if (MASK) sa = m0 ? 0.f : sa, sb = m1 ? 0.f : sb;
  const f2 s = f2_make(sa, sb);
  const f2 ci = f2_fma(nt[0], dx, f2_fma(nt[1], dy, f2_mul(nt[2], dz)));
  const f2 cj = f2_fma(ns[0], dx, f2_fma(ns[1], dy, f2_mul(ns[2], dz)));
  const f2 s2 = f2_mul(s, s), s3 = f2_mul(s2, s);
  if constexpr (LAPLACE) {
    const f2 E = f2_mul(f2_splat(1.f - c.eps), s3), F = f2_mul(f2_splat(1.f - c.inveps), s3);
    const f2 A = f2_mul(E, cj), B = f2_mul(F, ci), C = f2_mul(E, ci), D = f2_mul(F, cj);
    Pt = TRANS ? f2_fma(C, fs[0], Pt) : f2_fma(A, fs[1], Pt);
    Qt = TRANS ? f2_fma(D, fs[2], Qt) : f2_fma(B, fs[2], Qt);
    Ps = TRANS ? f2_fma(A, ft[2], Ps) : f2_fma(C, ft[2], Ps);
    Qs = TRANS ? f2_fma(B, ft[1], Qs) : f2_fma(D, ft[0], Qs);
  } else {
    const f2 kr = f2_mul(r2, s);
    float ea, eb;
    f2_get(f2_mul(kr, f2_splat(-1.4426950408889634f)), ea, eb);
    ea = ex2_approx(ea), eb = ex2_approx(eb);
    if (MASK) ea = m0 ? 0.f : ea, eb = m1 ? 0.f : eb;
    const f2 e = f2_make(ea, eb);
    const f2 t = f2_fma(e, kr, e);
    const f2 omt = f2_sub(f2_splat(1.f), t);
    const f2 w = f2_fma(omt, f2_mul(f2_splat(-3.f), s2), e);  // (w - 3) s^2
    const f2 cij = f2_fma(nt[0], ns[0], f2_fma(nt[1], ns[1], f2_mul(nt[2], ns[2])));
    const f2 V = f2_mul(f2_fma(w, f2_mul(ci, cj), f2_mul(omt, cij)), s3);  // -U s^3
    const f2 K1 = f2_fma(omt, s, e);
    const f2 ts3 = f2_mul(t, s3);
    const f2 E = f2_fma(f2_splat(-c.eps), ts3, s3), F = f2_fma(f2_splat(-c.inveps), ts3, s3);
    const f2 A = f2_mul(E, cj), B = f2_mul(F, ci), C = f2_mul(E, ci), D = f2_mul(F, cj);
    if (!TRANS) {
      Pt = f2_fma(A, fs[1], f2_fma(K1, fs[0], Pt));
      Qt = f2_fma(V, fs[1], f2_fma(B, fs[2], Qt));
      Ps = f2_fma(C, ft[2], f2_fma(K1, ft[0], Ps));
      Qs = f2_fma(V, ft[1], f2_fma(D, ft[0], Qs));
    } else {
      Pt = f2_fma(V, fs[1], f2_fma(C, fs[0], Pt));
      Qt = f2_fma(K1, fs[0], f2_fma(D, fs[2], Qt));
      Ps = f2_fma(V, ft[1], f2_fma(A, ft[2], Ps));
      Qs = f2_fma(K1, ft[0], f2_fma(B, ft[1], Qs));
    }
  }
}

// ------------------------------------------------------------------ kernel blocks
// The four kernel values of pair (target i, source j) times ds_j (times 4 pi),
// in FP32: returns (K2, K1) in v[0], v[1] and (K4, K3) in v[2], v[3].
// TRANS: the block of A^T instead, output element i gathering input element
// j (pair_transpose of pair.cuh with d = x_i - x_j): the phi row (K2_ji,
// K4_ji) in v[0], v[1], the psi row (K1_ji, K3_ji) in v[2], v[3], times the
// record's area field (the output's area is applied to the sums), i.e.
// ((1 - eps t) c_i s^3, K4, (1 - e) s, (1 - t/eps) c_j s^3).
// SCALED: positions, area and normal in kappa-scaled units (k_tc_colmax,
// mrhs_tc.cu: kappa r = r2 s and (w - 3) s^2 = 3 (t - 1) s^2 + e; one row
// comes out with an extra power of kappa); c.nkl2e and c.smax are then
// -log2(e) and the 1/r cap in those units.
template <bool SCALED, bool TRANS>
__device__ __forceinline__ void kernel_block(float xi, float yi, float zi, float nxi, float nyi, float nzi, float4 g,
                                             float4 nv, bool zero, const PairConst<float>& c, float* v) {
  const float dx = xi - g.x, dy = yi - g.y, dz = zi - g.z;
  const float r2 = dx * dx + dy * dy + dz * dz;
  float s = fminf(rsqrt_approx(r2), c.smax);
  s = zero ? 0.f : s;
  const float r = r2 * s;
  const float e = ex2_approx(r * c.nkl2e);
  const float kr = SCALED ? r : r * c.kappa;
  const float ci = nxi * dx + nyi * dy + nzi * dz;
  const float cj = nv.x * dx + nv.y * dy + nv.z * dz;
  const float cij = nxi * nv.x + nyi * nv.y + nzi * nv.z;
  const float t = e * kr + e;
  const float tm1 = t - 1.f;
  const float sa = s * g.w;
  const float s2 = s * s;
  const float s3a = s2 * sa;
  // (w - 3) s^2
  const float wm3s2 = SCALED ? (3.f * tm1) * s2 + e : ((t - e) * kr + 3.f * tm1) * s2;
  const float k4 = (tm1 * cij - wm3s2 * (ci * cj)) * s3a;
  if (!TRANS) {
    v[1] = sa - e * sa;                                  // K1 ds = (1 - e) s ds
    v[0] = ((c.eps * t - 1.f) * cj) * s3a;               // K2 ds
    v[3] = ((t * c.inveps - 1.f) * ci) * s3a;            // K3 ds
    v[2] = k4;                                           // K4 ds
  } else {
    v[0] = ((1.f - c.eps * t) * ci) * s3a;               // K2_ji
    v[1] = k4;                                           // K4_ji
    v[2] = sa - e * sa;                                  // K1_ji
    v[3] = ((1.f - t * c.inveps) * cj) * s3a;            // K3_ji
  }
}

}  // namespace bipb

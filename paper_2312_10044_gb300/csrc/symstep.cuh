// Device pieces of the symmetric mat-vec shared by its own pack and reduction
// kernels (sym.cu) and by the Krylov step that fuses them (gmres.cu).
#pragma once
#include "internal.cuh"

namespace bipb {

// Running sum of per-tile partial sums.  FP64 partials: FP64.  FP32 partials:
// a df64 sum on the FP32 pipe (TwoSum, the errors added up), exact to about
// 2^-48 of the sum, far below the partials' own 2^-24: GB300 has two FP64 lanes
// per SM, and converting and adding each FP32 partial in FP64 took most of a
// small system's Krylov step (34 us of 42 at N = 1280).
template <typename PT>
struct PartSum;
template <>
struct PartSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct PartSum<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    const df t = two_sum(hi, v);
    hi = t.hi;
    lo = __fadd_rn(lo, t.lo);
  }
  // of an infinite sum the TwoSum errors are NaN and the leading part is the sum
  __device__ __forceinline__ double value() const { return lo == lo ? (double)hi + (double)lo : (double)hi; }
};

// Sum of component c (0: phi, 1: psi) of one element of a system over a
// symmetric pass's partial sums: the i-side blocks of the element's row, then
// the j-side values of rows 0..E, in that order.  S = {n, first row entry,
// j-side base, T} of the system; tab[S.y + E] = {first i-side block, blocks, 0, 0}.
template <typename PT>
__device__ __forceinline__ double sym_sum(const int4* __restrict__ tab, const int4 S, const PT* __restrict__ part,
                                          int e, int c) {
  const int n = S.x, T = S.w, E = e / T;
  const int4 R = tab[S.y + E];
  PartSum<PT> p;
  const PT* b = part + (size_t)R.x + (size_t)c * T + (e - E * T);
#pragma unroll 16
  for (int k = 0; k < R.y; ++k) p.add(b[(size_t)k * 2 * T]);
  // row I starts at S.z + 2 (I n - T I (I - 1) / 2): element e of it at e - I T
#pragma unroll 8
  for (int I = 0; I <= E; ++I) {
    const PT* r = part + (int64_t)S.z + 2 * ((int64_t)I * n - (int64_t)T * I * (I - 1) / 2) + (e - I * T);
    p.add(r[c * (n - I * T)]);
  }
  return p.value();
}

// The FP32 record of one element (Sym32Policy, sym.cu) from its geometry g, v
// and its values phi, psi of the mat-vec's input.
__device__ __forceinline__ void sym32_record(const double4_32a& g, const double4_32a& v, double phi, double psi,
                                             bool transpose, double sigma, float4* __restrict__ o) {
  const float a = (float)(transpose ? phi : g.w * psi);
  const float al = (float)(sigma * (transpose ? psi : g.w * phi));
  const float x = (float)(sigma * g.x), y = (float)(sigma * g.y), z = (float)(sigma * g.z);
  const float nx = (float)v.x, ny = (float)v.y, nz = (float)v.z, f = transpose ? al : -a;
  o[0] = make_float4(x, x, y, y);
  o[1] = make_float4(z, z, a, a);
  o[2] = make_float4(nx, nx, ny, ny);
  o[3] = make_float4(nz, nz, -al, -al);
  o[4] = make_float4(f, f, 0.f, 0.f);
}

// The same when the record already holds this element's geometry: the fields
// a, -alpha and f only.
__device__ __forceinline__ void sym32_refresh(double area, double phi, double psi, bool transpose, double sigma,
                                              float4* __restrict__ o) {
  const float a = (float)(transpose ? phi : area * psi);
  const float al = (float)(sigma * (transpose ? psi : area * phi));
  const float f = transpose ? al : -a;
  reinterpret_cast<float2*>(o)[3] = make_float2(a, a);
  reinterpret_cast<float2*>(o)[7] = make_float2(-al, -al);
  reinterpret_cast<float2*>(o)[8] = make_float2(f, f);
}

}  // namespace bipb

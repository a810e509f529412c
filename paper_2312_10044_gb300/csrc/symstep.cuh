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
// A sum of FP32 values may leave their range although each of them is in it: the sum is
// then taken again in FP64 (also of infinities and NaN).
__device__ __forceinline__ bool left_range(const PartSum<double>&) { return false; }
__device__ __forceinline__ bool left_range(const PartSum<float>& p) { return !(fabsf(p.hi) <= 3.402823466e38f); }
template <typename PT>
__device__ __forceinline__ double sum_strided_fp64(const PT* __restrict__ p, size_t stride, int count) {
  double t = 0.0;
#pragma unroll 1
  for (int k = 0; k < count; ++k) t += (double)p[(size_t)k * stride];
  return t;
}

// Sum of count values stride apart, in order, U loads in flight at a time: the last
// batch is filled up with zeros, where a loop unrolled by U would leave up to U - 1
// values to a rolled remainder that waits for each load in turn.  (A guard around
// each addition lets the compiler move the load behind it, which is as slow.)
template <int U, typename PT>
__device__ __forceinline__ PartSum<PT> sum_strided(const PT* __restrict__ p, size_t stride, int count) {
  PartSum<PT> acc;
  for (int k = 0; k < count; k += U) {
    PT v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) v[q] = k + q < count ? p[(size_t)(k + q) * stride] : PT(0);
#pragma unroll
    for (int q = 0; q < U; ++q) acc.add(v[q]);
  }
  return acc;
}

// sym_sum in FP64
template <typename PT>
__device__ __noinline__ double sym_sum_fp64(const int4* __restrict__ tab, const int4 S, const PT* __restrict__ part,
                                            int e, int c) {
  const int n = S.x, T = S.w, E = e / T;
  const int4 R = tab[S.y + E];
  double t = sum_strided_fp64(part + (size_t)R.x + (size_t)c * T + (e - E * T), (size_t)2 * T, R.y);
#pragma unroll 1
  for (int I = 0; I <= E; ++I)
    t += (double)part[(int64_t)S.z + 2 * ((int64_t)I * n - (int64_t)T * I * (I - 1) / 2) + (e - I * T) + c * (n - I * T)];
  return t;
}

// Sum of component c (0: phi, 1: psi) of one element of a system over a
// symmetric pass's partial sums: the i-side blocks of the element's row, then
// the j-side values of rows 0..E, in that order.  S = {n, first row entry,
// j-side base, T} of the system; tab[S.y + E] = {first i-side block, blocks, 0, 0}.
template <typename PT>
__device__ __forceinline__ double sym_sum(const int4* __restrict__ tab, const int4 S, const PT* __restrict__ part,
                                          int e, int c) {
  const int n = S.x, T = S.w, E = e / T;
  const int4 R = tab[S.y + E];
  PartSum<PT> p = sum_strided<sizeof(PT) == 4 ? 24 : 8>(part + (size_t)R.x + (size_t)c * T + (e - E * T), (size_t)2 * T, R.y);
  // row I starts at S.z + 2 (I n - T I (I - 1) / 2): element e of it at e - I T
  constexpr int U = sizeof(PT) == 4 ? 8 : 4;
  for (int I0 = 0; I0 <= E; I0 += U) {
    PT v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int I = I0 + q;
      const int64_t o = (int64_t)S.z + 2 * ((int64_t)I * n - (int64_t)T * I * (I - 1) / 2) + (e - I * T);
      v[q] = I <= E ? part[o + c * (n - I * T)] : PT(0);
    }
#pragma unroll
    for (int q = 0; q < U; ++q) p.add(v[q]);
  }
  if (left_range(p)) return sym_sum_fp64(tab, S, part, e, c);
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

// Far-field (treecode) FP32 mat-vec of Eqs. 5-6, after Sec. 2.2.3.
//
// The mat-vec is an N-body sum per target over sources carrying
// a_j = ds_j psi_j and m_j = ds_j phi_j n_j (K2 and K4 are linear in the
// source normal, so m_j carries it).  The transpose A^T w is the same kind of
// sum: output element t gathers column t of A, whose entries of row element
// j depend on n_j only through K3 and K4, linearly, so the sources carry
// a_j = wphi_j and m_j = wpsi_j n_j, the pair is the transposed one
// (tree_pair2) and the output element's area multiplies the
// sums.  The tree, the lists and the proxies serve both directions.  The elements form a binary tree of
// clusters; a cluster holding more than `leaf` elements is split in two at
// the median of its longest box side (ties by element index), so every
// cluster is one range of element positions in tree order.  Targets are
// taken leaf by leaf: for target leaf B a cluster c is far when
//   r_c + theta r_B <= theta |x_B - x_c|
// (box centres, half box diagonals), which implies the paper's acceptance
// criterion r_c / |x - x_c| <= theta for every target of B.  Traversal from
// the root gives each leaf a list of source ranges:
//   far c with more elements than proxies -> the (p+1)^3 proxy sources of c,
//   far c otherwise, or a near leaf       -> c's elements (summed directly),
//   a near cluster                        -> its two children.
// A proxy source sits at a Chebyshev point s_k of c's box and carries
//   a_k = sum_{j in c} L_k(x_j) a_j,   m_k = sum_{j in c} L_k(x_j) m_j
// with L_k the tensor-product Lagrange basis of degree p per coordinate
// (barycentric form): a degree-p polynomial in the source position stands in
// for the kernel over a far cluster, as the Taylor series about the cluster
// centre does in the paper.  Because proxies and elements are records of the
// same form (position, a, m), every list entry is summed by the one ordered
// pair formula (tree_pair2) and the far-field pass has the shape
// of the direct pass.
//
// One mat-vec is five launches on the handle's stream:
//   k_tree_pack   element records in tree order (gathered through perm);
//   k_tree_up     partial proxy weights, one CTA per piece of <= 512
//                 elements of a far cluster (FP32 runs of 32 elements, TwoSums across);
//   k_tree_proxy  proxy records (pieces added in order, TwoSums);
//   k_tree_far    one CTA per work item: a target leaf (one target per thread)
//                 against a run of its list's records, streamed through shared
//                 memory; FP32 partial sums per item;
//   k_tree_reduce per target, its leaf's items in order (TwoSums), 1/(4 pi) and
//                 the diagonal, scattered back to element order.
// Every sum is in a fixed order, so the pass is bitwise reproducible.
#include <algorithm>
#include <cmath>
#include <numeric>

#include "internal.cuh"
#include "symstep.cuh"

namespace bipb {

namespace {

constexpr double kInv4PiT = 1.0 / (4.0 * kPi);
constexpr int kUpPiece = 512;  // elements per piece of the upward pass
constexpr int kUpRun = 32;      // elements per FP32 run of the upward pass
constexpr int kFarCH = 512;     // records per shared-memory chunk of the far-field kernel
constexpr int kMaxLeaf = 512;
constexpr int kFarMinB = 2;     // resident CTAs of kMaxLeaf threads the far-field kernel's registers allow

__device__ __forceinline__ bool tree_skipped(const int* skip, int stride, int sys) {
  return skip != nullptr && skip[(size_t)sys * stride] != 0;
}

// ------------------------------------------------------------------ kernels
// rec[k][t] = (sigma x, a = ds psi), (m = sigma ds phi n, 0) of element perm[t],
// system k; transposed: a = wphi, m = sigma wpsi n.  sigma: see tree_pair2.
__global__ void k_tree_pack(int n, int rec_stride, bool transpose, double sigma, const int* __restrict__ perm,
                            const double4_32a* __restrict__ tgt64, const int4* __restrict__ lay,
                            const double* __restrict__ u, float4* __restrict__ rec, const int* __restrict__ skip,
                            int skip_stride) {
  const int k = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n || tree_skipped(skip, skip_stride, k)) return;
  const int4 L = lay[k];
  const int e = perm[t];
  const double4_32a g = tgt64[2 * (L.x + e)], v = tgt64[2 * (L.x + e) + 1];
  const double phi = u[L.z + e], psi = u[L.z + L.y + e];
  const double a = transpose ? phi : g.w * psi, f = sigma * (transpose ? psi : g.w * phi);
  const size_t o = 2 * ((size_t)k * rec_stride + t);
  rec[o] = make_float4((float)(sigma * g.x), (float)(sigma * g.y), (float)(sigma * g.z), (float)a);
  rec[o + 1] = make_float4((float)(f * v.x), (float)(f * v.y), (float)(f * v.z), 0.f);
}

// Partial proxy weights of one piece of a far cluster: for proxy q = (q0, q1, q2),
//   upart[.][q] = sum over the piece's elements of l_q0(x) l_q1(y) l_q2(z) (a, m),
// with l_i the barycentric Lagrange basis at the cluster's Chebyshev nodes
// (weights (-1)^i, halved at both ends).  An element whose FP32 record is on a node
// takes the node's basis value 1 exactly; in kappa-scaled units node and element are
// rounded apart, and one on a node may come out an ulp beside it (its basis value then
// differs from 1 by that ulp's share of the node spacing: the error of the
// mat-vec is the same with nodes scaled in FP64).
//
// Bound by the FP32 pipe: thread (g, q0, q1) of G groups adds every G-th
// element of a chunk to its column of DEG + 1 proxies, one multiplication and
// four multiply-adds (two packed) each, so the product of the first two basis
// values and the loads are shared by the column.  FP32 over 32 elements, the
// runs and the groups by TwoSums (PartSum); upart holds (sum, trailing part).
// At N = 120001, degree 6, 0.10 ms; one proxy per thread with FP64 sums took
// 0.29 ms.
template <int DEG>
struct UpShape {
  static constexpr int NP = DEG + 1, P = NP * NP * NP, Q = NP * NP;
  static constexpr int NT = 256, G = NT / Q;  // groups of elements
  static constexpr int CH = kUpRun * G;       // elements staged at once
  static constexpr int NB = (NP + 3) / 4 * 4;
};
template <int DEG>
__global__ void __launch_bounds__(256) k_tree_up(const int4* __restrict__ pieces, const float* __restrict__ nodes,
                                                 float sigma, int rec_stride, const float4* __restrict__ rec,
                                                 float2* __restrict__ upart, int n_pieces,
                                                 const int* __restrict__ skip, int skip_stride) {
  using U = UpShape<DEG>;
  constexpr int NP = U::NP, P = U::P, G = U::G, CH = U::CH, NB = U::NB;
  __shared__ __align__(16) float bas[CH][3][NB];
  __shared__ float4 val[CH];
  __shared__ float nd[3][NP];
  __shared__ float2 comb[G * P];
  const int k = blockIdx.y;
  if (tree_skipped(skip, skip_stride, k)) return;
  const int4 pc = pieces[blockIdx.x];  // {slot, first position, count, 0}
  const int tid = threadIdx.x;
  if (tid < 3 * NP) nd[tid / NP][tid % NP] = sigma * nodes[(size_t)pc.x * 3 * NP + tid];
  const int g = tid / U::Q, q01 = tid % U::Q, q0 = q01 / NP, q1 = q01 % NP;  // g == G: idle
  PartSum<float> acc[NP][4];
  const float4* R = rec + 2 * (size_t)k * rec_stride;
  for (int c0 = 0; c0 < pc.z; c0 += CH) {
    const int cnt = min(CH, pc.z - c0);
    __syncthreads();  // nodes staged; the previous chunk consumed
    for (int q = tid; q < 3 * cnt; q += U::NT) {  // basis values of element q / 3 along coordinate q % 3
      const int e = q / 3, d = q % 3;
      const size_t o = 2 * (size_t)(pc.y + c0 + e);
      const float4 r0 = R[o];
      if (d == 0) {
        const float4 r1 = R[o + 1];
        val[e] = make_float4(r0.w, r1.x, r1.y, r1.z);
      }
      const float t = d == 0 ? r0.x : (d == 1 ? r0.y : r0.z);
      float w[NP];
      float sum = 0.f;
      int hit = -1;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const float diff = t - nd[d][i];
        const float wi = ((i & 1) ? -1.f : 1.f) * ((i == 0 || i == DEG) ? 0.5f : 1.f);
        if (fabsf(diff) < 1e-30f) hit = i;
        w[i] = wi / diff;
        sum += w[i];
      }
      const float inv = 1.f / sum;
#pragma unroll
      for (int i = 0; i < NP; ++i) bas[e][d][i] = hit >= 0 ? (i == hit ? 1.f : 0.f) : w[i] * inv;
    }
    __syncthreads();
    if (g < G) {
      f2 sa[NP], sm[NP];  // (a, mx), (my, mz)
#pragma unroll
      for (int i = 0; i < NP; ++i) sa[i] = sm[i] = f2_splat(0.f);
#pragma unroll 2
      for (int e = g; e < cnt; e += G) {
        const float4 v = val[e];
        const f2 va = f2_make(v.x, v.y), vm = f2_make(v.z, v.w);
        const float w01 = bas[e][0][q0] * bas[e][1][q1];
        float b2[NB];
#pragma unroll
        for (int i = 0; i < NB; i += 4) *reinterpret_cast<float4*>(b2 + i) = *reinterpret_cast<float4*>(&bas[e][2][i]);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const f2 w = f2_splat(w01 * b2[i]);
          sa[i] = f2_fma(w, va, sa[i]);
          sm[i] = f2_fma(w, vm, sm[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        float x, y;
        f2_get(sa[i], x, y);
        acc[i][0].add(x), acc[i][1].add(y);
        f2_get(sm[i], x, y);
        acc[i][2].add(x), acc[i][3].add(y);
      }
    }
  }
  // the groups in order, one component at a time
  float2* o = upart + 4 * (size_t)(k * n_pieces + blockIdx.x) * P;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    __syncthreads();
    if (g < G)
#pragma unroll
      for (int i = 0; i < NP; ++i) comb[g * P + q01 * NP + i] = make_float2(acc[i][c].hi, acc[i][c].lo);
    __syncthreads();
    for (int q = tid; q < P; q += U::NT) {
      PartSum<float> t;
      for (int x = 0; x < G; ++x) t.add(comb[x * P + q].x), t.lo += comb[x * P + q].y;
      o[c * P + q] = make_float2(t.hi, t.lo);
    }
  }
}

// Proxy records after the element records: (sigma s_q, a_q), (m_q, 0), the
// pieces of the slot's cluster added in order.
template <int DEG>
__global__ void k_tree_proxy(int n_slots, const int2* __restrict__ up_tab, const float* __restrict__ nodes, float sigma,
                             const float2* __restrict__ upart, int n_pieces, int n, int rec_stride,
                             float4* __restrict__ rec, const int* __restrict__ skip, int skip_stride) {
  constexpr int NP = DEG + 1, P = NP * NP * NP;
  const int k = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_slots * P || tree_skipped(skip, skip_stride, k)) return;
  const int slot = idx / P, kp = idx % P;
  const int k0 = kp / (NP * NP), k1 = (kp / NP) % NP, k2 = kp % NP;
  const int2 T = up_tab[slot];
  PartSum<float> s[4];
#pragma unroll 4
  for (int p = T.x; p < T.x + T.y; ++p) {
    const float2* v = upart + 4 * (size_t)(k * n_pieces + p) * P + kp;
#pragma unroll
    for (int c = 0; c < 4; ++c) s[c].add(v[c * P].x), s[c].lo += v[c * P].y;
  }
  const float* nd = nodes + (size_t)slot * 3 * NP;
  const size_t o = 2 * ((size_t)k * rec_stride + n + idx);
  rec[o] = make_float4(sigma * nd[k0], sigma * nd[NP + k1], sigma * nd[2 * NP + k2], s[0].hi + s[0].lo);
  rec[o + 1] = make_float4(s[1].hi + s[1].lo, s[2].hi + s[2].lo, s[3].hi + s[3].lo, 0.f);
}

// Two source records (packed) added to one target: S1 += s [(1 - e) a + E s^2
// (m.d)], S3 += s^3 [(1 - t) (n.m) + (n.d) ((w - 3) s^2 (m.d) + F a)] with d =
// target - source, which are the two outputs of both directions (pair.cuh):
//   A u:   E = eps t - 1, F = 1 - t / eps;  phi = S1, psi = -S3;
//   A^T w: E = 1 - t / eps, F = eps t - 1;  phi = -S3, psi = S1
// (d changes its sign against pair_transpose, hence E and F).  The formulas
// are placed so that no packed operand needs a negation (two logical
// operations each).  FORM:
//   kScaled (kappa >= kScaledKappaMin): positions and m times sigma = kappa, where kappa r
//     = r2 s, (1 - e) s = (1 - t) s + e and (w - 3) s^2 = 3 (t - 1) s^2 + e;
//     the sums take factors of kappa (S1) and kappa^2 (S3);
//   kPlain (0 < kappa below that): sigma = 1;
//   kLaplace (kappa = 0): e = t = 1, w = 3, only E and F remain.
enum TreeForm { kScaled, kPlain, kLaplace };
struct TreeConst {
  float ef, e0, ff, f0;  // E = ef t + e0, F = ff t + f0
  float kappa, smax;     // smax in the units of the positions
};
struct TreeTarget {
  f2 x[3], n[3];
};
template <TreeForm FORM, bool MASK>
__device__ __forceinline__ void tree_pair2(const TreeTarget& T, const f2* R, bool m0, bool m1, const TreeConst& c,
                                           f2& S1, f2& S3) {
  const f2 dx = f2_sub(T.x[0], R[0]), dy = f2_sub(T.x[1], R[1]), dz = f2_sub(T.x[2], R[2]);
  const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
  float sa, sb;
  f2_get(r2, sa, sb);
  sa = fminf(rsqrt_approx(sa), c.smax), sb = fminf(rsqrt_approx(sb), c.smax);
  if (MASK) sa = m0 ? 0.f : sa, sb = m1 ? 0.f : sb;
  const f2 s = f2_make(sa, sb);
  const f2 a = R[3];
  const f2 cd = f2_fma(T.n[0], dx, f2_fma(T.n[1], dy, f2_mul(T.n[2], dz)));  // n.d
  const f2 cm = f2_fma(R[4], dx, f2_fma(R[5], dy, f2_mul(R[6], dz)));        // m.d
  const f2 s2 = f2_mul(s, s), s3 = f2_mul(s2, s);
  if constexpr (FORM == kLaplace) {
    S1 = f2_fma(f2_mul(f2_splat(c.ef + c.e0), s3), cm, S1);
    S3 = f2_fma(f2_mul(f2_splat(c.ff + c.f0), s3), f2_mul(cd, a), S3);
  } else {
    const f2 cnm = f2_fma(T.n[0], R[4], f2_fma(T.n[1], R[5], f2_mul(T.n[2], R[6])));  // n.m
    const f2 r = f2_mul(r2, s);
    const f2 kr = FORM == kScaled ? r : f2_mul(r, f2_splat(c.kappa));
    float ea, eb;
    f2_get(f2_mul(kr, f2_splat(-1.4426950408889634f)), ea, eb);
    ea = ex2_approx(ea), eb = ex2_approx(eb);
    if (MASK) ea = m0 ? 0.f : ea, eb = m1 ? 0.f : eb;
    const f2 e = f2_make(ea, eb);
    const f2 t = f2_fma(e, kr, e);
    const f2 omt = f2_sub(f2_splat(1.f), t);
    f2 w, k1;  // (w - 3) s^2, (1 - e) s
    if constexpr (FORM == kScaled) {
      w = f2_fma(omt, f2_mul(f2_splat(-3.f), s2), e);
      k1 = f2_fma(omt, s, e);
    } else {
      w = f2_mul(f2_fma(f2_sub(t, e), kr, f2_mul(f2_splat(-3.f), omt)), s2);
      k1 = f2_sub(s, f2_mul(e, s));
    }
    const f2 E = f2_fma(f2_splat(c.ef), t, f2_splat(c.e0)), F = f2_fma(f2_splat(c.ff), t, f2_splat(c.f0));
    S1 = f2_fma(f2_mul(E, s3), cm, f2_fma(k1, a, S1));
    S3 = f2_fma(f2_fma(cd, f2_fma(w, cm, f2_mul(F, a)), f2_mul(omt, cnm)), s3, S3);
  }
}

// One work item: the targets of one leaf (thread t: position lf.x + t) against
// the records of segments [it.y, it.z).  The self pair is masked in the
// segments that overlap the leaf's own positions.
//
// Bound by the FP32 pipe: records are staged with the values of two
// consecutive ones side by side (an odd end padded by a record without
// strength), so each thread evaluates two pairs by 34 packed instructions, 18
// of them multiply-adds (three register operands, which take half as long
// again): 43 cycles a warp and source by that count, 47 measured (the scalar
// unscaled pair took 53).  At N = 120001 the pass takes 3.13 ms (3.92 before);
// the records of a chunk (512 against 256) and the unroll (2 against 4 and 8)
// are worth 1 % each.  A leaf's last, partly filled warp does not lengthen the
// pass when its idle lanes take part of the records: the other warps of its
// processor partition set the pace.
template <TreeForm FORM>
__global__ void __launch_bounds__(kMaxLeaf, kFarMinB)
    k_tree_far(const int4* __restrict__ items, const int2* __restrict__ segs, const int4* __restrict__ leaf_tab,
               const int* __restrict__ perm, const float4* __restrict__ tgt32, const float4* __restrict__ rec,
               int rec_stride, float* __restrict__ part, int n_items, int lmax, TreeConst c,
               const int* __restrict__ skip, int skip_stride) {
  // [record pair]: (x, x', y, y'), (z, z', a, a'), (mx, mx', my, my'), (mz, mz', -, -)
  __shared__ float4 sh[2 * kFarCH];
  float* shf = reinterpret_cast<float*>(sh);
  const int k = blockIdx.y;
  if (tree_skipped(skip, skip_stride, k)) return;
  const int4 it = items[blockIdx.x];
  const int4 lf = leaf_tab[it.x];
  const int t = threadIdx.x;
  const bool active = t < lf.y;
  const int pos = lf.x + min(t, lf.y - 1);
  const float4* R = rec + 2 * (size_t)k * rec_stride;
  const float4 g = R[2 * (size_t)pos], v = tgt32[2 * (size_t)perm[pos] + 1];
  const TreeTarget T{{f2_splat(g.x), f2_splat(g.y), f2_splat(g.z)}, {f2_splat(v.x), f2_splat(v.y), f2_splat(v.z)}};
  f2 S1 = f2_splat(0.f), S3 = f2_splat(0.f);
  auto load = [&](int jj, f2* w) {
    const float4* q = sh + 4 * jj;
    const float4 A = q[0], B = q[1], C = q[2];
    const float2 D = *reinterpret_cast<const float2*>(q + 3);
    w[0] = f2_make(A.x, A.y), w[1] = f2_make(A.z, A.w), w[2] = f2_make(B.x, B.y), w[3] = f2_make(B.z, B.w);
    w[4] = f2_make(C.x, C.y), w[5] = f2_make(C.z, C.w), w[6] = f2_make(D.x, D.y);
  };
  for (int sg = it.y; sg < it.z; ++sg) {
    const int2 S = segs[sg];
    const bool self = S.x < lf.x + lf.y && S.x + S.y > lf.x;
    for (int j0 = 0; j0 < S.y; j0 += kFarCH) {
      const int m = min(kFarCH, S.y - j0), mp = (m + 1) / 2;
      __syncthreads();
      const float4* src = R + 2 * (size_t)(S.x + j0);
      for (int q = t; q < 4 * mp; q += blockDim.x) {  // half q & 1 of record q / 2
        const bool pad = q >= 2 * m;
        float4 x = src[pad ? q - 2 : q];
        if (pad) x = q & 1 ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(x.x, x.y, x.z, 0.f);
        float* o = shf + 16 * (q >> 2) + 8 * (q & 1) + ((q >> 1) & 1);
        o[0] = x.x, o[2] = x.y, o[4] = x.z, o[6] = x.w;
      }
      __syncthreads();
      if (!active) continue;
      f2 w[7];
      if (!self) {
#pragma unroll 2
        for (int jj = 0; jj < mp; ++jj) {
          load(jj, w);
          tree_pair2<FORM, false>(T, w, false, false, c, S1, S3);
        }
      } else {
        const int own = pos - S.x - j0;
        for (int jj = 0; jj < mp; ++jj) {
          load(jj, w);
          tree_pair2<FORM, true>(T, w, 2 * jj == own, 2 * jj + 1 == own, c, S1, S3);
        }
      }
    }
  }
  if (active) {
    float* o = part + 2 * (size_t)lmax * ((size_t)k * n_items + blockIdx.x);
    o[t] = f2_sum(S1);
    o[lmax + t] = f2_sum(S3);
  }
}

// y of element perm[t]: diag u - f (sum over the leaf's items in order), with f1
// for S1 and f3 for S3 (1/(4 pi), their scale and the sign of S3); the sums
// times the element's area, and S3 the phi output, for the transpose (area_of given)
__global__ void k_tree_reduce(int n, const int* __restrict__ perm, const int* __restrict__ leaf_of,
                              const int4* __restrict__ leaf_tab, const float* __restrict__ part, int n_items,
                              int lmax, const int4* __restrict__ lay, const double4_32a* __restrict__ area_of,
                              const double* __restrict__ u, double* __restrict__ y, double dphi, double dpsi, double f1,
                              double f3, const int* __restrict__ skip, int skip_stride) {
  const int k = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n || tree_skipped(skip, skip_stride, k)) return;
  const int4 lf = leaf_tab[leaf_of[t]];
  const int local = t - lf.x;
  const float* o = part + 2 * (size_t)lmax * ((size_t)k * n_items + lf.z) + local;
  const PartSum<float> s1 = sum_strided<8>(o, (size_t)2 * lmax, lf.w), s3 = sum_strided<8>(o + lmax, (size_t)2 * lmax, lf.w);
  const int4 L = lay[k];
  const int e = perm[t];
  const bool tr = area_of != nullptr;
  const double w = tr ? area_of[2 * (L.x + e)].w : 1.0;
  const double t1 = left_range(s1) ? sum_strided_fp64(o, (size_t)2 * lmax, lf.w) : s1.value(),
               t3 = left_range(s3) ? sum_strided_fp64(o + lmax, (size_t)2 * lmax, lf.w) : s3.value();
  const double v1 = w * f1 * t1, v3 = w * f3 * t3;
  y[L.z + e] = dphi * u[L.z + e] - (tr ? v3 : v1);
  y[L.z + L.y + e] = dpsi * u[L.z + L.y + e] - (tr ? v1 : v3);
}

// ------------------------------------------------------------------ host: tree and lists
struct Node {
  int start, end;
  double lo[3], hi[3];
  int left, right;
};

// The tree of clusters over the centroids as given (FP64), in the order the
// definition above fixes (median split of the longest side, ties by index).
void build_nodes(const double* x, int n, int leaf, std::vector<int>& perm, std::vector<Node>& nodes) {
  perm.resize(n);
  std::iota(perm.begin(), perm.end(), 0);
  nodes.clear();
  auto make = [&](int s, int e) {
    Node nd;
    nd.start = s, nd.end = e, nd.left = nd.right = -1;
    for (int d = 0; d < 3; ++d) nd.lo[d] = INFINITY, nd.hi[d] = -INFINITY;
    for (int i = s; i < e; ++i)
      for (int d = 0; d < 3; ++d) {
        const double v = x[3 * (size_t)perm[i] + d];
        nd.lo[d] = std::min(nd.lo[d], v);
        nd.hi[d] = std::max(nd.hi[d], v);
      }
    nodes.push_back(nd);
    return (int)nodes.size() - 1;
  };
  std::vector<int> stack{make(0, n)};
  while (!stack.empty()) {
    const int k = stack.back();
    stack.pop_back();
    const Node nd = nodes[k];
    const int cnt = nd.end - nd.start;
    if (cnt <= leaf) continue;
    int d = 0;
    for (int q = 1; q < 3; ++q)
      if (nd.hi[q] - nd.lo[q] > nd.hi[d] - nd.lo[d]) d = q;
    std::sort(perm.begin() + nd.start, perm.begin() + nd.end, [&](int a, int b) {
      const double xa = x[3 * (size_t)a + d], xb = x[3 * (size_t)b + d];
      return xa < xb || (xa == xb && a < b);
    });
    const int h = cnt / 2;
    const int l = make(nd.start, nd.start + h);
    const int r = make(nd.start + h, nd.end);
    nodes[k].left = l;
    nodes[k].right = r;
    stack.push_back(r);
    stack.push_back(l);
  }
}

void centre_radius(const Node& nd, double c[3], double* r) {
  double s = 0.0;
  for (int d = 0; d < 3; ++d) {
    c[d] = 0.5 * (nd.lo[d] + nd.hi[d]);
    const double h = 0.5 * (nd.hi[d] - nd.lo[d]);
    s = s + h * h;
  }
  *r = std::sqrt(s);
}

struct Entry {
  bool far;
  int a, b;  // direct: positions [a, b); far: node a
};

void collect(const std::vector<Node>& nodes, int k, const double xb[3], double rb, double theta, int n_proxy,
             std::vector<Entry>& out) {
  const Node& nd = nodes[k];
  double xc[3], rc;
  centre_radius(nd, xc, &rc);
  double s = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double dd = xb[d] - xc[d];
    s = s + dd * dd;
  }
  const double dist = std::sqrt(s);
  const int count = nd.end - nd.start;
  if (rc + theta * rb <= theta * dist) {
    if (count > n_proxy)
      out.push_back(Entry{true, k, 0});
    else
      out.push_back(Entry{false, nd.start, nd.end});
  } else if (nd.left < 0) {
    out.push_back(Entry{false, nd.start, nd.end});
  } else {
    collect(nodes, nd.left, xb, rb, theta, n_proxy, out);
    collect(nodes, nd.right, xb, rb, theta, n_proxy, out);
  }
}

template <int DEG>
void launch_up(const FarField* f, cudaStream_t st, int K, float sigma, const int* skip, int skip_stride) {
  k_tree_up<DEG><<<dim3(f->n_up, K), 256, 0, st>>>(f->up_pieces.p, f->nodes.p, sigma, f->rec_stride, f->rec.p, f->upart.p,
                                                    f->n_up, skip, skip_stride);
}
template <int DEG>
void launch_proxy(const FarField* f, cudaStream_t st, int K, float sigma, const int* skip, int skip_stride) {
  constexpr int P = (DEG + 1) * (DEG + 1) * (DEG + 1);
  k_tree_proxy<DEG><<<dim3((f->n_slots * P + 255) / 256, K), 256, 0, st>>>(
      f->n_slots, f->up_tab.p, f->nodes.p, sigma, f->upart.p, f->n_up, f->n, f->rec_stride, f->rec.p, skip, skip_stride);
}

int far_occupancy(int nt) {  // the forms have one shape; the scaled kernel sets the plan
  int o = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_tree_far<kScaled>, nt, 0) != cudaSuccess) {
    (void)cudaGetLastError();
    o = 1;
  }
  return std::max(o, 1);
}

std::unique_ptr<FarField> build_far_field(Surface* s) {
  auto f = std::make_unique<FarField>();
  f->theta = s->far_theta;
  f->degree = s->far_degree;
  f->leaf = s->far_leaf;
  const int n = (int)s->n;
  f->n = n;
  const int np1 = f->degree + 1, P = np1 * np1 * np1;
  std::vector<int> perm;
  std::vector<Node> nodes;
  build_nodes(s->raw_centroids.data(), n, f->leaf, perm, nodes);
  // leaves in tree order
  std::vector<int> leaves;
  for (int k = 0; k < (int)nodes.size(); ++k)
    if (nodes[k].left < 0) leaves.push_back(k);
  std::sort(leaves.begin(), leaves.end(), [&](int a, int b) { return nodes[a].start < nodes[b].start; });
  f->n_leaves = (int)leaves.size();
  // interaction lists (adjacent direct ranges merged)
  std::vector<std::vector<Entry>> lists(leaves.size());
  std::vector<int> slot_of(nodes.size(), -1);
  for (size_t li = 0; li < leaves.size(); ++li) {
    double xb[3], rb;
    centre_radius(nodes[leaves[li]], xb, &rb);
    std::vector<Entry> raw;
    collect(nodes, 0, xb, rb, f->theta, P, raw);
    auto& out = lists[li];
    for (const Entry& e : raw) {
      if (!e.far && !out.empty() && !out.back().far && out.back().b == e.a)
        out.back().b = e.b;
      else
        out.push_back(e);
      if (e.far) slot_of[e.a] = 0;
    }
  }
  std::vector<int> slot_node;
  for (int k = 0; k < (int)nodes.size(); ++k)
    if (slot_of[k] >= 0) slot_of[k] = (int)slot_node.size(), slot_node.push_back(k);
  f->n_slots = (int)slot_node.size();
  f->rec_stride = n + f->n_slots * P;
  // segments of every leaf as record ranges, and their lengths
  std::vector<std::vector<int2>> lseg(leaves.size());
  std::vector<int64_t> lrec(leaves.size(), 0);
  int lmax = 1;
  for (size_t li = 0; li < leaves.size(); ++li) {
    lmax = std::max(lmax, nodes[leaves[li]].end - nodes[leaves[li]].start);
    for (const Entry& e : lists[li]) {
      const int2 sg = e.far ? make_int2(n + slot_of[e.a] * P, P) : make_int2(e.a, e.b - e.a);
      lseg[li].push_back(sg);
      lrec[li] += sg.y;
    }
  }
  f->lmax = lmax;
  f->nt = (lmax + 31) / 32 * 32;
  // cut every leaf's list into pieces of about L records; L keeps whole waves busy
  const int slots = s->num_sms * far_occupancy(f->nt);
  int64_t rmax = 1;
  for (auto r : lrec) rmax = std::max(rmax, r);
  auto n_items_for = [&](int64_t L) {
    int64_t c = 0;
    for (auto r : lrec) c += std::max<int64_t>(1, (r + L - 1) / L);
    return c;
  };
  int64_t bestL = rmax;
  double best = 1e300;
  for (int64_t L = 256; L < 2 * rmax; L = L + std::max<int64_t>(64, L / 16)) {
    const int64_t c = n_items_for(L);
    const double est = (double)((c + slots - 1) / slots) * (double)(std::min(L, rmax) + 256);
    if (est < best) best = est, bestL = L;
  }
  std::vector<int4> items, leaf_tab(leaves.size());
  std::vector<int2> segs;
  std::vector<int> leaf_of(n);
  f->pair_evals = 0;
  for (size_t li = 0; li < leaves.size(); ++li) {
    const Node& nd = nodes[leaves[li]];
    const int cnt = nd.end - nd.start;
    for (int p = nd.start; p < nd.end; ++p) leaf_of[p] = (int)li;
    f->pair_evals += (int64_t)cnt * lrec[li];
    const int64_t R = lrec[li];
    const int pieces = (int)std::max<int64_t>(1, (R + bestL - 1) / bestL);
    leaf_tab[li] = make_int4(nd.start, cnt, (int)items.size(), pieces);
    // walk the segments, cutting at q_p = p R / pieces
    size_t si = 0;
    int off = 0;  // records of segment si already given out
    for (int p = 0; p < pieces; ++p) {
      int64_t want = (int64_t)(p + 1) * R / pieces - (int64_t)p * R / pieces;
      const int first = (int)segs.size();
      while (want > 0 && si < lseg[li].size()) {
        const int2 sg = lseg[li][si];
        const int take = (int)std::min<int64_t>(want, sg.y - off);
        segs.push_back(make_int2(sg.x + off, take));
        want -= take;
        off += take;
        if (off == sg.y) ++si, off = 0;
      }
      items.push_back(make_int4((int)li, first, (int)segs.size(), 0));
    }
  }
  f->n_items = (int)items.size();
  // upward pieces and Chebyshev nodes of every far cluster (centred, FP32)
  std::vector<int4> up;
  std::vector<int2> up_tab(f->n_slots);
  std::vector<float> nd32((size_t)f->n_slots * 3 * np1);
  const double* ctr = &s->part_center[0];
  for (int sl = 0; sl < f->n_slots; ++sl) {
    const Node& nd = nodes[slot_node[sl]];
    up_tab[sl] = make_int2((int)up.size(), 0);
    for (int p = nd.start; p < nd.end; p += kUpPiece) up.push_back(make_int4(sl, p, std::min(kUpPiece, nd.end - p), 0));
    up_tab[sl].y = (int)up.size() - up_tab[sl].x;
    double ext[3], emax = 0.0;
    for (int d = 0; d < 3; ++d) ext[d] = nd.hi[d] - nd.lo[d], emax = std::max(emax, ext[d]);
    for (int d = 0; d < 3; ++d) {
      const double e = std::max(ext[d], 1e-3 * emax);
      const double c = 0.5 * (nd.lo[d] + nd.hi[d]);
      for (int i = 0; i <= f->degree; ++i)
        nd32[((size_t)sl * 3 + d) * np1 + i] = (float)(c + (0.5 * e) * std::cos(kPi * i / f->degree) - ctr[d]);
    }
  }
  f->n_up = (int)up.size();
  // device copies
  cudaStream_t st = s->stream;
  auto put = [&](auto& buf, const auto& v) {
    using T = typename std::decay_t<decltype(v)>::value_type;
    buf.ensure(std::max<size_t>(v.size(), 1), st);
    if (!v.empty())
      BIPB_CUDA(cudaMemcpyAsync(buf.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st));
  };
  put(f->perm, perm);
  put(f->leaf_of, leaf_of);
  put(f->leaf_tab, leaf_tab);
  put(f->items, items);
  put(f->segs, segs);
  put(f->up_pieces, up);
  put(f->up_tab, up_tab);
  put(f->nodes, nd32);
  BIPB_CUDA(cudaStreamSynchronize(st));  // the host vectors go out of scope
  ++s->alloc_gen;
  return f;
}

}  // namespace

FarField* far_field(Surface* s) {
  BIPB_REQUIRE(!s->batch, "the far-field mat-vec needs a single-surface handle");
  FarField* f = s->far.get();
  if (f && f->theta == s->far_theta && f->degree == s->far_degree && f->leaf == s->far_leaf) return f;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  BIPB_CUDA(cudaStreamIsCapturing(s->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) throw Error(BIPB_ERR_CUDA, "far-field tree built while recording a graph");
  s->far = build_far_field(s);
  return s->far.get();
}

void matvec_tree(Surface* s, const SysLayout& L, const PairConst<float>& c0, double kappa, bool transpose,
                 const double* u, double* y, double dphi, double dpsi, const int* skip, int skip_stride) {
  for (int k = 0; k < L.K; ++k)
    BIPB_REQUIRE(L.geo_off[k] == 0 && L.n[k] == (int)s->n, "the far-field mat-vec covers one surface");
  FarField* f = far_field(s);
  const int K = L.K;
  const int P = (f->degree + 1) * (f->degree + 1) * (f->degree + 1);
  if (f->rec.ensure(2 * (size_t)f->rec_stride * K, s->stream)) ++s->alloc_gen;
  if (f->part.ensure(2 * (size_t)f->lmax * f->n_items * K, s->stream)) ++s->alloc_gen;
  if (f->upart.ensure(std::max<size_t>(1, 4 * (size_t)P * f->n_up * K), s->stream)) ++s->alloc_gen;
  const int4* lay = s->lay_dev(L);
  const int nb = (f->n + 255) / 256;
  const TreeForm form = kappa == 0.0 ? kLaplace : kappa < kScaledKappaMin ? kPlain : kScaled;
  const double sigma = form == kScaled ? kappa : 1.0;
  const float sg = (float)sigma;
  TreeConst c;
  c.ef = transpose ? -c0.inveps : c0.eps, c.e0 = transpose ? 1.f : -1.f;
  c.ff = transpose ? c0.eps : -c0.inveps, c.f0 = transpose ? -1.f : 1.f;
  c.kappa = c0.kappa, c.smax = (float)(kSMaxD / sigma);
  k_tree_pack<<<dim3(nb, K), 256, 0, s->stream>>>(f->n, f->rec_stride, transpose, sigma, f->perm.p, s->tgt64.p, lay, u,
                                                  f->rec.p, skip, skip_stride);
  BIPB_LAUNCHED(s);
  if (f->n_up > 0) {
    switch (f->degree) {
      case 4: launch_up<4>(f, s->stream, K, sg, skip, skip_stride); break;
      case 6: launch_up<6>(f, s->stream, K, sg, skip, skip_stride); break;
      default: launch_up<8>(f, s->stream, K, sg, skip, skip_stride); break;
    }
    BIPB_LAUNCHED(s);
    switch (f->degree) {
      case 4: launch_proxy<4>(f, s->stream, K, sg, skip, skip_stride); break;
      case 6: launch_proxy<6>(f, s->stream, K, sg, skip, skip_stride); break;
      default: launch_proxy<8>(f, s->stream, K, sg, skip, skip_stride); break;
    }
    BIPB_LAUNCHED(s);
  }
  {
    TimedLaunch tl(s, kTMvTree);
    auto kernel = form == kScaled ? k_tree_far<kScaled> : form == kPlain ? k_tree_far<kPlain> : k_tree_far<kLaplace>;
    kernel<<<dim3(f->n_items, K), f->nt, 0, s->stream>>>(f->items.p, f->segs.p, f->leaf_tab.p, f->perm.p, s->tgt32.p,
                                                         f->rec.p, f->rec_stride, f->part.p, f->n_items, f->lmax, c,
                                                         skip, skip_stride);
    BIPB_LAUNCHED(s);
  }
  k_tree_reduce<<<dim3(nb, K), 256, 0, s->stream>>>(f->n, f->perm.p, f->leaf_of.p, f->leaf_tab.p, f->part.p,
                                                    f->n_items, f->lmax, lay, transpose ? s->tgt64.p : nullptr, u, y,
                                                    dphi, dpsi, kInv4PiT * sigma, -kInv4PiT * sigma * sigma, skip,
                                                    skip_stride);
  BIPB_LAUNCHED(s);
}

}  // namespace bipb

// Mat-vec of Eqs. 5-6 (and its transpose) visiting every unordered pair once.
//
// The four kernels of a pair share r, e^{-kappa r}, t and w; only the dot
// products with the normals and the sign of d differ between the two
// directions.  Each work item is one tile of T targets of a system (row I)
// against a range of sources at or after the tile's first element; every pair
// (i, j) with j > i is evaluated once and applied both ways:
//   target i gathers source j      -> register accumulators (i side)
//   target j gathers source i      -> summed over the CTA's T targets (j side)
// In the tile's own diagonal block the pairs with j <= i are masked (1/r = 0).
// The j side of a source is summed over a warp by accumulators that rotate
// through the lanes, and over the warps in a fixed order, so results are
// bitwise reproducible.
//
// Row I of a system has n - I T sources, so rows shrink down the system.
// Rows I and nT - 1 - I are folded together (about n + T sources between
// them) and the folded rows are cut into pieces of equal length; a piece is
// one work item and covers one or two segments (tile, source range).  All
// items thus carry the same work, and their number is chosen to fill whole
// waves of resident CTAs.
//
// Partial sums (per system, T = targets per tile, nT tiles):
//   i side: one block of 2 x T values per segment (a row's segments are
//           numbered consecutively, in source order);
//   j side: for row I, 2 x (n - I T) values (every element j >= I T).
// The reduction adds, for element e of tile E, the i-side blocks of row E and
// the j-side values of rows 0..E, in that fixed order: FP64 partials in FP64, FP32
// ones by TwoSums (PartSum, symstep.cuh).
#include <algorithm>
#include <cmath>
#include <map>
#include <memory>
#include <mutex>
#include <queue>
#include <type_traits>

#include "f32x2.cuh"
#include "internal.cuh"
#include "symstep.cuh"
#include "tf64.cuh"

namespace bipb {

namespace {

constexpr double kInv4PiS = 1.0 / (4.0 * kPi);

// ------------------------------------------------------------------ policies
// A policy: the record of an element (RW vectors of 4 values; both roles), a
// pack of PACK targets of one thread (Tgt, with its accumulators Acc), a source
// (Src), and the pair update of a pack with one source.  PACK = 2: two targets
// in packed FP32 (f32x2.cuh), the source's values duplicated in its record so
// that one 64-bit load gives a packed operand; the j side stays packed (one
// half per target of the pack) until a block of 32 sources is done.  Red is the
// j side of one source over a warp.

// FP64, one target per pack.  Record (a, alpha, n.x, n.y), (n.z, x.h, x.l), (x.m),
// (n as integers, fix2),
// where (a, alpha) = (ds psi, ds phi) for A u and (wphi, wpsi) for A^T w and the
// position is in three floats on the surface's grid (df_pos), 9 of them from the
// second vector's second value on.  LAPLACE: the kappa = 0 form (pair.cuh);
// otherwise the records are in kappa-scaled units (SCALED).
template <bool TRANS, bool LAPLACE>
struct Sym64Policy {
  using V4 = double4_32a;
  using PT = double;  // partial sums are stored in this type
  static constexpr bool SCALED = !LAPLACE;
  static constexpr int RW = 4, PACK = 1, UNROLL = 1;
  static constexpr bool CHUNKED = false;
  struct Tgt {
    df_pos x[3];
    double a, n[3], al;
    fix2 f[3];  // the normal as integers
  };
  using Src = Tgt;
  struct Acc {
    double p, q;
  };
  using Red = Acc;
  struct Args {
    TfConst c;
    const float4* tab;  // the exp table as kept by the surface (exp_table, capi.cu)
  };
  __device__ static float4* exp_tab() {
    __shared__ float4 tab[kTfTab];  // 2^(j/1024) as three floats
    return tab;
  }
  __device__ static void prologue(const Args& g) {
    if (LAPLACE) return;
    const float2* t2 = reinterpret_cast<const float2*>(g.tab);
    const float* t3 = reinterpret_cast<const float*>(g.tab + kExpTab / 2);
    for (int j = threadIdx.x; j < kTfTab; j += blockDim.x) exp_tab()[j] = make_float4(t2[j].x, t2[j].y, t3[j], 0.f);
  }
  __device__ static void load(const V4* rec, const int* i, Tgt& t) {
    const V4* r = rec + 4 * (size_t)i[0];
    unpack(r[0], r[1], r[2], r[3], t);
  }
  // record q of a chunk staged as planes (vector r of record q at sh[r * CH + q])
  template <int CH>
  __device__ static void load_src(const V4* sh, int q, Src& e) { unpack(sh[q], sh[CH + q], sh[2 * CH + q], sh[3 * CH + q], e); }
  static __device__ float2 floats(double v) { return make_float2(__int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v))); }
  static __device__ double pair_of(float a, float b) { return __hiloint2double(__float_as_int(b), __float_as_int(a)); }
  static __device__ fix2 ints(double v) { return fix2{__double2loint(v), __double2hiint(v)}; }
  __device__ static void unpack(const V4& A, const V4& B, const V4& C, const V4& F, Tgt& e) {
    e.f[0] = ints(F.x), e.f[1] = ints(F.y), e.f[2] = ints(F.z);
    e.a = A.x, e.al = A.y, e.n[0] = A.z, e.n[1] = A.w, e.n[2] = B.x;
    const float2 p = floats(B.y), q = floats(B.z), r = floats(B.w), s = floats(C.x);
    e.x[0] = df_pos{p.x, q.y, s.x}, e.x[1] = df_pos{p.y, r.x, s.y}, e.x[2] = df_pos{q.x, r.y, floats(C.y).x};
  }
  __device__ static void zero(Acc& v) { v.p = 0.0, v.q = 0.0; }
  // i side of the targets t and j side of source sj for the pairs d = x_t - x_sj
  template <bool MASK>
  __device__ static void pair(const Args& g, const Tgt& t, const Src& sj, const bool* masked, Acc& ti, Acc& tj) {
    const tf d[3] = {tf_diff(t.x[0], sj.x[0]), tf_diff(t.x[1], sj.x[1]), tf_diff(t.x[2], sj.x[2])};
    TfRadial R = tf_radial<LAPLACE>(tf_norm2(d[0], d[1], d[2]), g.c, LAPLACE ? nullptr : exp_tab());
    const double dx = tf_to_double<true>(d[0], 0), dy = tf_to_double<true>(d[1], 0), dz = tf_to_double<true>(d[2], 0);
    if (MASK && masked[0]) R.k1 = R.v = R.w = R.k2 = R.k3 = 0.0;
    const double cij = LAPLACE ? 0.0 : fix2_dot(t.f, sj.f);
    sym_pair64<TRANS, LAPLACE>(dx, dy, dz, cij, t.n, t.a, t.al, sj.n, sj.a, sj.al, R, ti.p, ti.q, tj.p, tj.q);
  }
  __device__ static void flush(Acc&, const Acc&) {}
  __device__ static Red reduced(const Acc& v) { return v; }
  __device__ static double add(double a, double b) { return a + b; }
  __device__ static void rotate(Acc& v, int src) {
    v.p = __shfl_sync(0xffffffffu, v.p, src);
    v.q = __shfl_sync(0xffffffffu, v.q, src);
  }
  // a source slot q past the end of a chunk: far away, no field, no normal (adds exact zeros)
  template <int CH>
  __device__ static void pad(V4* sh, int q) {
    sh[q] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    sh[CH + q] = make_double4_32a(0.0, pair_of(1e4f, 1e4f), pair_of(1e4f, 0.f), 0.0);
    sh[2 * CH + q] = sh[3 * CH + q] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
  }
  __device__ static PT out(double v) { return v; }
  __device__ static void store(PT* p, int T, const int* o, const bool* in, const Acc& v) {
    if (in[0]) p[o[0]] = v.p, p[T + o[0]] = v.q;
  }
};

// FP32, two targets per pack.  What bounds it: the FP32 pipe's register ports.  An
// FFMA with three register operands takes 1.5 issue cycles (FFMA2 three for two
// results; microbench/alu_peaks.cu), FADD and FMUL one, so a pair of 22 FFMA and 21
// others takes 54 cycles of a scheduler however it is issued, and the scalar form
// waited for its loads, shuffles and MUFU calls on top (64.5).  Packed, they
// hide behind it: N = 20480 0.387 -> 0.350 ms, N = 65537 3.43 -> 3.15 ms a
// mat-vec (59.7 cycles a pair).  Record, 5 float4, every value twice: (x, x, y, y),
// (z, z, a, a), (nx, nx, ny, ny), (nz, nz, -alpha, -alpha), (f, f, 0, 0) with f
// = -a (A u) or alpha (A^T w): packed FP32 has no negated operands, so every
// sign of sym_pair2 is one that a record, a constant or a subtraction brings.
template <bool TRANS, bool LAPLACE>
struct Sym32Policy {
  using V4 = float4;
  using PT = float;
  static constexpr bool SCALED = !LAPLACE;
  static constexpr int RW = 5, PACK = 2, UNROLL = 4;
  static constexpr bool CHUNKED = false;
  struct Tgt {
    f2 x[3], n[3], f[3];  // f: a, -alpha and alpha (A u) or -a (A^T w)
  };
  struct Src {
    f2 x[3], n[3], f[3];  // f: a, -alpha and -a (A u) or alpha (A^T w)
  };
  struct Acc {
    f2 p, q;
  };
  struct Red {
    float p, q;
  };
  struct Args {
    PairConst<float> c;
  };
  __device__ static void prologue(const Args&) {}
  __device__ static void load(const V4* rec, const int* i, Tgt& t) {
    const V4 *r = rec + 5 * (size_t)i[0], *q = rec + 5 * (size_t)i[1];
    const V4 A = r[0], B = r[1], C = r[2], D = r[3], E = q[0], F = q[1], G = q[2], H = q[3];
    t.x[0] = f2_make(A.x, E.x), t.x[1] = f2_make(A.z, E.z), t.x[2] = f2_make(B.x, F.x);
    t.n[0] = f2_make(C.x, G.x), t.n[1] = f2_make(C.z, G.z), t.n[2] = f2_make(D.x, H.x);
    t.f[0] = f2_make(B.z, F.z), t.f[1] = f2_make(D.z, H.z);
    t.f[2] = TRANS ? f2_make(-B.z, -F.z) : f2_make(-D.z, -H.z);
  }
  template <int CH>
  __device__ static void load_src(const V4* sh, int q, Src& e) {
    const ulonglong2* v = reinterpret_cast<const ulonglong2*>(sh);
    const ulonglong2 A = v[q], B = v[CH + q], C = v[2 * CH + q], D = v[3 * CH + q];
    e.x[0].v = A.x, e.x[1].v = A.y, e.x[2].v = B.x, e.f[0].v = B.y;
    e.n[0].v = C.x, e.n[1].v = C.y, e.n[2].v = D.x, e.f[1].v = D.y;
    e.f[2].v = v[4 * CH + q].x;
  }
  __device__ static void zero(Acc& v) { v.p = f2_splat(0.f), v.q = f2_splat(0.f); }
  template <bool MASK>
  __device__ static void pair(const Args& g, const Tgt& t, const Src& sj, const bool* masked, Acc& ti, Acc& tj) {
    sym_pair2<MASK, TRANS, LAPLACE>(t.x, t.n, t.f, sj.x, sj.n, sj.f, masked[0], masked[1], g.c, ti.p, ti.q, tj.p, tj.q);
  }
  __device__ static void flush(Acc&, const Acc&) {}
  __device__ static Red reduced(const Acc& v) { return Red{f2_sum(v.p), f2_sum(v.q)}; }
  __device__ static float add(float a, float b) { return a + b; }
  __device__ static void rotate(Acc& v, int src) {
    v.p.v = __shfl_sync(0xffffffffu, v.p.v, src);
    v.q.v = __shfl_sync(0xffffffffu, v.q.v, src);
  }
  template <int CH>
  __device__ static void pad(V4* sh, int q) {
    sh[q] = make_float4(1e4f, 1e4f, 1e4f, 1e4f);
    sh[CH + q] = make_float4(1e4f, 1e4f, 0.f, 0.f);
    sh[2 * CH + q] = sh[3 * CH + q] = sh[4 * CH + q] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ static PT out(float v) { return v; }
  __device__ static void store(PT* p, int T, const int* o, const bool* in, const Acc& v) {
    float a, b, c, d;
    f2_get(v.p, a, b);
    f2_get(v.q, c, d);
    if (in[0]) p[o[0]] = a, p[T + o[0]] = c;
    if (in[1]) p[o[1]] = b, p[T + o[1]] = d;
  }
};

__device__ df* sym_exp_table() {
  __shared__ __align__(16) df tab[kExpTab];
  return tab;
}

// df64 record, 5 float4: (x.h, a.hi), (x.l, a.lo), (n.hi, alpha.hi), (n.lo, alpha.lo),
// (x.m, 0), the position in three parts on the surface's grid (df_pos);
// SCALED: positions and alpha in kappa-scaled units (df_sym_pair)
template <bool TRANS, bool SCALED_>
struct SymDFPolicy {
  using V4 = float4;
  using PT = double;
  static constexpr bool SCALED = SCALED_;
  static constexpr int RW = 5, PACK = 1, UNROLL = 1;
  static constexpr bool CHUNKED = true;  // every chunk summed from zero, then added to the running sums
  struct Tgt {
    df_pos x[3];
    df a, n[3], al;
  };
  using Src = Tgt;
  struct Acc {
    df p, q;
  };
  using Red = Acc;
  struct Args {
    DFConst c;
  };
  __device__ static void prologue(const Args& g) { df_load_exp_table(sym_exp_table(), g.c); }
  __device__ static void load(const V4* rec, const int* i, Tgt& t) {
    const V4* r = rec + 5 * (size_t)i[0];
    unpack(r[0], r[1], r[2], r[3], r[4], t);
  }
  template <int CH>
  __device__ static void load_src(const V4* sh, int q, Src& e) {
    unpack(sh[q], sh[CH + q], sh[2 * CH + q], sh[3 * CH + q], sh[4 * CH + q], e);
  }
  __device__ static void unpack(const float4& A, const float4& B, const float4& C, const float4& D, const float4& M,
                                Tgt& e) {
    e.x[0] = df_pos{A.x, B.x, M.x}, e.x[1] = df_pos{A.y, B.y, M.y}, e.x[2] = df_pos{A.z, B.z, M.z};
    e.a = df{A.w, B.w};
    e.n[0] = df{C.x, D.x}, e.n[1] = df{C.y, D.y}, e.n[2] = df{C.z, D.z}, e.al = df{C.w, D.w};
  }
  __device__ static void zero(Acc& v) { v.p = df{0.f, 0.f}, v.q = df{0.f, 0.f}; }
  template <bool MASK>
  __device__ static void pair(const Args& g, const Tgt& t, const Src& sj, const bool* masked, Acc& ti, Acc& tj) {
    const df d[3] = {df_diff(t.x[0], sj.x[0]), df_diff(t.x[1], sj.x[1]), df_diff(t.x[2], sj.x[2])};
    df_sym_pair<MASK, TRANS, SCALED>(d, t.n, t.a, t.al, sj.n, sj.a, sj.al, masked[0], g.c, sym_exp_table(), ti.p, ti.q,
                                     tj.p, tj.q);
  }
  __device__ static void flush(Acc& sum, const Acc& v) {
    sum.p = df_add(sum.p, v.p);
    sum.q = df_add(sum.q, v.q);
  }
  // the accumulators are updated lazily (df_mac): bring them back to normal form
  __device__ static Red reduced(const Acc& v) { return Red{two_sum(v.p.hi, v.p.lo), two_sum(v.q.hi, v.q.lo)}; }
  __device__ static df add(df a, df b) { return df_add(a, b); }
  __device__ static df shfl(df v, int src) {
    return df{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
  }
  __device__ static void rotate(Acc& v, int src) { v.p = shfl(v.p, src), v.q = shfl(v.q, src); }
  template <int CH>
  __device__ static void pad(float4* sh, int q) {
    sh[q] = make_float4(1e4f, 1e4f, 1e4f, 0.f);
    sh[CH + q] = sh[2 * CH + q] = sh[3 * CH + q] = sh[4 * CH + q] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ static PT out(df v) { return df_to_double(v); }
  __device__ static void store(PT* p, int T, const int* o, const bool* in, const Acc& v) {
    if (in[0]) p[o[0]] = out(v.p), p[T + o[0]] = out(v.q);
  }
};

// ------------------------------------------------------------------ kernel
// One shared-memory chunk of cnt sources (starting at j0) against the
// thread's NP packs of targets.  MASK: the chunk overlaps the tile's own
// targets, and pairs with j <= i are masked.  The j side rotates through the
// warp: the chunk is taken in blocks of 32 sources (the slots past cnt padded
// with records that add exact zeros); at step k of a block, lane l evaluates
// source (l + k) mod 32 against its targets, then takes over the accumulator
// of the next source from lane l + 1.  After 32 steps lane l holds the
// complete j-side sum of source (l + 31) mod 32 over the warp's targets,
// accumulated in a fixed order; it leaves it in jred[warp][source].
template <class P, int NP, int CH, bool MASK>
__device__ __forceinline__ void sym_chunk(const typename P::Args& g, const typename P::Tgt* tg,
                                          const int (*idx)[P::PACK], typename P::Acc* acc, const typename P::V4* sh,
                                          int cnt, int j0, typename P::Red (*jred)[CH]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int next = (lane + 1) & 31;
  for (int r0 = 0; r0 < cnt; r0 += 32) {
    typename P::Acc tj;
    P::zero(tj);
#pragma unroll P::UNROLL
    for (int k = 0; k < 32; ++k) {
      const int jj = r0 + ((lane + k) & 31);
      typename P::Src sj;
      P::template load_src<CH>(sh, jj, sj);
#pragma unroll
      for (int t = 0; t < NP; ++t) {
        bool masked[P::PACK];
#pragma unroll
        for (int h = 0; h < P::PACK; ++h) masked[h] = MASK && j0 + jj <= idx[t][h];
        P::template pair<MASK>(g, tg[t], sj, masked, acc[t], tj);
      }
      if (k < 31) P::rotate(tj, next);
    }
    const int mine = r0 + ((lane + 31) & 31);
    if (mine < cnt) jred[warp][mine] = P::reduced(tj);
  }
}

// Item (three int4): {rec_off, n, sys, jbase}, then two segments
// {t0, s0, s1, ioff} (s0 == s1: empty): targets t0 + [0, T) of a system with n
// elements whose records start at rec_off, against sources [s0, s1) (s0 >=
// t0); i-side partials at part[ioff + c T + i - t0], j-side at part[jrow +
// c (n - t0) + j - t0] with jrow the start of row t0 / T after jbase.
template <class P, int NT, int TPT, int CH, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_sym(typename P::Args g, const int4* __restrict__ items,
                                            const typename P::V4* __restrict__ rec, typename P::PT* __restrict__ part,
                                            const int* __restrict__ skip, int skip_stride) {
  using V4 = typename P::V4;
  using Acc = typename P::Acc;
  constexpr int NW = NT / 32, T = NT * TPT, NP = TPT / P::PACK;
  static_assert(TPT % P::PACK == 0, "whole packs of targets");
  __shared__ V4 sh[CH * P::RW];
  __shared__ typename P::Red jred[NW][CH];
  chain_wait();  // the records of the pack kernel
  chain_release();  // the next kernel is placed once every block of this one is, and waits there
  const int4 H = items[3 * blockIdx.x];
  const int rec_off = H.x, n = H.y, sys = H.z, jbase = H.w;
  if (skip != nullptr && skip[(size_t)sys * skip_stride] != 0) return;
  P::prologue(g);  // per-CTA shared tables (made visible by the first barrier below)
  for (int seg = 0; seg < 2; ++seg) {
    const int4 S = items[3 * blockIdx.x + 1 + seg];
    const int t0 = S.x, s0 = S.y, s1 = S.z, ioff = S.w;
    if (s0 >= s1) continue;
    const int I = t0 / T;
    const int64_t jrow = jbase + 2 * ((int64_t)I * n - (int64_t)T * I * (I - 1) / 2);
    const int len = n - t0;  // j-side row length
    typename P::Tgt tg[NP];
    Acc acc[NP], sum[P::CHUNKED ? NP : 1];
    int idx[NP][P::PACK];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      int r[P::PACK];
#pragma unroll
      for (int h = 0; h < P::PACK; ++h) {
        idx[k][h] = t0 + (k * P::PACK + h) * NT + threadIdx.x;
        r[h] = rec_off + min(idx[k][h], n - 1);
      }
      P::load(rec, r, tg[k]);
      P::zero(acc[k]);
      if (P::CHUNKED) P::zero(sum[k]);
    }
    for (int j0 = s0; j0 < s1; j0 += CH) {
      const int cnt = min(CH, s1 - j0);
      __syncthreads();
      // stage the chunk as planes: vector r of record q at sh[r * CH + q] (the
      // lanes of a warp read consecutive records: no bank conflicts)
      const V4* src = rec + (size_t)(rec_off + j0) * P::RW;
      for (int e = threadIdx.x; e < cnt * P::RW; e += NT) sh[(e % P::RW) * CH + e / P::RW] = src[e];
      for (int q = cnt + threadIdx.x; q < ((cnt + 31) & ~31); q += NT) P::template pad<CH>(sh, q);
      __syncthreads();
      if (j0 < t0 + T)
        sym_chunk<P, NP, CH, true>(g, tg, idx, acc, sh, cnt, j0, jred);
      else
        sym_chunk<P, NP, CH, false>(g, tg, idx, acc, sh, cnt, j0, jred);
      if (P::CHUNKED)
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          P::flush(sum[k], acc[k]);
          P::zero(acc[k]);
        }
      __syncthreads();
      for (int q = threadIdx.x; q < cnt; q += NT) {
        typename P::Red v = jred[0][q];
#pragma unroll
        for (int w = 1; w < NW; ++w) v.p = P::add(v.p, jred[w][q].p), v.q = P::add(v.q, jred[w][q].q);
        const int o = j0 + q - t0;
        part[jrow + o] = P::out(v.p);
        part[jrow + len + o] = P::out(v.q);
      }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      int o[P::PACK];
      bool in[P::PACK];
#pragma unroll
      for (int h = 0; h < P::PACK; ++h) o[h] = idx[k][h] - t0, in[h] = idx[k][h] < n;
      P::store(part + ioff, T, o, in, P::CHUNKED ? sum[k] : acc[k]);
    }
  }
}

// ------------------------------------------------------------------ pack / reduce
// Records of every system at vec_off / 2 (RW vectors each).  lay[k] = {geo_off, n, vec_off, chg_off}.
// A u: a = ds psi, alpha = ds phi; A^T w: a = wphi, alpha = wpsi.
// sigma: the positions and alpha are multiplied by it (kappa-scaled records; 1 otherwise);
// gscale: the power of two at or above sigma, by which the surface's coordinate grid grows with it
__global__ void k_pack_sym64(const int4* __restrict__ lay, bool transpose, const double4_32a* __restrict__ tgt64,
                             const double* __restrict__ u, double4_32a* __restrict__ rec, const int* __restrict__ skip,
                             int skip_stride, double sigma, double gscale) {
  chain_wait();
  chain_release();
  const int k = blockIdx.y;
  const int4 L = lay[k];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= L.y || (skip != nullptr && skip[(size_t)k * skip_stride] != 0)) return;
  const double4_32a g = tgt64[2 * (L.x + j)], v = tgt64[2 * (L.x + j) + 1];
  const double phi = u[L.z + j], psi = u[L.z + L.y + j];
  const double a = transpose ? phi : g.w * psi;
  const double al = sigma * (transpose ? psi : g.w * phi);
  const double grid = gscale * v.w;  // of the scaled coordinates
  const df_pos x0 = df_split_grid(sigma * g.x, grid), x1 = df_split_grid(sigma * g.y, grid),
               x2 = df_split_grid(sigma * g.z, grid);
  auto two = [](float p, float q) { return __hiloint2double(__float_as_int(q), __float_as_int(p)); };
  auto fix = [](double n) {
    const fix2 f = fix2_from_double(n);
    return __hiloint2double(f.l, f.h);
  };
  double4_32a* o = rec + 4 * (size_t)(L.z / 2 + j);
  o[0] = make_double4_32a(a, al, v.x, v.y);
  o[1] = make_double4_32a(v.z, two(x0.h, x1.h), two(x2.h, x0.l), two(x1.l, x2.l));
  o[2] = make_double4_32a(two(x0.m, x1.m), two(x2.m, 0.f), 0.0, 0.0);
  o[3] = make_double4_32a(fix(v.x), fix(v.y), fix(v.z), 0.0);
}

// every value twice, with the negated fields (Sym32Policy)
__global__ void k_pack_sym32(const int4* __restrict__ lay, bool transpose, const double4_32a* __restrict__ tgt64,
                             const double* __restrict__ u, float4* __restrict__ rec, const int* __restrict__ skip,
                             int skip_stride, double sigma) {
  chain_wait();
  chain_release();
  const int k = blockIdx.y;
  const int4 L = lay[k];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= L.y || (skip != nullptr && skip[(size_t)k * skip_stride] != 0)) return;
  const double4_32a g = tgt64[2 * (L.x + j)], v = tgt64[2 * (L.x + j) + 1];
  const double phi = u[L.z + j], psi = u[L.z + L.y + j];
  sym32_record(g, v, phi, psi, transpose, sigma, rec + 5 * (size_t)(L.z / 2 + j));
}

__global__ void k_pack_sym_df(const int4* __restrict__ lay, bool transpose, const double4_32a* __restrict__ tgt64,
                              const double* __restrict__ u, float4* __restrict__ rec, const int* __restrict__ skip,
                              int skip_stride, double sigma, double gscale) {
  chain_wait();
  chain_release();
  const int k = blockIdx.y;
  const int4 L = lay[k];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= L.y || (skip != nullptr && skip[(size_t)k * skip_stride] != 0)) return;
  const double4_32a g = tgt64[2 * (L.x + j)], v = tgt64[2 * (L.x + j) + 1];
  const double phi = u[L.z + j], psi = u[L.z + L.y + j];
  const df a = df_from_double(transpose ? phi : g.w * psi);
  const df al = df_from_double(sigma * (transpose ? psi : g.w * phi));
  const double grid = gscale * v.w;  // of the scaled coordinates
  const df_pos x0 = df_split_grid(sigma * g.x, grid), x1 = df_split_grid(sigma * g.y, grid),
               x2 = df_split_grid(sigma * g.z, grid);
  const df n0 = df_from_double(v.x), n1 = df_from_double(v.y), n2 = df_from_double(v.z);
  float4* o = rec + 5 * (size_t)(L.z / 2 + j);
  o[0] = make_float4(x0.h, x1.h, x2.h, a.hi);
  o[1] = make_float4(x0.l, x1.l, x2.l, a.lo);
  o[2] = make_float4(n0.hi, n1.hi, n2.hi, al.hi);
  o[3] = make_float4(n0.lo, n1.lo, n2.lo, al.lo);
  o[4] = make_float4(x0.m, x1.m, x2.m, 0.f);
}

// y_i = diag u_i - (1/(4 pi)) scale_i f_c sym_sum, f_c = f.x for the phi rows
// and f.y for the psi rows (the factors of kappa-scaled records).
template <typename PT>
__global__ void k_reduce_sym(const int4* __restrict__ lay, const int4* __restrict__ tab, const PT* __restrict__ part,
                             const double* __restrict__ u, double* __restrict__ y, double d_phi, double d_psi,
                             const double4_32a* __restrict__ tgt64_for_area, const int* __restrict__ skip,
                             int skip_stride, double2 f) {
  chain_wait();
  chain_release();
  const int k = blockIdx.y;
  const int4 L = lay[k];
  const int n = L.y;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n || (skip != nullptr && skip[(size_t)k * skip_stride] != 0)) return;
  const int c = i < n ? 0 : 1, e = i - c * n;
  const double acc = sym_sum(tab, tab[k], part, e, c);
  const double sc = kInv4PiS * (tgt64_for_area ? tgt64_for_area[2 * (L.x + e)].w : 1.0);
  y[L.z + i] = (c == 0 ? d_phi : d_psi) * u[L.z + i] - sc * (c == 0 ? f.x : f.y) * acc;
}

int blocks_of(int64_t n, int bs) { return (int)std::max<int64_t>(1, (n + bs - 1) / bs); }

// ------------------------------------------------------------------ work list
// Folded rows (I, nT - 1 - I) of every system are cut into pieces of about
// Lsrc sources; Lsrc is the candidate (the length giving 1 .. 32 waves of
// equal pieces) whose greedy schedule (pieces sorted by size, each to the
// first free CTA slot) finishes first.  A piece costs its
// sources in blocks of 32 plus 32 per segment (loading a tile, storing its partials).
struct HostPlan {
  std::vector<int4> items, tab;
  int n_items = 0;
  int64_t part_len = 0;
};

HostPlan compute_sym_plan(const SysLayout& L, int T, int slots, int ch);

// The work list depends only on the layout, the tile and the CTA slots:
// handles of the same sizes share its host copy (a process-wide memo of at
// most 64 entries), and each uploads it once.
ItemPlan* plan_sym(Surface* s, uint64_t key, const SysLayout& L, int T, int slots, int ch) {
  auto it = s->plans.find(key);
  if (it != s->plans.end()) return it->second.get();
  uint64_t mk = 0xcbf29ce484222325ull;
  auto mix = [&](uint64_t v) { mk = (mk ^ v) * 0x100000001b3ull; };
  mix((uint64_t)T), mix((uint64_t)slots), mix((uint64_t)ch), mix((uint64_t)L.K);
  for (int k = 0; k < L.K; ++k) mix((uint64_t)L.n[k]), mix((uint64_t)L.vec_off[k]);
  static std::mutex mu;
  static std::map<uint64_t, std::shared_ptr<const HostPlan>> memo;
  std::shared_ptr<const HostPlan> hp;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto m = memo.find(mk);
    if (m != memo.end()) hp = m->second;
  }
  if (!hp) {
    hp = std::make_shared<const HostPlan>(compute_sym_plan(L, T, slots, ch));
    std::lock_guard<std::mutex> lock(mu);
    if (memo.size() >= 64) memo.erase(memo.begin());
    memo[mk] = hp;
  }
  auto plan = std::make_unique<ItemPlan>();
  plan->n_items = hp->n_items;
  plan->part_len = hp->part_len;
  plan->items.ensure(hp->items.size(), s->stream);
  plan->tab.ensure(hp->tab.size(), s->stream);
  BIPB_CUDA(cudaMemcpyAsync(plan->items.p, hp->items.data(), hp->items.size() * sizeof(int4), cudaMemcpyHostToDevice,
                            s->stream));
  BIPB_CUDA(cudaMemcpyAsync(plan->tab.p, hp->tab.data(), hp->tab.size() * sizeof(int4), cudaMemcpyHostToDevice,
                            s->stream));
  BIPB_CUDA(cudaStreamSynchronize(s->stream));
  ++s->alloc_gen;
  ItemPlan* raw = plan.get();
  s->plans[key] = std::move(plan);
  return raw;
}

HostPlan compute_sym_plan(const SysLayout& L, int T, int slots, int ch) {
  const int K = L.K;
  struct Fold {
    int k, Ia, Ib, la, lb;  // rows Ia and Ib (-1: none) with la and lb sources
  };
  std::vector<Fold> folds;
  int64_t total = 0;
  int n_max = 1;
  for (int k = 0; k < K; ++k) {
    const int n = L.n[k], nT = (n + T - 1) / T;
    n_max = std::max(n_max, n);
    for (int I = 0; I < nT / 2; ++I) {
      const int Ib = nT - 1 - I;
      folds.push_back(Fold{k, I, Ib, n - I * T, n - Ib * T});
    }
    if (nT % 2) folds.push_back(Fold{k, nT / 2, -1, n - (nT / 2) * T, 0});
  }
  for (const Fold& f : folds) total += f.la + f.lb;
  // pieces of fold f: cuts at equal parts moved to whole blocks of 32 sources of their
  // row (the kernel takes sources in blocks of 32, so a piece of 33 would cost 64: at n =
  // 1000, T = 64 half as many blocks again); emits (first, end) along the fold
  auto each_piece = [](const Fold& f, double Ls, auto&& emit) {
    const int len = f.la + f.lb, P = std::max(1, (int)std::lround(len / Ls));
    int a = 0;
    for (int p = 1; p <= P; ++p) {
      int b = len;
      if (p < P) {
        b = (int)((int64_t)p * len / P);
        b = b < f.la ? std::min(f.la, (b + 16) / 32 * 32) : f.la + std::min(f.lb, (b - f.la + 16) / 32 * 32);
      }
      if (b > a) emit(a, b);
      a = std::max(a, b);
    }
  };
  // cost of a piece: its sources in blocks of 32, plus 32 per segment
  auto cost_of = [](const Fold& f, int a, int b) {
    const int x = std::max(0, std::min(b, f.la) - a), y = b - std::max(a, f.la);
    return (x > 0 ? (x + 31) / 32 * 32 + 32 : 0) + (y > 0 ? (y + 31) / 32 * 32 + 32 : 0);
  };
  auto makespan = [&](double Ls) {
    std::vector<double> cost;
    for (const Fold& f : folds) each_piece(f, Ls, [&](int a, int b) { cost.push_back(cost_of(f, a, b)); });
    std::sort(cost.begin(), cost.end(), std::greater<double>());
    std::priority_queue<double, std::vector<double>, std::greater<double>> q;
    for (int i = 0; i < slots; ++i) q.push(0.0);
    double end = 0.0;
    for (double c : cost) {
      const double t = q.top() + c;
      q.pop();
      q.push(t);
      end = std::max(end, t);
    }
    return end;
  };
  // candidates: the piece length that gives w waves of equal pieces, w from 1
  // to 32 (uneven batches need many short pieces to balance); stop once the
  // schedule is within 1 % of the ideal total / slots
  const double ideal = (double)total / (double)slots;
  double best_L = 2.0 * n_max, best = makespan(best_L);
  static const double kWaves[] = {1, 1.5, 2, 3, 4, 6, 8, 12, 16, 24, 32};
  for (double w : kWaves) {
    if (best <= 1.01 * ideal) break;
    const double Ls = std::max((double)ch, (double)total / (w * slots));
    const double m = makespan(Ls);
    if (m < best * 0.995) best = m, best_L = Ls;
  }

  // segments: {k, row, s0, s1, piece}; a piece has one or two
  struct Seg {
    int k, I, s0, s1, piece;
  };
  std::vector<Seg> segs;
  std::vector<int> piece_cost;
  for (const Fold& f : folds)
    each_piece(f, best_L, [&](int a, int b) {
      const int id = (int)piece_cost.size();
      piece_cost.push_back(cost_of(f, a, b));
      const int ta = f.Ia * T;
      if (a < f.la) segs.push_back(Seg{f.k, f.Ia, ta + a, ta + std::min(b, f.la), id});
      if (b > f.la) {
        const int tb = f.Ib * T;
        segs.push_back(Seg{f.k, f.Ib, tb + std::max(a - f.la, 0), tb + (b - f.la), id});
      }
    });
  // i-side blocks numbered row by row (system, row, first source)
  std::vector<int> order(segs.size());
  for (size_t i = 0; i < segs.size(); ++i) order[i] = (int)i;
  std::sort(order.begin(), order.end(), [&](int x, int y) {
    const Seg &a = segs[x], &b = segs[y];
    if (a.k != b.k) return a.k < b.k;
    if (a.I != b.I) return a.I < b.I;
    return a.s0 < b.s0;
  });
  std::vector<int> block(segs.size());
  std::vector<int4> tab(K);
  std::vector<int> rowbase(K);
  int nrows = 0;
  for (int k = 0; k < K; ++k) {
    rowbase[k] = K + nrows;
    nrows += (L.n[k] + T - 1) / T;
  }
  std::vector<int4> rowtab(nrows, make_int4(0, 0, 0, 0));
  for (size_t r = 0; r < order.size(); ++r) {
    const Seg& g = segs[order[r]];
    block[order[r]] = (int)r;
    int4& e = rowtab[rowbase[g.k] - K + g.I];
    if (e.y == 0) e.x = (int)((int64_t)r * 2 * T);
    e.y += 1;
  }
  int64_t off = (int64_t)segs.size() * 2 * T;
  std::vector<int64_t> jbase(K);
  for (int k = 0; k < K; ++k) {
    const int n = L.n[k], nT = (n + T - 1) / T;
    jbase[k] = off;
    off += 2 * ((int64_t)nT * n - (int64_t)T * nT * (nT - 1) / 2);
    tab[k] = make_int4(n, rowbase[k], (int)jbase[k], T);
  }
  BIPB_REQUIRE(off < ((int64_t)1 << 31), "mat-vec too large for one symmetric work list");

  // items: three int4 per piece, largest piece first
  const int n_pieces = (int)piece_cost.size();
  std::vector<int4> items((size_t)3 * n_pieces, make_int4(0, 0, 0, 0));
  std::vector<int> nseg(n_pieces, 0);
  for (size_t i = 0; i < segs.size(); ++i) {
    const Seg& g = segs[i];
    const int p = g.piece;
    items[3 * p] = make_int4(L.vec_off[g.k] / 2, L.n[g.k], g.k, (int)jbase[g.k]);
    items[3 * p + 1 + nseg[p]++] = make_int4(g.I * T, g.s0, g.s1, (int)((int64_t)block[i] * 2 * T));
  }
  std::vector<int> porder(n_pieces);
  for (int p = 0; p < n_pieces; ++p) porder[p] = p;
  std::stable_sort(porder.begin(), porder.end(), [&](int x, int y) { return piece_cost[x] > piece_cost[y]; });
  std::vector<int4> sorted((size_t)3 * n_pieces);
  for (int p = 0; p < n_pieces; ++p)
    for (int c = 0; c < 3; ++c) sorted[(size_t)3 * p + c] = items[(size_t)3 * porder[p] + c];
  tab.insert(tab.end(), rowtab.begin(), rowtab.end());
  HostPlan hp;
  hp.items = std::move(sorted);
  hp.tab = std::move(tab);
  hp.n_items = n_pieces;
  hp.part_len = off;
  return hp;
}

// Plan-cache key of one symmetric pass over one layout (SplitMix64 finaliser,
// so that distinct (pass, layout) pairs do not collide by construction).
uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
uint64_t sym_key(int pass_id, uint64_t layout_key) {
  return mix64(layout_key ^ mix64(0x5e11000000000000ull + (uint64_t)pass_id));
}

// Partial sums a symmetric pass over L needs with tiles of T targets (the
// i-side blocks excluded), and whether they fit the 32-bit offsets.
bool sym_fits(const SysLayout& L, int T) {
  int64_t off = 0;
  for (int k = 0; k < L.K; ++k) {
    const int n = L.n[k], nT = (n + T - 1) / T;
    off += 2 * ((int64_t)nT * n - (int64_t)T * nT * (nT - 1) / 2);
  }
  return off < ((int64_t)1 << 30);
}

template <class P, int NT, int TPT, int CH, int MINB>
int sym_occupancy() {
  static int occ = [] {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_sym<P, NT, TPT, CH, MINB>, NT, 0) != cudaSuccess) {
      (void)cudaGetLastError();
      o = 1;
    }
    return std::max(o, 1);
  }();
  return occ;
}

template <class P, int NT, int TPT, int CH, int MINB>
void run_sym(Surface* s, int pass_id, int kind, const SysLayout& L, const typename P::Args& g, bool transpose,
             DevBuf<typename P::V4>& recbuf, DevBuf<typename P::PT>& partbuf, const double* u, double* y,
             double dphi, double dpsi, const int* skip, int skip_stride, double sigma = 1.0, int stages = kSymAll,
             SymStep* step = nullptr) {
  constexpr int T = NT * TPT;
  if (!P::SCALED) sigma = 1.0;
  // A u: P ~ sigma, Q ~ sigma^2; A^T w: P ~ sigma^2, Q ~ sigma (pair.cuh)
  const double2 f = transpose ? make_double2(sigma * sigma, sigma) : make_double2(sigma, sigma * sigma);
  const uint64_t key = sym_key(pass_id, L.key);
  ItemPlan* plan = plan_sym(s, key, L, T, s->num_sms * sym_occupancy<P, NT, TPT, CH, MINB>(), CH);
  s->grow(recbuf, (size_t)(L.len / 2) * P::RW);
  s->grow(partbuf, (size_t)plan->part_len);
  const int4* lay = s->lay_dev(L);
  if constexpr (std::is_same<typename P::PT, float>::value) {
    if (step != nullptr) *step = SymStep{plan->tab.p, partbuf.p, recbuf.p, sigma, f, dphi, dpsi, transpose};
  }
  const dim3 pgrid(blocks_of(L.max_n, 128), L.K);
  if (!(stages & kSymPack)) {
  } else if constexpr (std::is_same<typename P::V4, double4_32a>::value) {
    launch_chained(k_pack_sym64, pgrid, 128, 0, s->stream, lay, transpose, s->tgt64.p, u, recbuf.p, skip, skip_stride,
                   sigma, std::exp2(std::ceil(std::log2(sigma))));
  } else if constexpr (std::is_same<typename P::PT, double>::value) {
    launch_chained(k_pack_sym_df, pgrid, 128, 0, s->stream, lay, transpose, s->tgt64.p, u, recbuf.p, skip, skip_stride,
                   sigma, std::exp2(std::ceil(std::log2(sigma))));
  } else {
    launch_chained(k_pack_sym32, pgrid, 128, 0, s->stream, lay, transpose, s->tgt64.p, u, recbuf.p, skip, skip_stride,
                   sigma);
  }
  if (stages & kSymPack) BIPB_LAUNCHED(s);
  if (stages & kSymPairs) {
    TimedLaunch tl(s, kind);
    launch_chained(k_sym<P, NT, TPT, CH, MINB>, plan->n_items, NT, 0, s->stream, g, plan->items.p, recbuf.p,
                   partbuf.p, skip, skip_stride);
    BIPB_LAUNCHED(s);
  }
  if (stages & kSymReduce) {
    launch_chained(k_reduce_sym<typename P::PT>, dim3(blocks_of(2 * (int64_t)L.max_n, 128), L.K), 128, 0, s->stream, lay, plan->tab.p, partbuf.p, u, y, dphi,
                   dpsi, transpose ? s->tgt64.p : nullptr, skip, skip_stride, f);
    BIPB_LAUNCHED(s);
  }
}

}  // namespace

// The symmetric FP32 / FP64 forms: LAPLACE for kappa = 0, kappa-scaled
// records for kappa >= kSymKappaMin; in between (a Debye length above 1e6 A)
// the scaled 1/r^3 could leave the FP32 range, and the caller takes the
// ordered kernels.

template <typename T>
bool sym_form(double kappa, PairConst<T>& c, bool& laplace) {
  laplace = kappa == 0.0;
  if (!laplace && kappa < kSymKappaMin) return false;
  c.smax = (T)(laplace ? kSMaxD : kSMaxD / kappa);  // the 1/r cap at 1e-6 A, in the units of the records
  return true;
}

bool matvec_sym32(Surface* s, const SysLayout& L, const PairConst<float>& c0, double kappa, bool transpose,
                  int variant, const double* u, double* y, double dphi, double dpsi, const int* skip,
                  int skip_stride, int stages, SymStep* step) {
  if (variant < 0 || variant > 2) throw Error(BIPB_ERR_INVALID_ARG, "unknown symmetric FP32 mat-vec variant");
  // Shapes (threads, targets per thread, tile of targets): 0 (256, 2, 512), 1
  // (128, 4, 512), 2 (256, 4, 1024), 3 (128, 2, 256).  Variant 2 takes the
  // shape by size.  A tile of T targets evaluates n T / 2 masked pairs of its
  // own diagonal beside the n^2 / 2 real ones, and a small surface needs small
  // tiles to give every SM work, while the large tile shares each source load
  // among more targets.  Whole mat-vec, us, tile 1024 / 512 / 256: N = 1280 28.8
  // / 25.6 / 22; 2500 38.3 / 29.5 / 25.7; 3500 43.1 / 38.1 / 34.9; 4200 55 / 37.0 /
  // 39.2; 20480 358 / 351 / 356; 40000 1234 / 1196 / 1300; 46000 1574 / 1578 / 1778;
  // 65537 3138 / 3170 / 3584.
  int shape = variant;
  static const int kT[4] = {512, 512, 1024, 256};
  if (variant == 2) {
    shape = L.max_n < 4096 ? 3 : L.max_n < 45056 ? 1 : 2;
    if (!sym_fits(L, kT[shape])) shape = 2;  // a large batch: fewer partial sums
  }
  PairConst<float> c = c0;
  bool lap = false;
  if (!sym_fits(L, kT[shape]) || !sym_form(kappa, c, lap)) return false;
  const int kind = transpose ? kTMv32T : kTMv32;
#define BIPB_SYM32_RUN(TR_, LAP_, V_, NT_, TPT_, CH_, MINB_)                                                       \
  run_sym<Sym32Policy<TR_, LAP_>, NT_, TPT_, CH_, MINB_>(s, (TR_ ? 0x100 : 0x200) + V_, kind, L, {c}, TR_, s->rec32, \
                                                         s->part32, u, y, dphi, dpsi, skip, skip_stride, kappa, stages, step)
#define BIPB_SYM32(V_, NT_, TPT_, CH_, MINB_)                     \
  case V_:                                                         \
    if (transpose) {                                               \
      if (lap)                                                     \
        BIPB_SYM32_RUN(true, true, V_, NT_, TPT_, CH_, MINB_);     \
      else                                                         \
        BIPB_SYM32_RUN(true, false, V_, NT_, TPT_, CH_, MINB_);    \
    } else {                                                       \
      if (lap)                                                     \
        BIPB_SYM32_RUN(false, true, V_, NT_, TPT_, CH_, MINB_);    \
      else                                                         \
        BIPB_SYM32_RUN(false, false, V_, NT_, TPT_, CH_, MINB_);   \
    }                                                              \
    return true;
  switch (shape) {
    BIPB_SYM32(0, 256, 2, 64, 3)
    BIPB_SYM32(1, 128, 4, 64, 4)
    BIPB_SYM32(2, 256, 4, 64, 2)
    BIPB_SYM32(3, 128, 2, 32, 6)
  }
#undef BIPB_SYM32
#undef BIPB_SYM32_RUN
  return false;
}

// FP64 shapes: tiles of 64 targets in CTAs of 64 threads up to 32768 elements,
// tiles and CTAs of 256 above.  Small tiles leave less of the diagonal masked
// and more, shorter work items (N = 320 60 against 135 us, 1000 107 / 198, 7001
// 1062 / 1167, 20000 8330 / 8490), and
// the j-side partials (8 n^2 / T bytes: 134 MB at 32768 with T = 64) would only grow.
constexpr int kSym64Small = 32768;

bool matvec_sym64(Surface* s, const SysLayout& L, const PairConst<double>& c0, double kappa, bool transpose,
                  const double* u, double* y, double dphi, double dpsi, const int* skip, int skip_stride) {
  PairConst<double> c = c0;
  bool lap = false;
  const bool small = L.max_n <= kSym64Small && sym_fits(L, 64);  // else fewer partial sums
  if (!sym_fits(L, small ? 64 : 256) || !sym_form(kappa, c, lap)) return false;
  TfConst t;
  t.em1 = tf_from_double(c.eps - 1.0), t.eps = tf_from_double(c.eps);
  t.im1 = tf_from_double(c.inveps - 1.0), t.inv = tf_from_double(c.inveps);
  tf_set_cap(t, c.smax);
#define BIPB_SYM64_RUN(TR_, LAP_, V_, NT_, CH_, MINB_)                                                          \
  run_sym<Sym64Policy<TR_, LAP_>, NT_, 1, CH_, MINB_>(s, (TR_ ? 0x300 : 0x400) + V_, TR_ ? kTMv64T : kTMv64, L, \
                                                      {t, s->exptab.p}, TR_, s->rec64, s->part64, u, y, dphi,  \
                                                      dpsi, skip, skip_stride, kappa)
#define BIPB_SYM64(V_, NT_, CH_, MINB_)                    \
  if (transpose) {                                         \
    if (lap)                                               \
      BIPB_SYM64_RUN(true, true, V_, NT_, CH_, MINB_);     \
    else                                                   \
      BIPB_SYM64_RUN(true, false, V_, NT_, CH_, MINB_);    \
  } else {                                                 \
    if (lap)                                               \
      BIPB_SYM64_RUN(false, true, V_, NT_, CH_, MINB_);    \
    else                                                   \
      BIPB_SYM64_RUN(false, false, V_, NT_, CH_, MINB_);   \
  }
  if (small) {
    BIPB_SYM64(0, 64, 32, 8)
  } else {
    BIPB_SYM64(1, 256, 64, 1)
  }
#undef BIPB_SYM64
#undef BIPB_SYM64_RUN
  return true;
}

bool matvec_sym_df(Surface* s, const SysLayout& L, const DFConst& c, double kappa, bool transpose, const double* u,
                   double* y, double dphi, double dpsi, const int* skip, int skip_stride) {
  if (!sym_fits(L, 128)) return false;
  // kappa-scaled records for kappa >= kSymKappaMin (the FP32 rule), unscaled otherwise
  const bool scaled = kappa >= kSymKappaMin;
#define BIPB_SYMDF_RUN(TR_, SC_)                                                                                 \
  run_sym<SymDFPolicy<TR_, SC_>, 128, 1, 32, 1>(s, TR_ ? 0x500 : 0x600, TR_ ? kTMvDFT : kTMvDF, L, {c}, TR_,     \
                                               s->recdf, s->part64, u, y, dphi, dpsi, skip, skip_stride, kappa)
  if (transpose) {
    if (scaled)
      BIPB_SYMDF_RUN(true, true);
    else
      BIPB_SYMDF_RUN(true, false);
  } else {
    if (scaled)
      BIPB_SYMDF_RUN(false, true);
    else
      BIPB_SYMDF_RUN(false, false);
  }
#undef BIPB_SYMDF_RUN
  return true;
}

}  // namespace bipb

// Device-resident restarted GMRES (Saad & Schultz; the Krylov solver of
// Sec. 2.2.2) over a batch of independent systems, and mixed-precision
// iterative refinement.
//
// Unlike the paper's GPU pipeline (Sec. 2.4), which copies x and y across
// PCIe and runs the Arnoldi process on the host every iteration, every step
// here stays on the device: mat-vec, classical Gram-Schmidt with one
// re-orthogonalisation (CGS2, the same Krylov basis as modified Gram-Schmidt
// in exact arithmetic, but as matrix-vector shaped passes; one pass for the
// FP32 Krylov solve inside the mixed modes), Givens rotations and the
// convergence test.  K systems (right-hand sides of one surface, or
// surfaces of uneven size) advance together: one Krylov vector is the
// concatenation of the K systems' vectors, every kernel covers all of them,
// and a system that has converged skips its share.  The host reads one small
// status record per system per restart cycle.  One cycle (m Arnoldi steps,
// the least-squares update and the restart vector) is recorded once as a
// CUDA graph and replayed.
//
// Restart vector: after k steps the residual of the new iterate is
// r = V_{k+1} Q^T (g_k e_{k+1}) (Q the product of the Givens rotations), so
// the next cycle starts from it without another mat-vec; the true residual
// b - A x is computed when the recurrence reports convergence.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <map>
#include <mutex>

#include "internal.cuh"
#include "symstep.cuh"

namespace bipb {

namespace {

constexpr int kBS = 256;
constexpr double kInv4PiG = 1.0 / (4.0 * kPi);

struct DevState {
  int k;       // Arnoldi steps done in this cycle
  int skip;    // nonzero: the rest of the cycle does nothing for this system
  int conv;    // recurrence residual <= tol
  int stop;    // iteration cap reached
  int iters;   // Arnoldi steps in this call
  int max_iter;
  int m;
  int active;  // the system takes part in this call
  double tol;    // relative to bnorm
  double bnorm;  // norm of the right-hand side of this call
  double beta;   // norm of the current cycle's start residual
  double est;    // latest |g_k| / bnorm
  int arrive;    // blocks of this system done with the current normalisation step
  int pad_;
};
constexpr int kStateInts = (int)(sizeof(DevState) / sizeof(int));
static_assert(offsetof(DevState, skip) == sizeof(int), "skip must be the second int");

// Sum over the block in a fixed order, valid in thread 0.  One warp adds the
// values from shared memory: a tree of shuffles in every warp would take
// five times the FP64 additions (two lanes per SM).
template <int NT>
__device__ double block_sum(double v) {
  __shared__ double red[NT];
  __syncthreads();
  red[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    double p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) p[i & 3] += red[32 * i + threadIdx.x];
    t = (p[0] + p[1]) + (p[2] + p[3]);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  return t;
}

// Block table: blk[b] = {system, first element, end element, first block of
// the system}, sysb[k] = {first block, end block, 0, 0}, lay[k] = {geo_off, n,
// vec_off, chg_off}.  A block owns a range of one system's elements: their phi
// unknowns vec_off + e and their psi unknowns vec_off + n + e.

// Sum of v over a warp in a fixed order (tree of shuffles down), then
// broadcast from lane 0, so every lane holds the same, reproducible value.
__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}

// sum over blocks b in [b0, b1) of part[b * stride + i], by one warp, fixed order
__device__ __forceinline__ double warp_sum_parts(const double* part, int stride, int i, int b0, int b1) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  constexpr int U = 5;  // loads in flight, the last batch filled with zeros (sum_strided)
  for (int b = b0 + lane; b < b1; b += 32 * U) {
    double v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) v[q] = b + 32 * q < b1 ? part[(size_t)(b + 32 * q) * stride + i] : 0.0;
#pragma unroll
    for (int q = 0; q < U; ++q) s += v[q];
  }
  if (b1 - b0 > 8) return warp_sum(s);
  for (int o = 4; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);  // lanes 0..7 hold all of it
  return __shfl_sync(0xffffffffu, s, 0);
}

// The lines of V_0 .. V_j that the block reads, into L1 (they are read in two
// phases of the step, whose first loads would each wait for L2).
template <int NT>
__device__ __forceinline__ void prefetch_basis(int j, int64_t len, const double* V, int4 B, int4 Lk) {
  const int lines = ((B.z - B.y) * 8 + 127) / 128 + 1;
  for (int t = threadIdx.x; t < 2 * (j + 1) * lines; t += NT) {
    const int r = t / lines, q = t % lines;
    const double* p = V + (size_t)(r >> 1) * len + Lk.z + (r & 1) * Lk.y + min(B.y + 16 * q, B.z - 1);
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
  }
}

// part[b * m1 + i] = V_i . w over block b's unknowns, i <= j: one warp per
// vector (one tree of FP64 shuffles each), its phi and psi unknowns side by
// side.  V and w hold values that other threads of the cluster or block wrote in
// this kernel.
template <int NT>
__device__ __forceinline__ void block_dots(int j, int m1, int64_t len, const double* V, const double* w,
                                           double* part, int b, int4 B, int4 Lk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = warp; i <= j; i += NT / 32) {
    const double *v = V + (size_t)i * len + Lk.z, *x = w + Lk.z;
    double acc[2] = {0.0, 0.0};
    constexpr int U = 5;  // elements in flight, the last batch filled with zeros (sum_strided)
    for (int e = B.y + lane; e < B.z; e += 32 * U) {
      double p[2 * U], q[2 * U];
#pragma unroll
      for (int r = 0; r < 2 * U; ++r) {
        const int o = e + 32 * (r >> 1);
        const bool in = o < B.z;
        p[r] = in ? v[o + (r & 1) * Lk.y] : 0.0;
        q[r] = in ? x[o + (r & 1) * Lk.y] : 0.0;
      }
#pragma unroll
      for (int r = 0; r < 2 * U; ++r) acc[r & 1] += p[r] * q[r];
    }
    const double t = warp_sum(acc[0] + acc[1]);
    if (lane == 0) part[(size_t)b * m1 + i] = t;
  }
}

// Preconditioning by the element self blocks (Sec. 2.2.4 with one element per
// leaf): with the self pair omitted, element i's 2 x 2 block of A is
// diag(1/2 (1 + eps), 1/2 (1 + 1/eps)), so M^-1 scales the phi rows by pre.x
// and the psi rows by pre.y.  It is applied on the right, A M^-1 y = r,
// d = M^-1 y: GMRES then minimises the true residual, which is what the
// stopping tests and the refinement read.

// One Arnoldi step after the mat-vec, in three phases with a reduction over the
// system's blocks between them: the dot products V^T w (with FUSED, w first
// summed from the symmetric FP32 mat-vec's partial sums); w -= V h and ||w||;
// the next basis vector, the Givens rotation and (FUSED) the next mat-vec's
// records.  As three kernels (a block per about 128 elements), or, for small
// systems, as one kernel with one cluster of CTAs per system, whose barrier
// takes the place of the kernel boundaries.
// What bounds the cluster's step (10.6 us at N = 1280, the tenth vector; 14.2
// before): a chain of latencies.  So every loop keeps its loads in flight
// together (a rolled remainder waits for each), the basis is fetched into L1 beside
// the mat-vec's sums, tables are read before the previous kernel's end, and the Givens
// step's state and reciprocal beside the dot products; and FP64 additions
// (two lanes per SM), so a vector takes one tree of shuffles and a block's sum
// one warp.
struct StepArgs {
  int j, m;
  int64_t len;
  double *V, *w;
  double *part, *part2, *part1;  // per block: dots, second-pass dots, norm
  double *H, *cs, *sn, *g;
  DevState* st;
  const int4 *blk, *sysb, *lay;
  double* tz;    // M^-1 v_{j+1} (preconditioned), or nullptr
  double2 pre;   // M^-1
  SymStep mv;    // FUSED: the symmetric mat-vec
  const double* u;  // FUSED: its input
  const double4_32a* tgt64;
};

template <int NT, bool FUSED>
__device__ __forceinline__ void step_dots(const StepArgs& a, int b, int4 B, int4 Lk, int4 Sm) {
  if (FUSED) {
    const int cnt = B.z - B.y;
    for (int t = threadIdx.x; t < 2 * cnt; t += NT) {
      const int c = t < cnt ? 0 : 1, e = B.y + t - c * cnt;
      const int64_t x = Lk.z + (int64_t)c * Lk.y + e;
      const double ux = a.u[x];
      const double sc = kInv4PiG * (a.mv.transpose ? a.tgt64[2 * (Lk.x + e)].w : 1.0);
      const double acc = sym_sum(a.mv.tab, Sm, a.mv.part, e, c);
      a.w[x] = (c ? a.mv.dpsi : a.mv.dphi) * ux - sc * (c ? a.mv.f.y : a.mv.f.x) * acc;
    }
    __syncthreads();  // the block's w is visible to all its threads
  }
  block_dots<NT>(a.j, a.m + 1, a.len, a.V, a.w, a.part, b, B, Lk);
}

// h_i = sum over the system's blocks of part[.][i]; w -= sum_i h_i V_i; H[:, j] (+)= h;
// with NORM, also part1[b] = sum of the updated w^2 over block b's unknowns;
// otherwise the block's dot products of the updated w for the second
// Gram-Schmidt pass (block-local, so they need no reduction in between).
// col: the system's column of H as well, in the first block.
template <int NT, bool NORM>
__device__ __forceinline__ void step_orth(const StepArgs& a, const double* part, int accumulate, int b, int4 B,
                                          int4 S, int4 Lk, double* col) {
  const int j = a.j, m1 = a.m + 1;
  __shared__ double h[kMaxRestart + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();  // h of an earlier phase has been read
  for (int i = warp; i <= j; i += NT / 32) {
    const double v = warp_sum_parts(part, m1, i, S.x, S.y);
    if (lane == 0) h[i] = v;
  }
  __syncthreads();
  if (b == S.x) {
    double* Hs = a.H + (size_t)B.x * m1 * a.m + (size_t)j * m1;
    for (int i = threadIdx.x; i <= j; i += NT) {
      const double v = accumulate ? Hs[i] + h[i] : h[i];
      Hs[i] = v;
      if (col != nullptr) col[i] = v;
    }
  }
  double ss = 0.0;
  const int cnt = B.z - B.y;
  for (int t = threadIdx.x; t < 2 * cnt; t += NT) {
    const int64_t x = Lk.z + B.y + (t < cnt ? t : t - cnt + Lk.y);
    double p = a.w[x];
    constexpr int U = 4;
    for (int i0 = 0; i0 <= j; i0 += U) {
      double v[U];
#pragma unroll
      for (int q = 0; q < U; ++q) v[q] = i0 + q <= j ? a.V[(size_t)(i0 + q) * a.len + x] : 0.0;
#pragma unroll
      for (int q = 0; q < U; ++q) p -= h[min(i0 + q, j)] * v[q];
    }
    a.w[x] = p;
    ss += p * p;
  }
  if (NORM) {
    ss = block_sum<NT>(ss);
    if (threadIdx.x == 0) a.part1[b] = ss;
  } else {
    __syncthreads();  // the block's updated w is visible to all its threads
    block_dots<NT>(j, m1, a.len, a.V, a.w, a.part2, b, B, Lk);
  }
}

// What the Givens step reads beside the new column: the earlier rotations and
// the system's state.  Loaded by one warp of the system before it is needed.
struct GivensIn {
  double cs[kMaxRestart], sn[kMaxRestart], col[kMaxRestart + 1];
  double gj, inv_bnorm, tol;
  int iters, max_iter, m;
};
__device__ __forceinline__ void givens_load(const StepArgs& a, int sys, GivensIn& in) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < a.j; i += 32) in.cs[i] = a.cs[(size_t)sys * a.m + i], in.sn[i] = a.sn[(size_t)sys * a.m + i];
  if (lane == 0) {
    const DevState& S = a.st[sys];
    in.gj = a.g[(size_t)sys * (a.m + 1) + a.j];
    in.inv_bnorm = S.bnorm > 0.0 ? 1.0 / S.bnorm : 0.0;
    in.tol = S.tol, in.iters = S.iters, in.max_iter = S.max_iter, in.m = S.m;
  }
}

// Per system: apply earlier rotations to column j (in.col, then b = ||w||, given
// as b^2), make rotation j, update g, test.  One thread: the recurrence is
// serial, one FP64 multiply-add a rotation; b and 1/|(a, b)| are both
// taken from b^2, so the two 1/sqrt run side by side.
__device__ void givens_step(const StepArgs& A, int sys, const GivensIn& in, double b2) {
  const int j = A.j, m = A.m, m1 = m + 1;
  DevState& S = A.st[sys];
  double *cs = A.cs, *sn = A.sn;
  double* h = A.H + (size_t)sys * m1 * m + (size_t)j * m1;
  double* g_ = A.g + (size_t)sys * m1;
  const double gj = in.gj, tol = in.tol;
  const int iters = in.iters + 1, max_iter = in.max_iter, Sm = in.m;
  double a = in.col[0];
#pragma unroll 4
  for (int i = 0; i < j; ++i) {
    const double c = in.cs[i], t = in.sn[i], x = in.col[i + 1];
    h[i] = fma(c, a, t * x);
    a = fma(-t, a, c * x);
  }
  const double b = b2 > 0.0 ? b2 * rsqrt(b2) : 0.0;
  // den = sqrt(a^2 + b^2) = |(a, b)| of the pair scaled by a power of two near its
  // larger part; that of b is half the exponent of b^2
  const int eb = (((__double2hiint(b2) >> 20) & 0x7ff) + 1023) >> 1;
  const int big = max((__double2hiint(a) >> 20) & 0x7ff, b2 > 0.0 ? eb : 0);
  const int up = min(max(big, 1), 2045);
  const double down = __hiloint2double((2046 - up) << 20, 0), back = __hiloint2double(up << 20, 0);  // 2^(1023 - up), 2^(up - 1023)
  const double as = a * down, q = as * as + (b2 * down) * down;
  const double inv = q > 0.0 ? rsqrt(q) : 0.0;
  const double den = q * inv * back;
  const double c = q > 0.0 ? as * inv : 1.0, s = (b * down) * inv;
  h[j] = den;
  h[j + 1] = 0.0;
  cs[(size_t)sys * m + j] = c;
  sn[(size_t)sys * m + j] = s;
  const double gj1 = -s * gj;
  g_[j + 1] = gj1;
  g_[j] = c * gj;
  S.k = j + 1;
  S.iters = iters;
  const double est = fabs(gj1) * in.inv_bnorm;
  S.est = est;
  const int conv = est <= tol || b == 0.0;
  const int stop = iters >= max_iter;
  if (conv) S.conv = 1;
  if (stop) S.stop = 1;
  if (conv || stop || j + 1 == Sm) S.skip = 1;
}

// (||w||^2, 1 / ||w||) of the system from the blocks' sums, in each of the block's first NT threads (0, 0 for w = 0)
template <int NT = kBS>
__device__ __forceinline__ double2 step_norm(const double* part1, int4 S) {
  __shared__ double2 nrm;
  if (threadIdx.x < 32) {
    const double s = warp_sum_parts(part1, 1, 0, S.x, S.y);
    if (threadIdx.x == 0) nrm = make_double2(s, s > 0.0 ? rsqrt(s) : 0.0);
  }
  asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
  return nrm;
}

// v_{j+1} = inv w (and tz = M^-1 v_{j+1} when preconditioned, and FUSED the
// next mat-vec's records), by the block's first NT threads.
template <int NT, bool FUSED>
__device__ __forceinline__ void step_next(const StepArgs& a, double inv, int4 B, int4 Lk) {
  double* out = a.V + (size_t)(a.j + 1) * a.len;
  const bool pack = FUSED && a.j + 1 < a.m;
  for (int e = B.y + threadIdx.x; e < B.z; e += NT) {
    const int64_t x = Lk.z + e, y = x + Lk.y;
    double p = a.w[x] * inv, q = a.w[y] * inv;
    out[x] = p;
    out[y] = q;
    if (a.tz != nullptr) {
      p *= a.pre.x;
      q *= a.pre.y;
      a.tz[x] = p;
      a.tz[y] = q;
    }
    if (pack)
      sym32_refresh(a.tgt64[2 * (Lk.x + e)].w, p, q, a.mv.transpose, a.mv.sigma,
                    a.mv.rec + 5 * (size_t)(Lk.z / 2 + e));
  }
}

template <bool FUSED>
__global__ void __launch_bounds__(kBS) k_dots(StepArgs a) {
  // the tables are constant: read while the previous kernel ends
  const int4 B = a.blk[blockIdx.x], Lk = a.lay[B.x], Sm = FUSED ? a.mv.tab[B.x] : make_int4(0, 0, 0, 0);
  chain_wait();
  chain_release();
  if (a.st[B.x].skip) return;
  prefetch_basis<kBS>(a.j, a.len, a.V, B, Lk);
  step_dots<kBS, FUSED>(a, blockIdx.x, B, Lk, Sm);
}

template <bool NORM>
__global__ void __launch_bounds__(kBS) k_orth(StepArgs a, const double* part, int accumulate) {
  const int4 B = a.blk[blockIdx.x], S = a.sysb[B.x], Lk = a.lay[B.x];
  chain_wait();
  chain_release();
  if (a.st[B.x].skip) return;
  step_orth<kBS, NORM>(a, part, accumulate, blockIdx.x, B, S, Lk, nullptr);
}

// The Givens step is made by the last block of the system to finish (every
// block has then passed its skip test, so the step may set skip; the blocks'
// arrival is counted with an atomic after a fence, no block waits).
template <bool FUSED>
__global__ void __launch_bounds__(kBS) k_normalize(StepArgs a) {
  const int4 B = a.blk[blockIdx.x], S = a.sysb[B.x], Lk = a.lay[B.x];
  chain_wait();
  chain_release();
  if (a.st[B.x].skip) return;
  // every block reads what the Givens step needs, beside the norm: which one makes it is known
  // at the end only, and two rounds of loads and a division would follow
  __shared__ GivensIn in;
  if (threadIdx.x >= kBS - 32) {
    givens_load(a, B.x, in);
    const double* Hc = a.H + (size_t)B.x * (a.m + 1) * a.m + (size_t)a.j * (a.m + 1);
    for (int i = threadIdx.x - (kBS - 32); i <= a.j; i += 32) in.col[i] = Hc[i];
  }
  const double2 v = step_norm(a.part1, S);
  step_next<kBS, FUSED>(a, v.y, B, Lk);
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&a.st[B.x].arrive, 1) == S.y - S.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) {
    a.st[B.x].arrive = 0;
    givens_step(a, B.x, in, v.x);
  }
}

// The whole step in one launch: a cluster of kClu CTAs per system (its blocks).
// The cluster barrier orders the phases and makes each CTA's partial sums,
// w and H visible to the others.
constexpr int kClu = 8;      // CTAs of a cluster (the portable size)
constexpr int kCluNT = 512;  // threads of each
template <bool CGS2, bool FUSED>
__global__ void __cluster_dims__(kClu, 1, 1) __launch_bounds__(kCluNT) k_step(StepArgs a) {
  const int4 B = a.blk[blockIdx.x], S = a.sysb[B.x], Lk = a.lay[B.x];
  const int4 Sm = FUSED ? a.mv.tab[B.x] : make_int4(0, 0, 0, 0);
  chain_wait();
  chain_release();
  if (a.st[B.x].skip) return;  // the same for every CTA of the cluster
  __shared__ GivensIn in;
  const bool first = (int)blockIdx.x == S.x;
  prefetch_basis<kCluNT>(a.j, a.len, a.V, B, Lk);
  if (first && threadIdx.x >= kCluNT - 32) givens_load(a, B.x, in);
  step_dots<kCluNT, FUSED>(a, blockIdx.x, B, Lk, Sm);
  cluster_sync();
  if (CGS2) {
    step_orth<kCluNT, false>(a, a.part, 0, blockIdx.x, B, S, Lk, nullptr);
    cluster_sync();
    step_orth<kCluNT, true>(a, a.part2, 1, blockIdx.x, B, S, Lk, first ? in.col : nullptr);
  } else {
    step_orth<kCluNT, true>(a, a.part, 0, blockIdx.x, B, S, Lk, first ? in.col : nullptr);
  }
  cluster_sync();  // also: every CTA has passed its skip test
  // the last warp of the system's first block makes the Givens step beside the others' vector work
  if (threadIdx.x < kCluNT - 32) {
    const double2 v = step_norm<kCluNT - 32>(a.part1, S);
    step_next<kCluNT - 32, FUSED>(a, v.y, B, Lk);
  } else if (first) {
    const double b2 = warp_sum_parts(a.part1, 1, 0, S.x, S.y);
    if (threadIdx.x == kCluNT - 32) givens_step(a, B.x, in, b2);
  }
}

// part1[b] = sum of w^2 over block b's unknowns (mode 0: systems not skipped,
// mode 1: active systems, mode 2: every system)
__global__ void k_sumsq(const double* __restrict__ w, double* __restrict__ part1, const DevState* st,
                        const int4* __restrict__ blk, const int4* __restrict__ lay, int mode) {
  const int4 B = blk[blockIdx.x];
  if ((mode == 0 && st[B.x].skip) || (mode == 1 && !st[B.x].active)) return;
  const int4 Lk = lay[B.x];
  double acc = 0.0;
  for (int e = B.y + threadIdx.x; e < B.z; e += kBS) {
    const double p = w[Lk.z + e], q = w[Lk.z + Lk.y + e];
    acc += p * p + q * q;
  }
  acc = block_sum<kBS>(acc);
  if (threadIdx.x == 0) part1[blockIdx.x] = acc;
}

// Start of a solve, per active system: beta = bnorm = ||r0||, v_0 = r0 / beta
// (and tz = M^-1 v_0 when preconditioned).
__global__ void k_start(const double* __restrict__ r0, double* __restrict__ V, const double* __restrict__ part1,
                        DevState* st, const int4* __restrict__ blk, const int4* __restrict__ sysb,
                        const int4* __restrict__ lay, double* __restrict__ tz, double2 pre) {
  const int4 B = blk[blockIdx.x];
  if (!st[B.x].active) return;
  const int4 S = sysb[B.x], Lk = lay[B.x];
  const double2 v = step_norm(part1, S);
  const double inv = v.y;
  for (int e = B.y + threadIdx.x; e < B.z; e += kBS) {
    const int64_t x = Lk.z + e, y = x + Lk.y;
    const double p = r0[x] * inv, q = r0[y] * inv;
    V[x] = p;
    V[y] = q;
    if (tz != nullptr) tz[x] = pre.x * p, tz[y] = pre.y * q;
  }
  if (threadIdx.x == 0 && (int)blockIdx.x == S.x) {
    st[B.x].bnorm = v.x * inv;
    st[B.x].beta = v.x * inv;
  }
}

// Per system (one block): least squares R y = g (k x k) and the restart
// coefficients z = Q^T (g_k e_k) / |g_k|, from shared copies of the rotations
// and of g (one thread makes the serial recurrences).
__global__ void __launch_bounds__(64) k_lsq(int m, const double* __restrict__ H, const double* __restrict__ cs,
                      const double* __restrict__ sn, const double* __restrict__ g, double* __restrict__ y,
                      double* __restrict__ z, DevState* st) {
  chain_wait();
  chain_release();
  const int sys = blockIdx.x;
  DevState& S = st[sys];
  const int k = S.k;
  if (!S.active || k == 0) return;
  const int m1 = m + 1;
  __shared__ double c_[kMaxRestart], s_[kMaxRestart], r_[kMaxRestart + 1], z_[kMaxRestart + 1], d_[kMaxRestart];
  const double* Hs = H + (size_t)sys * m1 * m;
  for (int i = threadIdx.x; i <= k; i += 64) {
    // the reciprocals of the diagonal side by side: a division in each step of the
    // back substitution was most of this kernel
    if (i < k) c_[i] = cs[(size_t)sys * m + i], s_[i] = sn[(size_t)sys * m + i], d_[i] = 1.0 / Hs[(size_t)i * m1 + i];
    r_[i] = g[(size_t)sys * m1 + i];
  }
  // R as well, where it is small: each step would wait for its column from L2
  constexpr int kR = 32;
  __shared__ double R_[kR * kR];
  const bool small = k <= kR;
  if (small)
    for (int t = threadIdx.x; t < k * k; t += 64) R_[t / k * kR + t % k] = Hs[(size_t)(t / k) * m1 + t % k];
  __syncthreads();
  const double gk = r_[k], beta = fabs(gk);
  if (threadIdx.x >= 32) {  // second warp: the restart coefficients
    if (threadIdx.x == 32) {
      for (int i = 0; i <= k; ++i) z_[i] = 0.0;
      z_[k] = beta > 0.0 ? gk / beta : 0.0;
      for (int i = k - 1; i >= 0; --i) {
        const double a = z_[i], b = z_[i + 1];
        z_[i] = c_[i] * a - s_[i] * b;
        z_[i + 1] = s_[i] * a + c_[i] * b;
      }
      S.beta = beta;
    }
    __syncwarp();
    for (int i = threadIdx.x - 32; i <= k; i += 32) z[(size_t)sys * m1 + i] = z_[i];
  } else {  // first warp: back substitution by columns, the solved entries in r_
    for (int i = k - 1; i >= 0; --i) {
      const double yi = r_[i] * d_[i];
      const double* col = small ? R_ + i * kR : Hs + (size_t)i * m1;
      __syncwarp();
      for (int l = threadIdx.x; l < i; l += 32) r_[l] -= col[l] * yi;
      if (threadIdx.x == 0) y[(size_t)sys * m + i] = yi;
      __syncwarp();
    }
  }
}

// x += M^-1 sum_{i<k} y_i V_i ; V_0 <- sum_{i<=k} z_i V_i (per system); when
// preconditioned (tz != nullptr) also tz = M^-1 V_0, the next cycle's first input
__global__ void k_update(int m, int64_t len, double* __restrict__ V, double* __restrict__ x,
                         const double* __restrict__ y, const double* __restrict__ z, const DevState* st,
                         const int4* __restrict__ blk, double* __restrict__ tz, const int4* __restrict__ lay,
                         double2 pre) {
  chain_wait();
  chain_release();
  const int4 B = blk[blockIdx.x];
  const DevState& S = st[B.x];
  const int k = S.k;
  if (!S.active || k == 0) return;
  const int4 Lk = lay[B.x];
  const double* y_ = y + (size_t)B.x * m;
  const double* z_ = z + (size_t)B.x * (m + 1);
  for (int c = 0; c < 2; ++c) {
    const double f = c ? pre.y : pre.x;
    for (int o = B.y + threadIdx.x; o < B.z; o += kBS) {
      const int64_t e = Lk.z + c * Lk.y + o;
      double dx = 0.0, v0 = 0.0;
      constexpr int U = 4;
      for (int i0 = 0; i0 <= k; i0 += U) {
        double v[U];
#pragma unroll
        for (int q = 0; q < U; ++q) v[q] = i0 + q <= k ? V[(size_t)(i0 + q) * len + e] : 0.0;
#pragma unroll
        for (int q = 0; q < U; ++q) {
          dx += (i0 + q < k ? y_[i0 + q] : 0.0) * v[q];
          v0 += z_[min(i0 + q, k)] * v[q];
        }
      }
      if (tz != nullptr) {
        x[e] += f * dx;
        tz[e] = f * v0;
      } else {
        x[e] += dx;
      }
      V[e] = v0;
    }
  }
}

__global__ void k_next_cycle(int m, int K, double* __restrict__ g, DevState* st) {
  chain_wait();
  chain_release();
  const int sys = blockIdx.x * blockDim.x + threadIdx.x;
  if (sys >= K) return;
  DevState& S = st[sys];
  if (!S.active) return;
  double* g_ = g + (size_t)sys * (m + 1);
  g_[0] = S.beta;
  for (int i = 1; i <= m; ++i) g_[i] = 0.0;
  S.k = 0;
  S.est = S.bnorm > 0.0 ? S.beta / S.bnorm : 0.0;
  if (S.beta == 0.0 || S.est <= S.tol) S.conv = 1;
  S.skip = (S.conv || S.stop) ? 1 : 0;
}

__global__ void k_sub(int64_t len, const double* __restrict__ a, const double* __restrict__ b,
                      double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * kBS + threadIdx.x;
  if (i < len) out[i] = a[i] - b[i];
}
__global__ void k_add(int64_t len, const double* __restrict__ a, double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * kBS + threadIdx.x;
  if (i < len) out[i] += a[i];
}

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, (n + kBS - 1) / kBS); }

struct GraphTag {
  uint64_t gen;
  double eps_in, eps_out, kappa;
  bool timed;
  bool operator==(const GraphTag& o) const {
    return gen == o.gen && eps_in == o.eps_in && eps_out == o.eps_out && kappa == o.kappa && timed == o.timed;
  }
};
struct Recorded {
  cudaGraphExec_t exec;
  GraphTag tag;
  std::vector<EventPair> events;  // timing events recorded inside the graph
  long long kernels;              // kernel nodes in the graph
};

}  // namespace

struct GmresWork {
  uint64_t lay_key = 0;
  int m = 0, K = 0, nblk = 0;  // nblk: blocks of blk
  int precond = 0;  // bipb_precond of the current call
  int64_t len = 0;
  DevBuf<double> V, w, H, cs, sn, g, y, z, part, part2, part1, r, d, t, tz;
  DevBuf<int4> blk, sysb;      // blocks of about 128 elements
  DevBuf<int4> cblk, csysb;    // kClu blocks per system (the cluster step)
  DevBuf<int> mask;  // per system: 1 = leave out of the FP64 residual
  std::vector<int4> sysb_host;
  DevBuf<DevState> st_buf;
  DevState* st = nullptr;  // st_buf.p
  // host copies (pageable: every transfer of them is followed by a synchronisation)
  std::vector<DevState> st_host;
  std::vector<double> part1_host;
  std::vector<int> mask_host;
  std::map<int, Recorded> graphs;  // recorded cycles keyed by (precision, transpose, precond)
  const std::vector<EventPair>* replayed = nullptr;
  int device = 0;
  ~GmresWork();
};

namespace {

// Executable restart-cycle graphs of destroyed handles, kept for reuse: a new
// handle records its own cycle and, when a kept executable of the same kind
// accepts that graph (cudaGraphExecUpdate checks that the topology matches),
// updates it in place instead of instantiating a new one.  At most kPoolMax
// are kept; they are released with the process (the pool is never destroyed,
// so no CUDA call runs during static destruction).
struct PooledExec {
  int device, key;
  cudaGraphExec_t exec;
};
constexpr size_t kPoolMax = 16;
std::mutex& pool_mutex() {
  static auto* m = new std::mutex;
  return *m;
}
std::vector<PooledExec>& exec_pool() {
  static auto* v = new std::vector<PooledExec>;
  return *v;
}

void pool_put(int device, int key, cudaGraphExec_t exec) {
  std::lock_guard<std::mutex> lock(pool_mutex());
  if (exec_pool().size() < kPoolMax) {
    exec_pool().push_back(PooledExec{device, key, exec});
  } else {
    cudaGraphExecDestroy(exec);
  }
}

// An executable updated to run graph g, or nullptr.
cudaGraphExec_t pool_take(int device, int key, cudaGraph_t g) {
  std::lock_guard<std::mutex> lock(pool_mutex());
  auto& v = exec_pool();
  int tries = 0;
  for (size_t i = 0; i < v.size() && tries < 4; ++i) {
    if (v[i].device != device || v[i].key != key) continue;
    ++tries;
    cudaGraphExecUpdateResultInfo info;
    if (cudaGraphExecUpdate(v[i].exec, g, &info) == cudaSuccess) {
      cudaGraphExec_t e = v[i].exec;
      v.erase(v.begin() + (std::ptrdiff_t)i);
      return e;
    }
    (void)cudaGetLastError();  // a topology mismatch is not an error here
  }
  return nullptr;
}

}  // namespace

GmresWork::~GmresWork() {
  for (auto& kv : graphs) {
    if (kv.second.events.empty()) {
      pool_put(device, kv.first, kv.second.exec);  // untimed cycles only: no event nodes to carry over
    } else {
      cudaGraphExecDestroy(kv.second.exec);
      for (auto& e : kv.second.events) cudaEventDestroy(e.a), cudaEventDestroy(e.b);
    }
  }
}

void gmres_free(Surface* s) {
  delete s->gw;
  s->gw = nullptr;
}

namespace {

GmresWork* workspace(Surface* s, const SysLayout& L, int m) {
  GmresWork* w = s->gw;
  if (w && w->lay_key == L.key && w->m == m && w->K == L.K) return w;
  if (w) gmres_free(s);
  w = new GmresWork();
  w->device = s->device;
  s->gw = w;
  w->lay_key = L.key;
  w->m = m;
  w->K = L.K;
  w->len = L.len;
  // blocks: each covers a range of one system's elements, about 128 of them (at
  // most 1024 blocks per system); for the cluster step, kClu blocks per system
  std::vector<int4> blk, cblk;
  std::vector<int4> sysb(L.K), csysb(L.K);
  for (int k = 0; k < L.K; ++k) {
    const int n = L.n[k];
    auto cut = [&](int nb, std::vector<int4>& out, int4& range) {
      const int chunk = (n + nb - 1) / nb, first = (int)out.size();
      range = make_int4(first, first + nb, 0, 0);
      for (int b = 0; b < nb; ++b)
        out.push_back(make_int4(k, std::min(n, b * chunk), std::min(n, (b + 1) * chunk), first));
    };
    cut(std::min(1024, std::max(1, (n + 127) / 128)), blk, sysb[k]);
    cut(kClu, cblk, csysb[k]);
  }
  w->nblk = (int)blk.size();
  w->sysb_host = sysb;
  const int64_t len = L.len;
  w->V.ensure((size_t)(m + 1) * len, s->stream);
  w->w.ensure(len, s->stream);
  w->r.ensure(len, s->stream);
  w->d.ensure(len, s->stream);
  w->tz.ensure(len, s->stream);
  w->t.ensure(len, s->stream);
  w->H.ensure((size_t)L.K * (m + 1) * m, s->stream);
  w->cs.ensure((size_t)L.K * m, s->stream);
  w->sn.ensure((size_t)L.K * m, s->stream);
  w->g.ensure((size_t)L.K * (m + 1), s->stream);
  w->y.ensure((size_t)L.K * m, s->stream);
  w->z.ensure((size_t)L.K * (m + 1), s->stream);
  const size_t nb_max = std::max(blk.size(), cblk.size());
  w->part.ensure(nb_max * (m + 1), s->stream);
  w->part2.ensure(nb_max * (m + 1), s->stream);
  w->part1.ensure(nb_max, s->stream);
  w->blk.ensure(blk.size(), s->stream);
  w->sysb.ensure(L.K, s->stream);
  w->cblk.ensure(cblk.size(), s->stream);
  w->csysb.ensure(L.K, s->stream);
  w->mask.ensure(L.K, s->stream);
  w->st_buf.ensure(L.K, s->stream);
  w->st = w->st_buf.p;
  w->st_host.resize(L.K);
  w->part1_host.resize(w->nblk);
  w->mask_host.resize(L.K);
  BIPB_CUDA(cudaMemcpyAsync(w->blk.p, blk.data(), blk.size() * sizeof(int4), cudaMemcpyHostToDevice, s->stream));
  BIPB_CUDA(cudaMemcpyAsync(w->sysb.p, sysb.data(), sysb.size() * sizeof(int4), cudaMemcpyHostToDevice, s->stream));
  BIPB_CUDA(cudaMemcpyAsync(w->cblk.p, cblk.data(), cblk.size() * sizeof(int4), cudaMemcpyHostToDevice, s->stream));
  BIPB_CUDA(cudaMemcpyAsync(w->csysb.p, csysb.data(), csysb.size() * sizeof(int4), cudaMemcpyHostToDevice, s->stream));
  BIPB_CUDA(cudaStreamSynchronize(s->stream));
  ++s->alloc_gen;
  return w;
}

// One restart cycle: kernels only (no host synchronisation, no allocation).
// M^-1 of the self-block preconditioner: 1 / (1/2 (1 + eps)), 1 / (1/2 (1 + 1/eps))
double2 precond_factors(const bipb_medium& m) {
  const double eps = m.eps_out / m.eps_in;
  return make_double2(2.0 / (1.0 + eps), 2.0 / (1.0 + 1.0 / eps));
}

// Whether one cluster per system takes an Arnoldi step in one launch.  GB300
// has two FP64 lanes per SM, so eight SMs make the (j + 1) 4n multiply-adds of a
// step as fast as the three kernels' launches and block reductions take only
// for small systems, and only while every cluster has its SMs.  With the fused
// FP32 mat-vec they also sum its partial sums, one unknown per thread up to 2048
// elements.  Whole solves, cluster / kernels: one system of 320 elements 1.40 /
// 1.72 ms, 1280 1.55 / 1.76, 2560 2.24 / 2.15, 5120 4.20 / 3.48; 12 of 320 .. 5120,
// fused, 2.66 / 2.55; 16 charge sets on 5120 elements, not fused, 7.05 / 7.23 ms.
// (Clusters of 16, one system: 2560 elements 1.97 ms, 4000 3.17 / 3.25, 5120 4.1;
// four of up to 3000 1.23 / 1.19.)
bool cluster_step(const SysLayout& L, bool fused) {
  return L.max_n <= (fused ? 2048 : 5120) && L.K * kClu <= 160;
}

void issue_cycle(Surface* s, const SysLayout& L, GmresWork* w, const bipb_medium& med, int precision,
                 bool transpose) {
  const int4* lay = s->lay_dev(L);
  double* tz = w->precond ? w->tz.p : nullptr;
  const double2 pre = precond_factors(med);
  const int m = w->m, K = w->K, nb = w->nblk;
  const int64_t len = w->len;
  const int kg = (K + 127) / 128;
  const int* skip = &w->st->skip;
  // CGS2 for FP64 and df64 Krylov mat-vecs: the first pass also takes the
  // dot products of the second, the second also forms the block norms.
  // The FP32 / split-FP16 tensor-core Krylov solve of the mixed modes stops at a
  // relative 1e-6 (its true residual is measured in higher precision by
  // the refinement), and its FP64 basis of at most m vectors loses
  // orthogonality in one classical pass only at about eps_64 cond(A)^2:
  // one pass, which also forms the block norms.
  const bool cgs2 = precision == BIPB_FP64 || precision == BIPB_DF64;
  StepArgs a{0,       m,       len,     w->V.p, w->w.p, w->part.p, w->part2.p, w->part1.p, w->H.p, w->cs.p,
             w->sn.p, w->g.p, w->st, w->blk.p, w->sysb.p, lay,      tz,         pre,         {},     nullptr,
             s->tgt64.p};
  // the symmetric FP32 mat-vec fused into the step: its first records here, its
  // sums and the next records in the step's kernels
  const bool fused = precision == BIPB_FP32 &&
                     matvec_sym32_stages(s, L, med, transpose, tz ? tz : w->V.p, w->w.p, skip, kStateInts, kSymPack, &a.mv);
  const bool cluster = cluster_step(L, fused);
  if (cluster) a.blk = w->cblk.p, a.sysb = w->csysb.p;
  for (int j = 0; j < m; ++j) {
    double* vj = w->V.p + (size_t)j * len;
    a.j = j;
    a.u = tz ? tz : vj;
    if (fused)
      matvec_sym32_stages(s, L, med, transpose, a.u, w->w.p, skip, kStateInts, kSymPairs, nullptr);
    else
      matvec(s, L, med, precision, transpose, a.u, w->w.p, skip, kStateInts);
    if (cluster) {
      launch_chained(cgs2 ? k_step<true, false> : fused ? k_step<false, true> : k_step<false, false>, K * kClu, kCluNT, 0,
                     s->stream, a);
      BIPB_LAUNCHED(s);
      continue;
    }
    launch_chained(fused ? k_dots<true> : k_dots<false>, nb, kBS, 0, s->stream, a);
    BIPB_LAUNCHED(s);
    if (cgs2) {
      launch_chained(k_orth<false>, nb, kBS, 0, s->stream, a, a.part, 0);
      BIPB_LAUNCHED(s);
      launch_chained(k_orth<true>, nb, kBS, 0, s->stream, a, a.part2, 1);
    } else {
      launch_chained(k_orth<true>, nb, kBS, 0, s->stream, a, a.part, 0);
    }
    BIPB_LAUNCHED(s);
    launch_chained(fused ? k_normalize<true> : k_normalize<false>, nb, kBS, 0, s->stream, a);
    BIPB_LAUNCHED(s);
  }
  launch_chained(k_lsq, K, 64, 0, s->stream, m, w->H.p, w->cs.p, w->sn.p, w->g.p, w->y.p, w->z.p, w->st);
  BIPB_LAUNCHED(s);
  launch_chained(k_update, nb, kBS, 0, s->stream, m, len, w->V.p, w->d.p, w->y.p, w->z.p, w->st, w->blk.p, tz, lay,
                 pre);
  BIPB_LAUNCHED(s);
  launch_chained(k_next_cycle, kg, 128, 0, s->stream, m, K, w->g.p, w->st);
  BIPB_LAUNCHED(s);
}

void run_cycle(Surface* s, const SysLayout& L, GmresWork* w, const bipb_medium& med, int precision,
               bool transpose) {
  // A recorded cycle bakes in the medium and every buffer address, so it is
  // tagged with both and re-recorded when either changes.
  const int key = (precision * 2 + (transpose ? 1 : 0)) * 2 + (w->precond ? 1 : 0);
  const GraphTag tag{s->alloc_gen, med.eps_in, med.eps_out, med.kappa, s->timer.on};
  auto it = w->graphs.find(key);
  if (it != w->graphs.end() && it->second.tag == tag) {
    BIPB_CUDA(cudaGraphLaunch(it->second.exec, s->stream));
    s->launches += it->second.kernels;
    w->replayed = &it->second.events;
    return;
  }
  // a plain launch first: it runs this cycle and creates every scratch buffer
  issue_cycle(s, L, w, med, precision, transpose);
  const GraphTag after{s->alloc_gen, med.eps_in, med.eps_out, med.kappa, s->timer.on};
  // record a copy of the cycle for the next calls (recording does not run it)
  cudaGraph_t graph = nullptr;
  std::vector<EventPair> evs;
  BIPB_CUDA(cudaStreamBeginCapture(s->stream, cudaStreamCaptureModeThreadLocal));
  s->timer.capture = &evs;
  s->recording = true;
  s->recorded_launches = 0;
  try {
    issue_cycle(s, L, w, med, precision, transpose);
  } catch (...) {
    s->recording = false;
    s->timer.capture = nullptr;
    cudaStreamEndCapture(s->stream, &graph);
    if (graph) cudaGraphDestroy(graph);
    throw;
  }
  s->timer.capture = nullptr;
  s->recording = false;
  const long long kernels = s->recorded_launches;
  BIPB_CUDA(cudaStreamEndCapture(s->stream, &graph));
  if (!(s->alloc_gen == after.gen)) {  // a buffer moved while recording: do not keep it
    cudaGraphDestroy(graph);
    for (auto& e : evs) s->timer.pool.push_back(e.a), s->timer.pool.push_back(e.b);
    return;
  }
  cudaGraphExec_t exec = evs.empty() ? pool_take(s->device, key, graph) : nullptr;
  cudaError_t e = exec ? cudaSuccess : cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  BIPB_CUDA(e);
  if (it != w->graphs.end()) {
    cudaGraphExecDestroy(it->second.exec);
    for (auto& ev : it->second.events) s->timer.pool.push_back(ev.a), s->timer.pool.push_back(ev.b);
  }
  w->graphs[key] = Recorded{exec, after, std::move(evs), kernels};
}

void read_states(Surface* s, GmresWork* w) {
  BIPB_CUDA(cudaMemcpyAsync(w->st_host.data(), w->st, w->K * sizeof(DevState), cudaMemcpyDeviceToHost, s->stream));
  BIPB_CUDA(cudaStreamSynchronize(s->stream));
  if (s->timer.on) {
    s->timer.collect();
    if (w->replayed)
      for (auto& e : *w->replayed) s->timer.add(e);
  }
  w->replayed = nullptr;
}

// Per-system 2-norms of a batched vector (all systems, fixed summation order).
std::vector<double> norms(Surface* s, const SysLayout& L, GmresWork* w, const double* v) {
  k_sumsq<<<w->nblk, kBS, 0, s->stream>>>(v, w->part1.p, w->st, w->blk.p, s->lay_dev(L), 2);
  BIPB_LAUNCHED(s);
  BIPB_CUDA(cudaMemcpyAsync(w->part1_host.data(), w->part1.p, w->nblk * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
  BIPB_CUDA(cudaStreamSynchronize(s->stream));
  std::vector<double> out(w->K);
  for (int k = 0; k < w->K; ++k) {
    double acc = 0.0;
    for (int b = w->sysb_host[k].x; b < w->sysb_host[k].y; ++b) acc += w->part1_host[b];
    out[k] = std::sqrt(acc);
  }
  return out;
}

// GMRES on op(A) d = r0 for the active systems (d starts at zero; others are
// left alone).  Per system: stop at recurrence estimate <= tol[k] (relative
// to ||r0_k||) or after cap[k] iterations.  Returns iterations per system.
std::vector<int> gmres_core(Surface* s, const SysLayout& L, GmresWork* w, const bipb_medium& med, int precision,
                            bool transpose, const double* r0, const std::vector<char>& active,
                            const std::vector<double>& tol, const std::vector<int>& cap, std::vector<int>* conv) {
  const int K = w->K;
  BIPB_CUDA(cudaMemsetAsync(w->d.p, 0, (size_t)w->len * sizeof(double), s->stream));
  BIPB_CUDA(cudaStreamSynchronize(s->stream));  // st_host is about to be rewritten
  for (int k = 0; k < K; ++k) {
    DevState& S = w->st_host[k];
    S = DevState{};
    S.active = active[k] ? 1 : 0;
    S.skip = S.active ? 0 : 1;
    S.conv = S.active ? 0 : 1;
    S.stop = (S.active && cap[k] <= 0) ? 1 : 0;
    S.max_iter = cap[k];
    S.m = w->m;
    S.tol = tol[k];
    S.est = 1.0;
  }
  BIPB_CUDA(cudaMemcpyAsync(w->st, w->st_host.data(), K * sizeof(DevState), cudaMemcpyHostToDevice, s->stream));
  const int kg = (K + 127) / 128;
  const int4* lay = s->lay_dev(L);
  k_sumsq<<<w->nblk, kBS, 0, s->stream>>>(r0, w->part1.p, w->st, w->blk.p, lay, 1);
  BIPB_LAUNCHED(s);
  k_start<<<w->nblk, kBS, 0, s->stream>>>(r0, w->V.p, w->part1.p, w->st, w->blk.p, w->sysb.p, lay,
                                          w->precond ? w->tz.p : nullptr, precond_factors(med));
  BIPB_LAUNCHED(s);
  k_next_cycle<<<kg, 128, 0, s->stream>>>(w->m, K, w->g.p, w->st);
  BIPB_LAUNCHED(s);
  read_states(s, w);
  auto running = [&] {
    for (int k = 0; k < K; ++k)
      if (w->st_host[k].active && !w->st_host[k].conv && !w->st_host[k].stop) return true;
    return false;
  };
  while (running()) {
    run_cycle(s, L, w, med, precision, transpose);
    read_states(s, w);
  }
  std::vector<int> it(K);
  conv->assign(K, 0);
  for (int k = 0; k < K; ++k) {
    it[k] = w->st_host[k].iters;
    (*conv)[k] = w->st_host[k].conv;
  }
  return it;
}

}  // namespace

std::vector<SolveResult> gmres_solve(Surface* s, const SysLayout& L, const bipb_medium& med,
                                     const bipb_solve_params& p, bool transpose, const double* rhs, double* x,
                                     bool warm) {
  const int K = L.K;
  std::vector<SolveResult> res(K);
  const int m = p.restart > 0 ? p.restart : 10;
  const int max_iter = p.max_iter > 0 ? p.max_iter : 1000;
  GmresWork* w = workspace(s, L, m);
  w->precond = p.precond;
  const int64_t len = L.len;
  const int nb = grid_for(len);
  const std::vector<double> bnorm = norms(s, L, w, rhs);
  const bool mixed = p.precision == BIPB_MIXED || p.precision == BIPB_MIXED_DF64 || p.precision == BIPB_MIXED_TENSOR ||
                     p.precision == BIPB_MIXED_TREE;
  // arithmetic of the Krylov mat-vecs and of the residual r = b - A x
  int inner = !mixed ? p.precision : BIPB_FP32;
  if (p.precision == BIPB_MIXED_TENSOR) inner = BIPB_TENSOR;
  if (p.precision == BIPB_MIXED_TREE) inner = BIPB_TREE32;
  const int resid = (p.precision == BIPB_MIXED || p.precision == BIPB_FP64) ? BIPB_FP64 : BIPB_DF64;
  // r = rhs - A x (or rhs when starting from zero)
  if (warm) {
    matvec(s, L, med, resid, transpose, x, w->t.p, nullptr, 0);
    for (auto& r : res) r.matvecs64++;
    k_sub<<<nb, kBS, 0, s->stream>>>(len, rhs, w->t.p, w->r.p);
    BIPB_LAUNCHED(s);
  } else {
    BIPB_CUDA(cudaMemsetAsync(x, 0, (size_t)len * sizeof(double), s->stream));
    BIPB_CUDA(cudaMemcpyAsync(w->r.p, rhs, (size_t)len * sizeof(double), cudaMemcpyDeviceToDevice, s->stream));
  }
  std::vector<double> rel(K, 1.0);
  if (warm) {
    std::vector<double> rn = norms(s, L, w, w->r.p);
    for (int k = 0; k < K; ++k) rel[k] = bnorm[k] > 0 ? rn[k] / bnorm[k] : 0.0;
  }
  for (int k = 0; k < K; ++k)
    if (bnorm[k] == 0.0) rel[k] = 0.0;
  // inner solves stop near the inner operator's own accuracy (about 1e-7 for
  // FP32 pairs and for the split-FP16 tensor-core tiles): iterating further
  // does not reduce the true residual
  const double inner_floor = p.inner_tol > 0 ? p.inner_tol : 1e-6;
  const int inner_cap = p.inner_max_iter > 0 ? p.inner_max_iter : 200;
  std::vector<char> active(K), done(K, 0);
  std::vector<int> iters(K, 0);
  for (;;) {
    bool any = false;
    std::vector<double> tol_rel(K, 1.0);
    std::vector<int> cap(K, 0);
    for (int k = 0; k < K; ++k) {
      active[k] = !done[k] && rel[k] > p.tol && iters[k] < max_iter;
      if (!active[k]) continue;
      any = true;
      cap[k] = max_iter - iters[k];
      if (mixed) {
        tol_rel[k] = std::max(inner_floor, 0.3 * p.tol / rel[k]);
        cap[k] = std::min(cap[k], inner_cap);
      } else {
        tol_rel[k] = p.tol / rel[k];
      }
    }
    if (!any) break;
    std::vector<int> conv;
    std::vector<int> used = gmres_core(s, L, w, med, inner, transpose, w->r.p, active, tol_rel, cap, &conv);
    // x += d (d is zero outside the active systems); r = rhs - A x in FP64 for the active systems
    k_add<<<nb, kBS, 0, s->stream>>>(len, w->d.p, x);
    BIPB_LAUNCHED(s);
    for (int k = 0; k < K; ++k) w->mask_host[k] = active[k] ? 0 : 1;
    BIPB_CUDA(cudaMemcpyAsync(w->mask.p, w->mask_host.data(), K * sizeof(int), cudaMemcpyHostToDevice, s->stream));
    matvec(s, L, med, resid, transpose, x, w->t.p, w->mask.p, 1);
    k_sub<<<nb, kBS, 0, s->stream>>>(len, rhs, w->t.p, w->r.p);
    BIPB_LAUNCHED(s);
    std::vector<double> rn = norms(s, L, w, w->r.p);
    for (int k = 0; k < K; ++k) {
      if (!active[k]) continue;
      iters[k] += used[k];
      res[k].matvecs64++;
      if (mixed) {
        res[k].matvecs32 += used[k];
        res[k].refine_steps++;
      } else {
        res[k].matvecs64 += used[k];
      }
      const double new_rel = bnorm[k] > 0 ? rn[k] / bnorm[k] : 0.0;
      if (!mixed && !conv[k]) done[k] = 1;                                           // iteration cap
      if (mixed && res[k].refine_steps >= 3 && new_rel > 0.1 * rel[k]) done[k] = 1;  // refinement stalled
      rel[k] = new_rel;
    }
  }
  for (int k = 0; k < K; ++k) {
    res[k].iters = iters[k];
    res[k].rel_residual = rel[k];
    res[k].converged = rel[k] <= p.tol ? 1 : 0;
  }
  return res;
}

}  // namespace bipb

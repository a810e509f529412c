// Throughput microbenchmark of the pipes the pair kernels run on: FP32 FFMA,
// FP64 DFMA and the MUFU approximations (rsqrt.approx, ex2.approx).  A
// standalone program (not part of libbipb), built and run by
// `bench.py --mode peaks`; it prints one "name value" line per pipe, in
// lane-operations per second, after one warm-up launch.
//
// Every thread runs 8 (FFMA), 4 (DFMA) or 4 (MUFU) independent dependency
// chains, and the grid holds 8 CTAs of 256 threads per SM, so the issue
// slots, not latencies, bound each kernel.
//
// ffma shares two of its operands among all chains.  ffma3 is the FFMA the pair
// kernels are full of: three register operands, none the one of the FFMA before
// (2 CTAs per SM for its 24 registers of operands); ffma2 the packed form (results per
// second), fadd and fadd2 additions with two such operands.
#include <cstdio>
#include <cuda_runtime.h>

namespace {

constexpr int kIters = 4096;

__global__ void k_ffma(float* out, float a, float b) {
  float x[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) x[c] = threadIdx.x + c;
  for (int i = 0; i < kIters; ++i)
#pragma unroll
    for (int c = 0; c < 8; ++c) x[c] = fmaf(x[c], a, b);
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) s += x[c];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// 8 accumulators, each against another of 8 x and y every time.  PACKED: .f32x2
// instructions on both halves of 64-bit registers; ADD: additions of x.
__device__ __forceinline__ unsigned long long pair_of(float a, float b) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
template <bool PACKED, bool ADD>
__global__ void __launch_bounds__(256) k_three(float* out, float s0) {
  float a[8], x[8], y[8];
  unsigned long long A[8], X[8], Y[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    a[c] = s0 + c, x[c] = s0 * c + 0.01f * threadIdx.x, y[c] = s0 * 0.1f * c + 0.02f * threadIdx.x;
    A[c] = pair_of(a[c], (float)threadIdx.x), X[c] = pair_of(x[c], threadIdx.x + 0.5f), Y[c] = pair_of(y[c], s0 + threadIdx.x);
  }
  for (int i = 0; i < 2 * kIters; ++i)  // 64 instructions each: long enough for the launch not to count
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int p = (c + r) & 7, q = (3 * c + r) & 7;
        if (PACKED && ADD) asm volatile("add.rn.f32x2 %0, %1, %2;" : "=l"(A[c]) : "l"(X[p]), "l"(A[c]));
        if (PACKED && !ADD) asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(A[c]) : "l"(X[p]), "l"(Y[q]), "l"(A[c]));
        if (!PACKED && ADD) asm volatile("add.rn.f32 %0, %1, %2;" : "=f"(a[c]) : "f"(x[p]), "f"(a[c]));
        if (!PACKED && !ADD) asm volatile("fma.rn.f32 %0, %1, %2, %3;" : "=f"(a[c]) : "f"(x[p]), "f"(y[q]), "f"(a[c]));
      }
  float s = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) s += PACKED ? (float)(A[c] & 0xffff) + (float)(A[c] >> 48) : a[c];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

__global__ void k_dfma(double* out, double a, double b) {
  double x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = threadIdx.x + c;
  for (int i = 0; i < kIters / 32; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = fma(x[c], a, b);
  out[blockIdx.x * blockDim.x + threadIdx.x] = x[0] + x[1] + x[2] + x[3];
}

__global__ void k_mufu(float* out) {
  float x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = threadIdx.x + 1.0f + c;
  for (int i = 0; i < kIters / 4; ++i) {
    asm volatile("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(x[0]));
    asm volatile("rsqrt.approx.ftz.f32 %0, %0;" : "+f"(x[1]));
    asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[2]));
    asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[3]));
  }
  out[blockIdx.x * blockDim.x + threadIdx.x] = x[0] + x[1] + x[2] + x[3];
}

}  // namespace

int main() {
  cudaDeviceProp p;
  if (cudaGetDeviceProperties(&p, 0) != cudaSuccess) {
    std::printf("error no device\n");
    return 1;
  }
  const int blocks = p.multiProcessorCount * 8, threads = 256;
  const double n = (double)blocks * threads;
  void* buf = nullptr;
  if (cudaMalloc(&buf, (size_t)n * sizeof(double)) != cudaSuccess) {
    std::printf("error cudaMalloc\n");
    return 1;
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  auto timed = [&](auto launch) {
    launch();  // warm-up
    cudaEventRecord(e0);
    launch();
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    return (double)ms / 1e3;
  };
  const double t_ffma = timed([&] { k_ffma<<<blocks, threads>>>((float*)buf, 0.999f, 0.001f); });
  const double t_dfma = timed([&] { k_dfma<<<blocks, threads>>>((double*)buf, 0.999, 0.001); });
  const double t_mufu = timed([&] { k_mufu<<<blocks, threads>>>((float*)buf); });
  const int few = p.multiProcessorCount * 2;
  const double m = (double)few * threads;
  const double t_ffma3 = timed([&] { k_three<false, false><<<few, threads>>>((float*)buf, 1e-3f); });
  const double t_ffma2 = timed([&] { k_three<true, false><<<few, threads>>>((float*)buf, 1e-3f); });
  const double t_fadd = timed([&] { k_three<false, true><<<few, threads>>>((float*)buf, 1e-3f); });
  const double t_fadd2 = timed([&] { k_three<true, true><<<few, threads>>>((float*)buf, 1e-3f); });
  std::printf("sms %d\n", p.multiProcessorCount);
  std::printf("ffma_per_s %.6e\n", n * kIters * 8 / t_ffma);
  std::printf("dfma_per_s %.6e\n", n * (kIters / 32) * 4 / t_dfma);
  std::printf("mufu_per_s %.6e\n", n * kIters / t_mufu);
  std::printf("ffma3_per_s %.6e\n", m * kIters * 128 / t_ffma3);
  std::printf("ffma2_per_s %.6e\n", 2.0 * m * kIters * 128 / t_ffma2);
  std::printf("fadd_per_s %.6e\n", m * kIters * 128 / t_fadd);
  std::printf("fadd2_per_s %.6e\n", 2.0 * m * kIters * 128 / t_fadd2);
  const cudaError_t err = cudaGetLastError();
  std::printf("status %s\n", err == cudaSuccess ? "ok" : cudaGetErrorString(err));
  cudaFree(buf);
  return err == cudaSuccess ? 0 : 1;
}

// Pipe-rate microbenchmark for one B200: lane-operations per clock per SM of FFMA, packed FFMA2, MUFU.EX2, SHFL and a
// dependent LDS chain, alone and in the mixes the scan kernels use, at 128..1024 threads per SM (one CTA per SM).
// The benchmark's ALU roofline takes its MUFU and FP32 rates from this program's output.
// A second table mixes two instruction kinds with independent operands and prints the cycles one scheduler spends per
// warp on a group of them, a third what one instruction of a kind adds to a stream of packed FMAs, and a fourth what a packed FMA costs by
// the registers it reads.  Packed values are float2 throughout: as 64-bit integers the loops move both halves of each on every trip.
//   nvcc -gencode arch=compute_100a,code=sm_100a -O3 -o pipe_rates pipe_rates.cu && ./pipe_rates
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <cuda_runtime.h>
#include <cstdint>
#define ITERS 4096
template <int MODE>
__global__ void __launch_bounds__(1024) k(float* out, long long* cyc, float a, float b, int) {
  float x[8];
  float2 p[8];
  __shared__ float sm[4096];
  for (int i = 0; i < 8; ++i) { x[i] = threadIdx.x * 0.001f + i; p[i] = make_float2(x[i], x[i] + 1.f); }
  for (int i = threadIdx.x; i < 4096; i += blockDim.x) sm[i] = i;
  const float2 aa = make_float2(a, a), bb = make_float2(b, b);
  __syncthreads();
  long long t0 = clock64();
  for (int it = 0; it < ITERS; ++it) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (MODE == 0) x[i] = fmaf(x[i], a, b);
      if (MODE == 1) p[i] = __ffma2_rn(p[i], aa, bb);
      if (MODE == 2) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[i]));
      if (MODE == 3) x[i] = __shfl_xor_sync(0xffffffffu, x[i], 1 + (i & 15));
      if (MODE == 4) { x[i] = fmaf(x[i], a, b); if ((i & 7) == 0) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[i])); }
      if (MODE == 5) x[i] = sm[(threadIdx.x + (int)x[i]) & 4095];
      if (MODE == 6) { p[i] = __ffma2_rn(p[i], aa, bb); if ((i & 3) == 0) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[i])); }
      if (MODE == 7) { p[i] = __ffma2_rn(p[i], aa, bb); if ((i & 3) == 0) x[i] = __shfl_xor_sync(0xffffffffu, x[i], 1); }
      if (MODE == 8) { x[i] = fmaf(x[i], a, b); if ((i & 3) == 0) x[(i+1)&7] = __shfl_xor_sync(0xffffffffu, x[(i+1)&7], 1); }
      if (MODE == 9) { x[i] = fmaf(x[i], a, b); if ((i & 3) == 0) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(x[(i+1)&7])); }
    }
  }
  long long t1 = clock64();
  float s = 0; for (int i = 0; i < 8; ++i) s += x[i] + p[i].x + p[i].y;
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cyc[blockIdx.x] = t1 - t0;
}
void check(cudaError_t e) {
  if (e != cudaSuccess) { fprintf(stderr, "%s\n", cudaGetErrorString(e)); exit(1); }
}
typedef void (*Kern)(float*, long long*, float, float, int);
double cycles(Kern kern, int threads) {   // of a CTA's run, mean over the SMs, second launch
  int dev, sms;
  check(cudaGetDevice(&dev));
  check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  float* out; long long* cyc;
  check(cudaMalloc(&out, sizeof(float) * sms * threads));
  check(cudaMalloc(&cyc, sizeof(long long) * sms));
  for (int r = 0; r < 2; ++r) {
    kern<<<sms, threads>>>(out, cyc, 0.999f, 0.001f, 12345);
    check(cudaGetLastError());
    check(cudaDeviceSynchronize());
  }
  std::vector<long long> h(sms);
  check(cudaMemcpy(h.data(), cyc, sizeof(long long) * sms, cudaMemcpyDeviceToHost));
  check(cudaFree(out)); check(cudaFree(cyc));
  double c = 0;
  for (long long v : h) c += v;
  return c / sms;
}
double per_group(Kern kern, int threads) { return cycles(kern, threads) / ITERS / (threads / 128.0); }   // of a scheduler, per warp and group
template <int MODE> void run(const char* name, double ops_per_iter_per_thread, int threads) {
  const double c = cycles(k<MODE>, threads);
  printf("%-28s threads/SM %4d: %7.2f lane-ops/clk/SM (%.0f cycles)\n", name, threads, ops_per_iter_per_thread * ITERS * threads / c, c);
}

// ---- mixes: NA operations of kind KA interleaved with NB of kind KB, all on independent registers ----
// kinds: 0 FFMA, 1 FFMA2, 2 LOP3, 3 EX2, 5 SHFL, 6 IMAD, 7 SEL, 8 FMNMX, 9 PRMT, 10 IADD, 11 FADD, 12 FMUL2
template <int K> __device__ __forceinline__ void op(float& x, float2& p, int& q, float& e, float a, float b, float2 aa, float2 bb, int ia,
                                                    bool c) {
  if (K == 0) x = fmaf(x, a, b);
  if (K == 1) p = __ffma2_rn(p, aa, bb);
  if (K == 2) asm volatile("lop3.b32 %0, %0, %1, %2, 0x96;" : "+r"(q) : "r"(ia), "r"(ia));
  if (K == 3) asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+f"(e));
  if (K == 5) e = __shfl_xor_sync(0xffffffffu, e, 1);
  if (K == 6) asm volatile("mad.lo.s32 %0, %0, %1, %2;" : "+r"(q) : "r"(ia), "r"(ia));
  if (K == 7) { q = c ? q : ia; asm volatile("" : "+r"(q)); }
  if (K == 8) asm volatile("max.f32 %0, %0, %1;" : "+f"(x) : "f"(a));
  if (K == 9) asm volatile("prmt.b32 %0, %0, %1, 0x5410;" : "+r"(q) : "r"(ia));
  if (K == 10) asm volatile("add.s32 %0, %0, %1;" : "+r"(q) : "r"(ia));
  if (K == 11) asm volatile("add.f32 %0, %0, %1;" : "+f"(x) : "f"(a));
  if (K == 12) p = __fmul2_rn(p, aa);
}
template <int KA, int NA, int KB, int NB>
__global__ void __launch_bounds__(1024) mixk(float* out, long long* cyc, float a, float b, int ia) {
  float x[16]; float2 p[16]; int q[16]; float e[16];
  const bool c = (threadIdx.x * ia) & 4;
  for (int i = 0; i < 16; ++i) { x[i] = threadIdx.x * 0.001f + i; q[i] = threadIdx.x + i; e[i] = -0.001f * threadIdx.x - i;
    p[i] = make_float2(x[i], x[i] + 1.f); }
  const float2 aa = make_float2(a, a), bb = make_float2(b, b);
  __syncthreads();
  long long t0 = clock64();
  for (int it = 0; it < ITERS; ++it) {
    constexpr int N = NA > NB ? NA : NB;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (i < NA) op<KA>(x[i & 15], p[i & 15], q[i & 15], e[i & 15], a, b, aa, bb, ia, c);
      if (i < NB) op<KB>(x[(i + 8) & 15], p[(i + 8) & 15], q[(i + 8) & 15], e[(i + 8) & 15], a, b, aa, bb, ia, c);
    }
  }
  long long t1 = clock64();
  float s = 0; for (int i = 0; i < 16; ++i) s += x[i] + p[i].x + p[i].y + q[i] + e[i];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cyc[blockIdx.x] = t1 - t0;
}
template <int KA, int NA, int KB, int NB> void runmix(const char* name, int threads) {
  printf("%-28s threads/SM %4d: %6.2f cycles per warp and group on one scheduler\n", name, threads,
         per_group(mixk<KA, NA, KB, NB>, threads));
}
// ---- 64 operations of kind K spread over 128 packed FMAs: what one adds ----
template <int K, int NK>
__global__ void addk(float* out, long long* cyc, float a, float b, int ia) {
  float x[16]; float2 p[16], p2[8]; int q[16]; float e[16];
  const bool c = (threadIdx.x * ia) & 4;
  for (int i = 0; i < 16; ++i) { x[i] = threadIdx.x * 0.001f + i; q[i] = threadIdx.x + i; e[i] = -0.001f * threadIdx.x - i;
    p[i] = make_float2(x[i], x[i] + 1.f); p2[i & 7] = p[i]; }
  const float2 aa = make_float2(a, a), bb = make_float2(b, b);
  __syncthreads();
  long long t0 = clock64();
#pragma unroll 1
  for (int it = 0; it < ITERS; ++it) {
#pragma unroll
    for (int i = 0; i < 128; ++i) {
      p[i & 15] = __ffma2_rn(p[i & 15], aa, bb);
      if ((i & 1) && (i >> 1) < NK) op<K>(x[(i >> 1) & 15], p2[(i >> 1) & 7], q[(i >> 1) & 15], e[(i >> 1) & 15], a, b, aa, bb, ia, c);
    }
  }
  long long t1 = clock64();
  float s = 0; for (int i = 0; i < 16; ++i) s += x[i] + p[i].x + p[i].y + p2[i & 7].x + q[i] + e[i];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cyc[blockIdx.x] = t1 - t0;
}
// ---- 128 packed operations by what they read ----
// W: an FMA of 0 one pair of its own, 1 two, 2 three, 4 two and a single register for both halves; 3 a product of two
template <int W>
__global__ void readk(float* out, long long* cyc, float a, float b, int ia) {
  float2 p[8], u[8], v[8];
  for (int i = 0; i < 8; ++i) { p[i] = make_float2(threadIdx.x, i); u[i] = make_float2(a * i + threadIdx.x, b); v[i] = make_float2(b * i + ia, a * threadIdx.x); }
  __syncthreads();
  long long t0 = clock64();
#pragma unroll 1
  for (int it = 0; it < ITERS; ++it) {
#pragma unroll
    for (int i = 0; i < 128; ++i) {
      const int j = i & 7, r = (i >> 3) & 7;
      if (W == 0) p[j] = __ffma2_rn(p[j], u[0], v[0]);
      if (W == 1) p[j] = __ffma2_rn(u[j], v[0], p[j]);
      if (W == 2) p[j] = __ffma2_rn(u[j], v[(j + r) & 7], p[j]);
      if (W == 3) p[j] = __fmul2_rn(p[j], u[j]);
      if (W == 4) p[j] = __ffma2_rn(u[j], make_float2(v[r].x, v[r].x), p[j]);
    }
  }
  long long t1 = clock64();
  float s = 0; for (int i = 0; i < 8; ++i) s += p[i].x + p[i].y;
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cyc[blockIdx.x] = t1 - t0;
}
template <int K> void runadd(const char* name) {
  const double base = per_group(addk<K, 0>, 384), with = per_group(addk<K, 64>, 384);
  printf("%-28s adds %5.2f cycles beside packed FMAs (128 of them: %.0f)\n", name, (with - base) / 64, base);
}
int main() {
  for (int th : {128, 256, 512, 1024}) {
    run<0>("FFMA", 8, th);
    run<1>("FFMA2 (counted as 2 fma)", 16, th);
    run<2>("MUFU.EX2", 8, th);
    run<3>("SHFL", 8, th);
    run<5>("LDS.32", 8, th);
    run<4>("FFMA + 1/8 EX2 (fma count)", 8, th);
    run<9>("FFMA + 1/4 EX2 indep (fma)", 8, th);
    run<6>("FFMA2 + 1/4 EX2 (fma count)", 16, th);
    run<7>("FFMA2 + 1/4 SHFL (fma count)", 16, th);
    run<8>("FFMA + 1/4 SHFL (fma count)", 8, th);
  }
  for (int th : {384, 1024}) {
    runmix<0, 8, 0, 8>("16 FFMA", th);
    runmix<1, 8, 1, 8>("16 FFMA2", th);
    runmix<2, 8, 2, 8>("16 LOP3", th);
    runmix<6, 8, 6, 8>("16 IMAD", th);
    runmix<3, 4, 3, 4>("8 EX2", th);
    runmix<0, 16, 3, 2>("16 FFMA + 2 EX2", th);
    runmix<0, 16, 3, 4>("16 FFMA + 4 EX2", th);
    runmix<1, 16, 3, 4>("16 FFMA2 + 4 EX2", th);
    runmix<1, 16, 5, 8>("16 FFMA2 + 8 SHFL", th);
    runmix<0, 16, 2, 16>("16 FFMA + 16 LOP3", th);
    runmix<1, 16, 2, 16>("16 FFMA2 + 16 LOP3", th);
    runmix<0, 16, 6, 16>("16 FFMA + 16 IMAD", th);
    runmix<1, 16, 6, 16>("16 FFMA2 + 16 IMAD", th);
    runmix<1, 16, 0, 16>("16 FFMA2 + 16 FFMA", th);
  }
  runadd<7>("SEL"); runadd<8>("FMNMX"); runadd<5>("SHFL"); runadd<10>("IADD"); runadd<3>("EX2"); runadd<11>("FADD"); runadd<0>("FFMA");
  runadd<9>("PRMT"); runadd<6>("IMAD"); runadd<12>("FMUL2"); runadd<2>("LOP3");
  printf("packed FMA of one pair of its own %.2f cycles, two %.2f, three %.2f, two and a register %.2f; packed product %.2f\n",
         per_group(readk<0>, 384) / 128, per_group(readk<1>, 384) / 128, per_group(readk<2>, 384) / 128, per_group(readk<4>, 384) / 128,
         per_group(readk<3>, 384) / 128);
  return 0;
}

// Residual-stack glue: gain-free RMSNorm over d_model (forward and VJP), the residual add, and the residual add with the
// norm of its result.  One warp per token; fp32 arithmetic; I/O in the activation dtype.
//
// Bound by HBM: rows go in 16-byte pieces (d_model is a multiple of 8) and stay in registers up to NORM_REG elements per
// lane, so every tensor is read and written once.  65,536 tokens x 768, bf16, buffers larger than L2: norm 44 -> 32 us, add
// 152 -> 44 us (it moved one 2-byte element per thread), VJP 100 -> 59 us; the add with the norm (64 us) saves the norm's read.
#include <type_traits>

#include "as_norm.cuh"

namespace as {
namespace {
constexpr int NORM_REG = 64;   // elements of a row a lane keeps

// what a value is after it has been stored
__device__ __forceinline__ float stored(float v, float) { return v; }
__device__ __forceinline__ float stored(float v, __nv_bfloat16) { return __bfloat162float(__float2bfloat16_rn(v)); }

// The sums over a row, in bf16: lane l adds elements l, l + 32, ... in that order, whatever the layout of the loads, through a
// copy of the row in shared memory.  A deep stack of bf16 layers turns differences of one rounding unit of a norm into
// differences of some per cent of its gradients (12 layers: 2 %), so a wider load should not change the order.
// fp32 rows are added up as they lie.
template <typename IO> constexpr bool kOrdered = sizeof(IO) == 2;
// After a bf16 norm comes a contraction that takes whole SMs; it may come in at once.  After an fp32 norm come small CTAs, which would
// crowd on the SMs the norm leaves free: they come when it ends (12 layers of 1,024 x 64: 380 -> 352 us a step; 3 x 303 x 192: 335 -> 268;
// bf16 5,424 x 416: 412 | 415).
template <typename IO> __device__ __forceinline__ void norm_begin() {
  pdl_wait();
  if (sizeof(IO) == 2) pdl_launch();
}
constexpr int NORM_WARPS = 4;   // rows per CTA

// One row per warp.  NP = 16-byte pieces of a row per lane, or 0: any width, the row read again for the second pass.
// ADD: the row is a + b, stored to `sum` (which may alias a), and the norm, which may alias b, is that of the stored row.
// None of the four is __restrict__: a lane has read all its pieces of a and b before it stores to sum or yhat (NP > 0), or has
// read its pieces of b before the second pass stores yhat (NP = 0).
template <typename IO, int NP, bool ADD>
__global__ void rmsnorm_fwd_kernel(int64_t rows, int P, const IO* a, const IO* b, IO* sum, IO* yhat, float eps) {
  norm_begin<IO>();
  constexpr int N = Vec<IO>::N;
  extern __shared__ __align__(16) uint8_t row_s[];
  const int64_t row = (int64_t)blockIdx.x * NORM_WARPS + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  IO* copy = reinterpret_cast<IO*>(row_s) + (threadIdx.x / 32) * P;
  if (row >= rows) return;
  auto get = [&](int c, float (&v)[N]) {
    ld_vec<IO>(a + row * P + c, v);
    if (ADD) {
      float w[N];
      ld_vec<IO>(b + row * P + c, w);
#pragma unroll
      for (int e = 0; e < N; ++e) v[e] = stored(v[e] + w[e], IO());
    }
  };
  float ss = 0.f;
  if (NP > 0) {
    float v[NP > 0 ? NP : 1][N];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int c = (k * 32 + lane) * N;
#pragma unroll
      for (int e = 0; e < N; ++e) v[k][e] = 0.f;
      if (c < P) get(c, v[k]);
      if (kOrdered<IO>) {
        if (c < P) st_vec<IO>(copy + c, v[k]);
      } else {
#pragma unroll
        for (int e = 0; e < N; ++e) ss = fmaf(v[k][e], v[k][e], ss);
      }
    }
    if (kOrdered<IO>) {
      __syncwarp();
      for (int i = lane; i < P; i += 32) { const float t = (float)copy[i]; ss = fmaf(t, t, ss); }
    }
    const float rinv = 1.f / sqrtf(wsum(ss) / (float)P + eps);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int c = (k * 32 + lane) * N;
      if (c >= P) break;
      if (ADD) st_vec<IO>(sum + row * P + c, v[k]);
#pragma unroll
      for (int e = 0; e < N; ++e) v[k][e] *= rinv;
      st_vec<IO>(yhat + row * P + c, v[k]);
    }
  } else {
    float v[N];
    for (int c = lane * N; c < P; c += 32 * N) {
      get(c, v);
#pragma unroll
      for (int e = 0; e < N; ++e)
        if (!kOrdered<IO>) ss = fmaf(v[e], v[e], ss);
      if (ADD) st_vec<IO>(sum + row * P + c, v);
    }
    if (kOrdered<IO>) {
      __syncwarp();   // the row as the warp wrote it (ADD) or as it came
      for (int i = lane; i < P; i += 32) { const float t = (float)(ADD ? sum : a)[row * P + i]; ss = fmaf(t, t, ss); }
    }
    const float rinv = 1.f / sqrtf(wsum(ss) / (float)P + eps);
    for (int c = lane * N; c < P; c += 32 * N) {
      ld_vec<IO>((ADD ? sum : a) + row * P + c, v);   // a lane reads back what it wrote itself
#pragma unroll
      for (int e = 0; e < N; ++e) v[e] *= rinv;
      st_vec<IO>(yhat + row * P + c, v);
    }
  }
}

// The three rows are all requested before the first is used, and kept as they were loaded (half the registers in bf16).
template <typename IO, int NP>
__global__ void rmsnorm_bwd_add_kernel(int64_t rows, int P, const IO* __restrict__ y, const IO* __restrict__ dyhat,
                                       IO* __restrict__ G, float eps) {
  norm_begin<IO>();
  constexpr int N = Vec<IO>::N, NK = NP > 0 ? NP : 1;
  extern __shared__ __align__(16) uint8_t row_s[];
  const int64_t row = (int64_t)blockIdx.x * NORM_WARPS + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  IO* copy = reinterpret_cast<IO*>(row_s) + (threadIdx.x / 32) * 2 * P;   // y, then dyhat
  if (row >= rows) return;
  const IO* yr = y + row * P;
  const IO* dr = dyhat + row * P;
  IO* gr = G + row * P;
  float ss = 0.f, dot = 0.f;
  auto sums = [&](const uint4& yq, const uint4& dq) {
    float v[N], d[N];
    ld_vec<IO>(reinterpret_cast<const IO*>(&yq), v); ld_vec<IO>(reinterpret_cast<const IO*>(&dq), d);
#pragma unroll
    for (int e = 0; e < N; ++e) { ss = fmaf(v[e], v[e], ss); dot = fmaf(v[e], d[e], dot); }
  };
  auto add = [&](int c, const uint4& yq, const uint4& dq, const uint4& gq, float rinv, float m) {
    float v[N], d[N], g[N];
    ld_vec<IO>(reinterpret_cast<const IO*>(&yq), v); ld_vec<IO>(reinterpret_cast<const IO*>(&dq), d);
    ld_vec<IO>(reinterpret_cast<const IO*>(&gq), g);
#pragma unroll
    for (int e = 0; e < N; ++e) g[e] += (d[e] - v[e] * rinv * m) * rinv;
    st_vec<IO>(gr + c, g);
  };
  auto raw = [](const IO* p) { return *reinterpret_cast<const uint4*>(p); };
  if (NP > 0) {
    uint4 yq[NK], dq[NK], gq[NK];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int c = (k * 32 + lane) * N;
      yq[k] = dq[k] = gq[k] = make_uint4(0u, 0u, 0u, 0u);
      if (c < P) { yq[k] = raw(yr + c); dq[k] = raw(dr + c); gq[k] = raw(gr + c); }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int c = (k * 32 + lane) * N;
      if (!kOrdered<IO>) sums(yq[k], dq[k]);
      else if (c < P) { *reinterpret_cast<uint4*>(copy + c) = yq[k]; *reinterpret_cast<uint4*>(copy + P + c) = dq[k]; }
    }
    if (kOrdered<IO>) {
      __syncwarp();
      for (int i = lane; i < P; i += 32) {
        const float v = (float)copy[i];
        ss = fmaf(v, v, ss);
        dot = fmaf(v, (float)copy[P + i], dot);
      }
    }
    ss = wsum(ss); dot = wsum(dot);
    const float rinv = 1.f / sqrtf(ss / (float)P + eps), m = dot * rinv / (float)P;   // m = mean_p(dyhat * yhat)
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int c = (k * 32 + lane) * N;
      if (c < P) add(c, yq[k], dq[k], gq[k], rinv, m);
    }
  } else {
    if (kOrdered<IO>) {
      for (int i = lane; i < P; i += 32) {
        const float v = (float)yr[i];
        ss = fmaf(v, v, ss);
        dot = fmaf(v, (float)dr[i], dot);
      }
    } else {
      for (int c = lane * N; c < P; c += 32 * N) sums(raw(yr + c), raw(dr + c));
    }
    ss = wsum(ss); dot = wsum(dot);
    const float rinv = 1.f / sqrtf(ss / (float)P + eps), m = dot * rinv / (float)P;
    for (int c = lane * N; c < P; c += 32 * N) add(c, raw(yr + c), raw(dr + c), raw(gr + c), rinv, m);
  }
}

template <typename IO>
__global__ void residual_add_kernel(int64_t n, const IO* a, const IO* __restrict__ b, IO* out) {
  norm_begin<IO>();
  constexpr int N = Vec<IO>::N;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * N;
  if (i >= n) return;
  float v[N], w[N];
  ld_vec<IO>(a + i, v); ld_vec<IO>(b + i, w);
#pragma unroll
  for (int e = 0; e < N; ++e) v[e] += w[e];
  st_vec<IO>(out + i, v);
}

// pieces per lane for a width: rounded up to 1, 2, 3, 4, 6 or 8; 0 beyond NORM_REG elements
template <typename IO, typename F>
int with_pieces(int P, F f) {
  const int np = (P + 32 * Vec<IO>::N - 1) / (32 * Vec<IO>::N);
  if (np * Vec<IO>::N <= NORM_REG) {
    if (np <= 1) return f(std::integral_constant<int, 1>{});
    if (np <= 2) return f(std::integral_constant<int, 2>{});
    if (np <= 3) return f(std::integral_constant<int, 3>{});
    if (np <= 4) return f(std::integral_constant<int, 4>{});
    if (np <= 6) return f(std::integral_constant<int, 6>{});
    if (np <= 8) return f(std::integral_constant<int, 8>{});
  }
  return f(std::integral_constant<int, 0>{});
}

template <typename IO, bool ADD>
int norm_fwd(const as_shape_t* sh, const void* a, const void* b, void* sum, void* yhat, float eps, cudaStream_t st) {
  const int64_t rows = (int64_t)sh->batch * sh->seqlen;
  return with_pieces<IO>(sh->d_model, [&](auto np) {
    return launch_dependent(rmsnorm_fwd_kernel<IO, decltype(np)::value, ADD>, dim3((unsigned)((rows + NORM_WARPS - 1) / NORM_WARPS)),
                            dim3(32 * NORM_WARPS), kOrdered<IO> && decltype(np)::value > 0 ? NORM_WARPS * sh->d_model * sizeof(IO) : 0, st,
                            rows, sh->d_model, (const IO*)a, (const IO*)b, (IO*)sum, (IO*)yhat, eps);
  });
}
template <typename IO>
int norm_bwd(const as_shape_t* sh, const void* y, const void* dyhat, void* G, float eps, cudaStream_t st) {
  const int64_t rows = (int64_t)sh->batch * sh->seqlen;
  return with_pieces<IO>(sh->d_model, [&](auto np) {
    return launch_dependent(rmsnorm_bwd_add_kernel<IO, decltype(np)::value>, dim3((unsigned)((rows + NORM_WARPS - 1) / NORM_WARPS)),
                            dim3(32 * NORM_WARPS), kOrdered<IO> && decltype(np)::value > 0 ? 2 * NORM_WARPS * sh->d_model * sizeof(IO) : 0, st,
                            rows, sh->d_model, (const IO*)y, (const IO*)dyhat, (IO*)G, eps);
  });
}
template <typename IO>
int add_rows(const as_shape_t* sh, const void* a, const void* b, void* out, cudaStream_t st) {
  const int64_t n = (int64_t)sh->batch * sh->seqlen * sh->d_model;
  const int64_t pieces = n / Vec<IO>::N;
  return launch_dependent(residual_add_kernel<IO>, dim3((unsigned)((pieces + 255) / 256)), dim3(256), 0, st, n, (const IO*)a,
                          (const IO*)b, (IO*)out);
}
}  // namespace

int launch_rmsnorm_fwd(const as_shape_t* sh, const void* y, void* yhat, float eps, cudaStream_t st) {
  return sh->io == AS_BF16 ? norm_fwd<__nv_bfloat16, false>(sh, y, nullptr, nullptr, yhat, eps, st)
                           : norm_fwd<float, false>(sh, y, nullptr, nullptr, yhat, eps, st);
}

int launch_residual_add_rmsnorm(const as_shape_t* sh, const void* a, const void* b, void* out, void* yhat, float eps,
                                cudaStream_t st) {
  return sh->io == AS_BF16 ? norm_fwd<__nv_bfloat16, true>(sh, a, b, out, yhat, eps, st)
                           : norm_fwd<float, true>(sh, a, b, out, yhat, eps, st);
}

int launch_rmsnorm_bwd_add(const as_shape_t* sh, const void* y, const void* dyhat, void* G, float eps, cudaStream_t st) {
  return sh->io == AS_BF16 ? norm_bwd<__nv_bfloat16>(sh, y, dyhat, G, eps, st) : norm_bwd<float>(sh, y, dyhat, G, eps, st);
}

int launch_residual_add(const as_shape_t* sh, const void* a, const void* b, void* out, cudaStream_t st) {
  return sh->io == AS_BF16 ? add_rows<__nv_bfloat16>(sh, a, b, out, st) : add_rows<float>(sh, a, b, out, st);
}

// One launch clears every buffer a gradient call accumulates into (status block, the [dB|dC] accumulator and, unless
// the caller accumulates, the five parameter gradients) and packs the weights: separate memsets and kernels cost more in
// launch gaps than in bytes.  All regions are 16-byte aligned and a multiple of 16 bytes long; rows of the weights are
// copied in 16-byte pieces.
namespace {
__global__ void prepare_kernel(ZeroList z, int zblocks, int P, int layers, int reps, const uint4* __restrict__ Wd,
                               const uint4* __restrict__ WB, const uint4* __restrict__ WC, uint4* __restrict__ out) {
  pdl_begin();
  if ((int)blockIdx.x < zblocks) {
    clear_regions(z, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)zblocks * blockDim.x);
    return;
  }
  const int q = P / 8;                                  // 16-byte pieces of a bf16 row
  const int64_t n = (int64_t)(P + reps * NBC) * q;      // pieces of one layer's Wcat
  const int64_t i = ((int64_t)blockIdx.x - zblocks) * blockDim.x + threadIdx.x;
  if (i >= n * layers) return;
  const int64_t l = i / n, row = (i - l * n) / q, col = i % q;
  const int64_t e = (row - P) & (NBC - 1);
  out[i] = row < P ? Wd[(l * P + row) * q + col] : (e < NS ? WB[(l * NS + e) * q + col] : WC[(l * NS + e - NS) * q + col]);
}
}  // namespace

int launch_prepare(const ZeroList& z, int P, int layers, int reps, const as_params_t* pr, void* wcat, cudaStream_t st) {
  size_t total = 0;
  for (int r = 0; r < z.n; ++r) total += z.bytes[r];
  int64_t zblocks = (int64_t)((total / 16 + 255) / 256);
  const int64_t cap = (int64_t)sm_count() * 8;
  if (zblocks > cap) zblocks = cap;
  const int64_t pieces = pr ? (int64_t)layers * (P + reps * NBC) * (P / 8) : 0;
  const int64_t blocks = zblocks + (pieces + 255) / 256;
  if (blocks < 1) return 0;
  if (blocks > 0x7fffffff) return 1;
  return launch_dependent(prepare_kernel, dim3((unsigned)blocks), dim3(256), 0, st, z, (int)zblocks, P, layers, reps,
                          (const uint4*)(pr ? pr->W_delta : nullptr), (const uint4*)(pr ? pr->W_B : nullptr),
                          (const uint4*)(pr ? pr->W_C : nullptr), (uint4*)wcat);
}

}  // namespace as

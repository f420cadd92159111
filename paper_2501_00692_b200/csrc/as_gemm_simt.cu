// FP32-pipe contractions of the layer for fp32 I/O, where the 1e-4 parity bar rules out TF32 or single bf16 tensor-core
// inputs.  One kernel body covers the three contractions over the virtual matrices Wcat = [W_delta; W_B; W_C] ([P+32, P])
// and Gcat = [du | dB | dC] ([tokens, P+32]), whose parts are read where they lie:
//   PROJ : [Delta | B | C] = X Wcat^T            (softplus + bias on the Delta columns)
//   DW   : [dW_delta; dW_B; dW_C] += Gcat^T X    (split over the tokens, fp32 reductions)
//   DX   : dx = dx_dir + Gcat Wcat
// Bound: the FP32 pipe for large shapes (8 x 4 outputs per thread: 32 FFMA per three 16-byte shared-memory loads), latency
// for small ones.  So the three parts of a contraction and all layers of a call share one launch, and the two gradient
// contractions, which are independent, share one too: 2 launches where one per part, layer and operand made 9 per layer.
// Operands go global -> registers -> shared memory, one K-tile ahead, in 16-byte pieces (P is a multiple of 8, so no piece
// straddles two parts).
#include "as_internal.cuh"

namespace as {

namespace {
constexpr int BM = 64, BN = 64, BK = 16, TM = 8, TN = 4, NT = 128;
constexpr int PADM = BM + 4, PADN = BN + 4;
enum { C_PROJ = 0, C_DW = 1, C_DX = 2 };

struct SimtArgs {
  const float *x, *W_delta, *W_B, *W_C, *b_delta;
  float *delta, *bc;                 // PROJ outputs
  const float *du, *dbc, *dxdir;     // gradient inputs
  float *dW_delta, *dW_B, *dW_C, *dx;
  int64_t M;                         // token rows per layer
  int P, layers, splitk;
  ZeroList zero;                     // PROJ: regions to clear for the later kernels of the call
  int ndx;                           // gradient launch: number of DX blocks (they come first); 0 when dx is not wanted
};

__device__ __forceinline__ float softplus_f(float u) {
  return fmaxf(u, 0.f) + log1pf(expf(-fabsf(u)));
}
__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

// a 16-byte piece of row r of Wcat (columns c..c+3), of row m of Gcat
__device__ __forceinline__ const float* wcat_at(const SimtArgs& a, int64_t l, int r, int c) {
  const int64_t P = a.P;
  if (r < a.P) return a.W_delta + (l * P + r) * P + c;
  r -= a.P;
  return r < NS ? a.W_B + (l * NS + r) * P + c : a.W_C + (l * NS + r - NS) * P + c;
}
__device__ __forceinline__ const float* gcat_at(const SimtArgs& a, int64_t l, int64_t m, int c) {
  const int64_t row = l * a.M + m;
  return c < a.P ? a.du + row * a.P + c : a.dbc + row * NBC + c - a.P;
}

// one BM x BN output tile of one contraction; blk: tile index inside this contraction's grid
template <int KIND>
__device__ __forceinline__ void tile(const SimtArgs& a, int64_t blk, float (&As)[2][BK][PADM], float (&Bs)[2][BK][PADN]) {
  const int tid = threadIdx.x;
  const int P = a.P, NW = P + NBC;
  // output extent [R, N] and contraction length K of one layer
  const int64_t R = KIND == C_DW ? NW : a.M;
  const int N = KIND == C_PROJ ? NW : P;
  const int64_t K = KIND == C_PROJ ? P : (KIND == C_DW ? a.M : NW);
  const int nt = (N + BN - 1) / BN;
  const int64_t rt = (R + BM - 1) / BM;
  const int n0 = (int)(blk % nt) * BN;
  int64_t t = blk / nt;
  const int64_t m0 = (t % rt) * BM;
  t /= rt;
  const int splitk = KIND == C_DW ? a.splitk : 1;
  const int64_t lay = t / splitk;
  int64_t kbeg = 0, kend = K;
  if (KIND == C_DW) {
    const int64_t kchunk = ((K + splitk - 1) / splitk + BK - 1) / BK * BK;
    kbeg = (t % splitk) * kchunk;
    kend = min(K, kbeg + kchunk);
    if (kbeg >= kend) return;
  }

  constexpr bool A_K = KIND != C_DW, B_K = KIND == C_PROJ;   // operand contiguous along K (else along its own rows)
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 ra[2], rb[2];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int idx = tid + i * NT;
      {
        const int64_t m = m0 + (A_K ? idx >> 2 : (idx & 15) * 4), k = k0 + (A_K ? (idx & 3) * 4 : idx >> 4);
        const float* p = KIND == C_PROJ ? a.x + (lay * a.M + m) * P + k
                                        : (KIND == C_DX ? gcat_at(a, lay, m, (int)k) : gcat_at(a, lay, k, (int)m));
        ra[i] = m < R && k < kend ? ldg4(p) : zero4;
      }
      {
        const int n = n0 + (B_K ? idx >> 2 : (idx & 15) * 4);
        const int64_t k = k0 + (B_K ? (idx & 3) * 4 : idx >> 4);
        const float* p = KIND == C_PROJ ? wcat_at(a, lay, n, (int)k)
                                        : (KIND == C_DX ? wcat_at(a, lay, (int)k, n) : a.x + (lay * a.M + k) * P + n);
        rb[i] = n < N && k < kend ? ldg4(p) : zero4;
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int idx = tid + i * NT;
      if (A_K) {
        const int m = idx >> 2, k = (idx & 3) * 4;
        As[buf][k][m] = ra[i].x; As[buf][k + 1][m] = ra[i].y; As[buf][k + 2][m] = ra[i].z; As[buf][k + 3][m] = ra[i].w;
      } else {
        *reinterpret_cast<float4*>(&As[buf][idx >> 4][(idx & 15) * 4]) = ra[i];
      }
      if (B_K) {
        const int n = idx >> 2, k = (idx & 3) * 4;
        Bs[buf][k][n] = rb[i].x; Bs[buf][k + 1][n] = rb[i].y; Bs[buf][k + 2][n] = rb[i].z; Bs[buf][k + 3][n] = rb[i].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[buf][idx >> 4][(idx & 15) * 4]) = rb[i];
      }
    }
  };

  const int tx = tid & 15, ty = tid >> 4;   // this thread's rows ty*8 .. +7, columns tx*4 .. +3
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  fetch(kbeg);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < kend;
    if (more) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM + 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * TN]);
      const float av[TM] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[TN] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    if (more) {
      put(buf ^ 1);
      __syncthreads();
    }
  }

  const int n = n0 + tx * TN;   // four columns: all inside one part (its border is a multiple of 8) or all outside
  if (n >= N) return;
  float4 bias = zero4;
  if (KIND == C_PROJ && n < P) bias = ldg4(a.b_delta + lay * P + n);
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t m = m0 + ty * TM + i;
    if (m >= R) break;
    const int64_t row = lay * a.M + m;
    float4 v = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (KIND == C_PROJ) {
      if (n < P) {
        v = make_float4(softplus_f(v.x + bias.x), softplus_f(v.y + bias.y), softplus_f(v.z + bias.z), softplus_f(v.w + bias.w));
        *reinterpret_cast<float4*>(a.delta + row * P + n) = v;
      } else {
        *reinterpret_cast<float4*>(a.bc + row * NBC + n - P) = v;
      }
    } else if (KIND == C_DX) {
      const float4 d = ldg4(a.dxdir + row * P + n);
      *reinterpret_cast<float4*>(a.dx + row * P + n) = make_float4(v.x + d.x, v.y + d.y, v.z + d.z, v.w + d.w);
    } else {
      const int e = (int)m - P;
      float* dst = e < 0 ? a.dW_delta + (lay * P + m) * P + n
                         : (e < NS ? a.dW_B + (lay * NS + e) * P + n : a.dW_C + (lay * NS + e - NS) * P + n);
      atomicAdd(reinterpret_cast<float4*>(dst), v);
    }
  }
}

__global__ void __launch_bounds__(NT) simt_proj_kernel(const __grid_constant__ SimtArgs a) {
  __shared__ __align__(16) float As[2][BK][PADM];
  __shared__ __align__(16) float Bs[2][BK][PADN];
  pdl_begin();
  clear_regions(a.zero, (int64_t)blockIdx.x * NT + threadIdx.x, (int64_t)gridDim.x * NT);
  tile<C_PROJ>(a, blockIdx.x, As, Bs);
}
// both gradient contractions: the first ndx blocks compute dx, the rest the weight gradients
__global__ void __launch_bounds__(NT) simt_grad_kernel(const __grid_constant__ SimtArgs a) {
  __shared__ __align__(16) float As[2][BK][PADM];
  __shared__ __align__(16) float Bs[2][BK][PADN];
  pdl_begin();
  if ((int)blockIdx.x < a.ndx) tile<C_DX>(a, blockIdx.x, As, Bs);
  else tile<C_DW>(a, (int64_t)blockIdx.x - a.ndx, As, Bs);
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
SimtArgs base_args(const Plan& pl, const as_params_t* pr, const void* x) {
  SimtArgs a{};
  a.x = (const float*)x; a.W_delta = (const float*)pr->W_delta; a.W_B = (const float*)pr->W_B; a.W_C = (const float*)pr->W_C;
  a.b_delta = pr->b_delta; a.M = (int64_t)pl.Bg * pl.T; a.P = pl.P; a.layers = pl.KL; a.splitk = 1;
  return a;
}
}  // namespace

int simt_projections(const Plan& pl, const as_params_t* pr, const void* x, const ZeroList& z, char* ws, cudaStream_t st) {
  SimtArgs a = base_args(pl, pr, x);
  a.zero = z;
  a.delta = (float*)(ws + pl.off_delta); a.bc = (float*)(ws + pl.off_bc);
  const int64_t blocks = cdiv(a.M, BM) * cdiv(pl.P + NBC, BN) * a.layers;
  if (blocks > 0x7fffffff) return 1;
  return launch_dependent(simt_proj_kernel, dim3((unsigned)blocks), dim3(NT), 0, st, a);
}

int simt_gradients(const Plan& pl, const as_params_t* pr, const void* x, const as_grads_t* out, char* ws, cudaStream_t st) {
  SimtArgs a = base_args(pl, pr, x);
  a.du = (const float*)(ws + pl.off_du); a.dbc = (const float*)(ws + pl.off_dbc); a.dxdir = (const float*)(ws + pl.off_dxdir);
  a.dW_delta = out->dW_delta; a.dW_B = out->dW_B; a.dW_C = out->dW_C; a.dx = (float*)out->dx;
  const int64_t ndx = out->dx ? cdiv(a.M, BM) * cdiv(pl.P, BN) * a.layers : 0;
  const int64_t tiles = cdiv(pl.P + NBC, BM) * cdiv(pl.P, BN) * a.layers;
  // split over the tokens: about four CTAs per SM, 64 tokens or more each (below that the reductions outweigh the sums)
  int64_t s = cdiv((int64_t)sm_count() * 4, tiles);
  if (s > cdiv(a.M, 64)) s = cdiv(a.M, 64);
  a.splitk = (int)(s < 1 ? 1 : s);
  a.ndx = (int)ndx;
  const int64_t blocks = ndx + tiles * a.splitk;
  if (blocks > 0x7fffffff) return 1;
  return launch_dependent(simt_grad_kernel, dim3((unsigned)blocks), dim3(NT), 0, st, a);
}

}  // namespace as

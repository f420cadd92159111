// Internal declarations shared by the translation units of libadjoint_ssm (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "../../include/adjoint_ssm.h"

namespace as {

extern std::atomic<int64_t> g_launches;   // kernels launched by this library (diagnostic)
inline void count_launch(int n = 1) { g_launches.fetch_add(n); }

// Launches of this library are programmatically dependent: once all CTAs of a kernel have called pdl_launch() (or are done), the
// CTAs of the next one may take their places, set up what they need in their SM - barriers, tensor memory, descriptors in the
// constant cache - and wait in pdl_wait() until the kernel before has finished and its writes are visible.  That hides the
// launch latency and the set-up (1,600 of the 14,000 cycles of a 256 x 256 contraction).  Nothing may touch global memory
// before pdl_wait().
// pdl_launch() comes after pdl_wait(), never before: a kernel that lets the next one in while it waits itself has the CTAs of two,
// three kernels queue up on the SMs that happen to be free, several to an SM beside idle ones, and there they stay.  us, let in at
// once | after the wait: gradients 512 x 64 fp32 35.5 | 29.2, 4,655 x 128 84 | 76; forwards 3 x 1,177 x 256 59 | 39, 2 x 211 x 104 fp32
// 21.9 | 15.3; step of 5 layers of 799 x 704 947 | 730.  Contractions and the forward's two
// passes let the next one in when a CTA has sent for its last operands, or is done with its tile or its tokens (gradient of
// 477 x 1,768 90 -> 86; forwards of 3,040 x 1,448 79 -> 75, 571 x 512 fp32 53 -> 38, 4 x 970 x 128 fp32 35 -> 30); the gradient's segment
// pass and the main kernel later than after their wait are as often slower as faster (10,506 x 128 118 -> 110, but 4 x 218 x 64 fp32
// 40 -> 45; 348 x 128 48 -> 58).  The carries do it half way (gradients of 2 x 304 x 480 55 -> 50, 2 x 168 x 480 fp32 101 -> 87; at their end 2,301 x 376 fp32 99 -> 116).
template <typename... KA, typename... A>
inline int launch_dependent(void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, KA(args)...);
  count_launch();
  return (int)e;
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() { pdl_wait(); pdl_launch(); }
// a descriptor the kernel will use: into the constant cache
__device__ __forceinline__ void prefetch_map(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory");
}

// Function attributes (the dynamic shared-memory limit) belong to a device: remember per device, per kernel
// instantiation, whether the limit has been raised.  `done` is a static array of the launcher, one flag per device; host
// threads that make their first calls at once at worst repeat the (idempotent) setting.
constexpr int AS_MAX_DEVICES = 64;
typedef std::atomic<bool> DeviceFlags[AS_MAX_DEVICES];
template <typename K>
inline int ensure_dynamic_smem(K kern, int bytes, DeviceFlags& done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= AS_MAX_DEVICES) return 1;
  if (!done[dev].load(std::memory_order_acquire)) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return 1;
    done[dev].store(true, std::memory_order_release);
  }
  return 0;
}

// cuTensorMapEncodeTiled, looked up through the runtime once per process (as_api.cu); null if the driver does not have it
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled();

// Number of SMs of the current device (grids are sized in multiples of it); queried once per device.  The cache is
// a plain array of atomics: concurrent first calls from several host threads at worst query twice.
inline int sm_count() {
  static std::atomic<int> cached[AS_MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= AS_MAX_DEVICES) return 148;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n <= 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

constexpr int NS = 16;        // d_state handled by the scan kernels
constexpr int CK = 8;         // tokens per checkpoint chunk (h of one chunk lives in registers)
constexpr int NCH = 2;        // channels per thread of the scan kernels
constexpr int NTHR = 128;     // threads per CTA of the scan kernels; two threads share a channel set, 8 states each
constexpr int CH = NTHR / 2 * NCH;   // channels per CTA
constexpr int NU = 4 * NCH;   // packed state pairs (f32x2) a thread owns
constexpr int TILE_FLOATS = CH * NS;   // one (channel tile, all states) block of a per-segment / per-chunk array
constexpr int NBC = 2 * NS;   // per-token row of [B_t | C_t] (and of [dB_t | dC_t])
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;

// ---- I/O element access ---------------------------------------------------------------------
template <typename T> __device__ __forceinline__ float ld_io(const T* p);
template <> __device__ __forceinline__ float ld_io<float>(const float* p) { return __ldg(p); }
template <> __device__ __forceinline__ float ld_io<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(__ldg(p));
}
template <typename T> __device__ __forceinline__ void st_io(T* p, float v);
template <> __device__ __forceinline__ void st_io<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void st_io<__nv_bfloat16>(__nv_bfloat16* p, float v) {
  *p = __float2bfloat16_rn(v);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- packed fp32 arithmetic ------------------------------------------------------------------
// A value is a float2, never a 64-bit integer: a loop that carries 64-bit integers through inline assembly moves both halves of each
// on every trip (8 packed FMAs of a rolled loop: 27.8 cycles of a scheduler, 18.7 so).
typedef float2 f2;
struct __align__(16) f2x2 { f2 x, y; };
__device__ __forceinline__ f2 pk(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ void upk(f2 v, float& lo, float& hi) { lo = v.x; hi = v.y; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2x2 split4(float4 v) { return f2x2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ f2x2 ld2x2(const void* p) { return split4(*reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st2x2(void* p, f2 a, f2 b) { *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y); }

// ---- status block: the first STATUS_BYTES of the scratch ------------------------------------
// Word 0 is AS_OK or the code a kernel reported.  It is cleared by a kernel that reports nothing there, so a kernel that runs
// later may simply set it.  The bf16 projections clear it themselves where the weights are packed (there is no kernel before
// them), and a CTA that starts late would erase what another one has set: so they never set it.  Each of their CTAs owns one
// byte behind the word's 16-byte piece, which it (or the kernel before) zeroes when it starts and sets to 1 if a wait gives up.
// as_check_status looks at the whole block.  Ordered forward with packed weights, 256 x 256: 32.4 us with the race, 32.6 so,
// 33.9 with a clearing kernel in front; 2,048 x 512: 45.3, 45.4, 47.3.
constexpr int STATUS_BYTES = 256;
constexpr int STATUS_CTA = 16;                          // offset of the CTAs' bytes
constexpr int STATUS_CTAS = STATUS_BYTES - STATUS_CTA;  // as many CTAs can report

// ---- time segmentation and scratch layout ---------------------------------------------------
// Time is cut into S segments of L tokens (L a multiple of CK); a CTA owns (segment, batch element,
// CH channels).  Per-(segment, channel, state) and per-(chunk, channel, state) arrays are stored as
// blocks of TILE_FLOATS floats per channel tile, in the order the owning thread keeps them in registers
// (float4 q of thread tid at float offset (q*NTHR + tid)*4), so one bulk copy moves a CTA's block and
// every thread's access is a contiguous 16 bytes.  A thread's values are the state pairs of its channels, in the chunk
// checkpoints the channel pairs of its states.
struct Plan {
  int KL;           // layers handled by one call (independent problems that share dy); 1 for the single-layer entry points
  int Bg;           // batch elements per layer
  int B, P;         // B = KL * Bg: the kernels see (layer, batch element) as one batch index; layer = b / Bg
  int64_t T;
  int64_t tbar;     // clamped to T
  int full;         // tbar >= T
  int L;            // segment length (tokens)
  int S;            // number of segments
  int64_t NC;       // number of CK-token chunks = ceil(T/CK)
  int m;            // tbar / L   (whole segments inside a window that starts on a segment boundary)
  int direct;       // windows of at most four whole segments: the main kernel sums them from mu_loc, no block sums
  int r;            // tbar % L   (tokens of the following partial segment)
  int io;           // as_dtype_t
  int scalar;       // 1: one decay rate per channel (A_log is [P]), 0: one per (channel, state)
  int tiles;        // ceil(P / CH) channel tiles
  int tc;           // 1: bf16 tensor-core contractions (bf16 I/O), 0: FP32-pipe GEMMs
  int ordered;      // a call of a bf16 stack's step: as_ssm_forward_ordered, or a gradient with AS_ORDERED
  int ffma;         // projections of bf16 I/O on the fp32 pipe (as_ssm_forward_ordered, widths off the 32-element grid)
  int one_order;    // bf16 forwards of stacks and of the matmul form: one segmentation and one order of the carries for all sizes
  int split;        // fp32 I/O: contractions on the tensor cores, every operand as three bf16 terms (as_gemm_split.cu)
  int gsplit;       // bf16 terms per value of dB, dC in Gcat: 1, or 3 (exact) where d_model % 32 != 0
  int gcols;        // columns of Gcat = [du|dB|dC..]: P + 32 gsplit
  int du_ld;        // row pitch (elements) of the du buffer: P, or that of Gcat where it is the left part of it
  // byte offsets into the workspace
  size_t off_status, off_delta, off_bc, off_ckpt, off_cs, off_hend, off_muloc, off_mupart, off_segd,
      off_partd, off_hstart, off_suf, off_pre, off_total, off_live, off_du, off_dxdir, off_dbc,
      off_bptt_ckpt, off_wcat, off_wcatx, off_xs, off_wsp, off_gs, total_fwd, total_grad;
};

// PLAN_GRAD: gradient calls.  PLAN_FWD: as_ssm_forward.  PLAN_FWD_SMALL: as_ssm_forward_static where its array cannot hold
// PLAN_FWD (longer segments; fp32 I/O: projections on the FP32 pipe, which need no room for split operands).
// PLAN_FWD_ORDERED: as_ssm_forward_ordered.
enum { PLAN_GRAD = 0, PLAN_FWD = 1, PLAN_FWD_SMALL = 2, PLAN_FWD_ORDERED = 3 };
int make_plan(const as_shape_t* sh, int64_t tbar, int layers, Plan* pl, int kind = PLAN_GRAD);

// ---- launchers (each returns a cudaError_t as int) ------------------------------------------

// regions to clear in one launch (each 16-byte aligned, length a multiple of 16 bytes)
struct ZeroList { void* ptr[8]; size_t bytes[8]; int n; };
__device__ __forceinline__ void clear_regions(const ZeroList& z, int64_t first, int64_t stride) {
  for (int r = 0; r < z.n; ++r) {
    uint4* p = reinterpret_cast<uint4*>(z.ptr[r]);
    for (int64_t i = first; i < (int64_t)(z.bytes[r] / 16); i += stride) p[i] = make_uint4(0u, 0u, 0u, 0u);
  }
}
// one launch: clears the regions and (pr != null) packs Wcat[l] = [W_delta; (W_B; W_C) x reps] for every layer
int launch_prepare(const ZeroList& z, int P, int layers, int reps, const as_params_t* pr, void* wcat, cudaStream_t st);

// FP32-pipe contractions of fp32 I/O (as_gemm_simt.cu): projections (which also clear the regions that the later kernels
// of the call accumulate into), and the weight and input gradients in one launch
int simt_projections(const Plan& pl, const as_params_t* pr, const void* x, const ZeroList& z, char* ws, cudaStream_t st);
int simt_gradients(const Plan& pl, const as_params_t* pr, const void* x, const as_grads_t* out, char* ws, cudaStream_t st);

struct ScanPtrs {
  const void *x, *dy;
  const float* A_log;
  char* ws;
};
int launch_prepass(const Plan& pl, const ScanPtrs& sp, bool with_mu, cudaStream_t st);
int launch_fixup(const Plan& pl, const ScanPtrs& sp, bool with_mu, cudaStream_t st);
// res: a layer of a residual stack of one channel tile, y_out = y_in + y and yhat = norm(y_out) in place of y (yhat may be null)
struct Residual { const void* y_in; void* y_out; void* yhat; float eps; };
bool residual_applies(const Plan& pl);
bool residual_pays(const Plan& pl);
int launch_forward_y(const Plan& pl, const ScanPtrs& sp, void* y, const Residual* res, cudaStream_t st);
// matmul form of the y pass (as_scan_mm.cu): scalar structure with bf16 I/O and d_model % 128 == 0
bool forward_y_mm_applies(const Plan& pl);
int launch_forward_y_mm(const Plan& pl, const ScanPtrs& sp, void* y, cudaStream_t st);
int launch_forward_state_mm(const Plan& pl, const ScanPtrs& sp, cudaStream_t st);   // the segment pass in the same form
int launch_adjoint_main(const Plan& pl, const ScanPtrs& sp, float* dA_log, float* db_delta, cudaStream_t st);
int launch_wait_selftest(int* status, unsigned limit, cudaStream_t st);

// bf16 tensor-core path (as_gemm_tc.cu).  The projections clear the regions `z` (and the CTAs' bytes of the status block)
// where the call has no kernel before them.  wcat: the packed weights, or null: W_delta, W_B, W_C are read where they lie.
int tc_projections(const Plan& pl, const as_params_t* pr, const void* wcat, int wreps, const void* x,
                   const ZeroList& z, char* ws, cudaStream_t st);
// between: phase timing's event between weight and input gradient, which then are two launches at every size; or null.
int tc_gradients(const Plan& pl, const as_params_t* pr, const void* wcat, const void* x, const as_grads_t* out, char* ws, cudaStream_t st,
                 cudaEvent_t between);

// fp32 I/O on the tensor cores by exact three-term splits (as_gemm_split.cu), for large enough products
int split_projections(const Plan& pl, const as_params_t* pr, const void* x, const ZeroList& z, char* ws, cudaStream_t st);
int split_gradients(const Plan& pl, const as_grads_t* out, char* ws, cudaStream_t st);

int launch_bptt(const Plan& pl, const ScanPtrs& sp, float* dA_log, float* db_delta, cudaStream_t st);

// the layer forward behind as_ssm_forward, as_ssm_forward_ordered, as_ssm_forward_residual and as_ssm_forward_static; an AS_* code (as_api.cu)
int forward(const as_shape_t* shape, const as_params_t* params, const void* x, void* y, void* ws, size_t ws_bytes, void* stream,
            int kind, const Residual* res = nullptr);

// device address of the library's built-in scratch array on the current device (as_noalloc.cu); AS_OK or an error code
int static_scratch_address(void** out);

int launch_rmsnorm_fwd(const as_shape_t* sh, const void* y, void* yhat, float eps, cudaStream_t st);
int launch_residual_add(const as_shape_t* sh, const void* a, const void* b, void* out, cudaStream_t st);
int launch_residual_add_rmsnorm(const as_shape_t* sh, const void* a, const void* b, void* out, void* yhat, float eps,
                                cudaStream_t st);
int launch_rmsnorm_bwd_add(const as_shape_t* sh, const void* y, const void* dyhat, void* G, float eps,
                           cudaStream_t st);

}  // namespace as

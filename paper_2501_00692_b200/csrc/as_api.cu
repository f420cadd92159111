// extern "C" entry points: argument checks, scratch layout, and the launch sequence of each call.
#include <string.h>

#include <atomic>

#include "as_internal.cuh"

using namespace as;

namespace as {
std::atomic<int64_t> g_launches{0};

EncodeTiledFn encode_tiled() {
  static std::atomic<EncodeTiledFn> found{nullptr};   // host threads that come first at once look it up more than once
  EncodeTiledFn fn = found.load(std::memory_order_relaxed);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    found.store(fn, std::memory_order_relaxed);
  }
  return fn;
}
}  // namespace as

namespace {

// Phase timing is a diagnostic with process-wide state: one set of events, no locking.  It is meant for one host
// thread driving one stream (as the header says); everything else in the library is free of shared mutable state.
bool g_timing = false;
bool g_timing_valid = false;
cudaEvent_t g_ev[AS_NUM_PHASES + 1];

void mark(int i, cudaStream_t st) {
  if (g_timing) cudaEventRecord(g_ev[i], st);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_shape(const as_shape_t* sh) {
  if (!sh) return AS_ERR_NULL;
  if (sh->batch < 1 || sh->seqlen < 1 || sh->d_model < 1) return AS_ERR_SHAPE;
  if (sh->d_state != NS) return AS_ERR_SHAPE;
  if (sh->a_structure != AS_A_DIAGONAL && sh->a_structure != AS_A_SCALAR) return AS_ERR_SHAPE;
  if (sh->io != AS_F32 && sh->io != AS_BF16) return AS_ERR_DTYPE;
  if (sh->d_model % 8 != 0) return AS_ERR_ALIGN;
  if (sh->batch > 65535) return AS_ERR_SHAPE;
  // token rows are addressed with 32-bit TMA coordinates (row + window lookahead + one chunk), and the time
  // segments (at most 2048 tokens each) fill gridDim.y
  if ((int64_t)sh->batch * sh->seqlen + sh->seqlen + 2 * CK >= ((int64_t)1 << 31)) return AS_ERR_LIMIT;
  return AS_OK;
}

int check_params(const as_params_t* pr) {
  if (!pr || !pr->W_delta || !pr->b_delta || !pr->W_B || !pr->W_C || !pr->A_log) return AS_ERR_NULL;
  if (!aligned16(pr->W_delta) || !aligned16(pr->b_delta) || !aligned16(pr->W_B) || !aligned16(pr->W_C) ||
      !aligned16(pr->A_log) || !aligned16(pr->Wcat))
    return AS_ERR_ALIGN;
  return AS_OK;
}

#define AS_TRY(expr)                      \
  do {                                    \
    int e__ = (expr);                     \
    if (e__ != 0) return AS_ERR_CUDA;     \
  } while (0)

// Wcat of the call (null: none) and how often it holds W_B and W_C
struct Wcat { const void* p; int reps; };

// What every call begins with: the regions `z` are cleared, Wcat is the caller's packed copy if it gave one or else packed into
// the scratch, and steps 1-3 of SSM(.) run: Delta = softplus(x W_delta^T + b), B = x W_B^T, C = x W_C^T (every layer of the
// call).  The gradient of a width that is not a multiple of 32 needs W_B and W_C once per term of the dB, dC split.
int begin(const Plan& pl, const as_params_t* pr, const ZeroList& z, bool grad, const void* x, char* ws, cudaStream_t st,
          Wcat* wcat) {
  if (!pl.tc || pl.ffma) {
    AS_TRY(pl.split ? split_projections(pl, pr, x, z, ws, st) : simt_projections(pl, pr, x, z, ws, st));
    return AS_OK;
  }
  wcat->reps = grad ? pl.gsplit : 1;
  const bool packed = pr->Wcat && wcat->reps == 1;
  // Short runs read W_delta, W_B, W_C where they lie, at the price of a column tile's rows past P coming in pieces of 16: the packing
  // kernel in front is a tenth of such a call (us, with it | without: forwards 256 x 256 17.2 | 15.8, 512 x 1,024
  // 27.1 | 25.0, gradient of 601 x 64 30.4 | 29.5).  Longer ones have other things to wait for, and
  // read the packed copy once more per 256 tokens.
  const bool direct = !packed && pl.P % 16 == 0 && (int64_t)pl.B * pl.T <= 1024;
  char* at = ws + (grad ? pl.off_wcatx : pl.off_wcat);
  wcat->p = packed ? pr->Wcat : direct ? nullptr : at;
  ZeroList own{};
  if (packed || direct) {   // the projections clear the regions themselves, of the status block the word only
    own = z;
    own.bytes[0] = STATUS_CTA;
  } else AS_TRY(launch_prepare(z, pl.P, pl.KL, wcat->reps, pr, at, st));
  AS_TRY(tc_projections(pl, pr, wcat->p, wcat->reps, x, own, ws, st));
  return AS_OK;
}

// the net-VJPs: weight gradients (contractions over all tokens) and the input gradient, for every layer of the call
int contractions(const Plan& pl, const as_params_t* pr, const Wcat& wcat, const void* x, const as_grads_t* out, char* ws,
                 cudaStream_t st) {
  if (pl.tc) {
    AS_TRY(tc_gradients(pl, pr, wcat.p, x, out, ws, st, g_timing ? g_ev[5] : nullptr));
  } else {   // fp32: one launch for both, the first phase counts them, the second reads zero
    AS_TRY(pl.split ? split_gradients(pl, out, ws, st) : simt_gradients(pl, pr, x, out, ws, st));
    mark(5, st);
  }
  mark(6, st);
  return AS_OK;
}

int check_grad_args(const as_shape_t* sh, const as_params_t* pr, const void* x, const void* dy,
                    const as_grads_t* out, void* ws) {
  int e = check_shape(sh);
  if (e) return e;
  e = check_params(pr);
  if (e) return e;
  if (!x || !dy || !out || !ws) return AS_ERR_NULL;
  if (!out->dW_delta || !out->db_delta || !out->dW_B || !out->dW_C || !out->dA_log) return AS_ERR_NULL;
  if (!aligned16(x) || !aligned16(dy) || !aligned16(ws) || !aligned16(out->dW_delta) || !aligned16(out->db_delta) ||
      !aligned16(out->dW_B) || !aligned16(out->dW_C) || !aligned16(out->dA_log) || !aligned16(out->dx))
    return AS_ERR_ALIGN;
  return AS_OK;
}

// regions a call accumulates into (the status block is always the first)
void add_region(ZeroList* z, void* p, size_t bytes) { z->ptr[z->n] = p; z->bytes[z->n] = (bytes + 15) / 16 * 16; ++z->n; }
ZeroList grad_regions(const Plan& pl, uint32_t flags, const as_grads_t* out, char* ws) {
  const size_t P = pl.P, K = pl.KL;
  ZeroList z{};
  add_region(&z, ws + pl.off_status, STATUS_BYTES);
  add_region(&z, ws + pl.off_dbc, (size_t)pl.B * pl.T * NBC * 4);
  if (!(flags & AS_ACCUMULATE)) {
    add_region(&z, out->dW_delta, K * P * P * 4);
    add_region(&z, out->db_delta, K * P * 4);
    add_region(&z, out->dW_B, K * NS * P * 4);
    add_region(&z, out->dW_C, K * NS * P * 4);
    add_region(&z, out->dA_log, K * (pl.scalar ? P : P * NS) * 4);
  }
  return z;
}

}  // namespace

// The layer forward; `kind` (a forward kind of make_plan) alone decides which kernels run and how much scratch they need.
int as::forward(const as_shape_t* shape, const as_params_t* params, const void* x, void* y, void* ws, size_t ws_bytes,
                void* stream, int kind, const Residual* res) {
  int e = check_shape(shape);
  if (e) return e;
  e = check_params(params);
  if (e) return e;
  if (!x || !(res ? res->y_out : y) || !ws || (res && !res->y_in)) return AS_ERR_NULL;
  if (!aligned16(x) || !aligned16(y) || !aligned16(ws)) return AS_ERR_ALIGN;
  if (res && (!aligned16(res->y_in) || !aligned16(res->y_out) || !aligned16(res->yhat))) return AS_ERR_ALIGN;
  Plan pl;
  e = make_plan(shape, shape->seqlen, 1, &pl, kind);
  if (e) return e;
  if (res && !residual_applies(pl)) return AS_ERR_LIMIT;
  if (ws_bytes < pl.total_fwd) return AS_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* w = reinterpret_cast<char*>(ws);
  Wcat wcat{};
  ZeroList z{};
  add_region(&z, w + pl.off_status, STATUS_BYTES);
  e = begin(pl, params, z, false, x, w, st, &wcat);
  if (e) return e;
  ScanPtrs sp{x, nullptr, params->A_log, w};
  const bool mm = forward_y_mm_applies(pl);
  if (mm) AS_TRY(launch_forward_state_mm(pl, sp, st));
  else AS_TRY(launch_prepass(pl, sp, false, st));
  AS_TRY(launch_fixup(pl, sp, false, st));
  if (mm) AS_TRY(launch_forward_y_mm(pl, sp, y, st));
  else AS_TRY(launch_forward_y(pl, sp, y, res, st));
  return AS_OK;
}

extern "C" {

int as_version(void) { return AS_VERSION; }

const char* as_strerror(int code) {
  switch (code) {
    case AS_OK: return "ok";
    case AS_ERR_NULL: return "a required pointer is NULL";
    case AS_ERR_SHAPE: return "bad shape (non-positive dimension or d_state != 16)";
    case AS_ERR_DTYPE: return "unsupported io dtype";
    case AS_ERR_TBAR: return "tbar must be >= 1";
    case AS_ERR_WORKSPACE: return "workspace too small";
    case AS_ERR_ALIGN: return "pointer not 16-byte aligned or d_model not a multiple of 8";
    case AS_ERR_CUDA: return "CUDA runtime call or launch failed";
    case AS_ERR_TIMEOUT: return "bounded device-side wait gave up";
    case AS_ERR_LIMIT: return "size exceeds a fixed capacity of this entry point";
    default: return "unknown status code";
  }
}

int as_workspace_bytes(const as_shape_t* shape, int64_t tbar, size_t* fwd_bytes, size_t* grad_bytes) {
  int e = check_shape(shape);
  if (e) return e;
  if (tbar < 1) return AS_ERR_TBAR;
  Plan pl;
  e = make_plan(shape, tbar, 1, &pl);
  if (e) return e;
  if (fwd_bytes) {
    Plan pf;
    e = make_plan(shape, shape->seqlen, 1, &pf, PLAN_FWD);
    if (e) return e;
    *fwd_bytes = pf.total_fwd;
  }
  if (grad_bytes) {
    *grad_bytes = pl.total_grad;
    e = make_plan(shape, shape->seqlen, 1, &pl);   // as_full_bptt_grad and the full form cut the time differently
    if (e) return e;
    if (pl.total_grad > *grad_bytes) *grad_bytes = pl.total_grad;
    e = make_plan(shape, shape->seqlen, 1, &pl, PLAN_FWD);
    if (e) return e;
    if (pl.total_fwd > *grad_bytes) *grad_bytes = pl.total_fwd;
  }
  return AS_OK;
}

int as_check_status(const void* ws, void* stream) {
  if (!ws) {   // the built-in scratch array of as_ssm_forward_static on the current device
    void* p = nullptr;
    const int e = static_scratch_address(&p);
    if (e) return e;
    ws = p;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  alignas(int) unsigned char block[STATUS_BYTES];
  if (cudaMemcpyAsync(block, ws, STATUS_BYTES, cudaMemcpyDeviceToHost, st) != cudaSuccess) return AS_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return AS_ERR_CUDA;
  int word = 0;
  memcpy(&word, block, sizeof word);
  if (word != AS_OK) return word;
  for (int i = STATUS_CTA; i < STATUS_BYTES; ++i)
    if (block[i]) return AS_ERR_TIMEOUT;
  return AS_OK;
}

int as_ssm_forward(const as_shape_t* shape, const as_params_t* params, const void* x, void* y, void* ws,
                   size_t ws_bytes, void* stream) {
  return forward(shape, params, x, y, ws, ws_bytes, stream, PLAN_FWD);
}

int as_ssm_forward_ordered(const as_shape_t* shape, const as_params_t* params, const void* x, void* y, void* ws,
                           size_t ws_bytes, void* stream) {
  return forward(shape, params, x, y, ws, ws_bytes, stream, PLAN_FWD_ORDERED);
}

int as_ssm_forward_residual_applies(const as_shape_t* shape) {
  Plan pl;
  return check_shape(shape) == AS_OK && make_plan(shape, shape->seqlen, 1, &pl, PLAN_FWD_ORDERED) == AS_OK && residual_pays(pl) ? 1 : 0;
}

int as_ssm_forward_residual(const as_shape_t* shape, const as_params_t* params, const void* x, const void* y_in, void* y_out, void* yhat,
                            float eps, void* ws, size_t ws_bytes, void* stream) {
  const Residual res{y_in, y_out, yhat, eps};
  return forward(shape, params, x, nullptr, ws, ws_bytes, stream, PLAN_FWD_ORDERED, &res);
}

int as_adjoint_grad(const as_shape_t* shape, const as_params_t* params, const void* x, const void* dy, int64_t tbar,
                    uint32_t flags, const as_grads_t* out, void* ws, size_t ws_bytes, void* stream) {
  return as_adjoint_grad_layers(shape, 1, params, x, dy, tbar, flags, out, ws, ws_bytes, stream);
}

int as_workspace_bytes_layers(const as_shape_t* shape, int32_t layers, int64_t tbar, size_t* grad_bytes) {
  int e = check_shape(shape);
  if (e) return e;
  if (tbar < 1) return AS_ERR_TBAR;
  if (layers < 1) return AS_ERR_SHAPE;
  if ((int64_t)layers * shape->batch * shape->seqlen + shape->seqlen + 2 * CK >= ((int64_t)1 << 31)) return AS_ERR_LIMIT;
  Plan pl;
  e = make_plan(shape, tbar, layers, &pl);
  if (e) return e;
  if (grad_bytes) *grad_bytes = pl.total_grad;
  if (layers == 1) return as_workspace_bytes(shape, tbar, nullptr, grad_bytes);
  return AS_OK;
}

size_t as_wcat_bytes(const as_shape_t* shape, int32_t layers) {
  if (check_shape(shape) != AS_OK || layers < 1) return 0;
  return (size_t)layers * (shape->d_model + NBC) * shape->d_model * (shape->io == AS_BF16 ? 2 : 4);
}

int as_pack_weights(const as_shape_t* shape, int32_t layers, const as_params_t* params, void* wcat, void* stream) {
  int e = check_shape(shape);
  if (e) return e;
  e = check_params(params);
  if (e) return e;
  if (!wcat) return AS_ERR_NULL;
  if (!aligned16(wcat)) return AS_ERR_ALIGN;
  if (layers < 1) return AS_ERR_SHAPE;
  if (shape->io != AS_BF16) return AS_ERR_DTYPE;   // only the bf16 tensor-core contractions read a packed copy
  AS_TRY(launch_prepare(ZeroList{}, shape->d_model, layers, 1, params, wcat, reinterpret_cast<cudaStream_t>(stream)));
  return AS_OK;
}

int as_adjoint_grad_layers(const as_shape_t* shape, int32_t layers, const as_params_t* params, const void* x,
                           const void* dy, int64_t tbar, uint32_t flags, const as_grads_t* out, void* ws,
                           size_t ws_bytes, void* stream) {
  int e = check_grad_args(shape, params, x, dy, out, ws);
  if (e) return e;
  if (tbar < 1) return AS_ERR_TBAR;
  if (layers < 1) return AS_ERR_SHAPE;
  if ((int64_t)layers * shape->batch * shape->seqlen + shape->seqlen + 2 * CK >= ((int64_t)1 << 31)) return AS_ERR_LIMIT;
  Plan pl;
  e = make_plan(shape, tbar, layers, &pl);
  if (e) return e;
  pl.ordered = (flags & AS_ORDERED) != 0;
  if (ws_bytes < pl.total_grad) return AS_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* w = reinterpret_cast<char*>(ws);
  mark(0, st);
  Wcat wcat{};
  e = begin(pl, params, grad_regions(pl, flags, out, w), true, x, w, st, &wcat);
  if (e) return e;
  mark(1, st);
  ScanPtrs sp{x, dy, params->A_log, w};
  AS_TRY(launch_prepass(pl, sp, true, st));
  mark(2, st);
  AS_TRY(launch_fixup(pl, sp, true, st));
  mark(3, st);
  AS_TRY(launch_adjoint_main(pl, sp, out->dA_log, out->db_delta, st));
  mark(4, st);
  e = contractions(pl, params, wcat, x, out, w, st);
  if (g_timing && e == AS_OK) g_timing_valid = true;
  return e;
}

int as_full_bptt_grad(const as_shape_t* shape, const as_params_t* params, const void* x, const void* dy,
                      uint32_t flags, const as_grads_t* out, void* ws, size_t ws_bytes, void* stream) {
  int e = check_grad_args(shape, params, x, dy, out, ws);
  if (e) return e;
  Plan pl;
  e = make_plan(shape, shape->seqlen, 1, &pl);
  if (e) return e;
  pl.ordered = (flags & AS_ORDERED) != 0;
  if (ws_bytes < pl.total_grad) return AS_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  char* w = reinterpret_cast<char*>(ws);
  Wcat wcat{};
  e = begin(pl, params, grad_regions(pl, flags, out, w), true, x, w, st, &wcat);
  if (e) return e;
  ScanPtrs sp{x, dy, params->A_log, w};
  AS_TRY(launch_bptt(pl, sp, out->dA_log, out->db_delta, st));
  return contractions(pl, params, wcat, x, out, w, st);
}

int as_rmsnorm_fwd(const as_shape_t* shape, const void* y, void* yhat, float eps, void* stream) {
  int e = check_shape(shape);
  if (e) return e;
  if (!y || !yhat) return AS_ERR_NULL;
  if (!aligned16(y) || !aligned16(yhat)) return AS_ERR_ALIGN;
  AS_TRY(launch_rmsnorm_fwd(shape, y, yhat, eps, reinterpret_cast<cudaStream_t>(stream)));
  return AS_OK;
}

int as_residual_add(const as_shape_t* shape, const void* y_in, const void* ytilde, void* y_out, void* stream) {
  int e = check_shape(shape);
  if (e) return e;
  if (!y_in || !ytilde || !y_out) return AS_ERR_NULL;
  if (!aligned16(y_in) || !aligned16(ytilde) || !aligned16(y_out)) return AS_ERR_ALIGN;
  AS_TRY(launch_residual_add(shape, y_in, ytilde, y_out, reinterpret_cast<cudaStream_t>(stream)));
  return AS_OK;
}

int as_residual_add_rmsnorm(const as_shape_t* shape, const void* y_in, const void* ytilde, void* y_out, void* yhat,
                            float eps, void* stream) {
  int e = check_shape(shape);
  if (e) return e;
  if (!y_in || !ytilde || !y_out || !yhat) return AS_ERR_NULL;
  if (!aligned16(y_in) || !aligned16(ytilde) || !aligned16(y_out) || !aligned16(yhat)) return AS_ERR_ALIGN;
  AS_TRY(launch_residual_add_rmsnorm(shape, y_in, ytilde, y_out, yhat, eps, reinterpret_cast<cudaStream_t>(stream)));
  return AS_OK;
}

int as_rmsnorm_bwd_add(const as_shape_t* shape, const void* y, const void* dyhat, void* G_inout, float eps,
                       void* stream) {
  int e = check_shape(shape);
  if (e) return e;
  if (!y || !dyhat || !G_inout) return AS_ERR_NULL;
  if (!aligned16(y) || !aligned16(dyhat) || !aligned16(G_inout)) return AS_ERR_ALIGN;
  AS_TRY(launch_rmsnorm_bwd_add(shape, y, dyhat, G_inout, eps, reinterpret_cast<cudaStream_t>(stream)));
  return AS_OK;
}

int as_wait_selftest(void* ws, size_t ws_bytes, uint32_t poll_limit, void* stream) {
  if (!ws) return AS_ERR_NULL;
  if (ws_bytes < STATUS_BYTES) return AS_ERR_WORKSPACE;
  if (!aligned16(ws)) return AS_ERR_ALIGN;
  if (poll_limit == 0 || poll_limit > (1u << 20)) return AS_ERR_LIMIT;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  AS_TRY((int)cudaMemsetAsync(ws, 0, STATUS_BYTES, st));
  AS_TRY(launch_wait_selftest(reinterpret_cast<int*>(ws), poll_limit, st));
  return AS_OK;
}

int64_t as_launch_count(int reset) {
  const int64_t v = as::g_launches.load();
  if (reset) as::g_launches.store(0);
  return v;
}

int as_sm_count(void) { return sm_count(); }

int as_set_timing(int enable) {
  static bool created = false;
  if (enable && !created) {
    for (int i = 0; i <= AS_NUM_PHASES; ++i)
      if (cudaEventCreate(&g_ev[i]) != cudaSuccess) return AS_ERR_CUDA;
    created = true;
  }
  g_timing = enable != 0;
  g_timing_valid = false;
  return AS_OK;
}

int as_get_timing(float* ms, int n) {
  if (!ms) return AS_ERR_NULL;
  if (!g_timing || !g_timing_valid) return AS_ERR_NULL;
  if (cudaEventSynchronize(g_ev[AS_NUM_PHASES]) != cudaSuccess) return AS_ERR_CUDA;
  for (int i = 0; i < n && i < AS_NUM_PHASES; ++i)
    if (cudaEventElapsedTime(&ms[i], g_ev[i], g_ev[i + 1]) != cudaSuccess) return AS_ERR_CUDA;
  return AS_OK;
}

}  // extern "C"

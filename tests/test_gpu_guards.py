"""Out-of-bounds write detection without a sanitizer: every output and the scratch buffer sit between guard
regions filled with a pattern; after each entry point the guards must be untouched.  Plus run-to-run agreement."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GUARD = 4096


def guarded(nbytes):
    """(view of nbytes between two guards, whole buffer)."""
    n = (int(nbytes) + 255) // 256 * 256
    whole = torch.full((n + 2 * GUARD,), 0xA5, dtype=torch.uint8, device=DEV)
    return whole[GUARD:GUARD + n], whole, n


def guards_intact(whole, n):
    return bool((whole[:GUARD] == 0xA5).all()) and bool((whole[GUARD + n:] == 0xA5).all())


def typed(view, shape, dtype):
    numel = 1
    for s in shape:
        numel *= s
    return view[: numel * torch.empty((), dtype=dtype).element_size()].view(dtype).view(*shape)


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("batch,T,P,tbar", [(2, 300, 40, 70), (1, 1000, 136, 2000), (2, 5, 8, 2), (1, 2048, 256, 512)])
def test_no_write_outside_buffers(batch, T, P, tbar, io):
    build_library()
    w = synth.custom_workload("guard", 18, batch, T, P, tbar=tbar, io=io)
    theta = synth.layer_params(w, 0, DEV)
    x, dy = synth.activations(w, DEV)
    sh = B.shape_of(x)
    fb, gb = B.as_workspace_bytes(sh, tbar)
    esz = x.element_size()
    bufs = {}
    ws_v, ws_w, ws_n = guarded(gb)
    N = w.d_state
    shapes = {"dW_delta": (P, P), "db_delta": (P,), "dW_B": (N, P), "dW_C": (N, P), "dA_log": (P, N)}
    grads = {}
    for k, shp in shapes.items():
        numel = 1
        for s in shp:
            numel *= s
        v, wh, n = guarded(numel * 4)
        bufs[k] = (wh, n)
        grads[k] = typed(v, shp, torch.float32)
    v, wh, n = guarded(batch * T * P * esz)
    bufs["dx"] = (wh, n)
    grads["dx"] = typed(v, (batch, T, P), x.dtype)
    v, wh, n = guarded(batch * T * P * esz)
    bufs["y"] = (wh, n)
    y = typed(v, (batch, T, P), x.dtype)

    def check(what):
        torch.cuda.synchronize()
        assert guards_intact(ws_w, ws_n), f"{what}: wrote outside the workspace"
        for k, (wh_, n_) in bufs.items():
            assert guards_intact(wh_, n_), f"{what}: wrote outside {k}"

    B.as_ssm_forward(sh, theta, x, y, ws_v); check("as_ssm_forward")
    B.as_adjoint_grad(sh, theta, x, dy, tbar, grads, ws_v); check("as_adjoint_grad")
    first = {k: v.clone() for k, v in grads.items()}
    B.as_adjoint_grad(sh, theta, x, dy, tbar, grads, ws_v); check("as_adjoint_grad (second call)")
    # run-to-run: atomics make bitwise equality a non-promise, but the two runs must agree to rounding (with bf16
    # I/O a different summation order can flip the bf16 rounding of an intermediate or an output element)
    rtol = 1e-5 if io == "f32" else 1e-2
    for k in grads:
        a, b = first[k].double(), grads[k].double()
        assert float((a - b).abs().max()) <= rtol * float(a.abs().max()) + 1e-30, k
    B.as_adjoint_grad(sh, theta, x, dy, T, grads, ws_v); check("as_adjoint_grad (full)")
    B.as_full_bptt_grad(sh, theta, x, dy, grads, ws_v); check("as_full_bptt_grad")
    yh = torch.empty_like(x)
    B.as_rmsnorm_fwd(sh, x, y); B.as_rmsnorm_bwd_add(sh, x, dy, grads["dx"]); B.as_residual_add(sh, x, dy, y)
    check("glue")
    assert B.as_check_status(ws_v) == 0


def test_bounded_wait_reports_timeout_and_context_survives():
    """A device-side wait that can never be satisfied gives up after its poll limit, the host reads AS_ERR_TIMEOUT
    from the status word, and the next call on the same context works and reports AS_OK."""
    build_library()
    ws = torch.zeros(4096, dtype=torch.uint8, device=DEV)
    B.as_wait_selftest(ws, poll_limit=2048)
    assert B.as_check_status(ws) == B.AS_ERR_TIMEOUT
    w = synth.custom_workload("after", 19, 1, 64, 32, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, _ = synth.activations(w, DEV)
    sh = B.shape_of(x)
    fb, _ = B.as_workspace_bytes(sh, 64)
    ws2 = B.alloc_workspace(fb, DEV)
    y = torch.empty_like(x)
    B.as_ssm_forward(sh, theta, x, y, ws2)
    assert B.as_check_status(ws2) == B.AS_OK
    assert torch.isfinite(y).all()


@pytest.mark.parametrize("T,P", [(100, 64), (9000, 256)])   # fewer CTAs than bytes in the status block; one per SM
def test_status_block_of_packed_weights_calls(T, P):
    """With packed weights the projections both clear the status word and may report, each CTA through a byte of its own:
    every byte of a stale block has to be written, and any byte set counts."""
    build_library()
    w = synth.custom_workload("status", 20, 1, T, P, tbar=T, io="bf16")
    theta = dict(synth.layer_params(w, 0, DEV))
    x, dy = synth.activations(w, DEV)
    sh = B.shape_of(x)
    theta["Wcat"] = torch.empty(B.as_wcat_bytes(sh), dtype=torch.uint8, device=DEV)
    B.as_pack_weights(sh, 1, theta, theta["Wcat"])
    fb, gb = B.as_workspace_bytes(sh, T)
    ws = B.alloc_workspace(max(fb, gb), DEV)
    y, grads = torch.empty_like(x), B.alloc_grads(sh, DEV)
    for call in (lambda: B.as_ssm_forward(sh, theta, x, y, ws), lambda: B.as_ssm_forward_ordered(sh, theta, x, y, ws),
                 lambda: B.as_adjoint_grad(sh, theta, x, dy, T, grads, ws)):
        ws[:256] = 0xFF
        call()
        assert B.as_check_status(ws) == B.AS_OK
        for cta in (0, 1, 147, 239):
            ws[16 + cta] = 1
            assert B.as_check_status(ws) == B.AS_ERR_TIMEOUT, cta
            ws[16 + cta] = 0
        assert B.as_check_status(ws) == B.AS_OK


@pytest.mark.parametrize("io", ["f32", "bf16"])
def test_host_threads_on_their_own_streams(io):
    """Several host threads may call at once, each with its own stream and scratch; what the launchers remember per process
    is shared between them.  Sequential calls before and after give the same outputs, to the rounding of the atomics."""
    import threading
    build_library()
    w = synth.custom_workload("threads", 24, 1, 700, 136, tbar=90, io=io)
    theta = synth.layer_params(w, 0, DEV)
    x, dy = synth.activations(w, DEV)
    sh = B.shape_of(x)
    _, gb = B.as_workspace_bytes(sh, w.tbar)
    n = 4
    ws = [B.alloc_workspace(gb, DEV) for _ in range(n)]
    ys = [torch.empty_like(x) for _ in range(n)]
    grads = [B.alloc_grads(sh, DEV) for _ in range(n)]
    streams = [torch.cuda.Stream() for _ in range(n)]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            for _ in range(5):
                B.as_ssm_forward(sh, theta, x, ys[i], ws[i], stream=streams[i])
                B.as_adjoint_grad(sh, theta, x, dy, w.tbar, grads[i], ws[i], stream=streams[i])
        except Exception as e:   # an assertion in a thread would be lost
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(B.as_check_status(ws[i], streams[i]) == B.AS_OK for i in range(n))
    y, ref = torch.empty_like(x), B.alloc_grads(sh, DEV)
    B.as_ssm_forward(sh, theta, x, y, ws[0])
    B.as_adjoint_grad(sh, theta, x, dy, w.tbar, ref, ws[0])
    rtol = 1e-5 if io == "f32" else 1e-2
    for i in range(n):
        assert torch.equal(ys[i], y)
        for k, v in ref.items():
            a, b = grads[i][k].double(), v.double()
            assert float((a - b).abs().max()) <= rtol * float(b.abs().max()) + 1e-30, k

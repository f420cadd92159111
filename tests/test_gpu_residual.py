"""A layer of a residual stack in one call against its parts, bit for bit, at ragged lengths and widths, in place and without the norm
(needs a B200)."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library
from paper_2501_00692_b200.stack import Stack

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("T,P", [(1, 8), (7, 128), (8, 64), (129, 72), (600, 120), (5000, 96)])
def test_one_call_and_its_parts(T, P):
    build_library()
    w = synth.custom_workload("residual", 59, 2, T, P, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, acc = synth.activations(w, DEV)
    sh = B.shape_of(x)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, T)[0], DEV)
    tilde, total, norm = (torch.empty_like(x) for _ in range(3))
    B.as_ssm_forward_ordered(sh, theta, x, tilde, ws)
    B.as_residual_add_rmsnorm(sh, acc, tilde, total, norm)
    out, yhat = torch.empty_like(x), torch.empty_like(x)
    B.as_ssm_forward_residual(sh, theta, x, acc, out, yhat, ws)
    assert B.as_check_status(ws) == B.AS_OK
    assert torch.equal(out, total) and torch.equal(yhat, norm)
    out.zero_()
    B.as_ssm_forward_residual(sh, theta, x, acc, out, None, ws)
    assert torch.equal(out, total)
    B.as_ssm_forward_residual(sh, theta, x, acc, acc, x, ws)   # the sum over y_in, the norm over the layer's input
    assert torch.equal(acc, total) and torch.equal(x, norm)


@pytest.mark.parametrize("T,P", [(8192, 64), (8193, 64), (9000, 72)])   # both sides of the line from which a stack makes two calls
def test_stack_forward_by_either_form(T, P):
    build_library()
    w = synth.custom_workload("residual", 59, 1, T, P, layers=3, io="f32")
    thetas = [synth.layer_params(w, k, DEV) for k in range(3)]
    y0, _ = synth.activations(w, DEV)
    st = Stack(thetas, 1, T, P, dtype=torch.float32, device=DEV)
    assert st._residual == (T <= 8192 or P > 64)
    got = st.forward(y0)
    yhat, tilde, cur = torch.empty_like(y0), torch.empty_like(y0), y0.clone()
    B.as_rmsnorm_fwd(st.shape, cur, yhat)
    for th in thetas:
        B.as_ssm_forward_ordered(st.shape, th, yhat, tilde, st.ws)
        B.as_residual_add_rmsnorm(st.shape, cur, tilde, cur, yhat)
    assert B.as_check_status(st.ws) == B.AS_OK and torch.equal(got, cur)


@pytest.mark.parametrize("P,scalar,io", [(136, False, "f32"), (64, True, "f32"), (64, False, "bf16")])
def test_other_shapes_are_refused(P, scalar, io):
    build_library()
    w = synth.custom_workload("residual", 59, 1, 40, P, io=io)
    theta = synth.layer_params(w, 0, DEV)
    if scalar:
        theta["A_log"] = theta["A_log"][:, 0].contiguous()
    x, acc = synth.activations(w, DEV)
    sh = B.shape_of(x, 16, a_scalar=scalar)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, 40)[0], DEV)
    with pytest.raises(B.AsError) as e:
        B.as_ssm_forward_residual(sh, theta, x, acc, torch.empty_like(x), None, ws)
    assert e.value.code == B.AS_ERR_LIMIT


# two batch elements whose projections take the tensor cores (split operands are part of the scratch), in place too
@pytest.mark.parametrize("T,P", [(4003, 128), (9603, 104)])
def test_one_call_and_its_parts_with_split_projections(T, P):
    assert B.as_workspace_bytes(B.make_shape(2, T, P), T)[0] > 14 * 2 * T * P
    test_one_call_and_its_parts(T, P)


def test_residual_call_clears_a_stale_status():
    build_library()
    w = synth.custom_workload("residual", 59, 1, 100, 64, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, acc = synth.activations(w, DEV)
    sh = B.shape_of(x)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, 100)[0], DEV)
    ws[:256] = 0xFF
    B.as_ssm_forward_residual(sh, theta, x, acc, torch.empty_like(x), None, ws)
    assert B.as_check_status(ws) == B.AS_OK

"""Forward and gradient of a bf16 layer see the same Delta, and it is the softplus to the last bits (needs a B200).  Delta [B T, P] fp32 lies
behind the status block (256 bytes) of either call's scratch."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def delta_of(ws, n):
    return ws[256:256 + 4 * n].view(torch.float32).clone()


# on the 32-element grid; short runs with the weights in place, longer ones with packed weights, the widths' last tile full and ragged
@pytest.mark.parametrize("T,P,layers", [(200, 64, 1), (1500, 96, 1), (700, 256, 2), (2100, 416, 1)])
@pytest.mark.parametrize("ordered", [False, True])
def test_forward_and_gradient_form_the_same_delta(T, P, layers, ordered):
    build_library()
    w = synth.custom_workload("delta", 67, 1, T, P, tbar=T // 3, io="bf16")
    thetas = [synth.layer_params(w, k, DEV, slow_decay=k > 0) for k in range(layers)]
    x, dy = synth.activations(w, DEV)
    sh = B.shape_of(x, w.d_state)
    ws = B.alloc_workspace(B.as_workspace_bytes_layers(sh, layers, w.tbar) + B.as_workspace_bytes(sh, w.tbar)[0], DEV)
    y, n = torch.empty_like(x), T * P
    seen = []
    for th in thetas:
        (B.as_ssm_forward_ordered if ordered else B.as_ssm_forward)(sh, th, x, y, ws)
        seen.append(delta_of(ws, n))
    th = {k: torch.stack([t[k] for t in thetas]).contiguous() for k in thetas[0]}
    g = B.alloc_grads_layers(sh, layers, DEV, with_dx=True)
    B.as_adjoint_grad_layers(sh, layers, th, torch.stack([x] * layers), dy, w.tbar, g, ws, B.AS_ORDERED if ordered else 0)
    assert B.as_check_status(ws) == B.AS_OK
    assert torch.equal(delta_of(ws, layers * n), torch.cat(seen))
    if not ordered:   # and it is the softplus: fp32 sums of P products of bf16 values, 2e-6 for the polynomial and its argument
        u = x[0].double() @ thetas[0]["W_delta"].double().T + thetas[0]["b_delta"].double()
        size = x[0].double().abs() @ thetas[0]["W_delta"].double().abs().T + thetas[0]["b_delta"].double().abs()
        want = torch.nn.functional.softplus(u)
        off = (seen[0].view(T, P).double() - want).abs()
        assert bool((off <= want * (2e-6 + P * 2.0 ** -24 * size)).all())

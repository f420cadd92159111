"""fp32 contractions on the tensor cores (exact three-term bf16 splits) against the FP32-pipe kernels' accuracy: projections
and all dense gradients, measured against fp64 products of the same operands; shapes with ragged tiles and K blocks, several
layers, and forwards on both sides of the width from which they take them (needs a B200).  The fixed scratch that has no room
for the splits: tests/test_zz_no_alloc.py."""
import pytest
import torch

from oracle import ssm_oracle as O
from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, compare_grads, oracle_adjoint, theta_f64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# tokens * P * (P + 32) >= 2^28 takes the tensor cores
@pytest.mark.parametrize("layers,batch,T,P", [(1, 1, 4100, 248), (1, 2, 2500, 200), (2, 1, 17000, 104), (1, 1, 700, 648)])
def test_split_contractions(layers, batch, T, P):
    build_library()
    w = synth.custom_workload("split", 45, batch, T, P, tbar=max(1, T // 9), io="f32")
    thetas = [synth.layer_params(w, k, DEV, slow_decay=True) for k in range(layers)]
    x, dy = synth.activations(w, DEV)
    xs = torch.stack([x.roll(k, 1) for k in range(layers)]).contiguous()
    stacked = {k: torch.stack([t[k] for t in thetas]).contiguous() for k in thetas[0]}
    sh = B.shape_of(x, w.d_state)
    ws = B.alloc_workspace(B.as_workspace_bytes_layers(sh, layers, w.tbar), DEV)
    g = B.alloc_grads_layers(sh, layers, DEV, with_dx=True)
    B.as_adjoint_grad_layers(sh, layers, stacked, xs, dy, w.tbar, g, ws)
    assert B.as_check_status(ws) == B.AS_OK
    refs = [oracle_adjoint(thetas[k], xs[k], dy, w.tbar, channel_block=64) for k in range(layers)]
    for k in range(layers):
        compare_grads({n: v[k] for n, v in g.items()}, refs[k], TOL["f32"])
        for n in ("dW_delta", "dW_B", "dW_C", "dx"):   # well inside the bar: what fp32 multiply-adds give
            assert_close(synth.to_f64(g[n][k]), refs[k][n], 2e-5, n)
    y = torch.empty_like(x)
    B.as_ssm_forward(sh, thetas[0], x, y, ws)
    assert_close(synth.to_f64(y), refs[0]["y"], 1e-5, "y")


# forwards take the tensor cores from two column tiles on (P + 32 > 128)
@pytest.mark.parametrize("T,P", [(21900, 96), (19000, 104)])
def test_forward_on_both_sides_of_the_width_rule(T, P):
    build_library()
    w = synth.custom_workload("split-width", 46, 1, T, P, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, _ = synth.activations(w, DEV)
    sh = B.shape_of(x, w.d_state)
    fwd = B.as_workspace_bytes(sh, T)[0]
    assert (fwd > 10 * T * P) == (P > 96)      # the split operands are part of the scratch
    ws, y = B.alloc_workspace(fwd, DEV), torch.full_like(x, float("nan"))
    B.as_ssm_forward(sh, theta, x, y, ws)
    assert B.as_check_status(ws) == B.AS_OK
    assert_close(synth.to_f64(y[0]), O.ssm_forward(theta_f64(theta), synth.to_f64(x[0])), 1e-5, "y")

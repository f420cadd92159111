"""bf16 widths off the 32-element grid: the tensor-core contractions where a tile, a 16-column chunk or the border between
Delta and [B | C] cuts across the width, one layer and several layers in one launch (needs a B200)."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, compare_grads, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# P % 32 in {8, 16, 24}; widths below one tile, one row group past a 128-row tile, past a 208-column tile; T * batch with
# and without a ragged last tile (a multiple of 128 lets all layers go out as one launch)
@pytest.mark.parametrize("layers,T,P", [(1, 70, 8), (1, 200, 48), (1, 333, 104), (1, 130, 184), (1, 300, 216), (2, 64, 72), (3, 128, 136), (2, 50, 24)])
def test_bf16_width_off_the_grid(layers, T, P):
    build_library()
    w = synth.custom_workload("width", 41, 2, T, P, tbar=max(1, T // 3), io="bf16")
    thetas = [synth.layer_params(w, k, DEV, slow_decay=True) for k in range(layers)]
    x, dy = synth.activations(w, DEV)
    xs = torch.stack([x.roll(k, 1) for k in range(layers)]).contiguous()
    stacked = {k: torch.stack([t[k] for t in thetas]).contiguous() for k in thetas[0]}
    sh = B.shape_of(x, w.d_state)
    ws = B.alloc_workspace(B.as_workspace_bytes_layers(sh, layers, w.tbar), DEV)
    g = B.alloc_grads_layers(sh, layers, DEV, with_dx=True)
    B.as_adjoint_grad_layers(sh, layers, stacked, xs, dy, w.tbar, g, ws)
    assert B.as_check_status(ws) == B.AS_OK
    for k in range(layers):
        ref = oracle_adjoint(thetas[k], xs[k], dy, w.tbar)
        compare_grads({n: v[k] for n, v in g.items()}, ref, TOL["bf16"])
    # the forward, packing its weights itself and with the packed copy
    th = dict(thetas[0])
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, T)[0], DEV)
    for packed in (False, True):
        if packed:
            th["Wcat"] = torch.empty(B.as_wcat_bytes(sh), dtype=torch.uint8, device=DEV)
            B.as_pack_weights(sh, 1, th, th["Wcat"])
        y = torch.empty_like(x)
        B.as_ssm_forward(sh, th, x, y, ws)
        assert B.as_check_status(ws) == B.AS_OK
        assert_close(synth.to_f64(y), oracle_adjoint(thetas[0], x, dy, T)["y"], TOL["bf16"], "y")

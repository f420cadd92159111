"""The forward at the edges of its passes: sequence ends at every token of a chunk pair, widths below and just past a channel
tile, one segment and more segments than the carry loads ahead, both rate structures (needs a B200)."""
import pytest
import torch

from oracle import ssm_oracle as O
from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, theta_f64

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [(1, 1, 8), (2, 15, 72), (3, 66, 136), (1, 769, 264), (1, 4099, 520), (2, 1543, 384)]


@pytest.mark.parametrize("entry", [B.as_ssm_forward, B.as_ssm_forward_ordered], ids=["plain", "ordered"])
@pytest.mark.parametrize("scalar", [False, True], ids=["diagonal", "scalar"])
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d-T%d-P%d" % c)
def test_forward_edges(case, io, scalar, entry):
    build_library()
    batch, T, P = case
    w = synth.custom_workload("forward", 59, batch, T, P, tbar=T, io=io)
    theta = dict(synth.layer_params(w, 0, DEV))
    if scalar:
        theta["A_log"] = theta["A_log"][:, 0].contiguous()
    x, _ = synth.activations(w, DEV)
    sh = B.shape_of(x, w.d_state, a_scalar=scalar)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, T)[0], DEV)
    y = torch.full_like(x, float("nan"))
    entry(sh, theta, x, y, ws)
    assert B.as_check_status(ws) == 0
    ref = theta_f64(theta)
    if scalar:
        ref["A_log"] = ref["A_log"][:, None].repeat(w.d_state, axis=1)
    for b in range(batch):
        assert_close(synth.to_f64(y[b]), O.ssm_forward(ref, synth.to_f64(x[b])), TOL[io], f"y[{b}]")

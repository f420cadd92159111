"""The forward's decay factors from the smallest step sizes to those that leave nothing of a state, in the two states of a channel
whose factors the segment pass forms on the FP32 pipe (needs a B200)."""
import pytest

from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, gpu_forward, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# step sizes softplus(b): exponents of a token from some 1e-5 to beyond -1,000; 37 segments and a ragged chunk
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("b_range", [(-12, -9), (-4, -2), (-1, 1), (4, 8), (30, 60)])
def test_factors_of_two_states(b_range, io):
    build_library()
    w = synth.custom_workload("factors", 53, 2, 589, 72, io=io)
    theta = synth.layer_params(w, 0, DEV, b_delta_range=b_range)
    keep = theta["W_B"].clone()
    theta["W_B"].zero_()
    for n in (7, 15):
        theta["W_B"][n] = keep[n]
    x, dy = synth.activations(w, DEV)
    ref = oracle_adjoint(theta, x, dy, w.seqlen)["y"]
    assert_close(synth.to_f64(gpu_forward(w, theta, x)), ref, TOL[io], "y")

"""The forward's decay factors from the smallest step sizes to those that leave nothing of a state, in the two states of a channel
whose factors the segment pass forms on the FP32 pipe (needs a B200)."""
import math

import numpy as np
import pytest
import torch

from oracle import ssm_oracle as O
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, gpu_forward, oracle_adjoint, theta_f64

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


@pytest.mark.parametrize("io", ["f32", "bf16"])
def test_nothing_is_left_of_a_large_state(io):
    """A state of some 1e36, then a token whose factors lie far below the smallest fp32 number, then tokens that hardly decay and
    look at the state: nothing of it is left.  The large tokens stand third, the decays last in every four, so that each segment (a
    multiple of eight tokens) ends right after a decay."""
    build_library()
    P, T = 8, 640
    w = synth.custom_workload("left", 71, 1, T, P, io=io)
    theta = synth.layer_params(w, 0, DEV)
    for k in ("W_delta", "W_B", "W_C"):
        theta[k].zero_()
    theta["A_log"].fill_(math.log(16.0))
    theta["b_delta"].fill_(-20.0)
    theta["W_delta"][0, 1] = 1.0   # Delta of channel 0 by x of channel 1, B by channel 0, C by channel 2
    theta["W_B"][:, 0] = 0.25
    theta["W_C"][:, 2] = 1.0
    x = torch.zeros(1, T, P, device=DEV, dtype=w.torch_dtype)
    x[:, 2::4, 0], x[:, 2::4, 1] = 1e19, 18.0   # Delta 0.13
    x[:, 3::4, 1] = 120.0                        # Delta 100
    x[:, 0::4, 0], x[:, 0::4, 2] = 1.0, 1.0      # Delta 2e-9
    y = synth.to_f64(gpu_forward(w, theta, x))[..., 0]
    ref = oracle_adjoint(theta, x, torch.zeros_like(x), T)["y"][..., 0]
    assert abs(ref).max() < 1e-6
    assert abs(y - ref).max() < 1e-6, abs(y - ref).max()


# 41,428 tokens of one channel tile: on 148 SMs segments of 96 (fp32) and 40 (bf16) tokens, more chunks than the staging ring holds, so the
# two states go from chunk to chunk and from segment to segment through the polynomial factors; a ragged last chunk
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("b_range", [(-9, -7), (-4, -2), (-1, 1)])
def test_factors_of_two_states_over_many_chunks(b_range, io):
    build_library()
    w = synth.custom_workload("factors", 54, 4, 10357, 72, io=io)
    theta = synth.layer_params(w, 0, DEV, b_delta_range=b_range)
    for n in range(16):
        if n not in (7, 15):
            theta["W_B"][n].zero_()
    x, _ = synth.activations(w, DEV)
    y = synth.to_f64(gpu_forward(w, theta, x))
    th = theta_f64(theta)
    assert_close(y, np.stack([O.ssm_forward(th, one) for one in synth.to_f64(x)]), TOL[io], "y")

"""Scan kernels at CTA counts around whole multiples of the SM count, where the shared memory that spreads a launch changes, and
beyond the count from which on none is added (needs a B200)."""
import pytest

from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, compare_grads, gpu_adjoint, gpu_forward, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# one channel tile in segments of 16 tokens: a CTA for every 16 tokens, on 148 SMs
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("ctas", [1, 147, 148, 149, 296, 297, 445, 593])
def test_around_whole_shares(ctas, io):
    build_library()
    w = synth.custom_workload("spread", 47, 1, 16 * ctas, 40, tbar=35, io=io)
    theta = synth.layer_params(w, 0, DEV, slow_decay=True)
    x, dy = synth.activations(w, DEV)
    ref = oracle_adjoint(theta, x, dy, 35)
    compare_grads(gpu_adjoint(w, theta, x, dy, 35), ref, TOL[io])
    assert_close(synth.to_f64(gpu_forward(w, theta, x)), ref["y"], TOL[io], "y")

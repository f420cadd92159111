"""Scan kernels at CTA counts around whole multiples of the SM count, where the shared memory that spreads a launch changes, and
beyond the count from which on none is added (needs a B200)."""
import numpy as np
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import PARAM, TOL, assert_close, compare_grads, gpu_adjoint, gpu_forward, oracle_adjoint

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


# 40 tokens and so many batch elements that each is one segment: a CTA per element, up to the share of an SM from which on no shared
# memory is added (5 in fp32, 8 in bf16)
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("share", [2, 3, 4, 5, 7, 8])
def test_one_cta_per_batch_element(share, more, io):
    build_library()
    kinds, n = 4, share * B.as_sm_count() + more
    w = synth.custom_workload("shares", 48, kinds, 40, 40, tbar=13, io=io)
    theta = synth.layer_params(w, 0, DEV, slow_decay=True)
    x, dy = synth.activations(w, DEV)
    of = torch.arange(n, device=DEV) % kinds
    g = gpu_adjoint(w, theta, x[of].contiguous(), dy[of].contiguous(), 13)
    refs = [oracle_adjoint(theta, x[k:k + 1], dy[k:k + 1], 13) for k in range(kinds)]
    want = {name: sum(int((of == k).sum()) * refs[k][name] for k in range(kinds)) for name in PARAM}
    want["dx"] = np.concatenate([r["dx"] for r in refs])[of.cpu().numpy()]
    compare_grads(g, want, TOL[io])

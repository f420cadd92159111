"""Carries across time segments at the edges of their forms: windows shorter than a segment, of up to four whole segments
(summed directly), of five and more (block sums), blocks that do not divide the segments, one segment, the full form with
one- and two-chunk segments, runs with and without segments whose window-exit terms are ruled out (needs a B200)."""
import pytest

from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, compare_grads, gpu_adjoint, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# segments are 16 tokens at these widths in the truncated form and 8 in the full form up to 1,024 tokens
CASES = [(1, 16, 8, 5, "slow"), (1, 17, 8, 16, "slow"), (2, 250, 72, 15, "slow"), (2, 250, 72, 79, "slow"), (2, 250, 72, 80, "slow"),
         (1, 1000, 40, 83, "slow"), (1, 1000, 40, 501, "slow"), (1, 1000, 40, 999, "slow"), (1, 1000, 136, 1000, "slow"),
         (1, 1030, 40, 1030, "slow"), (1, 3000, 64, 1500, "standard"), (1, 3000, 64, 1500, "fast"), (2, 2500, 200, 700, "fast")]


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d-T%d-P%d-tb%d-%s" % c)
def test_carry_forms(case, io):
    build_library()
    batch, T, P, tbar, law = case
    w = synth.custom_workload("carry", 43, batch, T, P, tbar=tbar, io=io)
    rng = {"slow": (-9.0, -7.0), "standard": None, "fast": (-1.0, 1.0)}[law]
    theta = synth.layer_params(w, 0, DEV, b_delta_range=rng)
    x, dy = synth.activations(w, DEV)
    compare_grads(gpu_adjoint(w, theta, x, dy, tbar), oracle_adjoint(theta, x, dy, tbar), TOL[io])

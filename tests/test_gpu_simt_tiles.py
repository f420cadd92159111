"""The fp32-pipe contractions on both tile sizes: remainders of the 32- and 64-wide tiles and of their K-tiles, one token,
and the last shape of the small tiles with the first one of the large (needs a B200)."""
import pytest

from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, compare_grads, gpu_adjoint, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [(1, 1, 8), (1, 33, 24), (1, 63, 40), (2, 97, 72), (1, 129, 136), (1, 4700, 64), (1, 4800, 64)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d-T%d-P%d" % c)
def test_simt_tiles(case):
    build_library()
    batch, T, P = case
    w = synth.custom_workload("simt", 61, batch, T, P, tbar=T, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, dy = synth.activations(w, DEV)
    compare_grads(gpu_adjoint(w, theta, x, dy, T), oracle_adjoint(theta, x, dy, T), TOL["f32"])

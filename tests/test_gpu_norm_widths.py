"""Norm kernels at the edges of their row layouts: widths below, at and past the 16-byte pieces a lane keeps in registers,
ragged last pieces, widths beyond them; in-place sums (needs a B200)."""
import pytest
import torch

from oracle import ssm_oracle as O
from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import assert_close

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("io,tol", [("f32", 1e-5), ("bf16", 8e-3)])
@pytest.mark.parametrize("P", [8, 120, 128, 136, 256, 264, 520, 768, 1032, 1288, 1544, 2048, 2056, 4104])
def test_norm_and_add(P, io, tol):
    build_library()
    w = synth.custom_workload("norms", 44, 2, 13, P, io=io)
    y, d = synth.activations(w, DEV)
    sh = B.shape_of(y)
    yhat, out, both = torch.empty_like(y), torch.empty_like(y), torch.empty_like(y)
    B.as_rmsnorm_fwd(sh, y, yhat)
    assert_close(synth.to_f64(yhat), O.rmsnorm(synth.to_f64(y)), tol, "norm")
    G = d.clone()
    B.as_rmsnorm_bwd_add(sh, y, d, G)
    assert_close(synth.to_f64(G), synth.to_f64(d) + O.rmsnorm_vjp(synth.to_f64(y), synth.to_f64(d)), tol, "norm vjp")
    B.as_residual_add(sh, y, d, out)
    assert torch.equal(out, y + d)
    B.as_rmsnorm_fwd(sh, out, yhat)
    acc, tilde = y.clone(), d.clone()
    B.as_residual_add_rmsnorm(sh, acc, tilde, acc, both)      # in place, then also over its second operand
    assert torch.equal(acc, out) and torch.equal(both, yhat)
    B.as_residual_add_rmsnorm(sh, y, tilde, acc, tilde)
    assert torch.equal(acc, out) and torch.equal(tilde, yhat)

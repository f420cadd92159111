"""Window exits and where they are left out (EXIT_LOG2 and EXIT_MARGIN_LOG2 in as_scan.cuh): the truncated gradient against the oracle,
with windows whose slowest exit factors lie on both sides of 2^-30 and 2^-64, and with upstream gradients that make an exit the whole
answer (needs a B200)."""
import numpy as np
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, assert_close, gpu_adjoint, oracle_adjoint, theta_f64, PARAM

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# standard law, 16 channels: the slowest state decays by some 0.04 log2 units a token, so the largest W of Tbar = 400 .. 1600 is 2^-14 .. 2^-65
@pytest.mark.parametrize("tbar", [400, 800, 1000, 1300, 1600])
@pytest.mark.parametrize("late", [False, True])
def test_exit_factors_around_the_cut(tbar, late):
    build_library()
    T = 3000
    w = synth.custom_workload("exitcut", 47, 1, T, 16, tbar=tbar, io="f32")
    theta = synth.layer_params(w, 0, DEV)
    x, dy = synth.activations(w, DEV)
    if late:
        dy[:, : T - 8] = 0   # tokens more than a window before the end get nothing once the last ones have left
    g = gpu_adjoint(w, theta, x, dy, tbar)
    ref = oracle_adjoint(theta, x, dy, tbar)
    # fp32 sums over up to 3,000 tokens (fixed-order part below 3000 * 2^-24 of the largest term; measured 1e-6): 1e-5
    for k in PARAM + ("dx",):
        assert_close(synth.to_f64(g[k]), ref[k], 1e-5, k)
    if late:
        # what exits leave behind: a W (the largest there is) of the cotangents, times the tbar roundings by which W and the recurrence differ
        x64, th = synth.to_f64(x)[0], theta_f64(theta)
        sums = np.cumsum(np.logaddexp(0.0, x64 @ th["W_delta"].T + th["b_delta"]), axis=0)
        W = np.exp(-np.exp(th["A_log"]).min(axis=1) * (sums[tbar:] - sums[:-tbar]).min(axis=0)).max()
        early = synth.to_f64(g["dx"])[:, : T - 8 - tbar]
        want = ref["dx"][:, : T - 8 - tbar]
        assert np.abs(early - want).max() <= (W * tbar * 2.0 ** -22 + 2.0 ** -64) * np.abs(ref["dx"]).max()


def _rates(kind, T, tbar, delta):
    """A_log whose window factors W = exp(A delta tbar) are 2^-log2w, per state: one state at `kind` among faster ones, or all of them."""
    which, log2w = kind
    fast = 90.0 + 2.0 * torch.arange(16, device=DEV)
    l2 = torch.full((16,), log2w, device=DEV) if which is None else torch.where(torch.arange(16, device=DEV) == which, log2w, fast)
    return torch.log(l2 * (np.log(2.0) / (delta * tbar)))


# One cotangent is larger than the others by `up` powers of two.  Its term leaves the tokens more than a window before it at W times that,
# 2^-4 of an ordinary cotangent (bf16: as large as one), whether W is 2^-42 or 2^-60; below 2^-64 nothing of it is to be seen.
@pytest.mark.parametrize("io,scalar,which", [(io, False, which) for io in ("f32", "bf16") for which in (None, 0, 7, 10)] + [("f32", True, None)])
@pytest.mark.parametrize("log2w,up", [(42.0, 38), (52.0, 48), (60.0, 56), (75.0, 40)])
def test_exit_of_a_cotangent_above_all_others(io, scalar, which, log2w, up):
    build_library()
    T, P, tbar, at = 1500, 40, 512, 1480
    delta = 0.05
    dt = torch.float32 if io == "f32" else torch.bfloat16
    gen = torch.Generator(device=DEV).manual_seed(11)
    normal = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    A_log = _rates((which, log2w), T, tbar, delta).expand(P, 16).contiguous()
    theta = {"W_delta": torch.zeros(P, P, device=DEV).to(dt), "b_delta": torch.full((P,), float(np.log(np.expm1(delta))), device=DEV),
             "W_B": (normal(16, P) / P ** 0.5).to(dt), "W_C": (normal(16, P) / P ** 0.5).to(dt), "A_log": A_log}
    x, dy = normal(1, T, P).to(dt), normal(1, T, P).to(dt)
    dy[:, at] *= 2.0 ** (up + (4 if io == "bf16" else 0))
    ref = oracle_adjoint(theta, x, dy, tbar)
    if scalar:
        theta["A_log"] = A_log[:, 0].contiguous()
    sh = B.shape_of(x, 16, a_scalar=scalar)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, tbar)[1], DEV)
    g = B.alloc_grads(sh, DEV)
    B.as_adjoint_grad(sh, theta, x, dy, tbar, g, ws)
    assert B.as_check_status(ws) == B.AS_OK
    # the tokens just before the window of token `at`.  fp32: W and the recurrence it is taken from agree to some T tbar-fold product
    # roundings, 512 * 2^-22 of the 2^-4 that leaves, beside the sums' own 1e-5; bf16 outputs 2^-9, operands of the input gradient likewise
    rows = slice(at - tbar - 39, at - tbar + 1)
    assert_close(synth.to_f64(g["dx"])[:, rows], ref["dx"][:, rows], 2e-5 if io == "f32" else TOL["bf16"], "dx")

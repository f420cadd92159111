"""Weight and input gradient of bf16 I/O in one launch and in two, several layers at once; phase timing, which makes them two and
tells them apart (needs a B200)."""
import pytest
import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library

from gpu_util import TOL, compare_grads, oracle_adjoint

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def stacked_call(w, layers, with_dx, timed):
    thetas = [synth.layer_params(w, k, DEV) for k in range(layers)]
    x, dy = synth.activations(w, DEV)
    xs = torch.stack([x.roll(k, 1) for k in range(layers)]).contiguous()
    th = {k: torch.stack([t[k] for t in thetas]).contiguous() for k in thetas[0]}
    sh = B.shape_of(x, w.d_state)
    ws = B.alloc_workspace(B.as_workspace_bytes_layers(sh, layers, w.tbar), DEV)
    g = B.alloc_grads_layers(sh, layers, DEV, with_dx=with_dx)
    B.as_set_timing(timed)
    try:
        phases = []
        for _ in range(3):
            B.as_adjoint_grad_layers(sh, layers, th, xs, dy, w.tbar, g, ws)
            phases.append(B.as_get_timing() if timed else None)
    finally:
        B.as_set_timing(False)
    assert B.as_check_status(ws) == B.AS_OK
    return thetas, xs, dy, g, phases


# widths on the 32-element grid and 16 off it; up to 1,024 tokens in all the weights are read where they lie, beyond that packed
@pytest.mark.parametrize("timed", [False, True])
@pytest.mark.parametrize("layers,T,P", [(3, 300, 80), (2, 511, 48), (3, 300, 96), (2, 700, 80), (1, 130, 16)])
def test_layers_in_one_launch_and_two(layers, T, P, timed):
    build_library()
    w = synth.custom_workload("launches", 53, 1, T, P, tbar=T // 2, io="bf16")
    thetas, xs, dy, g, _ = stacked_call(w, layers, True, timed)
    for k in range(layers):
        compare_grads({n: v[k] for n, v in g.items()}, oracle_adjoint(thetas[k], xs[k], dy, w.tbar), TOL["bf16"])


@pytest.mark.parametrize("with_dx", [True, False])
def test_phases_tell_the_contractions_apart(with_dx):
    """40,000 x 512: some 30 us for either contraction; two events with nothing between them are some 3 us apart."""
    build_library()
    w = synth.custom_workload("phases", 59, 1, 40000, 512, tbar=64, io="bf16")
    *_, phases = stacked_call(w, 1, with_dx, True)
    best = {k: min(p[k] for p in phases) for k in B.PHASES}
    assert all(v > 0 for v in best.values())
    assert best["weight_grads"] > 0.01
    assert (best["input_grad"] > 0.01) == with_dx, best


def test_large_layers_take_two_launches():
    """3 x 10,001 x 2,048: 960 tiles of 33 blocks for the input gradient, past the line of 400 blocks a pair of CTAs; rows that end inside
    a tile.  Every layer against a call of its own, which makes one launch: the same sums in another order, rounded to bf16 on the way
    (dx, and du as the operand of both contractions)."""
    build_library()
    w = synth.custom_workload("large", 61, 1, 10001, 2048, tbar=300, io="bf16")
    B.as_launch_count(reset=True)
    thetas, xs, dy, g, _ = stacked_call(w, 3, True, False)
    two = B.as_launch_count() // 3
    sh = B.shape_of(dy, w.d_state)
    ws = B.alloc_workspace(B.as_workspace_bytes(sh, w.tbar)[1], DEV)
    one = B.alloc_grads(sh, DEV, with_dx=True)
    for k in range(3):
        B.as_launch_count(reset=True)
        B.as_adjoint_grad(sh, thetas[k], xs[k], dy, w.tbar, one, ws)
        assert B.as_check_status(ws) == B.AS_OK
        assert two == B.as_launch_count() + 1
        for name, v in one.items():
            assert float((g[name][k].float() - v.float()).norm() / v.float().norm()) <= 2.0 ** -8, name

"""A stack whose parameters are updated in place between two steps, as training does it: the next step's results are those of a stack
built on the new values (needs a B200)."""
import pytest
import torch

from paper_2501_00692_b200 import synth
from paper_2501_00692_b200.build import build_library
from paper_2501_00692_b200.stack import Stack

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
K, T, P, TBAR = 3, 300, 64, 70
RTOL = {"f32": 1e-5, "bf16": 1e-2}   # the order of the atomic additions; every update below moves the results by far more


def setting(io):
    build_library()
    w = synth.custom_workload("updates", 61, 2, T, P, layers=K, tbar=TBAR, io=io)
    return w, [synth.layer_params(w, k, DEV) for k in range(K)], *synth.activations(w, DEV)


def step(st, x, g, mode):
    y = st.forward(x)
    grads, g0 = st.adjoint_grad(g, mode)
    out = {"y": y, **{f"{n} {k}": v for k, one in enumerate(grads) for n, v in one.items() if v is not None}}
    return out if g0 is None else {**out, "g0": g0}


def build(w, thetas):
    return Stack(thetas, w.batch, T, P, dtype=w.torch_dtype, device=DEV, tbar=TBAR)


def update(thetas):
    for th in thetas:
        th["W_delta"].neg_()
        th["b_delta"].add_(1.0)
        th["W_B"].mul_(2.0)
        th["W_C"].mul_(-1.5)
        th["A_log"].add_(0.7)


def check(got, want, io):
    torch.cuda.synchronize()
    assert got.keys() == want.keys() and torch.equal(got["y"], want["y"])
    for k in want:
        a, b = got[k].double(), want[k].double()
        assert float((a - b).abs().max()) <= RTOL[io] * float(b.abs().max()), k


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["chained", "paper"])
def test_update_between_steps(io, mode):
    w, thetas, x, g = setting(io)
    st = build(w, thetas)
    step(st, x, g, mode)
    update(thetas)
    check(step(st, x, g, mode), step(build(w, thetas), x, g, mode), io)
    st.forward(x)
    update(thetas)   # after the forward: the gradients are those at the new values
    got, _ = st.adjoint_grad(g, mode)
    fresh = build(w, thetas)
    fresh.ys = st.ys
    want, _ = fresh.adjoint_grad(g, mode)
    for k in range(K):
        one = {n: v for n, v in got[k].items() if v is not None}
        check({"y": x, **one}, {"y": x, **{n: want[k][n] for n in one}}, io)


@pytest.mark.parametrize("mode", ["chained", "paper"])
def test_writes_that_are_not_counted(mode):
    w, thetas, x, g = setting("bf16")
    st = build(w, thetas)
    step(st, x, g, mode)
    for th in thetas:
        for v in th.values():
            v.data.mul_(0.5)   # leaves the tensor's count of writes alone
    st.parameters_changed()
    check(step(st, x, g, mode), step(build(w, thetas), x, g, mode), "bf16")


@pytest.mark.parametrize("mode", ["chained", "paper"])
def test_update_between_replays(mode):
    w, thetas, x, g = setting("bf16")
    st = build(w, thetas)
    step(st, x, g, mode)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = step(st, x, g, mode)
    update(thetas)
    graph.replay()
    check(out, step(build(w, thetas), x, g, mode), "bf16")
    update(thetas)
    check(step(st, x, g, mode), step(build(w, thetas), x, g, mode), "bf16")


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["chained", "paper"])
def test_step_of_a_fused_optimizer(io, mode):
    """Fused optimizers write the parameters without counting it."""
    w, thetas, x, g = setting(io)
    st = build(w, thetas)
    step(st, x, g, mode)
    params = [v for th in thetas for v in th.values()]
    for v in params:
        v.grad = -v   # p - 0.5 * -p
    torch.optim.SGD(params, lr=0.5, fused=True).step()
    check(step(st, x, g, mode), step(build(w, thetas), x, g, mode), io)

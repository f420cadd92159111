"""Performance cases: what a program that uses this library has it do.

Three kinds of work, all through the public entry points:

  grad     one layer's gradients by the adjoint method (``binding.as_adjoint_grad``), full or truncated: the library's
           main product, called once per layer and training step;
  forward  one layer's forward (``binding.as_ssm_forward``), or the same for a caller that may not allocate device
           memory (``binding.as_ssm_forward_static``);
  stack    one training step of a residual stack (``stack.Stack``): the forward, then the gradients of every layer,
           chained through the stack or with the layers independent ("paper").

The sizes are the five workloads of ``synth.WORKLOADS`` and what lies between and beside them.  ``as_full_bptt_grad`` is
left out: it is a plain comparator that exists to check the adjoint path.
"""
import math

import torch

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200.stack import Stack

DEV = "cuda:0"
N = 16  # d_state


def listed():
    return [
        # C1, the smallest configuration (and what a unit test or a notebook runs): launches and latency count
        dict(name="grad_c1", kind="grad", io="f32", batch=1, seqlen=512, d_model=64, tbar=512, scalar=False, slow=False, dx=True),
        # C2: fp32 with a short window over a long sequence
        dict(name="grad_c2", kind="grad", io="f32", batch=1, seqlen=8192, d_model=256, tbar=64, scalar=False, slow=False, dx=True),
        # C3, the benchmark: a layer of the 127M-class width at 64K context
        dict(name="grad_c3", kind="grad", io="bf16", batch=2, seqlen=65536, d_model=768, tbar=2048, scalar=False, slow=False, dx=True),
        # C5's width and window on a quarter of its context: the largest single layer
        dict(name="grad_c5_part", kind="grad", io="bf16", batch=1, seqlen=262144, d_model=2048, tbar=4096, scalar=False, slow=False, dx=True),
        # a width, length and window that no tile divides, at an ordinary size
        dict(name="grad_ragged", kind="grad", io="bf16", batch=3, seqlen=5003, d_model=1000, tbar=777, scalar=False, slow=False, dx=True),
        # one C4 layer whose state decays slowly, so that the window's edge matters in every chunk; parameter gradients only
        dict(name="grad_slow", kind="grad", io="bf16", batch=2, seqlen=32768, d_model=768, tbar=1024, scalar=False, slow=True, dx=False),
        # the scalar structure (one decay rate per channel), full adjoint
        dict(name="grad_scalar", kind="grad", io="bf16", batch=2, seqlen=20000, d_model=512, tbar=20000, scalar=True, slow=False, dx=True),
        # inference / evaluation over the benchmark's batch
        dict(name="forward_c3", kind="forward", io="bf16", batch=2, seqlen=65536, d_model=768, scalar=False, slow=False, static=False),
        # the same for the scalar structure at C4's size
        dict(name="forward_scalar", kind="forward", io="bf16", batch=2, seqlen=32768, d_model=768, scalar=True, slow=False, static=False),
        # a short prompt inside a latency-critical host program
        dict(name="forward_guest", kind="forward", io="bf16", batch=1, seqlen=256, d_model=256, scalar=False, slow=False, static=True),
        # a training step of a stack at C4's width, length and window
        dict(name="stack_chained", kind="stack", io="bf16", batch=2, seqlen=32768, d_model=768, tbar=1024, layers=12, mode="chained", slow=False),
        # a small stack with independent layers, where the host's part of a step shows
        dict(name="stack_paper", kind="stack", io="f32", batch=1, seqlen=1024, d_model=64, tbar=256, layers=12, mode="paper", slow=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "grad", "forward", "forward", "stack"])
    io = rng.choice(["bf16", "bf16", "f32"])
    # widths: model widths are usually multiples of 64; any multiple of 8 is allowed
    width = _log_int(rng, 64, 2048 if io == "bf16" else 768)
    width = max(64, width // 64 * 64) if rng.random() < 0.6 else max(64, width // 8 * 8)
    batch = rng.choice([1, 1, 2, 3, 4])
    layers = rng.randint(2, 12) if kind == "stack" else 1
    # tokens of the batch; fp32 and widths off the 32-element grid are used for shorter runs
    most = 1 << 27 if io == "bf16" and width % 32 == 0 else 1 << 23
    tokens = _log_int(rng, 256, max(512, min(131072, most // width) // layers))
    seqlen = max(16, tokens // batch)
    case = dict(kind=kind, io=io, batch=batch, seqlen=seqlen, d_model=width, slow=rng.random() < 0.25)
    if kind != "stack":
        case["scalar"] = rng.random() < 0.2
    if kind == "forward":
        # the guest entry point has a fixed scratch: short sequences only
        case["static"] = batch * seqlen * width <= 1 << 20 and width <= 1024 and rng.random() < 0.5
    else:
        case["tbar"] = seqlen if rng.random() < 0.35 else _log_int(rng, min(16, seqlen), seqlen)
    if kind == "grad":
        case["dx"] = rng.random() < 0.75
    if kind == "stack":
        case["layers"], case["mode"] = layers, rng.choice(["chained", "paper"])
    return case


def _dtype(case):
    return torch.float32 if case["io"] == "f32" else torch.bfloat16


def _layer(case, gen):
    """Parameters of one layer, by the laws of ``synth``."""
    P, dt = case["d_model"], _dtype(case)

    def normal(*shape):
        return (torch.randn(*shape, generator=gen, device=DEV) / math.sqrt(P)).to(dt)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=gen, device=DEV)

    return {
        "W_delta": normal(P, P),
        "b_delta": uniform(-9.0, -7.0, P) if case["slow"] else uniform(-4.0, -2.0, P),
        "W_B": normal(N, P),
        "W_C": normal(N, P),
        "A_log": uniform(0.0, math.log(16.0), *((P,) if case.get("scalar") else (P, N))),
    }


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shape, dt = (case["batch"], case["seqlen"], case["d_model"]), _dtype(case)
    s = {"case": case}
    if case["kind"] == "stack":
        s["stack"] = Stack([_layer(case, gen) for _ in range(case["layers"])], *shape, dtype=dt, device=DEV, tbar=case["tbar"])
    else:
        s["theta"] = _layer(case, gen)
    s["x"] = torch.randn(shape, generator=gen, device=DEV, dtype=dt)
    if case["kind"] != "forward":
        s["dy"] = torch.randn(shape, generator=gen, device=DEV, dtype=dt)
    if case["kind"] == "grad":
        s["shape"] = B.shape_of(s["x"], N, a_scalar=case["scalar"])
        s["ws"] = B.alloc_workspace(B.as_workspace_bytes(s["shape"], case["tbar"])[1], DEV)
        s["grads"] = B.alloc_grads(s["shape"], DEV, with_dx=case["dx"])
    if case["kind"] == "forward":
        s["shape"] = B.shape_of(s["x"], N, a_scalar=case["scalar"])
        s["y"] = torch.empty_like(s["x"])
        if not case["static"]:
            s["ws"] = B.alloc_workspace(B.as_workspace_bytes(s["shape"], case["seqlen"])[0], DEV)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "grad":
        B.as_adjoint_grad(s["shape"], s["theta"], s["x"], s["dy"], case["tbar"], s["grads"], s["ws"])
        return s["grads"]
    if case["kind"] == "forward":
        if case["static"]:
            B.as_ssm_forward_static(s["shape"], s["theta"], s["x"], s["y"])
        else:
            B.as_ssm_forward(s["shape"], s["theta"], s["x"], s["y"], s["ws"])
        return s["y"]
    y = s["stack"].forward(s["x"])
    grads, g0 = s["stack"].adjoint_grad(s["dy"], mode=case["mode"])
    return {"y": y, "grads": grads, "g0": g0}


def work(case):
    """Each input read once and each output written once; two operations per multiply-add of the dense products
    (projections; for the gradients also the weight and, where it is wanted, the input gradient) and of the recurrences:
    per token, channel and state 3 multiply-adds for the state and y, 12 for the state and the adjoint."""
    e = 4 if case["io"] == "f32" else 2
    P, M, K = case["d_model"], case["batch"] * case["seqlen"], case.get("layers", 1)
    act = M * P * e
    a_log = 4 * P * (1 if case.get("scalar") else N)
    params = (P + 2 * N) * P * e + 4 * P + a_log
    pgrads = (P + 2 * N) * P * 4 + 4 * P + a_log
    dense, step = 2.0 * M * P * (P + 2 * N), 2.0 * M * P * N
    if case["kind"] == "forward":
        return {"bytes": 2 * act + params, "flops": dense + 3 * step}
    if case["kind"] == "grad":
        return {"bytes": (3 if case["dx"] else 2) * act + params + pgrads, "flops": (3 if case["dx"] else 2) * dense + 12 * step}
    chained = case["mode"] == "chained"
    return {"bytes": (4 if chained else 3) * act + K * (params + pgrads),
            "flops": K * ((4 if chained else 3) * dense + 15 * step)}


def tolerance(case):
    if case["io"] == "f32":
        # sums over up to a hundred thousand tokens in fp32; a stack carries one layer's rounding into the next
        return {"rel": 5e-5}
    # bf16 activations between the phases; a stack also rounds every layer's output to bf16
    return {"rel": 2e-2 if case["kind"] == "stack" else 1e-2, "max": 0.3}

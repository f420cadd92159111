"""Residual stack of K selective-SSM layers (Section 3.2; Algorithms 1 and 4 on one device):
y_k = y_{k-1} + SSM_k(Norm(y_{k-1})).  This module only sequences calls of the C-ABI library - every
tensor operation (RMSNorm, the layer forward, the residual add, the adjoint gradients, the RMSNorm VJP)
runs in the library's kernels; torch supplies device buffers.

Two gradient modes:
  "paper"   - Proposition 3 as printed: every layer receives the top gradient dL/dy_K itself and treats its
              input Norm(y_{k-1}) as a constant, so all layers are independent given the stored activations.
  "chained" - backpropagation through the whole stack: G_K = dL/dy_K, and going down
              G_{k-1} = G_k + RMSNormVJP(y_{k-1}, dx_k) with layer k driven by G_k.
"""
from __future__ import annotations

from operator import is_

import torch
from torch.optim.optimizer import register_optimizer_step_post_hook

from . import binding as B


_optimizer_steps = 0   # of any optimizer: fused ones write parameters without PyTorch counting it


def _after_optimizer_step(*_):
    global _optimizer_steps
    _optimizer_steps += 1


register_optimizer_step_post_hook(_after_optimizer_step)

WEIGHTS = ("W_delta", "W_B", "W_C")   # what a packed copy is made of


class Stack:
    """The parameters stay the caller's tensors and may be updated in place between two calls.  The copies of them that this object
    keeps, packed weights (bf16) and, for the batched "paper" gradients, all parameters stacked, are made again by the next call
    after a write that PyTorch counts and after the step of any torch.optim optimizer; after any other write (through `.data`, by
    a kernel of one's own, by replaying a graph that does not hold the stack's calls) call parameters_changed()."""

    def __init__(self, thetas, batch, seqlen, d_model, d_state=16, dtype=torch.float32, device="cuda:0", tbar=None,
                 eps=1e-6):
        self.thetas = [dict(t) for t in thetas]   # own dicts: a packed copy of the weights is added below
        self.K = len(thetas)
        self.eps = eps
        self.device = device
        io = B.AS_F32 if dtype == torch.float32 else B.AS_BF16
        self.shape = B.make_shape(batch, seqlen, d_model, d_state, io)
        self.tbar = seqlen if tbar is None else tbar
        _, gbytes = B.as_workspace_bytes(self.shape, self.tbar)
        self.ws = B.alloc_workspace(gbytes, device)
        self.ys = None       # y_0 .. y_K
        self.yhat = torch.empty(batch, seqlen, d_model, dtype=dtype, device=device)
        self._residual = B.as_ssm_forward_residual_applies(self.shape)   # a layer's last kernel ends in the sum and the norm
        self.ytilde = None if self._residual else torch.empty_like(self.yhat)
        # the bf16 tensor-core contractions read [W_delta; W_B; W_C] as one matrix: packed per layer, but for the layers whose
        # packed copy is the caller's
        self._own = [th for th in self.thetas if th.get("Wcat") is None] if io == B.AS_BF16 else []
        for th in self._own:
            th["Wcat"] = torch.empty(B.as_wcat_bytes(self.shape), dtype=torch.uint8, device=device)
        self._stacked = None   # parameters with a leading [K] dimension, built on first use of the batched call
        self._ws_layers = None
        self._captured = False
        self.parameters_changed()
        self._pack()

    def parameters_changed(self):
        """The copies of the parameters are made again before their next use."""
        self._packed_of = self._stacked_of = None

    def _contents(self, thetas, keys):
        """The parameters `keys`, how often each has been written, and the optimizers' steps so far; None where that cannot be told:
        inference tensors do not count writes, and a graph's replays write without a count, to the stack's parameters or
        before its captured calls."""
        self._captured = self._captured or torch.cuda.is_current_stream_capturing()
        if self._captured:
            return None
        ts = [th[k] for th in thetas for k in keys]
        try:
            return ts, [t._version for t in ts] + [_optimizer_steps]
        except RuntimeError:
            return None

    @staticmethod
    def _same(a, b):
        return a is not None and b is not None and a[1] == b[1] and all(map(is_, a[0], b[0]))

    def _pack(self):
        """Brings the packed weights in line with the parameters."""
        if not self._own:
            return
        now = self._contents(self._own, WEIGHTS)
        if self._same(now, self._packed_of):
            return
        for th in self._own:
            B.as_pack_weights(self.shape, 1, th, th["Wcat"])
        self._packed_of = now

    def forward(self, y0: torch.Tensor):
        """Runs the stack, keeping y_0..y_K (the per-layer inputs are re-normalised in the backward)."""
        self._pack()
        self.ys = [y0]
        # y_1 .. y_{K-1} in one block (one allocation, and the paper mode normalises them in one launch); y_K, which the
        # caller may keep, on its own
        block = torch.empty(max(self.K - 1, 0), *y0.shape, dtype=y0.dtype, device=y0.device)
        outs = [*block.unbind(0), torch.empty_like(y0)] if self.K else []
        B.as_rmsnorm_fwd(self.shape, y0, self.yhat, self.eps)
        for k, th in enumerate(self.thetas):
            if self._residual:
                B.as_ssm_forward_residual(self.shape, th, self.yhat, self.ys[-1], outs[k], self.yhat if k + 1 < self.K else None, self.ws,
                                          self.eps)
                self.ys.append(outs[k])
                continue
            B.as_ssm_forward_ordered(self.shape, th, self.yhat, self.ytilde, self.ws)
            yk = outs[k]
            if k + 1 < self.K:   # the next layer's input is the norm of the sum: both in one pass
                B.as_residual_add_rmsnorm(self.shape, self.ys[-1], self.ytilde, yk, self.yhat, self.eps)
            else:
                B.as_residual_add(self.shape, self.ys[-1], self.ytilde, yk)
            self.ys.append(yk)
        return self.ys[-1]

    def adjoint_grad(self, g: torch.Tensor, mode: str = "chained", record=None, batched=True):
        """Per-layer parameter gradients from the top gradient g = dL/dy_K.  Returns (list of grads, G_0 or None).
        `record`, if a dict, receives {k: (layer input, upstream gradient)} copies for the layers it has keys for.
        In "paper" mode the layers are independent and go to the library as one call (`batched=False`: layer by layer)."""
        assert self.ys is not None, "call forward() first"
        dev = g.device
        if mode == "paper" and batched:
            return self._paper_grad_batched(g, record), None
        self._pack()
        grads = [None] * self.K
        G = g.clone() if mode == "chained" else g
        for k in range(self.K - 1, -1, -1):
            B.as_rmsnorm_fwd(self.shape, self.ys[k], self.yhat, self.eps)
            if record is not None and k in record:
                record[k] = (self.yhat.clone(), G.clone())
            gk = B.alloc_grads(self.shape, dev, with_dx=(mode == "chained"))
            B.as_adjoint_grad(self.shape, self.thetas[k], self.yhat, G, self.tbar, gk, self.ws, B.AS_ORDERED)
            if mode == "chained":
                B.as_rmsnorm_bwd_add(self.shape, self.ys[k], gk["dx"], G, self.eps)
                gk["dx"] = None
            grads[k] = gk
        return grads, (G if mode == "chained" else None)

    def _paper_grad_batched(self, g: torch.Tensor, record=None):
        """Proposition 3: all K layers in one as_adjoint_grad_layers call (stacked parameters, stacked layer inputs,
        the one upstream gradient shared)."""
        K, sh = self.K, self.shape
        keys = ("W_delta", "b_delta", "W_B", "W_C", "A_log")
        if self._stacked is None:
            self._stacked = {k: torch.empty(K, *self.thetas[0][k].shape, dtype=self.thetas[0][k].dtype, device=self.device) for k in keys}
            if sh.io == B.AS_BF16:
                self._stacked["Wcat"] = torch.empty(B.as_wcat_bytes(sh, K), dtype=torch.uint8, device=self.device)
            self._ws_layers = B.alloc_workspace(B.as_workspace_bytes_layers(sh, K, self.tbar), self.device)
            self._xall = torch.empty(K, sh.batch, sh.seqlen, sh.d_model, dtype=self.yhat.dtype, device=self.device)
            self._x = self._xall.unbind(0)
        now = self._contents(self.thetas, keys)
        if not self._same(now, self._stacked_of):
            with torch.no_grad():
                for k in keys:
                    torch.stack([th[k] for th in self.thetas], out=self._stacked[k])
            if sh.io == B.AS_BF16:
                B.as_pack_weights(sh, K, self._stacked, self._stacked["Wcat"])
            self._stacked_of = now
        # norms row by row: layers whose inputs lie one behind the other (as forward() leaves y_1 .. y_{K-1}) take one launch
        step = self._x[0].numel() * self._x[0].element_size()
        at = [y.data_ptr() for y in self.ys[:K]]
        k = 0
        while k < K:
            e = k + 1
            while e < K and at[e] == at[e - 1] + step:
                e += 1
            run = B.make_shape(sh.batch * (e - k), sh.seqlen, sh.d_model, sh.d_state, sh.io)
            B.as_rmsnorm_fwd(run, self.ys[k], self._x[k], self.eps)
            k = e
        if record is not None:
            for k in record:
                if 0 <= k < K:
                    record[k] = (self._x[k].clone(), g.clone())
        gl = B.alloc_grads_layers(sh, K, g.device)
        B.as_adjoint_grad_layers(sh, K, self._stacked, self._xall, g, self.tbar, gl, self._ws_layers, B.AS_ORDERED)
        self.ws_last = self._ws_layers
        per_layer = {k: (v.unbind(0) if v is not None else [None] * K) for k, v in gl.items()}
        return [{k: v[i] for k, v in per_layer.items()} for i in range(K)]

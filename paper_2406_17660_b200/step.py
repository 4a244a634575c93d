"""Sequencing of the five library calls into the paper's Algorithm 1, per layer.

Nothing here computes: GrassLayer owns the caller-side buffers (torch device
memory) and issues grass_* calls in the order of Algorithm 1 -- every K
iterations compute_P (dense gradient -> row norms -> select, optional state
reset), then projected gradient, Adam, row-sparse apply (one grass_layer_step where
the update is fused).
"""
from __future__ import annotations

import torch

from . import binding as B


class GrassWorkspace:
    """Scratch shared by all layers of a model: sized for the largest layer.

    Holds the norms and the byte workspaces of grass_project_grad,
    grass_refresh_step and grass_select.  No m x n gradient buffer of a large layer
    exists: refresh iterations take the row norms straight from the GEMM's epilogue.
    """

    def __init__(self, shapes, T, r, dtype, method, device="cuda"):
        dt = B.BF16 if dtype == torch.bfloat16 else B.F32
        max_m = max(m for m, _ in shapes)
        proj = 256
        sel = 256
        nrm = 256
        for m, n in shapes:
            rr = min(r, m)
            proj = max(proj, B.grass_project_workspace_bytes(T, m, n, rr, dt))
            nrm = max(nrm, B.grass_refresh_workspace_bytes(T, m, n, rr, dt))
            sel = max(sel, B.grass_select_workspace_bytes(m, rr, method))
        self.norm_ws = torch.empty(nrm, dtype=torch.uint8, device=device)
        self.norms = torch.empty(max_m, dtype=torch.float32, device=device)
        self.project_ws = torch.empty(proj, dtype=torch.uint8, device=device)
        self.select_ws = torch.empty(sel, dtype=torch.uint8, device=device)


class GrassLayer:
    """State of one linear layer W (m x n) trained by GRASS with rank r."""

    def __init__(self, W, r, method, K, alpha, lr, beta1=0.9, beta2=0.999, eps=1e-8,
                 reset_state=True, seed=0, layer_id=0, workspace=None, side="rows",
                 fused_update=True, keep_U=True):
        """side = "rows": P selects r of the m output features (rows of W).
        side = "cols": P selects r of the n input features (columns of W), the paper's choice
        when m > n; the same library calls are used with dY and X exchanged, the state is
        r x m, and the apply step is the column form."""
        self.W = W
        self.side = side
        # Adam and the apply step in one kernel; keep_U=False also skips writing U
        self.fused_update = fused_update
        self.keep_U = keep_U
        self.m, self.n = W.shape if side == "rows" else (W.shape[1], W.shape[0])
        self.r, self.method, self.K = r, method, K
        self.alpha, self.lr, self.beta1, self.beta2, self.eps = alpha, lr, beta1, beta2, eps
        self.reset_state, self.seed, self.layer_id = reset_state, seed, layer_id
        dev = W.device
        self.idx = torch.zeros(r, dtype=torch.int32, device=dev)
        self.rho = torch.ones(r, dtype=torch.float32, device=dev)
        self.M = torch.zeros((r, self.n), dtype=torch.float32, device=dev)
        self.V = torch.zeros((r, self.n), dtype=torch.float32, device=dev)
        self.U = torch.empty((r, self.n), dtype=torch.float32, device=dev)
        self.Gc = torch.empty((r, self.n), dtype=torch.float32, device=dev)
        self.ws = workspace
        self.stream = None    # optional: the caller may pin a layer to a stream
        self.t = 0            # iteration counter of Algorithm 1
        self.adam_step = 0    # updates since the state was last zeroed
        self._call = None

    def refresh(self, dY, X):
        """compute_P from this iteration's gradient (Algorithm 1, every K iterations)."""
        ws = self.ws
        norms = ws.norms[: self.m]
        B.grass_grad_row_norms(dY, X, norms, ws.norm_ws)
        B.grass_select(norms, self.r, self.method, self.seed, self.layer_id, self.t // self.K,
                       self.idx, self.rho, ws.select_ws)
        if self.reset_state:
            self.M.zero_()
            self.V.zero_()
            self.adam_step = 0

    def _own_refresh(self):
        """Whether a program has put its own in the place of refresh(): then it is that which is called."""
        return type(self).refresh is not GrassLayer.refresh or "refresh" in self.__dict__

    def _refresh_step(self, dY, X, of, step):
        """A refresh iteration in one call, with the hyper-parameters of layer `of`."""
        ws, call = self.ws, self._call
        if call is None:
            call = self._call = B.LayerStepCall()
        call.state(0, self.idx, self.rho, self.Gc, self.M, self.V, self.U if self.keep_U else None,
                   self.W, self.side == "cols")
        call.inputs(0, dY, X)
        call.refresh(ws.project_ws, of.lr, of.beta1, of.beta2, of.eps, step, of.alpha,
                     self.method, self.seed, self.layer_id, self.t // self.K,
                     self.reset_state, ws.norms, ws.norm_ws, ws.select_ws)

    def step(self, dY, X):
        """One iteration of Algorithm 1 for this layer; dY (T x m), X (T x n) on the device."""
        if self.side == "cols":
            dY, X = X, dY        # select columns of X, contract with dY: G_C^T = P^T (X^T dY)
        refresh = self.t % self.K == 0
        if self.fused_update and not (refresh and self._own_refresh()):
            step = 1 if refresh and self.reset_state else self.adam_step + 1
            if refresh:
                self._refresh_step(dY, X, self, step)
            else:
                call = self._call
                if call is None:
                    call = self._call = B.LayerStepCall()
                call.state(0, self.idx, self.rho, self.Gc, self.M, self.V, self.U if self.keep_U else None,
                           self.W, self.side == "cols")
                call.inputs(0, dY, X)
                call.launch(1, self.ws.project_ws, self.lr, self.beta1, self.beta2, self.eps, step, self.alpha)
            self.adam_step = step              # (a call that was refused has changed nothing)
            self.t += 1
            return
        if refresh:
            self.refresh(dY, X)
        self.adam_step += 1
        B.grass_project_grad(dY, X, self.idx, self.rho, self.r, self.Gc, self.ws.project_ws)
        B.grass_subspace_adam(self.Gc, self.M, self.V, self.U, self.lr, self.beta1, self.beta2,
                              self.eps, self.adam_step)
        if self.side == "cols":
            B.grass_scatter_update_cols(self.W, self.U, self.idx, self.rho, self.alpha)
        else:
            B.grass_scatter_update(self.W, self.U, self.idx, self.rho, self.alpha)
        self.t += 1


class GrassLayerGroup:
    """Up to 8 layers of one shape (row selection, bf16) stepped together: their projections
    run as one set of launches and so do their Adam + apply updates.  The layers keep their
    own selection, state and weights; rows are re-selected layer by layer.  The iteration, lr, betas,
    eps, alpha and the step count of Adam are those of layer 0, on every iteration."""

    def __init__(self, layers, T, device="cuda"):
        if not 1 <= len(layers) <= 8:
            raise ValueError("a group holds 1 to 8 layers")
        first = layers[0]
        for l in layers:
            if (l.W.shape, l.r, l.K, l.side) != (first.W.shape, first.r, first.K, "rows"):
                raise ValueError("layers of a group must share shape, r, K and select rows")
        self.layers = layers
        nbytes = B.grass_project_batched_workspace_bytes(len(layers), T, first.m, first.n, first.r)
        self.ws = torch.empty(nbytes, dtype=torch.uint8, device=device)
        self.stream = None
        self._call = B.LayerStepCall()
        self._marshal()                     # layers that do not go together are refused here

    def _marshal(self):
        """The buffers that the layers have now: a layer may have been given others since the last step."""
        state = self._call.state
        for g, l in enumerate(self.layers):
            state(g, l.idx, l.rho, l.Gc, l.M, l.V, l.U if l.keep_U else None, l.W)

    def step(self, dYs, Xs):
        ls = self.layers
        first = ls[0]
        self._marshal()
        inputs = self._call.inputs
        for g in range(len(ls)):
            inputs(g, dYs[g], Xs[g])
        refresh, kept = first.t % first.K == 0, False
        if refresh:
            # the dense gradient that the norms need may already hold the selected rows
            kept = all(l.fused_update and not l._own_refresh() for l in ls) and B.grass_refresh_keeps_gradient(
                dYs[0].shape[0], first.m, first.n, first.r, B.BF16)
            if not kept:
                for l, dY, X in zip(ls, dYs, Xs):
                    l.refresh(dY, X)
        step = 1 if kept and first.reset_state else first.adam_step + 1
        if kept:
            for l, dY, X in zip(ls, dYs, Xs):
                l._refresh_step(dY, X, first, step)
        elif refresh and dYs[0].dtype == torch.bfloat16:
            # with the token slices, hence the bits, of the projection calls: after a reset they decide signs
            idxs, rhos, Gcs = [l.idx for l in ls], [l.rho for l in ls], [l.Gc for l in ls]
            B.grass_project_grad_batched(dYs, Xs, idxs, rhos, first.r, Gcs, self.ws)
            B.grass_adam_scatter_batched(Gcs, [l.M for l in ls], [l.V for l in ls],
                                         [l.U if l.keep_U else None for l in ls], [l.W for l in ls], idxs, rhos,
                                         first.lr, first.beta1, first.beta2, first.eps, step, first.alpha)
        else:
            self._call.launch(len(ls), self.ws, first.lr, first.beta1, first.beta2, first.eps, step, first.alpha)
        for l in ls:
            l.adam_step = 1 if kept and l.reset_state else l.adam_step + 1
            l.t += 1

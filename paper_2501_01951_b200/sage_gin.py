"""Buffer plumbing for the two other architectures the paper's evaluation names (Section 5, "The Model
and Datasets"): mean-aggregator GraphSAGE and GIN, full-graph training.  The paper does not define
them; the layers are their textbook forms, built from the same C-ABI steps as the GCN layer:

  GraphSAGE (mean):  H' = sigma([H | M H] [W_self; W_neigh] + b),  M = D^-1 A on a graph made with
                     GRAPH_NORM_ROW (no self loops);
  GIN:               H' = sigma(relu(((1 + eps) H + A H) W1 + b1) W2 + b2),  A on a graph made with
                     GRAPH_NORM_NONE (no self loops); the (1 + eps) H term is the aggregation
                     epilogue's residual.

As in ``train.py`` nothing is computed here: every value comes out of a kernel of ``libmixgcn.so``
(``spmm``, ``gemm``, ``weight_grad``, ``colsum``, ``loss_softmax_xent``, ``adam_step``).

Both aggregations are linear and stand before a product, so each layer picks the side of the product it aggregates on, by
the width it costs, as the GCN layers do: M H W_neigh = M (H W_neigh) and ((1 + eps) H + A H) W1 = (1 + eps) U + A U with
U = H W1.  A layer from 256 to 47 columns then gathers 47 instead of 256 in both directions.
"""
from __future__ import annotations

import torch

from . import binding as mg


def round4(x: int) -> int:
    return (x + 3) // 4 * 4


def update_first(d_in: int, d_out: int, first: bool, precision: int, relu: bool) -> bool:
    """Whether aggregating after the product (at width d_out, forward and backward) is cheaper than before it (at width
    d_in, forward and -- unless the layer is the first -- backward); ties aggregate first.  A product that rounds its operands
    rounds others on the other side of the aggregation: where a ReLU follows, signs near zero would change with them (GIN in
    bf16, whose sums grow with the degree: 1.4e-2 -> 5e-2 against fp32), so those layers keep the defining order."""
    if relu and precision != mg.PREC_FP32:
        return False
    return 2 * d_out < (1 if first else 2) * d_in


def product_precision(precision: int, relu: bool) -> int:
    """Precision of an update-first product: where a ReLU is taken of what the aggregation makes of it, fp32 sums keep the one
    order that GCN layers keep under a ReLU, and signs near zero with it."""
    return mg.PREC_FP32_FMA if relu and precision == mg.PREC_FP32 else precision


class _Base:
    def __init__(self, ctx, graph, dims, precision):
        self.ctx, self.g, self.precision = ctx, graph, precision
        self.tiles = precision != mg.PREC_FP32      # as in train.py
        self.dims = tuple(int(d) for d in dims)
        self.L = len(self.dims) - 1
        self.n = graph.n
        self.device = torch.device("cuda", ctx.device)
        self.ld = [round4(d) for d in self.dims]
        self.loss = torch.zeros(1, dtype=torch.float32, device=self.device)
        self.pred = torch.zeros(self.n, dtype=torch.int32, device=self.device)
        self.n_correct = torch.zeros(1, dtype=torch.int64, device=self.device)
        self.params, self.grads, self.m, self.v = [], [], [], []
        self._replay = mg.Replayer(ctx)      # the calls of an iteration, recorded once they have come twice with the same buffers

    def _layout_tiles(self, widths):
        if self.tiles:
            mg.graph_layout_tiles(self.g, widths, self.ctx)

    def _spmm(self, *args, **kwargs):
        mg.spmm(self.ctx, self.g, *args, tiles=self.tiles, **kwargs)

    def _z(self, r, c):
        return torch.zeros((r, c), dtype=torch.float32, device=self.device)

    def _bits(self, d):
        return torch.zeros((self.n, (d + 31) // 32), dtype=torch.int32, device=self.device)

    def _set_params(self, tensors):
        self.params = [t.to(self.device, torch.float32).contiguous().clone() for t in tensors]
        self.grads = [torch.zeros_like(t) for t in self.params]
        self.m = [torch.zeros_like(t) for t in self.params]
        self.v = [torch.zeros_like(t) for t in self.params]

    def compute_loss(self):
        mg.loss_softmax_xent(self.ctx, self.logits, self.labels, self.train_mask, self.loss, dlogits=self.logits,
                             pred=self.pred, n_correct=self.n_correct, C_=self.dims[-1])

    def step(self, t, lr=0.01, beta1=0.9, beta2=0.999, eps=1e-8):
        mg.adam_step(self.ctx, self.params, self.grads, self.m, self.v, t, lr, beta1, beta2, eps)

    def _calls_key(self):
        """Everything the issued calls depend on: every tensor the trainer holds, and the context's options."""
        held = []
        for v in self.__dict__.values():
            for t in v if isinstance(v, list) else (v,):
                held.append(t.data_ptr() if isinstance(t, torch.Tensor) else 0)
        return tuple(held), self.precision, self.g.h.value, self.ctx.h.value, tuple(self.ctx.options.items()), getattr(self, "gin_eps", None)

    def _iteration(self):
        self.forward()
        self.compute_loss()
        self.backward()

    def epoch(self, t, lr=0.01):
        self._replay.run(self._calls_key, self._iteration)
        self.step(t, lr)


class SageTrainer(_Base):
    """Mean-aggregator GraphSAGE.  ``graph`` must carry row-mean values (GRAPH_NORM_ROW, no self loops).
    A layer that aggregates first keeps S_l = [H_l | M H_l] (n x 2 ld_l): the left half is written by the layer below (or is
    the input), the right half by the aggregation, and one product with W_l = [W_self; W_neigh] (2 d_l x d_{l+1}) does the
    update.  A layer that updates first keeps S_l = H_l; one product with [W_self | W_neigh] gives both terms side by side,
    and the aggregation of the second adds the first as its residual."""

    def __init__(self, ctx, graph, dims, precision=mg.PREC_FP32):
        super().__init__(ctx, graph, dims, precision)
        n, L, ld = self.n, self.L, self.ld
        self.upd = [update_first(self.dims[l], self.dims[l + 1], l == 0, precision, l < L - 1) for l in range(L)]
        self._layout_tiles([self.dims[l + 1] if self.upd[l] else self.dims[l] for l in range(L)])
        self.S = [self._z(n, ld[l] if self.upd[l] else 2 * ld[l]) for l in range(L)]
        # gradients w.r.t. the layers' outputs: [G | M^T G] where the layer updates first, G otherwise; the hidden ones take
        # turns in two buffers, which the forward pass uses for the update-first products
        self.wide = [2 * ld[l + 1] if self.upd[l] else ld[l + 1] for l in range(L)]
        pool_w = max([self.wide[l] for l in range(L) if l < L - 1 or self.upd[l]] + [4])
        self.pool = [self._z(n, pool_w), self._z(n, pool_w if L >= 3 else 4)]
        self.G = [self.pool[l % 2 if L >= 3 else 0].view(-1)[: n * self.wide[l]].view(n, self.wide[l]) for l in range(L - 1)]
        self.G.append(self._z(n, self.wide[L - 1]))
        self.logits = self.G[L - 1][:, : ld[L]]
        agg_hidden = [2 * ld[l] for l in range(1, L) if not self.upd[l]]
        self.dS = self._z(n, max(agg_hidden)) if agg_hidden else None        # gradient w.r.t. [H_l | M H_l]
        # update-first layers: [W_self | W_neigh], its gradient and the column sums of [G | M^T G]
        self.Wc = [self._z(self.dims[l], self.wide[l]) if self.upd[l] else None for l in range(L)]
        self.dWc = [self._z(self.dims[l], self.wide[l]) if self.upd[l] else None for l in range(L)]
        self.dbc = [torch.zeros(self.wide[l], dtype=torch.float32, device=self.device) if self.upd[l] else None for l in range(L)]
        # signs of the hidden activations that a product writes (one bit per element), read by the backward gates
        self.signs = [None] + [None if self.upd[l - 1] else self._bits(self.dims[l]) for l in range(1, L)]

    def set_params(self, Ws_self, Ws_neigh, bs):
        """Parameter order: W_cat[0..L) (rows [W_self; W_neigh]), b[0..L)."""
        cats = []
        for l in range(self.L):
            W = torch.zeros(2 * self.ld[l], self.dims[l + 1])
            W[: self.dims[l]] = Ws_self[l]
            W[self.ld[l]: self.ld[l] + self.dims[l]] = Ws_neigh[l]
            cats.append(W)
        self._set_params(cats + list(bs))

    def set_inputs(self, X0, labels, train_mask):
        """X0: n x ld[0] device tensor (pads zero); it is copied once into the left half of S_0."""
        self.S[0][:, : self.ld[0]].copy_(X0)
        self.labels, self.train_mask = labels, train_mask

    def _halves(self, l, stacked, beside):
        """Pairs of the two d_l x d_{l+1} blocks in the stacked ([self; neigh]) and the side-by-side ([self | neigh]) layout."""
        d, ld, dout, do4 = self.dims[l], self.ld[l], self.dims[l + 1], self.ld[l + 1]
        return ((stacked[:d], beside[:, :dout]), (stacked[ld: ld + d], beside[:, do4: do4 + dout]))

    def forward(self):
        L, ld = self.L, self.ld
        for l in range(L):
            S, d, dout, do4 = self.S[l], ld[l], self.dims[l + 1], ld[l + 1]
            last = l == L - 1
            out = self.logits if last else self.S[l + 1][:, : do4]
            bias, relu = self.params[L + l], not last
            if self.upd[l]:
                for stacked, beside in self._halves(l, self.params[l], self.Wc[l]):
                    beside.copy_(stacked)
                P = self.pool[0].view(-1)[: self.n * self.wide[l]].view(self.n, self.wide[l])
                mg.gemm(self.ctx, product_precision(self.precision, relu), False, False, self.n, self.wide[l], self.dims[l], S, self.Wc[l], P)
                self._spmm(P[:, do4:], out, dout, epi=mg.make_epilogue(residual=P[:, :do4], residual_scale=1.0, bias=bias, relu=relu))
            else:
                self._spmm(S[:, :d], S[:, d:], self.dims[l])
                mg.gemm(self.ctx, self.precision, False, False, self.n, dout, 2 * d, S, self.params[l], out,
                        epi=mg.make_epilogue(bias=bias, relu=relu, sign_bits=None if last else self.signs[l + 1]))

    def backward(self):
        L, ld = self.L, self.ld
        for l in range(L - 1, -1, -1):
            d, dout, do4 = ld[l], self.dims[l + 1], ld[l + 1]
            Gc = self.G[l]                                      # gradient w.r.t. the layer's pre-activation, left half
            G = Gc[:, :do4]
            if l > 0:
                Gn = self.G[l - 1][:, :d]
                gate = dict(gate_bits=self.signs[l]) if self.signs[l] is not None else dict(gate=self.S[l][:, :d])
            if self.upd[l]:
                self._spmm(G, Gc[:, do4:], dout, transposed=True)
                mg.weight_grad(self.ctx, self.precision, self.dims[l], self.wide[l], self.n, self.S[l], Gc, self.dWc[l], self.dbc[l])
                for stacked, beside in self._halves(l, self.grads[l], self.dWc[l]):
                    stacked.copy_(beside)
                self.grads[L + l].copy_(self.dbc[l][:dout])
                if l > 0:
                    mg.gemm(self.ctx, self.precision, False, True, self.n, self.dims[l], self.wide[l], Gc, self.Wc[l], Gn, epi=mg.make_epilogue(gate_scale=1.0, **gate))
                continue
            mg.weight_grad(self.ctx, self.precision, 2 * d, dout, self.n, self.S[l], G, self.grads[l], self.grads[L + l])
            if l > 0:
                dS = self.dS.view(-1)[: self.n * 2 * d].view(self.n, 2 * d)
                mg.gemm(self.ctx, self.precision, False, True, self.n, 2 * d, dout, G, self.params[l], dS)
                # G_in = relu'(H_l) * (dS_left + M^T dS_right): residual and gate in the aggregation's epilogue
                self._spmm(dS[:, d:], Gn, self.dims[l], transposed=True,
                        epi=mg.make_epilogue(residual=dS[:, :d], residual_scale=1.0, gate_scale=1.0, **gate))


class GinTrainer(_Base):
    """GIN with a two-layer perceptron per layer.  ``graph`` must carry unit values (GRAPH_NORM_NONE, no
    self loops); ``gin_eps`` is the constant eps of the (1 + eps) self term."""

    def __init__(self, ctx, graph, dims, hidden, precision=mg.PREC_FP32, gin_eps=0.0):
        super().__init__(ctx, graph, dims, precision)
        n, L, ld = self.n, self.L, self.ld
        self.hidden, self.ldh, self.gin_eps = int(hidden), round4(hidden), float(gin_eps)
        self.upd = [update_first(self.dims[l], self.hidden, l == 0, precision, True) for l in range(L)]
        self._layout_tiles([self.hidden if self.upd[l] else self.dims[l] for l in range(L)])
        self.H = [None] + [self._z(n, ld[l]) for l in range(1, L)]
        # aggregate-first layers keep (1 + eps) H + A H for their weight gradient; update-first ones share scratch for H W1
        # and its gradient
        self.Z = [None if self.upd[l] else self._z(n, ld[l]) for l in range(L)]
        self.U = self._z(n, self.ldh) if any(self.upd) else None
        self.T = [self._z(n, self.ldh) for l in range(L)]
        self.logits = self._z(n, ld[L])
        wmax = max(ld[1:L]) if L >= 2 else 4
        self.dT, self.dZ = self._z(n, self.ldh), self._z(n, wmax)
        self.Ga, self.Gb = self._z(n, wmax), self._z(n, wmax)
        # signs of the activations that a product writes (one bit per element), read by the backward gates
        self.signs_H = [None] + [self._bits(self.dims[l]) for l in range(1, L)]
        self.signs_T = [None if self.upd[l] else self._bits(self.hidden) for l in range(L)]

    def set_params(self, W1s, b1s, W2s, b2s):
        """Parameter order: W1[0..L), b1[0..L), W2[0..L), b2[0..L)."""
        self._set_params(list(W1s) + list(b1s) + list(W2s) + list(b2s))

    def set_inputs(self, X0, labels, train_mask):
        self.H[0], self.labels, self.train_mask = X0, labels, train_mask

    def forward(self):
        L, h, keep = self.L, self.hidden, 1.0 + self.gin_eps
        for l in range(L):
            H, d = self.H[l], self.dims[l]
            if self.upd[l]:
                mg.gemm(self.ctx, product_precision(self.precision, True), False, False, self.n, h, d, H, self.params[l], self.U)
                self._spmm(self.U, self.T[l], h, epi=mg.make_epilogue(residual=self.U, residual_scale=keep, bias=self.params[L + l], relu=True))
            else:
                self._spmm(H, self.Z[l], d, epi=mg.make_epilogue(residual=H, residual_scale=keep))
                mg.gemm(self.ctx, self.precision, False, False, self.n, h, d, self.Z[l], self.params[l], self.T[l],
                        epi=mg.make_epilogue(bias=self.params[L + l], relu=True, sign_bits=self.signs_T[l]))
            last = l == L - 1
            out = self.logits if last else self.H[l + 1]
            mg.gemm(self.ctx, self.precision, False, False, self.n, self.dims[l + 1], h, self.T[l], self.params[2 * L + l], out,
                    epi=mg.make_epilogue(bias=self.params[3 * L + l], relu=not last, sign_bits=None if last else self.signs_H[l + 1]))

    def backward(self):
        L, h, keep = self.L, self.hidden, 1.0 + self.gin_eps
        G = self.logits
        for l in range(L - 1, -1, -1):
            d, dout = self.dims[l], self.dims[l + 1]
            mg.weight_grad(self.ctx, self.precision, h, dout, self.n, self.T[l], G, self.grads[2 * L + l], self.grads[3 * L + l])
            # dT = relu'(T) * (dP W2^T)
            gate = dict(gate_bits=self.signs_T[l]) if self.signs_T[l] is not None else dict(gate=self.T[l])
            mg.gemm(self.ctx, self.precision, False, True, self.n, h, dout, G, self.params[2 * L + l], self.dT, epi=mg.make_epilogue(gate_scale=1.0, **gate))
            if l > 0:
                Gn = (self.Ga if (L - 1 - l) % 2 == 0 else self.Gb).view(-1)[: self.n * self.ld[l]].view(self.n, self.ld[l])   # the two buffers alternate
            if self.upd[l]:
                mg.colsum(self.ctx, self.dT, self.grads[L + l], h)
                self._spmm(self.dT, self.U, h, transposed=True, epi=mg.make_epilogue(residual=self.dT, residual_scale=keep))
                mg.weight_grad(self.ctx, self.precision, d, h, self.n, self.H[l], self.U, self.grads[l])
                if l > 0:
                    mg.gemm(self.ctx, self.precision, False, True, self.n, d, h, self.U, self.params[l], Gn, epi=mg.make_epilogue(gate_bits=self.signs_H[l], gate_scale=1.0))
                    G = Gn
                continue
            mg.weight_grad(self.ctx, self.precision, d, h, self.n, self.Z[l], self.dT, self.grads[l], self.grads[L + l])
            if l > 0:
                dZ = self.dZ.view(-1)[: self.n * self.ld[l]].view(self.n, self.ld[l])
                mg.gemm(self.ctx, self.precision, False, True, self.n, d, h, self.dT, self.params[l], dZ)
                # G_in = relu'(H_l) * ((1 + eps) dZ + A^T dZ)
                self._spmm(dZ, Gn, d, transposed=True,
                        epi=mg.make_epilogue(residual=dZ, residual_scale=keep, gate_bits=self.signs_H[l], gate_scale=1.0))
                G = Gn

"""torch.autograd.Function wrappers whose backward is the library's hand-written
force vector-Jacobian product (the double backward of the energy).

    E, F = NNPFunction.apply(coords, weights, potential, species, box, mask)
    loss = ((F - F_target) ** 2).sum()
    loss.backward()        # coords.grad and weights.grad from nnp_force_vjp

`weights` is the flat parameter vector the potential was created with (the
library holds its own device copy; the tensor carries the gradient).
"""
from __future__ import annotations

import operator

import torch


class NNPFunction(torch.autograd.Function):
    @staticmethod
    def forward(ctx, coords, weights, potential, species, box=None, mask=None):
        E, F = potential.energy_forces(coords.detach().contiguous(), species, box, mask)
        ctx.set_materialize_grads(False)   # an unused output's gradient stays None
        ctx.potential, ctx.species, ctx.box, ctx.mask = potential, species, box, mask
        ctx.save_for_backward(coords)
        return E, F

    @staticmethod
    def backward(ctx, gE, gF):
        (coords,) = ctx.saved_tensors
        pot = ctx.potential
        gE = 0.0 if gE is None else float(gE.reshape(-1)[0])
        gF = torch.zeros_like(coords) if gF is None else gF
        sys = {"coords": coords.detach().contiguous(), "species": ctx.species, "box": ctx.box,
               "mask": ctx.mask}
        _, _, G, W = pot.force_vjp_batch([sys], [gE], [gF])
        return G[0], W, None, None, None, None


class NNPBatchFunction(torch.autograd.Function):
    """Batch of independent systems concatenated along the atom axis.
    sizes: atoms per system.  Returns energies [n_sys] and forces [sum(sizes), 3]."""

    @staticmethod
    def forward(ctx, coords, weights, potential, species, sizes, boxes=None):
        x, sp = coords.detach().contiguous(), species.contiguous()
        if isinstance(sizes, int):   # systems of one size, as torch.split takes it
            sizes = [len(t) for t in torch.split(sp, sizes)]
        if not isinstance(sizes, (list, tuple)):
            raise TypeError(f"sizes: an int or a list of ints, not {type(sizes).__name__}")
        sizes = [operator.index(n) for n in sizes]
        E, F = potential.energy_forces_flat(x, sp, sizes, boxes)
        ctx.set_materialize_grads(False)   # an unused output's gradient stays None
        ctx.potential, ctx.x, ctx.sp, ctx.sizes, ctx.boxes = potential, x, sp, sizes, boxes
        return E, F

    @staticmethod
    def backward(ctx, gE, gF):
        n = len(ctx.sizes)
        gEs = [0.0] * n if gE is None else gE.detach().double().cpu().tolist()
        gFs = torch.zeros_like(ctx.x) if gF is None else gF.detach().float().contiguous()
        G, W = ctx.potential.force_vjp_flat(ctx.x, ctx.sp, ctx.sizes, ctx.boxes, gEs, gFs)
        return G, W, None, None, None, None

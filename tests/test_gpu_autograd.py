"""GBEnergy's backward: weights per replica reach that replica's atoms, with
one replica and with several (an empty one among them), and the gradient is
itself differentiable in the weights."""
import numpy as np
import pytest

import synth
from gpu_common import device, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[130], [1], [100, 0, 77]])
def test_weighted_gradient(sizes):
    import torch

    import paper_1803_09652_gb300 as pkg
    b = synth.random_batch(sizes, seed=8, sites=False)
    xyzq, rad = to_dev(b, device())
    ctx = pkg.Context(b.atom_off)
    out = ctx.energy_forces(xyzq, rad)
    w = torch.linspace(0.5, 2.0, len(sizes), dtype=torch.float64, device=xyzq.device).requires_grad_(True)
    x = xyzq.clone().requires_grad_(True)
    g, = torch.autograd.grad((pkg.GBEnergy.apply(ctx, x, rad) * w).sum(), x, create_graph=True)
    wa = w.detach().repeat_interleave(torch.as_tensor(np.diff(b.atom_off), device=x.device))
    assert torch.equal(g.detach()[:, :3], (-out["F"].double() * wa[:, None]).float())
    assert torch.equal(g.detach()[:, 3], (out["dEdq"] * wa).float())
    dw, = torch.autograd.grad(g.double().square().sum(), w)
    one = (out["F"].double().square().sum(1) + out["dEdq"].square())
    off = b.atom_off
    ref = torch.stack([2 * w.detach()[r] * one[off[r]:off[r + 1]].sum() for r in range(len(sizes))])
    assert torch.allclose(dw, ref, rtol=1e-6)

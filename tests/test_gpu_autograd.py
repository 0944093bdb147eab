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


def test_backward_on_another_stream_keeps_the_atom_counts():
    """The context's atom counts live in the memory of the stream that first
    asked for them.  A backward pass enqueued on another stream still reads them
    after the context and the graph are gone: the first stream may not be given
    their memory before that work is done."""
    import torch

    import paper_1803_09652_gb300 as pkg
    b = synth.random_batch([100, 0, 77], seed=9, sites=False)
    xyzq, rad = to_dev(b, device())
    x = xyzq.clone().requires_grad_(True)
    ctx = pkg.Context(b.atom_off)
    ref, = torch.autograd.grad(pkg.GBEnergy.apply(ctx, x, rad).sum(), x)
    address = ctx.atom_counts(x.device).data_ptr()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        energy = pkg.GBEnergy.apply(ctx, x, rad).sum()
    del ctx                                    # waits for the device, then drops its counts
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)         # a fifth of a second before the backward pass
        grad, = torch.autograd.grad(energy, x)
    del energy
    fresh = [torch.empty(3, dtype=torch.int64, device=x.device) for _ in range(64)]
    busy = not side.query()
    assert address not in [t.data_ptr() for t in fresh]
    side.synchronize()
    assert busy and torch.equal(grad, ref)

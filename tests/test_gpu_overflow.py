"""Finite coordinates so far apart that the square of a distance overflows (only
a run that has blown up has them) are reported as non-finite, without and with
cutoffs, and the context evaluates valid input afterwards."""
import numpy as np
import pytest

import synth
from gpu_common import device, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1803_09652_gb300 as p
    return p


@pytest.mark.parametrize("cut", [{}, dict(rgbmax=12.0, cut=12.0), dict(rgbmax=12.0), dict(cut=12.0)])
@pytest.mark.parametrize("n,atom", [(33, 32), (96, 5), (96, 70), (300, 170), (1300, 700), (6500, 3201)])
def test_overflowing_distances_are_reported(pkg, n, atom, cut):
    import torch
    rep = synth.make_replica(n, 7, [])
    b = synth.Batch([rep], pH=np.zeros(1), E=np.zeros(1))
    xyzq, rad = to_dev(b, device())
    ctx = pkg.Context(b.atom_off, pkg.default_params(**cut))
    good = ctx.energy_forces(xyzq, rad, want=("R", "F"))
    ctx.sync_status()
    far = xyzq.clone()
    far[atom, 0] = 3.0e19
    for call in (lambda: ctx.born_radii(far, rad), lambda: ctx.energy_forces(far, rad, want=("R", "F")),
                 lambda: ctx.energy_forces(far, rad)):
        call()
        with pytest.raises(RuntimeError, match="NONFINITE"):
            ctx.sync_status()
    again = ctx.energy_forces(xyzq, rad, want=("R", "F"))
    ctx.sync_status()
    for k in good:
        assert torch.equal(again[k], good[k])


@pytest.mark.parametrize("n,atom", [(96, 70), (1300, 700)])
def test_far_coordinates_that_do_not_overflow_are_taken(pkg, n, atom):
    import torch
    rep = synth.make_replica(n, 7, [])
    rep.xyz[atom, 0] = 4.0e18
    xyzq, rad = to_dev(synth.Batch([rep], pH=np.zeros(1), E=np.zeros(1)), device())
    ctx = pkg.Context([0, n])
    out = ctx.energy_forces(xyzq, rad)
    ctx.sync_status()
    a = np.float32(rep.rho[atom]) - np.float32(0.09)
    assert out["R"][atom].item() == pytest.approx(float(a), rel=1e-7)      # no neighbour descreens it
    assert torch.all(out["F"][atom] == 0)

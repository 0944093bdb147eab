"""Finite coordinates so far apart that the square of a distance overflows: an
atom whose neighbours in the same 64 x 32 block are that far is reported as
non-finite (distances of 1e19 A and more only come from a run that has blown
up), without and with cutoffs, and the context evaluates valid input
afterwards."""
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

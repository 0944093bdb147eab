"""Blocks that straddle the Born-radius cutoff: pairs wholly inside it, pairs
whose sphere may cross it, close pairs and pairs past its reach, on full and
on diagonal tiles with ragged ends, with the cutoff from below every screened
radius (all pairs in reach are evaluated exactly) to past most of the
molecule, against the FP64 oracle.  The bars are those of the cutoff tests."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import F_ABS, device, f32, oracle_params, to_dev
from test_gpu_cutoff import born_bar

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1803_09652_gb300 as p
    return p


@pytest.mark.parametrize("rgbmax", [0.5, 1.9, 2.6, 5.0, 9.0, 14.0, 22.0])
def test_radii_and_forces_about_the_cutoff(pkg, rgbmax):
    import torch
    b = synth.random_batch([400, 129, 97, 65, 33, 32, 1], seed=83, sites=False)
    xyzq, rad = to_dev(b, device())
    ctx = pkg.Context(b.atom_off, pkg.default_params(rgbmax=rgbmax))
    out = ctx.energy_forces(xyzq, rad, want=("R", "F"))
    torch.cuda.synchronize()
    ctx.sync_status()
    p = oracle_params(rgbmax=f32(rgbmax))
    ref = oracle.batch_energy_forces(b, p)
    R, F = out["R"].cpu().numpy(), out["F"].cpu().numpy()
    assert np.all(np.abs(R - ref["R"]) <= born_bar(b, p) * ref["R"])
    assert np.abs(F - ref["F"]).max() <= F_ABS
    ctx.close()

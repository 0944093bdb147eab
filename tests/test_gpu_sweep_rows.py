"""Site rows and sweeps at the sizes where their work is cut differently:
numbers of site atoms around a warp's 32 and around the eight groups whose
slices two warps share, up to the limit of 1024, chains around a 256-atom
slice, and two sites that share atoms.  Against the oracle's sweep, with the
bars of test_gpu_sweep."""
import numpy as np
import pytest

import synth
from test_gpu_sweep import _sweep_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1803_09652_gb300 as p
    return p


@pytest.mark.parametrize("n,sizes", [
    (40, [1]), (255, [31]), (256, [32]), (257, [20, 13]), (300, [16] * 16), (520, [16] * 15 + [17]),
    (513, [128, 128, 33]), (1100, [16] * 64)])
def test_rows_at_group_and_slice_edges(pkg, n, sizes):
    rep = synth.make_replica(n, 200 + n, [(0, k, 3) for k in sizes])
    b = synth.Batch([rep], pH=np.array([4.6]), E=np.array([synth.E0_REF_V]))
    _sweep_case(pkg, b, 1)


def test_sites_that_share_atoms(pkg):
    """The second site holds four atoms of the first: an accepted move of one
    changes the charges the other starts from."""
    rep = synth.make_replica(120, 7, [(0, 10, 3), (0, 12, 4), (0, 9, 2)])
    first, second = rep.sites[0], rep.sites[1]
    second.atoms = np.concatenate([first.atoms[:4], second.atoms[4:]]).astype(np.int32)
    second.q_state[0, :4] = first.q_state[0, :4]
    b = synth.Batch([rep], pH=np.array([4.6]), E=np.array([synth.E0_REF_V]))
    accepted, _ = _sweep_case(pkg, b, 12)
    assert accepted > 3

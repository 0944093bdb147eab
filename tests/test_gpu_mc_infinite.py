"""Monte Carlo rows with an infinite term (a site atom at another atom's
position): the change of energy is the infinity that plain FP64 sums give, a
move of minus infinity is taken and one of plus infinity (or NaN) is not, for
single attempts and sweeps, and an accepted move's infinity reaches the rows of the
sites after it."""
import numpy as np
import pytest

import synth
from gpu_common import KT, device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1803_09652_gb300 as p
    return p


def _call(pkg, b, sweep):
    import torch
    dev = device()
    t = b.site_tables()
    ctx = pkg.Context(b.atom_off)
    xyzq = torch.as_tensor(b.xyzq(), device=dev)
    R = torch.full((b.n_atoms,), 2.0, device=dev)
    state = torch.zeros(t["n_sites"], dtype=torch.int32, device=dev)
    pH, E = torch.as_tensor(b.pH, device=dev), torch.as_tensor(b.E, device=dev)
    dG, acc = (ctx.mc_sweep if sweep else ctx.mc_step)(pkg.SiteTables(t, b.n_rep, dev), xyzq, R, pH, E, KT, 3, 0, 0, state)
    ctx.sync_status()
    return dG.cpu().numpy(), acc.cpu().numpy(), state.cpu().numpy(), xyzq[:, 3].cpu().numpy()


def _site_charges(site, q, dq):
    """State 0 has the charges q; state 1 differs at the site's first atom alone."""
    site.q_state[:] = q
    site.q_state[1, 0] += dq


@pytest.mark.parametrize("sweep", [False, True])
@pytest.mark.parametrize("n,other", [(40, 1), (300, 1), (300, 299), (700, 450)])
def test_site_atom_on_another_atom(pkg, n, other, sweep):
    reps, want = [], []
    for dq, q_other in ((0.25, 0.5), (0.25, -0.5), (-0.25, 0.5), (-0.25, -0.5)):
        rep = synth.make_replica(n, 17, [(0, 6, 2)])
        a = int(rep.sites[0].atoms[0])
        j = (int(rep.sites[0].atoms[-1]) + other) % n
        rep.xyz[j], rep.q[j] = rep.xyz[a], q_other
        _site_charges(rep.sites[0], rep.q[rep.sites[0].atoms], dq)
        reps.append(rep)
        # an atom of the site itself: its unchanged charge meets the infinite site-site term, 0 * inf
        want.append(np.nan if j in rep.sites[0].atoms else np.inf * dq * q_other)
    dG, acc, state, q = _call(pkg, synth.Batch(reps, pH=np.full(4, 4.6), E=np.zeros(4)), sweep)
    want = np.array(want)
    assert np.array_equal(dG, want, equal_nan=True)
    assert np.array_equal(acc, want < 0) and np.array_equal(state, want < 0)
    for r, rep in enumerate(reps):
        atoms = rep.sites[0].atoms
        assert np.array_equal(q[r * n + atoms], rep.sites[0].q_state[int(want[r] < 0)])


def test_accepted_move_reaches_the_next_site(pkg):
    """Two sites share a position; their charges grow apart in both moves, so
    that both are taken in either order."""
    rep = synth.make_replica(90, 18, [(0, 5, 2), (0, 7, 2)])
    first, second = rep.sites
    rep.xyz[second.atoms[0]] = rep.xyz[first.atoms[0]]
    rep.q[first.atoms[0]], rep.q[second.atoms[0]] = 0.25, -0.25
    _site_charges(first, rep.q[first.atoms], 0.125)
    _site_charges(second, rep.q[second.atoms], -0.125)
    dG, acc, state, _ = _call(pkg, synth.Batch([rep], pH=np.array([4.6]), E=np.zeros(1)), True)
    assert np.all(dG == -np.inf) and np.all(acc == 1) and np.all(state == 1)

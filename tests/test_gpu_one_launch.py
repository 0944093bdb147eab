"""Small batches run a force evaluation, or a run of MD steps, in one launch
(fused.cu).  Its results are those of the pass-by-pass launches bit for bit:
forces and radii against the same molecule in a batch that is too large for
one launch, MD against the same run with profiling on (which times the passes
one by one), at sizes around a tile, a row pair, the number of thread blocks
of a cluster and the largest replica that is taken."""
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


@pytest.mark.parametrize("kappa", [0.0, 0.125])
@pytest.mark.parametrize("sizes", [[1], [32], [33], [64, 0, 65], [128, 129], [237], [512], [673], [100] * 40, [290] * 80])
def test_forces_and_radii(pkg, sizes, kappa):
    import torch
    b = synth.random_batch(sizes[:3], seed=61, sites=False)
    b = synth.Batch(b.replicas + b.replicas[:1] * (len(sizes) - len(b.replicas)), pH=np.zeros(len(sizes)),
                    E=np.zeros(len(sizes)))
    big = synth.make_replica(1300, 5, [])
    wide = synth.Batch(b.replicas + [big], pH=np.zeros(len(sizes) + 1), E=np.zeros(len(sizes) + 1))
    n = b.n_atoms
    res = []
    for batch in (b, wide):
        xyzq, rad = to_dev(batch, device())
        ctx = pkg.Context(batch.atom_off, pkg.default_params(kappa=kappa))
        for _ in range(2):                     # the second call finds what the first left behind
            out = ctx.energy_forces(xyzq, rad, want=("R", "F", "F_fixed"))
        res.append((out["R"][:n], out["F"][:n], out["F_fixed"][:, :n], ctx.born_radii(xyzq, rad)[:n]))
        torch.cuda.synchronize()
        ctx.sync_status()
    for x, y in zip(*res):
        assert torch.equal(x, y)


@pytest.mark.parametrize("sizes", [[40], [256], [300, 0, 64, 129], [97] * 40])
def test_md_steps(pkg, sizes):
    import torch
    b = synth.random_batch(sizes[:4], seed=62)
    b = synth.Batch(b.replicas + b.replicas[:1] * (len(sizes) - len(b.replicas)), pH=np.full(len(sizes), 4.85),
                    E=np.full(len(sizes), synth.E0_REF_V))
    runs = []
    for prof in (False, True):
        sim = pkg.Simulation(b.atom_off, b.xyzq(), b.rad_screen(), pkg.default_params(rep_k=100.0, rep_sigma=2.5),
                             sites=b.site_tables(), pH=b.pH, E=b.E, seed=9, mc_every=5)
        sim.ctx.set_profiling(prof)
        sim.run(20).run(3)                     # captured blocks of five, then direct launches
        sim.sync()
        runs.append(sim)
    for k in ("xyzq", "vel", "force", "R", "state"):
        assert torch.equal(getattr(runs[0], k), getattr(runs[1], k)), k


@pytest.mark.parametrize("persistent", [False, True])
def test_autotune_md_leaves_caps_it_does_not_use(pkg, persistent):
    """A segment that runs in one launch reads no register caps: tuning on it
    keeps those the context has, refuses what a segment refuses, and moves no
    state; with profiling on the passes run one by one and are tuned."""
    import torch
    b = synth.random_batch([300, 180], seed=63)
    sim = pkg.Simulation(b.atom_off, b.xyzq(), b.rad_screen(), pkg.default_params(rep_k=100.0, rep_sigma=2.5),
                         sites=b.site_tables(), pH=b.pH, E=b.E, seed=9, mc_every=5)
    sim.ctx.set_persistent(persistent)
    x = sim.xyzq.clone()
    for caps in ((4, 3, 1), (1, 4, 4), (3, 1, 3)):
        for p, c in enumerate(caps):
            sim.ctx.set_reg_cap(c, p)
        assert sim.ctx.autotune_md(sim.st, sim.sites, 10) == caps
    assert sim.step == 0 and torch.equal(sim.xyzq, x)
    state, sim.st.state = sim.st.state, None
    with pytest.raises(pkg.GBError):
        sim.ctx.autotune_md(sim.st, sim.sites, 10)
    sim.st.state = state
    if not persistent:
        sim.ctx.set_profiling(True)
        assert all(c in (1, 3, 4) for c in sim.ctx.autotune_md(sim.st, sim.sites, 10))
    sim.sync()
    assert torch.equal(sim.xyzq, x)

"""What the pass-by-pass launches promise for batches beyond the one-launch
kernel's sizes: forces without energies are the same bit for bit whatever the
warps a block, the task length and the register caps, in 64 x 32 and in 128 x 32
blocks; MD segments are the same from captured blocks, from direct launches,
after tuning and from the persistent kernel; and the forms that only a salt run has agree with the oracle in 128 x 32
blocks."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from gpu_common import F_ABS, R_REL, device, oracle_params, to_dev

pytestmark = pytest.mark.gpu

WIDE = 12833                                   # 402 tiles: 128 x 32 blocks, the last tile of one atom
FIELDS = [{}, dict(rep_k=100.0, rep_sigma=2.5), dict(rep_k=100.0, rep_sigma=2.5, kappa=0.125)]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1803_09652_gb300 as p
    return p


def kernel_launches(pkg, ctx, xyzq, rad):
    """Kernels of one born_radii call, counted in a captured graph."""
    import torch
    R = torch.empty(xyzq.shape[0], dtype=torch.float32, device=xyzq.device)
    lib, s, graph, n = pkg.load(), torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    stream = ctypes.c_void_p(s.cuda_stream)
    assert lib.cudaStreamBeginCapture(stream, 2) == 0          # relaxed mode
    ctx.born_radii(xyzq, rad, R_out=R, stream=s)
    assert lib.cudaStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert lib.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert lib.cudaGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("sizes,one", [([1], True), ([237], True), ([672], True), ([673], False), ([1024], False),
                                       ([1300], False), ([100] * 40, True), ([290] * 80, True)])
def test_which_batches_run_in_one_launch(pkg, sizes, one):
    """672 atoms are 121 blocks for the 128 warps of a cluster of 16, 673 are 132."""
    b = synth.Batch([synth.make_replica(n, 3, []) for n in sizes], pH=np.zeros(len(sizes)), E=np.zeros(len(sizes)))
    xyzq, rad = to_dev(b, device())
    ctx = pkg.Context(b.atom_off)
    assert (kernel_launches(pkg, ctx, xyzq, rad) == 1) == one
    ctx.sync_status()


def _forces(pkg, sizes, field, tiles=None, caps=None, seed=41):
    import torch
    reps = [synth.make_replica(n, seed + k, []) for k, n in enumerate(sizes)]
    b = synth.Batch(reps, pH=np.zeros(len(sizes)), E=np.zeros(len(sizes)))
    xyzq, rad = to_dev(b, device())
    ctx = pkg.Context(b.atom_off, pkg.default_params(**field))
    if tiles:
        ctx.set_tiles(*tiles)
    if caps:
        for p, c in enumerate(caps):
            ctx.set_reg_cap(c, p)
    out = ctx.energy_forces(xyzq, rad, want=("R", "F", "F_fixed"))
    torch.cuda.synchronize()
    ctx.sync_status()
    return {k: v.cpu().numpy() for k, v in out.items()}, b


@pytest.mark.parametrize("field", FIELDS)
@pytest.mark.parametrize("sizes", [[1300], [1057, 33, 2000], [6433], [12800], [WIDE], [1300, WIDE]])
def test_forces_do_not_depend_on_the_split(pkg, sizes, field):
    ref, _ = _forces(pkg, sizes, field)
    for tiles, caps in [((1, 1), None), ((2, 2), (1, 1, 1)), ((8, 4), (3, 3, 3)), ((4, 64), (4, 4, 4)),
                        ((8, 1), (1, 3, 4)), ((3, 17), (4, 1, 3))]:
        out, _ = _forces(pkg, sizes, field, tiles, caps)
        for k in ref:
            assert np.array_equal(out[k], ref[k]), (tiles, caps, k)


@pytest.mark.parametrize("field", FIELDS)
def test_replica_does_not_depend_on_the_batch(pkg, field):
    """A replica of 128 x 32 blocks and one of 64 x 32 blocks, alone and together
    (alone the smaller one runs the kernel without 128 x 32 code)."""
    both, _ = _forces(pkg, [WIDE, 1300], field)
    first, _ = _forces(pkg, [WIDE], field)
    second, _ = _forces(pkg, [1300], field, seed=42)
    for k, axis in (("R", 0), ("F", 0), ("F_fixed", 1)):
        assert np.array_equal(both[k], np.concatenate([first[k], second[k]], axis)), k


@pytest.mark.parametrize("sizes,field", [([237, 672], FIELDS[2]), ([237, 672], dict(kappa=0.125)), ([WIDE], FIELDS[2])])
def test_salt_against_the_oracle(pkg, sizes, field):
    out, b = _forces(pkg, sizes, field)
    for k, rep in enumerate(b.replicas):
        x = [np.asarray(v, np.float32).astype(np.float64) for v in (rep.xyz, rep.q, rep.rho, rep.screen)]
        p = oracle_params(**{"bond_k": 0.0, "rep_k": 0.0, **field})
        ref = oracle.energy_forces(*x, p)
        ref["F"] += oracle.restraints(x[0], p)[1]                  # the soft repulsion
        a, c = b.atom_off[k], b.atom_off[k + 1]
        assert np.max(np.abs(out["R"][a:c] / ref["R"] - 1)) < R_REL
        assert np.max(np.abs(out["F"][a:c] - ref["F"])) < F_ABS


def _sim(pkg, b, **kw):
    field = kw.pop("field", FIELDS[1])
    return pkg.Simulation(b.atom_off, b.xyzq(), b.rad_screen(), pkg.default_params(**field), sites=b.site_tables(),
                          pH=b.pH, E=b.E, seed=9, **kw)


def _equal(a, b):
    import torch
    a.sync()
    b.sync()
    for k in ("xyzq", "vel", "force", "R", "state", "E", "grid"):
        assert torch.equal(getattr(a, k), getattr(b, k)), k


@pytest.mark.parametrize("field", FIELDS[1:])
@pytest.mark.parametrize("persistent", [False, True])
def test_captured_blocks_equal_direct_launches(pkg, persistent, field):
    device()                                   # skips without a GPU
    b = synth.config_eremd(4, 1100)
    runs = []
    for calls in (1, 40):
        sim = _sim(pkg, b, field=field, mc_every=5, ex_every=20, E_ladder=synth.e_ladder(4), pH_ladder=[b.pH[0]])
        sim.ctx.set_persistent(persistent)
        for _ in range(calls):
            sim.run(40 // calls)
        runs.append(sim)
    _equal(*runs)


def test_tuned_caps_change_no_result(pkg):
    """The run after tuning equals one with other caps: the segment reads them
    (more than one launch), and the tuner moves no state."""
    device()                                   # skips without a GPU
    b = synth.random_batch([1300, 1100], seed=64)
    runs = []
    for tune in (False, True):
        sim = _sim(pkg, b, mc_every=5)
        if tune:
            assert all(c in (1, 3, 4) for c in sim.ctx.autotune_md(sim.st, sim.sites, 10))
        else:
            for p, c in enumerate((4, 3, 4)):
                sim.ctx.set_reg_cap(c, p)
        assert sim.step == 0
        runs.append(sim.run(30))
    _equal(*runs)


@pytest.mark.parametrize("sizes", [[1100, 33, 64, 1], [WIDE]])
def test_persistent_kernel_equals_the_launches(pkg, sizes):
    """Both drivers add the same fixed-point forces: results are equal bit for bit."""
    device()                                   # skips without a GPU
    b = synth.random_batch(sizes, seed=13)
    runs = []
    for persistent in (False, True):
        sim = _sim(pkg, b, mc_every=5)
        sim.ctx.set_persistent(persistent)
        runs.append(sim.run(10))
    _equal(*runs)


@pytest.mark.parametrize("sizes", [[256], [300, 0, 64, 672]])
def test_one_launch_steps_with_salt(pkg, sizes):
    """One launch for a run of steps in salt water with repulsion: bit for bit the
    passes one by one (profiling on)."""
    device()                                   # skips without a GPU
    b = synth.random_batch(sizes, seed=62)
    runs = []
    for prof in (False, True):
        sim = _sim(pkg, b, field=FIELDS[2], mc_every=5)
        sim.ctx.set_profiling(prof)
        runs.append(sim.run(20).run(3))
    _equal(*runs)


@pytest.mark.parametrize("field", [dict(rgbmax=12.0, cut=12.0), dict(rgbmax=9.0), dict(cut=25.0, kappa=0.125)])
def test_cutoff_forces_do_not_depend_on_the_batch(pkg, field):
    """Few blocks in the batch: every block in range is a task; many: runs of them."""
    few, _ = _forces(pkg, [500, 1057, 33], field)
    many, _ = _forces(pkg, [500, 1057, 33, 12000, 12000], field)
    n = 500 + 1057 + 33
    for k in few:
        a, b = (few[k], many[k][:, :n]) if k == "F_fixed" else (few[k], many[k][:n])
        assert np.array_equal(a, b), k


@pytest.mark.parametrize("field", [{}, dict(rgbmax=12.0, cut=12.0)])
@pytest.mark.parametrize("n", [1, 33, 65, 129, 3840, 3841])
def test_static_entry_at_the_edges_of_its_task_lists(pkg, n, field):
    """Every block a task up to 3840 atoms, runs of columns beyond.  Without tile boxes
    a block may take another form than the context's; each is within its tolerance of
    the oracle, so the two are within twice that."""
    import torch
    out, b = _forces(pkg, [n], field)
    xyzq, rad = to_dev(b, device())
    R, F = torch.empty(n, device=xyzq.device), torch.empty((n, 3), device=xyzq.device)
    call = ctypes.CDLL(pkg.LIB_PATH).gb_energy_forces_static
    call.argtypes = [ctypes.c_int32, ctypes.c_void_p] + [ctypes.c_void_p] * 8
    params = pkg.default_params(**field)
    assert call(n, ctypes.byref(params), xyzq.data_ptr(), rad.data_ptr(), R.data_ptr(), None, F.data_ptr(), None, None,
                torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert np.max(np.abs(R.cpu().numpy() / out["R"] - 1)) < 2 * R_REL
    assert np.max(np.abs(F.cpu().numpy() - out["F"])) < 2 * F_ABS

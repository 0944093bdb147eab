"""The forms the pair passes take by distance (near with close pairs apart,
far, and the two distant fits), in 64 x 32 and in 128 x 32 blocks, against the
FP64 oracle: two chains at gaps on either side of every form's limit, chains
crowded into one another (every pair close), and one molecule just past the
size where 128 x 32 blocks begin, with a one-atom last tile."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import F_ABS, R_REL, device, oracle_params

pytestmark = pytest.mark.gpu


def _run(pkg, x, q, rho, scr, r_rel=R_REL, **kw):
    import torch
    dev = device()
    xyzq = np.concatenate([x, q[:, None]], 1).astype(np.float32)
    rad = np.stack([rho, scr], 1).astype(np.float32)
    ctx = pkg.Context([0, len(q)], pkg.default_params(**kw))
    out = ctx.energy_forces(torch.as_tensor(xyzq, device=dev), torch.as_tensor(rad, device=dev), want=("R", "F"))
    torch.cuda.synchronize()
    ctx.sync_status()
    ref = oracle.energy_forces(xyzq[:, :3].astype(np.float64), xyzq[:, 3].astype(np.float64), rad[:, 0].astype(np.float64),
                               rad[:, 1].astype(np.float64), oracle_params(**kw))
    R, F = out["R"].cpu().numpy(), out["F"].cpu().numpy()
    assert np.max(np.abs(R / ref["R"] - 1)) < r_rel
    assert np.max(np.abs(F - ref["F"])) < F_ABS


@pytest.fixture(scope="module")
def pkg():
    import paper_1803_09652_gb300 as p
    return p


def _two_chains(gap):
    a, b = synth.make_replica(150, 5, []), synth.make_replica(171, 6, [])
    shift = a.xyz[:, 0].max() - b.xyz[:, 0].min() + gap
    x = np.concatenate([a.xyz, b.xyz + np.array([shift, 0, 0], np.float32)])
    return x, np.concatenate([a.q, b.q]), np.concatenate([a.rho, b.rho]), np.concatenate([a.screen, b.screen])


# gaps around (s/r)^2 = 0.1, 0.025 / 0.0185 and 0.009 / 0.006 for s = 1.53 A
@pytest.mark.parametrize("gap", [2.0, 4.7, 5.0, 9.5, 9.9, 11.1, 11.4, 15.9, 16.3, 19.6, 20.0, 60.0])
def test_two_chains_at_every_form(pkg, gap):
    _run(pkg, *_two_chains(gap))


def test_two_chains_in_salt_water(pkg):
    _run(pkg, *_two_chains(7.0), kappa=0.125)


@pytest.mark.parametrize("n", [33, 97, 257])
def test_crowded_atoms_are_all_close_pairs(pkg, n):
    """A jittered lattice 1.3 A apart : every
    block is near, and its queue of close pairs runs full.  The closed form of an
    overlapping pair cancels about tenfold (1e-6 of a term, 2.5e-7 of a sum of
    twenty), and R moves by up to 3 Phi ~ 10 times that where tanh turns over:
    5e-6 with a factor of two."""
    rng = np.random.default_rng(n)
    k = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    x = (1.3 * g + rng.uniform(-0.1, 0.1, (n, 3))).astype(np.float32)
    q = rng.normal(0, 0.05, n).astype(np.float32)
    rho = np.asarray(synth.RADIUS_SET, np.float32)[rng.integers(0, 5, n)]
    scr = rng.uniform(0.2, 0.5, n).astype(np.float32)
    _run(pkg, x, q, rho, scr, r_rel=5e-6)


def test_first_size_with_row_pair_blocks(pkg):
    r = synth.make_replica(6433, 9, [])          # 202 tiles, the last of one atom
    _run(pkg, r.xyz, r.q, r.rho, r.screen)

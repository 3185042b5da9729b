"""Pure tree mode in boxes of any side, down to the closest pairs.

A term's offset and |d|^2 + eps^2 carry one FP32 rounding each, whatever the
separation: positions are held as two floats, and where a pair is closer than
these can tell, the FP64 positions are taken. Counts stay bit-exact and forces
within the bounds of the unit box in boxes of 3.7 and 64."""
import math

import numpy as np
import pytest

import oracle
from common import device_arrays, ng_params, oracle_params
from metrics import rel_err
from paper_1502_07442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1502_07442_gb300 import binding, build
    build.build()
    return binding


def _force(ng, w, count=False):
    import torch
    pos, typ, mass = device_arrays(w)
    n = typ.numel()
    sim = ng.Simulation(ng_params(w["params"]))
    ng.ng_build_tree(sim.ctx, pos, typ, mass)
    acc = torch.empty((3, n), dtype=torch.float32, device=pos.device)
    nint = ng.ng_tree_force(sim.ctx, acc, count=True)
    counts = torch.empty(n, dtype=torch.int64, device=pos.device)
    ng.ng_count_interactions(sim.ctx, counts)
    torch.cuda.synchronize()
    sim.close()
    return acc.cpu().numpy().astype(np.float64), counts.cpu().numpy(), nint


@pytest.mark.parametrize("L", [1.0, 3.7, 64.0])
def test_pairs_at_any_separation(ng, L):
    """Isolated pairs (cut-off 0.03 L, pairs 0.1 L apart) of separations 2e-2 to
    1e-12 L. Roundings of one Newtonian term, in units of 2^-24: offset 1, q 1.5
    (to the power -3/2), the root 1 and its product with q 1, coupling times mass
    2, quotient 1, product and sum 2: below 10."""
    rng = inputs.rng_for(17)
    c = (np.stack(np.meshgrid(*[np.arange(10)] * 3, indexing="ij")).reshape(3, -1) + 0.5) / 10
    m = c.shape[1]
    sep = 10.0 ** rng.uniform(-12, math.log10(0.02), m)
    u = rng.standard_normal((3, m))
    u /= np.linalg.norm(u, axis=0)
    c = c + rng.uniform(-0.02, 0.02, c.shape)
    pos = np.ascontiguousarray(np.concatenate([c, c + sep * u], axis=1) * L)
    n = 2 * m
    prm = dict(D=1, G=[[1.0]], law=[[0]], ya=[[0.0]], yl=[[1.0]], box=L, eps=1e-13 * L, rs=0.03 * L / 4.5,
               rcut=0.03 * L, theta=0.5, pm_mesh=0, leaf_size=8, pure_tree=1, beta=0.0)
    w = dict(pos=pos, type=np.zeros(n, np.uint8), mass=np.full(n, 1e-3, np.float32), params=prm)
    got, _, _ = _force(ng, w)
    x = pos * (1.0 / L)
    d = (x[:, m:] - x[:, :m]) * L
    q = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + prm["eps"] ** 2
    f = float(np.float32(1e-3)) * d / q ** 1.5
    want = np.concatenate([f, -f], axis=1)
    err = np.linalg.norm(got - want, axis=0) / np.linalg.norm(want, axis=0)
    assert err.max() <= 10 * 2.0 ** -24, (err.max(), sep[int(np.argmax(err)) % m])


def _boxed(L, n, seed, law, theta):
    rng = inputs.rng_for(seed)
    pos = inputs.clustered(n, rng, nspheres=8, a=0.02) * L
    typ = inputs.species_uniform(n, 2, rng)
    mass = np.full(n, 1.0 / n, np.float32)
    prm = dict(D=2, G=[[1.0, 0.8], [0.8, 1.2]], law=law, ya=[[0.3, 0.5], [0.5, 0.7]],
               yl=(np.array([[0.05, 0.03], [0.03, 0.02]]) * L).tolist(), box=L, eps=1e-4 * L, rs=0.1 * L,
               rcut=0.45 * L, theta=theta, pm_mesh=0, leaf_size=8, pure_tree=1, ignore_nperp=0,
               beta=(1.0 / n) / (4 * math.pi * 0.004 * L))
    return dict(pos=np.ascontiguousarray(pos), type=typ, mass=mass, params=prm)


@pytest.mark.parametrize("L", [3.7, 64.0])
@pytest.mark.parametrize("law", [[[0, 1], [1, 2]], [[0, 3], [3, 3]]], ids=["newton_yukawa", "mahalo"])
def test_other_boxes_match_the_oracle(ng, L, law):
    w = _boxed(L, 9001, 18, law, 0.5)
    acc, counts, nint = _force(ng, w)
    ref, c_ref = oracle.tree_walk(oracle_params(w["params"]), w["pos"], w["type"], w["mass"])
    assert np.array_equal(counts, c_ref) and nint == int(c_ref.sum())
    e, _ = rel_err(acc, ref)
    assert np.median(e) <= 1e-5 and np.percentile(e, 99) <= 1e-4


def test_lattice_corrections_scale_with_the_box(ng):
    """Newtonian forces in a box of side L are 1 / L^2 of those in the unit box
    (both within the bounds above of the exact ones: twice them here)."""
    out = []
    for L in (1.0, 3.7):
        w = _boxed(L, 3001, 19, [[0, 0], [0, 0]], 0.5)
        w["params"].update(pure_tree=2)
        out.append(_force(ng, w)[0] * L * L)
    e, _ = rel_err(out[1], out[0])
    assert np.median(e) <= 2e-5 and np.percentile(e, 99) <= 2e-4

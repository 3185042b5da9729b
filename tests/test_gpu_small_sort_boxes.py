"""The sort by counting and the radix sort on both sides of their line in boxes
that are not a power of two (5120 bodies; 8192 in those that are): keys,
permutation and type-major order bit-exact against the oracle, in a build and in
steps that stop at a level cap."""
import numpy as np
import pytest

import oracle
from common import device_arrays, ng_params, small_clustered
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


def _boxed(n, D, L, seed):
    w = small_clustered(n, D, seed)
    rng = inputs.rng_for(seed + 1)
    shift = rng.choice([-1.0, 1.0, 2.0], size=n) * (rng.random(n) < 0.1)
    prm = w["params"]
    w["params"] = dict(prm, box=L, eps=prm["eps"] * L, rs=prm["rs"] * L, rcut=prm["rcut"] * L)
    w["pos"] = np.ascontiguousarray(w["pos"] * L + shift[None, :] * L)
    w["pos"][:, ::3] = w["pos"][:, :1]          # a third of the bodies in one place
    return w


@pytest.mark.parametrize("n,D,L", [(1, 1, 3.7), (65, 2, 3.7), (4097, 6, 100.0), (5120, 3, 3.7), (5121, 3, 3.7),
                                   (8192, 2, 0.3), (8193, 2, 3.7), (8192, 4, 64.0)])
def test_sort_at_its_line(ng, n, D, L):
    import torch
    w = _boxed(n, D, L, 700 + n % 89)
    pos, typ, mass = device_arrays(w)
    sim = ng.Simulation(ng_params(w["params"]))
    keys = torch.empty(n, dtype=torch.int64, device=pos.device)
    perm = torch.empty(n, dtype=torch.int32, device=pos.device)
    order = torch.empty(n, dtype=torch.int32, device=pos.device)
    ng.ng_build_tree(sim.ctx, pos, typ, mass, keys, perm)
    offs = ng.ng_type_order(sim.ctx, D, order)
    sim.close()
    k_ref = oracle.keys(w["pos"], w["type"], box=L)
    p_ref = np.argsort(k_ref, kind="stable").astype(np.uint32)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), p_ref)
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), k_ref[p_ref])
    assert np.array_equal(order.cpu().numpy().view(np.uint32),
                          p_ref[np.argsort(w["type"][p_ref], kind="stable")])
    assert np.array_equal(offs, np.concatenate([[0], np.cumsum(np.bincount(w["type"], minlength=D))]))


@pytest.mark.parametrize("n", [5120, 5121])
def test_steps_at_its_line(ng, n):
    """Four steps (two of them replayed under the level cap) against four single
    ones, without couplings: the same drift, bit for bit."""
    import torch
    w = _boxed(n, 2, 3.7, 800)
    prm = dict(w["params"], G=np.zeros((2, 2)), pm_mesh=0)
    rng = inputs.rng_for(801)
    v0 = rng.uniform(-1, 1, (3, n)).astype(np.float32)
    out = []
    for calls, k in ((1, 4), (4, 1)):
        pos, typ, mass = device_arrays(w)
        vel = torch.from_numpy(v0.copy()).to(pos.device)
        acc = torch.zeros((3, n), dtype=torch.float32, device=pos.device)
        sim = ng.Simulation(ng_params(prm))
        for _ in range(calls):
            ng.ng_step(sim.ctx, pos, vel, typ, mass, acc, True, k, 2.0 ** -10)
        sim.close()
        out.append((pos.cpu().numpy(), vel.cpu().numpy(), acc.cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)

"""GPU parity of the sort, tree, monopoles and type-major order at the edges of
their tiles (keys, permutation and tree bit-exact against the oracle): radix
tiles of 1024 or 4096 keys (the larger from 1245184 bodies) in groups of 16, tree
tiles of 1024 bodies, leaf tiles of 256, type-order tiles of 4096, subtrees of
256 or 512 bodies; leaves of 1, 8 and 64 bodies, one to six species; and the
return of a stepped state to the caller's order in tiles of 256 bodies."""
import numpy as np
import pytest

import oracle
from common import device_arrays, ng_params, oracle_params, small_clustered
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


CASES = [(1, 6, 1), (2, 1, 1), (255, 2, 8), (256, 3, 8), (257, 4, 8), (1023, 5, 64), (1024, 6, 1),
         (1025, 1, 8), (4097, 2, 1), (16384, 3, 8), (16385, 6, 64), (65537, 4, 1),
         (600001, 5, 8), (1245183, 2, 32), (1245185, 3, 32)]


@pytest.mark.parametrize("n,D,leaf", CASES, ids=[f"n{c[0]}_d{c[1]}_leaf{c[2]}" for c in CASES])
def test_sort_and_tree_at_tile_edges(ng, n, D, leaf):
    import torch
    w = small_clustered(n, D, 300 + n % 97, leaf=leaf)
    if n > 1000:
        w["pos"][:, 500:600] = w["pos"][:, 499:500]     # equal keys: a level-20 leaf, ties in order
    rng = inputs.rng_for(n)
    w["mass"] = (rng.uniform(0.5, 1.5, n) / n).astype(np.float32)
    prm = w["params"]
    pos, typ, mass = device_arrays(w)
    sim = ng.Simulation(ng_params(prm))
    keys = torch.empty(n, dtype=torch.int64, device=pos.device)
    perm = torch.empty(n, dtype=torch.int32, device=pos.device)
    order = torch.empty(n, dtype=torch.int32, device=pos.device)
    ng.ng_build_tree(sim.ctx, pos, typ, mass, keys, perm)
    offs = ng.ng_type_order(sim.ctx, D, order)
    T = ng.ng_tree_export(sim.ctx, D)
    sim.close()
    k_ref = oracle.keys(w["pos"], w["type"])
    p_ref = np.argsort(k_ref, kind="stable").astype(np.uint32)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), p_ref)
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), k_ref[p_ref])
    t_sorted = w["type"][p_ref]
    assert np.array_equal(order.cpu().numpy().view(np.uint32), p_ref[np.argsort(t_sorted, kind="stable")])
    assert np.array_equal(offs, np.concatenate([[0], np.cumsum(np.bincount(w["type"], minlength=D))]))
    R = oracle.tree(oracle_params(prm), w["pos"], w["type"], w["mass"])
    for f in ("level", "prefix", "first", "count", "nchild", "child_first", "cnt"):
        assert np.array_equal(T[f], R[f].astype(T[f].dtype)), f
    # FP64 sums of the same terms in another order
    assert np.all(np.abs(T["mass"] - R["mass"]) <= 2.0 ** -53 * (R["cnt"].astype(float) + 2) * R["mass"])
    bound = 2.0 ** -53 * 4 * (R["cnt"].astype(np.float64) + 2)
    assert np.all(np.abs(T["com"] - R["com"]).max(axis=2) <= bound)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 5000])
def test_state_returns_to_caller_order(ng, n):
    """One step with unit masses' couplings off (G = 0): every body drifts
    freely, so positions and velocities of the caller's order follow in closed
    form, each operation exactly as the step rounds it."""
    import torch
    w = small_clustered(n, 2, 40 + n)
    prm = dict(w["params"], G=np.zeros((2, 2)), pm_mesh=0)
    pos, typ, mass = device_arrays(w)
    rng = inputs.rng_for(7 + n)
    vel = torch.from_numpy(rng.uniform(-1, 1, (3, n)).astype(np.float32)).to(pos.device)
    acc = torch.zeros((3, n), dtype=torch.float32, device=pos.device)
    x0, v0 = pos.cpu().numpy().copy(), vel.cpu().numpy().copy()
    sim = ng.Simulation(ng_params(prm))
    ng.ng_step(sim.ctx, pos, vel, typ, mass, acc, True, 1, 2.0 ** -10)
    sim.close()
    x = x0 + v0.astype(np.float64) * 2.0 ** -10          # exact product, one rounding: as the FMA
    assert np.array_equal(pos.cpu().numpy(), x - np.floor(x))
    assert np.array_equal(vel.cpu().numpy(), v0)
    assert np.all(acc.cpu().numpy() == 0)


@pytest.mark.parametrize("n,D", [(31, 1), (32, 6), (33, 2), (63, 3), (65, 4), (2047, 6), (4095, 1), (4096, 3),
                                 (8191, 2), (8192, 6), (8193, 5)])
def test_small_sort_at_its_edges(ng, n, D):
    """Sorts by counting (up to 8192 bodies, in blocks of 32 or 64) and the
    first size past them: duplicates keep their order."""
    import torch
    w = small_clustered(n, D, 500 + n)
    w["pos"][:, ::3] = w["pos"][:, :1]          # a third of the bodies in one place
    prm = w["params"]
    pos, typ, mass = device_arrays(w)
    sim = ng.Simulation(ng_params(prm))
    keys = torch.empty(n, dtype=torch.int64, device=pos.device)
    perm = torch.empty(n, dtype=torch.int32, device=pos.device)
    order = torch.empty(n, dtype=torch.int32, device=pos.device)
    ng.ng_build_tree(sim.ctx, pos, typ, mass, keys, perm)
    offs = ng.ng_type_order(sim.ctx, D, order)
    sim.close()
    k_ref = oracle.keys(w["pos"], w["type"])
    p_ref = np.argsort(k_ref, kind="stable").astype(np.uint32)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), p_ref)
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), k_ref[p_ref])
    assert np.array_equal(order.cpu().numpy().view(np.uint32),
                          p_ref[np.argsort(w["type"][p_ref], kind="stable")])
    assert np.array_equal(offs, np.concatenate([[0], np.cumsum(np.bincount(w["type"], minlength=D))]))


@pytest.mark.parametrize("n", [300, 20000, 131071, 131072, 131101])
def test_bodies_outside_the_box_and_bad_species(ng, n):
    """Every path of the sort (counting, radix passes, packed records from 131072
    bodies) wraps positions as the keys do and refuses a species out of range,
    after which the context takes good input."""
    import torch
    w = small_clustered(n, 3, 600 + n % 101)
    rng = inputs.rng_for(n + 1)
    w["pos"] = w["pos"] + rng.integers(-2, 3, w["pos"].shape)
    pos, typ, mass = device_arrays(w)
    bad = typ.clone()
    bad[n // 2] = 3
    sim = ng.Simulation(ng_params(w["params"]))
    keys = torch.empty(n, dtype=torch.int64, device=pos.device)
    with pytest.raises(ng.NgError):
        ng.ng_build_tree(sim.ctx, pos, bad, mass)
    ng.ng_build_tree(sim.ctx, pos, typ, mass, keys)
    T = ng.ng_tree_export(sim.ctx, 3)
    sim.close()
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), np.sort(oracle.keys(w["pos"], w["type"])))
    R = oracle.tree(oracle_params(w["params"]), w["pos"], w["type"], w["mass"])
    assert np.array_equal(T["cnt"], R["cnt"].astype(T["cnt"].dtype))
    bound = 2.0 ** -53 * 4 * (R["cnt"].astype(np.float64) + 2)
    assert np.all(np.abs(T["com"] - R["com"]).max(axis=2) <= bound)


@pytest.mark.parametrize("n,D,leaf", [(1048576, 2, 8), (1048577, 3, 1), (1048577, 6, 9)])
def test_large_trees_of_small_leaves(ng, n, D, leaf):
    """From 2^20 bodies: leaves by tiles up to 8 bodies, binned above."""
    test_sort_and_tree_at_tile_edges(ng, n, D, leaf)

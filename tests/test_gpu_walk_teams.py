"""Walks in which teams of 8, 4 or 2 warps share a group, against the walk of
whole groups per warp on the same bodies (a law table that leaves shared memory
for one warp a block makes no teams). Every list entry is evaluated once
whoever holds it: the executed interactions are the same number. The two law
tables (169 and 560 segments) are within 1.9e-5 and 1.8e-6 of the law's value 1
at zero separation, so forces differ by at most that share, and 80 FP32
roundings, of the sum of the terms' magnitudes, here bounded by 1.5 times the
sum of G m / rho^2 over all bodies within 1.3 cut-offs (a node stands for bodies
up to half its distance nearer or farther)."""
import numpy as np
import pytest

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


def _force(ng, w, **over):
    import torch
    pos, typ, mass = device_arrays(w)
    n = typ.numel()
    sim = ng.Simulation(ng_params(dict(w["params"], **over)))
    if over.get("opening"):
        ng.ng_set_acc_old(sim.ctx, torch.from_numpy(w["old"]).to(pos.device))
    ng.ng_build_tree(sim.ctx, pos, typ, mass)
    acc = torch.empty((3, n), dtype=torch.float32, device=pos.device)
    nint = ng.ng_tree_force(sim.ctx, acc, count=True)
    torch.cuda.synchronize()
    sim.close()
    return acc.cpu().numpy().astype(np.float64), nint


# bodies, cut-off in box units (0.07: split level 4; 0.45: level 2), leaf size
# (64: trees above the split level). With 16 warps a block and about 28 bodies a
# group, teams of 8 up to some 8000 bodies, of 4 to 34000, of 2 to 200000.
@pytest.mark.parametrize("n,rcut,leaf", [(20, 0.07, 8), (500, 0.07, 64), (3000, 0.07, 8), (3000, 0.45, 1),
                                         (20000, 0.07, 8), (20000, 0.45, 16), (120000, 0.07, 8)])
@pytest.mark.parametrize("opening", [0, 1], ids=["geometric", "relative"])
def test_teams_walk_what_one_warp_walks(ng, n, rcut, leaf, opening):
    w = small_clustered(n, 6, 60 + n % 31, leaf=leaf)
    w["params"].update(rs=rcut / 4.5, rcut=rcut, pm_mesh=0)
    w["old"] = (10.0 * inputs.rng_for(n).standard_normal((3, n))).astype(np.float32)
    over = dict(opening=opening, alpha=0.005)
    team, nt = _force(ng, w, **over)
    one, n1 = _force(ng, w, table_size=560, **over)
    assert nt == n1 > 0
    if n > 3000:
        return
    p = w["params"]
    tot = np.zeros(n)
    for j in range(n):
        d = w["pos"] - w["pos"][:, j:j + 1]
        d -= np.rint(d)
        r2 = (d ** 2).sum(axis=0)
        g = np.asarray(p["G"])[w["type"], w["type"][j]] * w["mass"][j]
        tot += np.where((r2 < (1.3 * rcut) ** 2) & (np.arange(n) != j), g / (r2 + p["eps"] ** 2), 0.0)
    err = np.linalg.norm(team - one, axis=0)
    assert np.all(err <= 1.5 * (2.1e-5 + 80 * 2.0 ** -24) * tot), (err / np.maximum(tot, 1e-300)).max()

"""The periodic local search where its work splits or its O(1) forms end: one
vehicle (no relocation target), more vehicles than ops (empty routes), one
customer, teams of one and of many CTAs, and matrices in which most gaps are
shortcuts (both simulated forms).  Whole runs equal to the oracle's, step by
step (whole numbers, no tolerance)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

FIELDS = ("accepted", "improved", "new_best", "rejected_infeasible", "ls_moves", "ls_new_best")


def same(vrp, inst, oi, iters, seed, ls, team_blocks, q=(1, 2)):
    init = vrp.initial_solution(inst)
    g = vrp.alns_run(inst, vrp.alns_params(iters, *q, 3, team_blocks, destroy_mask=63, ls_pickup_every=ls[0],
                                           ls_relocate_every=ls[1]), seed=seed, init=init)
    o = oracle.alns_run(oi, init[0], init[1], oracle.alns_params(iters, *q, 3, destroy_mask=63, ls_pickup_every=ls[0],
                                                                 ls_relocate_every=ls[1]), seed)
    assert np.array_equal(g["trace"], o["trace"]), np.argwhere(g["trace"] != o["trace"])[:3]
    for f in FIELDS:
        assert getattr(g["stats"], f) == getattr(o["stats"], f), f
    assert np.array_equal(g["best_ops"], o["best_ops"]) and np.array_equal(g["best_off"], o["best_off"])
    return g


@pytest.mark.parametrize("n,m,R,Q,tb", [(1, 1, 1, 1, 1), (1, 3, 3, 2, 4), (2, 32, 32, 1, 3), (5, 1, 2, 2, 2),
                                        (9, 32, 12, 2, 5), (17, 2, 4, 3, 1), (33, 6, 8, 3, 64), (47, 9, 20, 4, 7)])
@pytest.mark.parametrize("full", [False, True])
def test_local_search_edges(vrp, n, m, R, Q, tb, full):
    w = workloads.make_instance(n, m, m * Q if full else R, Q, "5x", "clustered", seed=n + m)
    inst = vrp.Instance.from_workload(w, load_full=full)
    oi = oracle.OracleInstance.from_workload(w, load_full=full)
    same(vrp, inst, oi, 12, 3, (1, 1), tb, q=(1, min(n, 3)))


@pytest.mark.parametrize("n,m,top,seed", [(12, 3, 40, 1), (20, 4, 400, 2), (30, 2, 3, 3), (26, 7, 100, 4)])
def test_local_search_on_matrices_of_shortcuts(vrp, n, m, top, seed):
    # independent legs of 0..top: for most gaps (x, y) and customers c,
    # d(x,c) + d(c,y) < d(x,y) or it ties
    rng = np.random.default_rng(seed)
    d = rng.integers(0, top + 1, size=(n + 1, n + 1)).astype(np.int32)
    p = rng.integers(0, 3 * top, size=n).astype(np.int32)
    inst = vrp.Instance(m, n, 4, p, d=d)
    oi = oracle.OracleInstance(d, p, m, n, 4)
    g = same(vrp, inst, oi, 10, seed, (1, 2), 6)
    assert g["stats"].fallback_entries > 0

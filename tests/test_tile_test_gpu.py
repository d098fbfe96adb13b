"""The matrix phase's first test of its tiles, on teams with fewer CTAs than
tiles: tile counts around a byte and a word of the mask, one CTA for all of
them, more groups of eight than CTAs, all customers removed at once, every
repair rule's bound, and shortcut gaps enough that the simulating CTAs leave
too few to test (then every tile runs).  Whole runs equal to the oracle's, step
by step (whole numbers, no tolerance)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def same(vrp, inst, oi, iters, seed, tb, q, mask, dmask):
    init = vrp.initial_solution(inst)
    g = vrp.alns_run(inst, vrp.alns_params(iters, *q, mask, tb, destroy_mask=dmask), seed=seed, init=init)
    o = oracle.alns_run(oi, init[0], init[1], oracle.alns_params(iters, *q, mask, destroy_mask=dmask), seed)
    assert np.array_equal(g["trace"], o["trace"]), np.argwhere(g["trace"] != o["trace"])[:3]
    assert np.array_equal(g["cur_ops"], o["cur_ops"]) and np.array_equal(g["cur_off"], o["cur_off"])
    assert np.array_equal(g["best_ops"], o["best_ops"]) and np.array_equal(g["best_off"], o["best_off"])
    return g["stats"]


# 2n + m gaps (less the removed customers') give 2 x 1, 3 x 2, 4 x 2 (a byte), 5 x 3, 8 x 4 (a word), 9 x 5 tiles
@pytest.mark.parametrize("n,m,tb", [(18, 2, 1), (40, 6, 2), (60, 7, 1), (66, 3, 5), (126, 5, 2), (131, 12, 1)])
@pytest.mark.parametrize("mask", [1, 2, 4, 8])
def test_tile_counts_and_repair_rules(vrp, n, m, tb, mask):
    w = workloads.make_instance(n, m, 4 * m, 4, "5x" if n % 4 else "2x", "clustered", seed=n)
    inst = vrp.Instance.from_workload(w)
    oi = oracle.OracleInstance.from_workload(w)
    st = same(vrp, inst, oi, 2 if n < 100 else 1, n + tb, tb, (2, 3), mask, 1)
    assert st.matrix_entries >= st.pruned_entries and st.tiles >= st.tiles_pruned


@pytest.mark.parametrize("mask", [1, 2, 4, 8])
def test_all_customers_out(vrp, mask):
    w = workloads.make_instance(20, 4, 12, 4, "2x", "clustered", seed=5)
    inst = vrp.Instance.from_workload(w)
    oi = oracle.OracleInstance.from_workload(w)
    same(vrp, inst, oi, 2, 4, 1, (20, 20), mask, 1)


@pytest.mark.parametrize("n,m,top,tb", [(40, 3, 40, 2), (70, 5, 400, 9), (50, 2, 3, 8)])
@pytest.mark.parametrize("mask", [1, 6])
def test_matrices_of_shortcuts(vrp, n, m, top, tb, mask):
    rng = np.random.default_rng(n)
    d = rng.integers(0, top + 1, size=(n + 1, n + 1)).astype(np.int32)
    p = rng.integers(0, 3 * top, size=n).astype(np.int32)
    inst = vrp.Instance(m, n, 4, p, d=d)
    oi = oracle.OracleInstance(d, p, m, n, 4)
    st = same(vrp, inst, oi, 2, 7, tb, (1, 2), mask, 63)
    assert st.fallback_entries > 0

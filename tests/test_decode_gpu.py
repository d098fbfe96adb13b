"""The decoder where its sort, list chunks and vehicle selection change form:
op counts around the sort's sizes (in registers up to 1024, in shared memory
beyond), lists of one entry more or less than a chunk, one and 32 vehicles,
many passes (Q = 1, R = 1), times too long for the packed key, equal keys, and
each source of distances.  Equal to the oracle (whole numbers, no tolerance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def check(vrp, n, m, R, Q, layout, keys, coords=None, d=None, p=None, full=False):
    import torch
    inst = vrp.Instance(m, R, Q, p, coords=coords, d=d, load_full=full)
    oi = oracle.OracleInstance(inst.dist(), p, m, R, Q, load_full=full)
    ops, off, z, un, fit = (t.cpu().numpy() for t in vrp.brkga_decode(inst, torch.from_numpy(keys).cuda(), layout))
    for k in range(len(keys)):
        oo, of, zo, uo, fo = oracle.decode(oi, keys[k], layout)
        done = int(of[m])
        assert (z[k], un[k], fit[k]) == (zo, uo, fo) and np.array_equal(off[k], of), k
        assert np.array_equal(ops[k][:done], oo[:done]), k


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("n,m,R,Q", [(1, 1, 1, 1), (2, 32, 3, 1), (15, 3, 1, 1), (16, 2, 4, 4), (17, 4, 2, 1), (32, 5, 8, 2),
                                     (33, 1, 3, 3), (64, 7, 1, 1), (65, 31, 65, 2), (129, 6, 9, 9), (257, 12, 26, 10),
                                     (512, 4, 20, 6), (513, 20, 52, 10)])
def test_decode_edges(vrp, n, m, R, Q, layout):
    rng = np.random.default_rng(n + m)
    coords = rng.integers(0, 1001, size=(n + 1, 2)).astype(np.int32)
    p = rng.integers(0, 300, size=n).astype(np.int32)
    L = 4 * n if layout else 2 * n + m
    keys = rng.random((5, L)).astype(np.float32)
    keys[1] = np.round(keys[1] * 4) / 4          # few distinct keys: ties by op and by vehicle
    keys[2] = 0.0
    keys[3, 0:2 * n:2] *= 0.25                   # drops first
    check(vrp, n, m, R, Q, layout, keys, coords=coords, p=p, full=n % 3 == 0)


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("top,pmax", [(60000, 1 << 20), (500000, 1 << 16), (30, 5)])
def test_decode_long_times(vrp, top, pmax, layout):
    # explicit matrices: 16-bit and 32-bit distances, and schedule times from 2^22 on
    n, m = 40, 6
    rng = np.random.default_rng(top)
    d = rng.integers(0, top + 1, size=(n + 1, n + 1)).astype(np.int32)
    p = rng.integers(0, pmax + 1, size=n).astype(np.int32)
    keys = rng.random((6, 4 * n if layout else 2 * n + m)).astype(np.float32)
    check(vrp, n, m, 8, 3, layout, keys, d=d, p=p)


@pytest.mark.parametrize("pop,layout", [(2, 0), (63, 1), (65, 0), (2049, 1)])
def test_generations_over_ranking_tiles(vrp, pop, layout):
    # populations around the ranking's element groups and key tile: the last
    # population and every generation's best equal the oracle's
    import workloads
    w = workloads.make_instance(9, 2, 3, 2, "2x", seed=pop)
    inst = vrp.Instance.from_workload(w)
    oi = oracle.OracleInstance.from_workload(w)
    g = vrp.brkga_run(inst, vrp.brkga_params(pop, 3, layout=layout), seed=5, final_keys=True)
    o = oracle.brkga_run(oi, oracle.brkga_params(pop, 3, layout=layout), None, None, 5)
    assert np.array_equal(g["trace"], o["trace"]) and g["best_fitness"] == o["best_fitness"]
    assert np.array_equal(g["keys"].cpu().numpy().view(np.uint32), o["keys"].view(np.uint32))
    assert np.array_equal(g["best_ops"], o["best_ops"])

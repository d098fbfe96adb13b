"""Default shapes where distances are gathered from L2 (an explicit matrix, or
points too far apart, too large for shared memory) and of the coordination
counts: results by the oracle whatever the batch size makes of the shape, and no
shape whose shared memory or second row costs more than its lanes give."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def instance(vrp, n, m, form):
    rng = np.random.default_rng(n + m)
    p = rng.integers(0, 300, size=n).astype(np.int32)
    if form == "wide":
        coords = rng.integers(0, 40000, size=(n + 1, 2)).astype(np.int32)
        return vrp.Instance(m, n, 8, p, coords=coords), oracle.OracleInstance(oracle.euc2d(coords), p, m, n, 8)
    d = rng.integers(0, 900 if form == "d16" else 100000, size=(n + 1, n + 1)).astype(np.int32)
    return vrp.Instance(m, n, 8, p, d=d), oracle.OracleInstance(d, p, m, n, 8)


# few and many routes, the sizes where the tile, the block or the routes per lane change
@pytest.mark.parametrize("n,m,form", [(240, 2, "d32"), (350, 5, "d16"), (300, 8, "d32"), (550, 12, "d16"),
                                      (500, 20, "d32"), (500, 20, "wide"), (700, 32, "d16"), (2047, 17, "d32")])
def test_results_whatever_the_shape(vrp, n, m, form):
    inst, oi = instance(vrp, n, m, form)
    po, pf = workloads.precedence_candidates(n, m, 24, seed=1)
    ro, rf = workloads.random_candidates(n, m, 16, seed=2)
    ops, off = np.concatenate([po, ro]), np.concatenate([pf, rf])
    ops[3, 5] = ops[3, 9]
    ops[30, 0] = 2 * n + 2
    zo, so = oracle.evaluate_batch(oi, ops, off, threads=8)
    counts = np.array([oracle.coordination(oi, o, f)[:2] for o, f in zip(ops, off)])
    for num in (1, 40, 700, 9000):
        if num * n > 4000000:
            continue
        ix = np.arange(num) % len(ops)
        to, tf = dev(ops[ix]), dev(off[ix])
        z, st = vrp.evaluate(inst, to, tf)
        cr, il = vrp.coordination(inst, to, tf)
        vrp.sync(inst)
        assert np.array_equal(z.cpu().numpy(), zo[ix]) and np.array_equal(st.cpu().numpy().astype(np.uint32), so[ix])
        assert np.array_equal(cr.cpu().numpy(), counts[ix, 0]) and np.array_equal(il.cpu().numpy(), counts[ix, 1])


# 20 of 32 lanes with one route each, 60 of 64 with two: two routes lose to the
# L1 that their tiles' shared memory takes
@pytest.mark.parametrize("form", ["d16", "d32", "wide"])
def test_one_route_per_lane_where_the_l1_counts(vrp, form):
    inst, _ = instance(vrp, 500, 20, form)
    cfg = vrp.get_eval_config(inst)
    assert cfg["dist_mode"] == ("global32" if form == "d32" else "global16")
    assert cfg["walk"] == "staged"

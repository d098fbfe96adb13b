"""Malformed candidates whose walk comes to its end: every sequence of codes at
the smallest sizes, in every distance form and with one and two routes per lane,
against the oracle (whole numbers, no tolerance)."""
import itertools

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(mode, walk, gw) for mode in ("smem32", "smem16", "global16", "global32", "coords")
          for walk, gw in (("staged", 1), ("streamed", 1), ("streamed", 2))]


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def same(z, st, zo, so):
    return np.array_equal(z.cpu().numpy(), zo) and np.array_equal(st.cpu().numpy().astype(np.uint32), so)


def check(vrp, ops, cuts, p, coords=None, d=None, full=False):
    """Every candidate in ops with every row of cuts, by every entry point and shape."""
    cuts = np.asarray(cuts, np.int32)
    m, n, p = cuts.shape[1] - 1, len(p), np.asarray(p, np.int32)
    off = np.repeat(cuts, len(ops), axis=0)
    ops = np.tile(np.asarray(ops, np.int32), (len(cuts), 1))
    inst = vrp.Instance(m, n, 2, p, coords=coords, d=d, load_full=full)
    d = oracle.euc2d(np.asarray(coords, np.int32)) if d is None else d
    oi = oracle.OracleInstance(d, p, m, n, 2, load_full=full)
    zo, so = oracle.evaluate_batch(oi, ops, off, threads=8)
    assert same(*vrp.evaluate_plain(inst, dev(ops), dev(off)), zo, so)
    to, tf = dev(ops), dev(off)
    assert same(*vrp.evaluate(inst, to, tf), zo, so)
    if ops.min() >= 0:
        assert same(*vrp.evaluate(inst, to.short(), tf.short()), zo, so)
    cross, inter = (t.cpu().numpy() for t in vrp.coordination(inst, to, tf))
    assert np.array_equal(cross == -1, so == vrp.MALFORMED)
    assert np.array_equal(inter == -1, (so & (vrp.MALFORMED | vrp.CYCLE)) != 0)
    mb = vrp.MultiBatch([(inst, to, tf)])
    assert same(*(t[0] for t in mb.evaluate()), zo, so)
    wide = coords is None or int((np.ptp(coords, axis=0).astype(np.int64) ** 2).sum()) >= 1 << 24
    big = d.max() >= 1 << 16
    for mode, walk, gw in SHAPES:
        if (mode == "coords" and wide) or (mode.endswith("16") and big):
            continue
        vrp.set_eval_config(inst, mode, 4, walk=walk, group_warps=gw)
        assert same(*vrp.evaluate(inst, to, tf), zo, so), (mode, walk, gw)
        if mode.startswith("global") and gw == 1:
            mb.set_config(mode, 4, walk)
            assert same(*(t[0] for t in mb.evaluate()), zo, so), ("multi", mode, walk)
    vrp.sync(inst)
    return zo, so


def sequences(codes, length):
    return np.array(list(itertools.product(codes, repeat=length)), np.int32)


# A drop of a customer already picked up must leave no slot that a pickup takes, or
# that a drop with travel plus processing time of 1 turns into "picked up".
def test_repeated_drop_behind_its_pickup(vrp):
    zo, so = check(vrp, [[2, 3, 2, 3, 4, 6]], [[0, 6]], [0, 1, 1], coords=np.zeros((4, 2), np.int32))
    assert so[0] == vrp.MALFORMED
    # the same in the integer-leg and the matrix forms: customer 4 far away, on its own
    for far in (3000, 70000):
        coords = np.array([[0, 0]] * 4 + [[far, 0]], np.int32)
        check(vrp, [[2, 3, 2, 3, 4, 6, 8, 9], [2, 3, 2, 3, 6, 4, 8, 9], [8, 9, 2, 3, 2, 3, 4, 6]],
              [[0, 6, 8], [0, 8, 8], [0, 2, 8]], [0, 1, 1, 0], coords=coords)


@pytest.mark.parametrize("p,leg,full", [((0, 1), 0, False), ((1, 0), 1, True), ((3, 2), 2, False)])
def test_all_sequences_of_two_customers(vrp, p, leg, full):
    coords = np.array([[0, 0], [leg, 0], [0, leg]], np.int32)
    ops = sequences(range(0, 8), 4)            # 0, 1, 6 and 7 are no op's code
    check(vrp, ops, [[0, 4]], p, coords=coords, full=full)
    check(vrp, ops, [[0, k, 4] for k in range(5)], p, coords=coords, full=full)


@pytest.mark.parametrize("p", [(0, 1, 1), (0, 0, 2), (2, 1, 0)])
def test_all_sequences_of_three_customers(vrp, p):
    ops = sequences(range(2, 8), 6)
    check(vrp, ops, [[0, 6]], p, coords=np.zeros((4, 2), np.int32))
    d = np.ones((4, 4), np.int32) - np.eye(4, dtype=np.int32)
    check(vrp, ops, [[0, 3, 6], [0, 2, 6]], p, d=d)


# the largest processing times an instance may have, where a slot not dropped yet
# comes closest to the word that means "picked up"
@pytest.mark.parametrize("p", [(2**31 - 2,), (2**31 - 3,), (2**31 - 4,), (2**30 - 1, 2**30 - 1)])
def test_largest_processing_times(vrp, p):
    n = len(p)
    ops = sequences(range(0, 2 * n + 4), 2 * n)
    zo, so = check(vrp, ops, [[0, 2 * n]], p, coords=np.zeros((n + 1, 2), np.int32))
    assert zo[so == 0].max() >= max(p)
    check(vrp, ops, [[0, k, 2 * n] for k in range(2 * n + 1)], p, d=np.zeros((n + 1, n + 1), np.int32))

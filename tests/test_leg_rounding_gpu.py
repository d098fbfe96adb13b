"""The evaluator's legs from fp16 points (the default where the points' box has a
squared diagonal below 2^21 - 2^12) where rounding is closest to a tie: squared
lengths r^2 + r, which round to r, and r^2 + r + 1, which round to r + 1."""
import math

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

LIMIT = 2**21 - 2**12


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def ties():
    """(dx, dy, rounded length) of every squared length r^2 + r and r^2 + r + 1 below the
    limit that is a sum of two squares, a few of its forms each."""
    out = []
    for r in range(1, math.isqrt(LIMIT) + 1):
        for s, want in ((r * r + r, r), (r * r + r + 1, r + 1)):
            if s >= LIMIT:
                continue
            forms = [(dx, math.isqrt(s - dx * dx)) for dx in range(math.isqrt(s // 2) + 1)
                     if math.isqrt(s - dx * dx) ** 2 == s - dx * dx]
            out += [(dx, dy, want) for dx, dy in forms[:1] + forms[-1:]]
    return sorted(set(out))


def test_every_near_tie(vrp):
    legs = ties()
    assert max(want for _, _, want in legs) >= 1440 and len(legs) > 500
    ops, off = dev(np.array([[2, 3]], np.int32)), dev(np.array([[0, 2]], np.int32))
    got = []
    for k, (dx, dy, want) in enumerate(legs):
        # the box anywhere, the leg in every direction
        base = np.array([[0, 0], [-700, 300], [(1 << 20) - 1448, -(1 << 20) + 1448], [17, -5]][k % 4], np.int32)
        far = base + np.array([[dx, dy], [-dx, dy], [dy, -dx], [-dy, -dx]][k // 4 % 4], np.int32)
        inst = vrp.Instance(1, 1, 1, np.zeros(1, np.int32), coords=np.array([base, far], np.int32))
        got.append(vrp.evaluate(inst, ops, off)[0])
    got = np.array([int(z[0]) for z in got])
    want = np.array([2 * w for _, _, w in legs])
    assert np.array_equal(got, want), [legs[i] for i in np.nonzero(got != want)[0][:10]]


# boxes whose squared diagonal is just below the limit: square, flat, upright
@pytest.mark.parametrize("w,h", [(1022, 1023), (1446, 40), (46, 1446), (1400, 364)])
def test_largest_boxes(vrp, w, h):
    assert w * w + h * h < LIMIT
    rng = np.random.default_rng(w)
    n, m = 300, 7
    coords = np.stack([rng.integers(0, w + 1, n + 1), rng.integers(0, h + 1, n + 1)], axis=1).astype(np.int32)
    coords[:4] = (0, 0), (w, h), (w, 0), (0, h)
    p = rng.integers(0, 40, n).astype(np.int32)
    inst = vrp.Instance(m, n, 4, p, coords=coords - 500)
    oi = oracle.OracleInstance(oracle.euc2d(coords), p, m, n, 4)
    po, pf = workloads.precedence_candidates(n, m, 600, seed=1)
    ro, rf = workloads.random_candidates(n, m, 200, seed=2)
    ops, off = np.concatenate([po, ro]), np.concatenate([pf, rf])
    zo, so = oracle.evaluate_batch(oi, ops, off, threads=8)
    z, st = vrp.evaluate(inst, dev(ops), dev(off))
    vrp.sync(inst)
    assert np.array_equal(z.cpu().numpy(), zo) and np.array_equal(st.cpu().numpy().astype(np.uint32), so)


# the largest n of the counting walk, and the next, which takes the kernel beside it
@pytest.mark.parametrize("n,m", [(2047, 20), (2047, 3), (2048, 20)])
def test_coordination_at_the_walks_limit(vrp, n, m):
    rng = np.random.default_rng(n + m)
    coords = rng.integers(0, 1000, size=(n + 1, 2)).astype(np.int32)
    p = rng.integers(0, 200, n).astype(np.int32)
    inst = vrp.Instance(m, n, 9, p, coords=coords)
    oi = oracle.OracleInstance(oracle.euc2d(coords), p, m, n, 9)
    po, pf = workloads.precedence_candidates(n, m, 6, seed=1)
    ro, rf = workloads.random_candidates(n, m, 4, seed=2)
    ops, off = np.concatenate([po, ro]), np.concatenate([pf, rf])
    ops[1, 7] = ops[1, 8]
    ops[7, 2] = 2 * n + 2
    cr, il = (t.cpu().numpy() for t in vrp.coordination(inst, dev(ops), dev(off)))
    for k in range(len(ops)):
        assert (cr[k], il[k]) == oracle.coordination(oi, ops[k], off[k])[:2], k

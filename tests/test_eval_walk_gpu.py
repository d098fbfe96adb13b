"""The evaluator's walk where its tiles, rows and chunks end: every result equal
to the plain GPU form's and the oracle's (whole numbers, no tolerance)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def population(n, m, count, seed):
    """Acyclic and random candidates, some with codes or offsets no candidate may have."""
    rng = np.random.default_rng(seed)
    po, pf = workloads.precedence_candidates(n, m, count, seed=seed)
    ro, rf = workloads.random_candidates(n, m, count, seed=seed + 1)
    ops, off = np.concatenate([po, ro]).copy(), np.concatenate([pf, rf]).copy()
    perm = rng.permutation(len(ops))
    ops, off = ops[perm], off[perm]
    odd = [0, 1, 2 * n + 2, 2 * n + 3, 4095, 65535, 65536 + 2, -1, 2**31 - 1, -2**31]
    for k in range(0, len(ops), 3):
        i = int(rng.integers(2 * n))
        ops[k, i] = ops[k, int(rng.integers(2 * n))] if k % 2 else odd[k // 3 % len(odd)]
    for k in range(1, len(ops), 7):
        off[k, int(rng.integers(m + 1))] += int(rng.integers(-2, 3))
    return ops, off


# row padding (n + 2 mod 4), one and two routes per lane, tiles of 1 to 32 candidates
@pytest.mark.parametrize("n,m", [(1, 1), (2, 3), (3, 2), (4, 1), (5, 32), (30, 11), (31, 12), (61, 17), (62, 21),
                                 (127, 16), (333, 5), (1001, 20), (2047, 32), (2046, 3)])
@pytest.mark.parametrize("box", [1000, 1447, 1500, 4000, 0])
def test_walk_edges(vrp, n, m, box):
    # box: points as fp16 pairs up to 1447, integer legs below 2^24, then the
    # matrix in memory; 0: an asymmetric matrix without points
    import torch
    if n > 1000 and box in (1500, 4000):
        pytest.skip("covered by the smaller sizes")
    rng = np.random.default_rng(n * 41 + m)
    full = bool(n % 2)
    p = rng.integers(0, 300, size=n).astype(np.int32)
    R, Q = max(1, n // 2), 3
    if box:
        coords = rng.integers(-box // 2, box - box // 2 + 1, size=(n + 1, 2)).astype(np.int32)
        if n > 1:
            coords[0], coords[1] = (-(box // 2), 0), (box - box // 2, 0)
        inst = vrp.Instance(m, R, Q, p, coords=coords, load_full=full)
        oi = oracle.OracleInstance(oracle.euc2d(coords), p, m, R, Q, load_full=full)
    else:
        d = rng.integers(0, 900, size=(n + 1, n + 1)).astype(np.int32)
        inst = vrp.Instance(m, R, Q, p, d=d, load_full=full)
        oi = oracle.OracleInstance(d, p, m, R, Q, load_full=full)
    count = 70 if n < 1000 else 12
    ops, off = population(n, m, count, seed=n + m + box)
    zo, so = oracle.evaluate_batch(oi, ops, off, threads=8)
    zp, sp = vrp.evaluate_plain(inst, dev(ops), dev(off))
    assert np.array_equal(zp.cpu().numpy(), zo) and np.array_equal(sp.cpu().numpy().astype(np.uint32), so)
    flat = torch.empty(ops.size + 8, dtype=torch.int32, device="cuda")
    per = 64 // m
    for walk, gw, shift, num in (("auto", 0, 0, len(ops)), ("auto", 0, 1, 1), ("staged", 1, 2, max(1, 32 // m)),
                                 ("staged", 1, 3, min(len(ops), 32 // m + 1)), ("streamed", 2, 1, min(len(ops), per + 1)),
                                 ("streamed", 2, 0, len(ops))):
        if walk == "auto":
            vrp.set_eval_config(inst, "auto")
        else:
            try:
                vrp.set_eval_config(inst, "coords" if 0 < box < 2800 else "global32", 2, walk=walk, group_warps=gw)
            except vrp.VrpError:
                continue
        # the codes from any 4-byte boundary on
        view = flat[shift:shift + num * 2 * n].view(num, 2 * n)
        view.copy_(dev(ops[:num]))
        z, st = vrp.evaluate(inst, view, dev(off[:num]))
        vrp.sync(inst)
        assert np.array_equal(z.cpu().numpy(), zo[:num]), (walk, shift, num)
        assert np.array_equal(st.cpu().numpy().astype(np.uint32), so[:num]), (walk, shift, num)
    # 16-bit codes where the values fit, from both 4-byte phases of a 16-byte chunk
    vrp.set_eval_config(inst, "auto")
    fits = ((ops >= 0) & (ops < 65536)).all(1) & ((off >= 0) & (off < 65536)).all(1)
    o16, f16 = ops[fits].astype(np.uint16).view(np.int16), off[fits].astype(np.uint16).view(np.int16)
    flat16 = torch.empty(o16.size + 16, dtype=torch.int16, device="cuda")
    for shift in (0, 2, 6):
        view = flat16[shift:shift + o16.size].view(len(o16), 2 * n)
        view.copy_(dev(o16))
        z, st = vrp.evaluate(inst, view, dev(f16))
        vrp.sync(inst)
        assert np.array_equal(z.cpu().numpy(), zo[fits]) and np.array_equal(st.cpu().numpy().astype(np.uint32), so[fits])


# one and two routes per lane, empty routes; p from 2^25 on takes the other kernel
@pytest.mark.parametrize("n,m,pmax", [(1, 1, 9), (3, 2, 9), (5, 32, 50), (61, 17, 300), (62, 21, 300), (333, 5, 300),
                                      (20, 3, 1 << 25)])
def test_coordination_edges(vrp, n, m, pmax):
    rng = np.random.default_rng(n)
    p = rng.integers(0, pmax + 1, size=n).astype(np.int32)
    p[0] = pmax
    coords = rng.integers(0, 900, size=(n + 1, 2)).astype(np.int32)
    inst = vrp.Instance(m, n, 3, p, coords=coords)
    oi = oracle.OracleInstance(oracle.euc2d(coords), p, m, n, 3)
    ops, off = population(n, m, 60, seed=n + m)
    cr, il = vrp.coordination(inst, dev(ops), dev(off))
    cr, il = cr.cpu().numpy(), il.cpu().numpy()
    for k in range(len(ops)):
        assert (cr[k], il[k]) == oracle.coordination(oi, ops[k], off[k])[:2], k

"""Shapes of a many-instance plan: what the tuner returns can be set again, and
every shape gives the oracle's results (whole numbers, no tolerance)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def make(vrp, points, seed, box=900):
    """(items, expected) of uneven instances; blocked and malformed candidates among them."""
    import torch
    rng = np.random.default_rng(seed)
    items, expect = [], []
    for n, m in ((1, 1), (5, 3), (18, 11), (40, 20), (33, 32), (61, 17)):
        p = rng.integers(0, 60, size=n).astype(np.int32)
        coords = rng.integers(0, box, size=(n + 1, 2)).astype(np.int32)
        d = oracle.euc2d(coords) if points else rng.integers(0, box, size=(n + 1, n + 1)).astype(np.int32)
        inst = vrp.Instance(m, n, 3, p, coords=coords) if points else vrp.Instance(m, n, 3, p, d=d)
        po, pf = workloads.precedence_candidates(n, m, 45, seed=n)
        ro, rf = workloads.random_candidates(n, m, 38, seed=n)
        ops, off = np.concatenate([po, ro]), np.concatenate([pf, rf])
        for k in range(0, len(ops), 5):
            ops[k, int(rng.integers(2 * n))] = [2 * n + 2, 0, 1, 2, 2 * n + 1, -7][k % 6]
        items.append((inst, torch.from_numpy(ops).cuda(), torch.from_numpy(off).cuda()))
        expect.append(oracle.evaluate_batch(oracle.OracleInstance(d, p, m, n, 3), ops, off))
    return items, expect


def check(mb, expect, what):
    for z, s in zip(mb.z, mb.st):
        z.fill_(-5), s.fill_(-5)
    z, s = mb.evaluate()
    for (zo, so), zi, si in zip(expect, z, s):
        assert np.array_equal(zi.cpu().numpy(), zo), what
        assert np.array_equal(si.cpu().numpy().astype(np.uint32), so), what


# points as fp16 pairs; points too far apart for them; explicit matrices
@pytest.mark.parametrize("points,box", [(True, 900), (True, 5000), (False, 900), (False, 90000)])
def test_tuned_shape_can_be_set_again(vrp, points, box):
    items, expect = make(vrp, points, 3, box)
    mb = vrp.MultiBatch(items)
    check(mb, expect, "default")
    cfg = mb.autotune()
    check(mb, expect, cfg)
    again = vrp.MultiBatch(items)
    again.set_config(cfg["dist_mode"], cfg["warps_per_block"], cfg["walk"], cfg["group_warps"])
    check(again, expect, cfg)
    # a program that passes mode, warps and walk only
    again.set_config(cfg["dist_mode"], cfg["warps_per_block"], cfg["walk"])
    check(again, expect, cfg)


@pytest.mark.parametrize("points", [True, False])
def test_every_shape(vrp, points):
    items, expect = make(vrp, points, 4)
    mb = vrp.MultiBatch(items)
    for mode in ("coords", "global16", "global32"):
        for walk, gw in (("staged", 1), ("streamed", 1), ("streamed", 2)):
            for warps in (1, 4, 24):
                if mode == "coords" and not points:
                    with pytest.raises(vrp.VrpError):
                        mb.set_config(mode, warps, walk, gw)
                    continue
                mb.set_config(mode, warps, walk, gw)
                check(mb, expect, (mode, walk, gw, warps))
    for bad in (("smem16", 4, "staged", 1), ("smem32", 4, "staged", 1), ("auto", 4, "staged", 1),
                ("global16", 0, "staged", 1), ("global16", 33, "staged", 1), ("global16", 4, "streamed", 0),
                ("global16", 4, "streamed", 3)):
        with pytest.raises(vrp.VrpError):
            mb.set_config(*bad)
    check(mb, expect, "after refusals")

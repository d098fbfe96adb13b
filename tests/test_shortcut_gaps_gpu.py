"""Many shortcut gaps: matrices without the triangle inequality, where a gap's
simulations outnumber the tiles.  The sizes where more warps of a CTA simulate at
once (eight below n = 300, two from n = 1000 on), one CTA and many, few and more
than the simulated number of such gaps."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def make(vrp, n, m):
    rng = np.random.default_rng(n)
    d = rng.integers(1, 400, size=(n + 1, n + 1)).astype(np.int32)
    np.fill_diagonal(d, 0)
    p = rng.integers(0, 90, size=n).astype(np.int32)
    R, Q = max(m, n // 6), 3
    return vrp.Instance(m, R, Q, p, d=d), oracle.OracleInstance(d, p, m, R, Q)


def run(vrp, inst, init, n, iters, blocks):
    par = vrp.alns_params(iters, repair_mask=15, destroy_mask=63, team_blocks=blocks, q_min=min(2, n), q_max=min(6, n))
    return vrp.alns_run(inst, par, seed=n, init=init)


@pytest.mark.parametrize("n,m,blocks,iters", [(4, 1, 1, 12), (13, 2, 1, 12), (15, 3, 0, 12), (30, 32, 3, 6),
                                              (60, 4, 2, 3)])
def test_small_runs_by_the_oracle(vrp, n, m, blocks, iters):
    inst, oi = make(vrp, n, m)
    init = vrp.initial_solution(inst)
    g = run(vrp, inst, init, n, iters, blocks)
    assert g["stats"].fallback_entries > 0
    o = oracle.alns_run(oi, init[0], init[1], oracle.alns_params(iters, min(2, n), min(6, n), 15, 63), n)
    assert np.array_equal(g["trace"], o["trace"])
    assert np.array_equal(g["best_ops"], o["best_ops"]) and np.array_equal(g["best_off"], o["best_off"])
    assert oracle.evaluate(oi, g["best_ops"], g["best_off"]) == (g["z_best"], 0)
    assert np.array_equal(g["cur_ops"], o["cur_ops"]) and np.array_equal(g["cur_off"], o["cur_off"])


# the same run whatever the team: each share of the simulations differs
@pytest.mark.parametrize("n,m,iters", [(130, 6, 4), (299, 8, 2), (333, 9, 2), (420, 7, 2), (1000, 20, 1)])
def test_teams_agree(vrp, n, m, iters):
    inst, oi = make(vrp, n, m)
    init = vrp.initial_solution(inst)
    runs = [run(vrp, inst, init, n, iters, b) for b in (0, 40, 3)]
    for r in runs:
        assert r["stats"].fallback_entries == runs[0]["stats"].fallback_entries > 0
        assert np.array_equal(r["trace"], runs[0]["trace"])
        assert np.array_equal(r["cur_ops"], runs[0]["cur_ops"]) and np.array_equal(r["best_ops"], runs[0]["best_ops"])
        assert oracle.evaluate(oi, r["best_ops"], r["best_off"]) == (r["z_best"], 0)

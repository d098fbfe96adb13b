"""Counters of an ALNS run that describe the work and not its order: the same on
every run, with the relocation's bound (other CTAs lower it at their own pace)
at work."""
import pytest

import workloads

pytestmark = pytest.mark.gpu

FIXED = ("iterations", "accepted", "improved", "new_best", "matrix_entries", "fallback_entries", "incremental_steps",
         "full_steps", "ls_moves", "ls_new_best", "tiles")


@pytest.mark.parametrize("n,m,layout,blocks,replicas", [(60, 5, "clustered", 12, 2), (200, 8, "uniform", 0, 1),
                                                        (300, 20, "clustered", 0, 1)])
def test_counters_repeat(vrp, n, m, layout, blocks, replicas):
    w = workloads.make_instance(n, m, max(m, n // 10), 6, "2x", layout, seed=n)
    inst = vrp.Instance.from_workload(w)
    p = vrp.alns_params(12, team_blocks=blocks, destroy_mask=63, repair_mask=15, ls_pickup_every=3,
                        ls_relocate_every=2, replicas=replicas)
    runs = [vrp.alns_run(inst, p, seed=4) for _ in range(4)]
    first = runs[0]["stats"]
    assert first.matrix_entries > 0 and 0 <= first.pruned_entries <= first.matrix_entries
    for r in runs[1:]:
        assert r["z_best"] == runs[0]["z_best"]
        for name in FIXED:
            assert getattr(r["stats"], name) == getattr(first, name), name

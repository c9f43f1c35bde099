"""Refined partner lists where some particles moved too far and only their
groups and their partners' groups are walked again (sizes with more groups than
a walk has warps): states equal those of steps that walk at every evaluation
bit for bit, and the walks test fewer candidates than those, but more than a
run in which nobody moves far."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _impact():
    ps = wl.al_impact(seed=41, n_side=46)
    ps.params = replace(ps.params, tree_reuse=3, dt_fixed=3.0 * ps.h.min() / 64 / 7000.0)
    return ps


def _rings():
    # the left ring at rest, the right one crossing half its shell per step
    ps = wl.rings_2d(seed=42, dx=1 / 60, h=2.5 / 60)
    ps.v[:, : ps.n // 2] = 0.0
    ps.params = replace(ps.params, tree_reuse=2, dt_fixed=0.5 * ps.h[0] / 64 / 0.059)
    return ps


def _batch():
    ps = wl.batched_impacts(seed=43, ninst=10, nmin=8000, nmax=20000, with_flaws=False)
    ps.materials = [replace(m, damage=False) for m in ps.materials]
    ps.dmg = None
    ps.params = replace(ps.params, tree_reuse=2, dt_fixed=1.5 * ps.h[0] / 64 / 6000.0)
    return ps


@pytest.mark.parametrize("make", [_impact, _rings, _batch])
def test_partial_walks(make):
    from paper_1604_03290_gb300 import sph
    ps = make()
    assert ps.n > 75000
    prm = replace(ps.params, precision="mixed")
    res = {}
    for name, p, every in (("refined", prm, 0), ("walked", prm, 1), ("still", replace(prm, dt_fixed=1e-6 * prm.dt_fixed), 0)):
        ctx = sph.Context(ps.dim, ps.n, max_instances=max(ps.ninst, 1), max_neighbours=200)
        ctx.set_tuning(walk_every_eval=every)
        ds = sph.DeviceState(ps)
        ctx.profile(True)
        sph.step(ctx, ds, ps.materials, p, p.tree_reuse)
        res[name] = (ds.to_numpy(), ctx.profile_counters()["walk_tests"])
    a, b = res["refined"][0], res["walked"][0]
    for k in ("x", "v", "rho", "u", "S", "id"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    assert res["still"][1] < res["refined"][1] < 0.9 * res["walked"][1], {k: v[1] for k, v in res.items()}

"""A tree window continued over calls (params.tree_continue) while the walk's
mode changes between them (sph_tuning.walk_every_eval): the lists are refined
only where the window's lists and shells are those of its own build walk, so the
states equal those of walking at every evaluation bit for bit."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def moving_impact():
    ps = wl.al_impact(seed=51, n_side=20)
    ps.params = replace(ps.params, precision="mixed", tree_reuse=4, dt_fixed=3.0 * ps.h.min() / 64 / 7000.0)
    return ps


def run(ps, modes):
    from paper_1604_03290_gb300 import sph
    ctx = sph.Context(ps.dim, ps.n, max_neighbours=200)
    ds = sph.DeviceState(ps)
    for i, every in enumerate(modes):
        ctx.set_tuning(walk_every_eval=every)
        sph.step(ctx, ds, ps.materials, ps.params, 1, cont=i > 0)
    return ds.to_numpy()


@pytest.mark.parametrize("modes", [(0, 0, 0, 0), (0, 1, 0, 0), (0, 0, 1, 0), (1, 0, 0, 0), (1, 0, 1, 0, 0, 0)])
def test_mode_changes_inside_a_window(modes):
    ps = moving_impact()
    want, got = run(ps, (1,) * len(modes)), run(ps, modes)
    for k in ("x", "v", "rho", "u", "S", "id"):
        np.testing.assert_array_equal(got[k], want[k], err_msg=k)

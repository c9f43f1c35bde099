"""States that a call must answer with SPH_ERR_NONFINITE: the partner walk still
runs over them, and its lists name particles of the state only.  With an
infinite support radius every other particle is a partner (r^2 < inf), both
ways; a particle whose position is not a number has none."""
import ctypes
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def state(n, dim):
    rng = np.random.default_rng(n + dim)
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x, ps.h = rng.uniform(0.0, 1.0, (dim, n)), rng.uniform(0.2, 0.4, n)
    return ps


def lists(ps):
    """The CSR lists sph_neighbours leaves, whatever it answers."""
    import torch
    from paper_1604_03290_gb300 import sph
    ctx = sph.Context(ps.dim, ps.n, max_neighbours=ps.n)
    ds = sph.DeviceState(ps)
    off = torch.zeros(ps.n + 1, dtype=torch.int64, device="cuda")
    idx = torch.full((ps.n * ps.n,), -7, dtype=torch.int32, device="cuda")
    st = ds.struct()
    r = ctx._lib.sph_neighbours(ctx.h, ctypes.byref(st), 16, 21, sph._ptr(off), sph._ptr(idx), idx.numel(), sph._stream(None))
    assert r == sph.SPH_ERR_NONFINITE
    return off.cpu().numpy(), idx.cpu().numpy()


# candidate counts of every remainder by four, in one group and in several
@pytest.mark.parametrize("n", [5, 6, 7, 8, 30, 33, 70, 131])
@pytest.mark.parametrize("dim", [2, 3])
def test_infinite_support_radius(n, dim):
    ps = state(n, dim)
    ps.h[n // 2] = np.inf
    off, idx = lists(ps)
    d = ps.x[:, :, None] - ps.x[:, None, :]
    r2 = d[0] * d[0] + d[1] * d[1]
    r2 = r2 + d[2] * d[2] if dim == 3 else r2
    hab = 0.5 * (ps.h[:, None] + ps.h[None, :])
    near = r2 < hab * hab
    np.fill_diagonal(near, False)
    a, b = np.nonzero(near)
    np.testing.assert_array_equal(off, np.concatenate([[0], np.cumsum(near.sum(1))]))
    np.testing.assert_array_equal(idx[: off[-1]], b)


@pytest.mark.parametrize("n", [6, 7, 33, 70])
def test_position_not_a_number(n):
    ps = state(n, 3)
    k = n // 2
    ps.x[1, k] = np.nan
    off, idx = lists(ps)
    assert off[k + 1] == off[k]
    assert (idx[: off[-1]] >= 0).all() and (idx[: off[-1]] < n).all() and not (idx[: off[-1]] == k).any()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("what", ["h", "x"])
def test_steps_report_it_and_the_context_goes_on(prec, what):
    from paper_1604_03290_gb300 import sph
    ps = state(70, 3)
    prm = replace(ps.params, precision=prec, tree_reuse=2)
    ctx = sph.Context(3, ps.n, max_neighbours=ps.n)
    good = sph.DeviceState(ps)
    bad = sph.DeviceState(ps)
    if what == "h":
        bad.h[35] = np.inf
    else:
        bad.x[1, 35] = np.nan
    with pytest.raises(sph.SphError) as e:
        sph.step(ctx, bad, ps.materials, prm, 2)
    assert e.value.status == sph.SPH_ERR_NONFINITE
    with pytest.raises(sph.SphError) as e:
        c = sph.DeviceState(ps)
        c.h[35] = np.inf
        sph.adapt_h(ctx, c, 20.0, 2, 4)
    assert e.value.status == sph.SPH_ERR_NONFINITE
    sph.step(ctx, good, ps.materials, prm, 2)

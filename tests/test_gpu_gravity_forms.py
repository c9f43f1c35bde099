"""The mixed Barnes-Hut walk's instances (with and without the containment test
and the counters, packed and unpacked node words) accept the same sets and give
the same sums bit for bit: theta on both sides of D theta^2 = 1, 2D and 3D,
ragged chunks, several instances, coincident particles; the sums follow the
FP64 walk's."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,theta,leaf,parts", [
    (1, 3, 0.5, 16, 1), (31, 3, 0.5, 8, 1), (3001, 3, 0.5, 16, 1), (3001, 3, 0.8, 16, 1), (3001, 3, 0.5, 32, 4),
    (2050, 2, 0.65, 8, 1), (2050, 2, 0.75, 8, 3), (2050, 3, 0.0, 16, 1)])
def test_instances_agree(n, dim, theta, leaf, parts):
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(n + dim)
    x = rng.normal(size=(dim, n))
    if n > 2500:
        x[:, :50] = x[:, :1]
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x, ps.m, ps.h = x, rng.uniform(0.5, 1.5, n), rng.uniform(0.05, 0.2, n)
    if parts > 1:
        ps.inst_off = np.linspace(0, n, parts + 1).astype(np.int64)
    P = replace(ps.params, gravity=True, G=1.0, theta=theta, leaf_size=leaf, max_depth=18, precision="mixed")
    out = []
    for plain, count in ((0, False), (0, True), (1, False)):
        ctx = sph.Context(dim, n, max_instances=parts, max_neighbours=8, leaf_size=leaf)
        ctx.set_tuning(plain_forms=plain)
        ctx.profile(count)
        out.append(sph.gravity(ctx, sph.DeviceState(ps), P).cpu().numpy())
    np.testing.assert_array_equal(out[1], out[0])
    np.testing.assert_array_equal(out[2], out[0])
    ctx = sph.Context(dim, n, max_instances=parts, max_neighbours=8, leaf_size=leaf)
    ref = sph.gravity(ctx, sph.DeviceState(ps), replace(P, precision="fp64")).cpu().numpy()
    # FP32 terms of a few ulps each, compensated sums: far below 1e-4 of the largest sum
    assert np.abs(out[0] - ref).max() <= 1e-4 * max(np.abs(ref).max(), 1e-30)

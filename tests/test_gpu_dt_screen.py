"""The time-step reduction where the limiting derivative lies below the range of
its FP32 screening (2^-60): the step equals the oracle's over the same
derivatives.  Scales on both sides of 2^-60 = 8.7e-19, in one instance and with
instances that share blocks and warps."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("parts", [1, 9])
@pytest.mark.parametrize("scale", [1.0, 3e-18, 1e-18, 1e-20, 1e-28])
def test_limit_below_the_screen(orc, scale, parts, precision):
    from paper_1604_03290_gb300 import sph
    ps = wl.lattice_block(seed=7, nx=10, ny=9, nz=9)
    rng = np.random.default_rng(8)
    ps.v = 1e-3 * scale * rng.normal(size=ps.x.shape)
    if parts > 1:
        ps.inst_off = np.linspace(0, ps.n, parts + 1).astype(np.int64)
    prm = replace(ps.params, precision=precision, max_depth=18, S_floor=1e-6 * scale, u_floor=1e-9 * scale)
    ctx = sph.Context(3, ps.n, max_instances=parts, max_neighbours=200)
    ds = sph.DeviceState(ps)
    d = {k: v.cpu().numpy() for k, v in sph.rhs(ctx, ds, ps.materials, prm).items()}
    want = orc.timestep(ps, ps.materials, prm, d)
    courant = 0.5 * (prm.c_courant * ps.h / d["cs"]).min()
    assert want.max() < courant  # the strain rates limit
    got = sph.step(ctx, sph.DeviceState(ps), ps.materials, prm, 1).cpu().numpy()
    # the same FP64 expressions; FP32 sums of up to 200 terms in mixed precision
    np.testing.assert_allclose(got, want, rtol=1e-12 if precision == "fp64" else 1e-4)

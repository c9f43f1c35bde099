"""Pairs at the edge of the kernel's support in FP64.  Pairs of particles (an
instance each) one support radius apart, to a few roundings: q = r/h of a
partner (r^2 < h^2) may round above 1 there.  Its kernel value is 0, and so is
any power of it: the artificial stress with a non-integer exponent equals the
oracle's."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def edge_pairs(seed, n_as, npairs=12000):
    rng = np.random.default_rng(seed)
    n = 2 * npairs
    ps = wl.lattice_block(nx=n, ny=1, dim=2, jitter=0.0)
    h = rng.uniform(0.5, 2.0, npairs)
    ang = rng.uniform(0.0, 2.0 * np.pi, npairs)
    ps.x = np.zeros((2, n))
    ps.x[:, 1::2] = h * np.array([np.cos(ang), np.sin(ang)])
    ps.h = np.repeat(h, 2)
    ps.v = rng.normal(0.0, 0.1, (2, n))
    ps.rho = rng.uniform(0.9, 1.1, n)
    ps.S = rng.normal(0.0, 0.1, ps.S.shape)
    ps.inst_off = np.arange(0, n + 1, 2, dtype=np.int64)
    ps.params = replace(ps.params, eps_s=0.2, n_as=n_as, xsph=0.5, dmpd=0.3, max_depth=20)
    return ps


@pytest.mark.parametrize("n_as", [4.0, 4.5])
def test_artificial_stress_at_the_support_edge(n_as):
    import oracle
    from paper_1604_03290_gb300 import sph
    ps = edge_pairs(1, n_as)
    o = oracle.rhs(ps, ps.materials, ps.params)
    assert 0.2 < o["nnb"].mean() < 0.8  # about half of the pairs are partners
    ctx = sph.Context(2, ps.n, max_instances=ps.n // 2, max_neighbours=8)
    out = sph.rhs(ctx, sph.DeviceState(ps), ps.materials, ps.params)
    g = {k: v.cpu().numpy() for k, v in out.items()}
    np.testing.assert_array_equal(g["nnb"], o["nnb"])
    # 1 - q is at most eight roundings (2^-50) on either side, so that a pair's
    # kernel slope is at most 6 sigma / h^3 2^-100 = 7e-29, and its terms (V_b,
    # m_b, stresses and velocities of order one to ten) stay below 1e-26
    for f in ("drho", "dv", "du", "dS"):
        err = np.abs(g[f] - o[f])
        assert (err <= 1e-26).all(), (f, np.isnan(g[f]).sum(), np.nanmax(err))

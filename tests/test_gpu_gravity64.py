"""The FP64 Barnes-Hut walk where its lists and lane sharing can go wrong:
sizes with 8, 4 and 2 lanes per particle and ragged last chunks, leaves of one
and of 32 members, theta = 0 (every term a list entry), coincident particles
(leaves at full depth longer than 32), 2D and several instances (one lane per
particle), against the oracle's walk."""
import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _scale(x, m, h, P):
    """Per particle G sum_b m_b r_ab / (r_ab^2 + eps_a^2)^1.5, the magnitude of the direct sum."""
    out = np.empty(x.shape[1])
    for a in range(x.shape[1]):
        d = x - x[:, a:a + 1]
        r2 = (d ** 2).sum(0)
        q = r2 + (P.eps_grav * h[a]) ** 2
        q[a] = np.inf
        out[a] = P.G * (m * np.sqrt(r2) / q ** 1.5).sum()
    return out


@pytest.mark.parametrize("n,dim,theta,leaf,twins", [
    (1, 3, 0.5, 16, 0), (33, 3, 0.5, 1, 0), (1000, 3, 0.5, 32, 0), (1000, 3, 0.0, 16, 0), (777, 2, 0.6, 8, 0),
    (900, 3, 0.9, 16, 70), (20011, 3, 0.5, 16, 0)])
def test_against_oracle(n, dim, theta, leaf, twins):
    import oracle
    from dataclasses import replace
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(n)
    x = rng.normal(size=(dim, n))
    if twins:
        x[:, :twins] = x[:, :1]
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x, ps.m, ps.h = x, rng.uniform(0.5, 1.5, n), rng.uniform(0.05, 0.2, n)
    P = replace(ps.params, gravity=True, G=1.0, theta=theta, leaf_size=leaf, precision="fp64")
    ctx = sph.Context(dim, n, max_neighbours=8, leaf_size=leaf)
    g = sph.gravity(ctx, sph.DeviceState(ps), P).cpu().numpy()
    o = oracle.gravity_bh(ps.x, ps.m, ps.h, dim, P.G, P.theta, P.eps_grav, P.leaf_size, P.max_depth)
    err = np.abs(g - o[:dim]).max(0)
    # n roundings of the terms' magnitude at most, well below 1e-12 of it
    pick = slice(None) if n < 2000 else slice(0, n, 97)
    scale = _scale(ps.x, ps.m, ps.h, P)[pick] if n < 2000 else np.abs(o).max()
    assert (err[pick] <= 1e-12 * scale + 1e-300).all()


def test_instances():
    import oracle
    from dataclasses import replace
    from paper_1604_03290_gb300 import sph
    ps = wl.batched_impacts(seed=5, ninst=3, nmin=200, nmax=700, with_flaws=False)
    ps.materials = [replace(m, damage=False) for m in ps.materials]
    P = replace(ps.params, gravity=True, G=1.0, precision="fp64", max_depth=19)
    ctx = sph.Context(3, ps.n, max_instances=3, max_neighbours=8)
    g = sph.gravity(ctx, sph.DeviceState(ps), P).cpu().numpy()
    for k in range(3):
        s = slice(int(ps.inst_off[k]), int(ps.inst_off[k + 1]))
        o = oracle.gravity_bh(ps.x[:, s], ps.m[s], ps.h[s], 3, P.G, P.theta, P.eps_grav, P.leaf_size, P.max_depth)
        assert (np.abs(g[:, s] - o).max(0) <= 1e-12 * _scale(ps.x[:, s], ps.m[s], ps.h[s], P)).all()

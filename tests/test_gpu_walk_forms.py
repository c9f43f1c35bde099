"""The partner walk where its buffers and batches can go wrong: groups of one
particle, instances smaller than a group, smoothing lengths so large that a
group's ranges or the node stack overflow (the one-by-one walk) and so small
that nobody has a partner, coincident particles (leaves at full depth), 2D, and
single-particle leaves, against the oracle's lists."""
import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dim,h,leaf,twins", [
    (1, 3, 0.2, 16, 0), (31, 3, 0.3, 16, 0), (33, 3, 5.0, 1, 0), (65, 2, 0.3, 4, 0), (6000, 3, 0.02, 16, 0),
    (6000, 3, 0.12, 1, 0), (9000, 3, 0.6, 1, 0), (4000, 3, 2.0, 8, 0), (3000, 3, 0.1, 16, 100), (20011, 3, 0.07, 32, 0)])
def test_lists_match_oracle(n, dim, h, leaf, twins):
    import oracle
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(n)
    x = rng.uniform(0.0, 1.0, (dim, n))
    if twins:
        x[:, :twins] = x[:, :1]
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x, ps.h = x, h * rng.uniform(0.8, 1.2, n)
    roff, ridx = oracle.neighbours(ps.x, ps.h, dim)
    kmax = max(int(np.diff(roff).max()), 1)
    ctx = sph.Context(dim, n, max_neighbours=kmax, leaf_size=leaf)
    off, idx = sph.neighbours(ctx, sph.DeviceState(ps), leaf_size=leaf)
    np.testing.assert_array_equal(off.cpu().numpy(), roff)
    np.testing.assert_array_equal(idx.cpu().numpy(), ridx)


def test_small_instances():
    import oracle
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(2)
    sizes = [1, 2, 31, 32, 33, 400, 1, 7]
    n = sum(sizes)
    ps = wl.lattice_block(nx=n, ny=1, nz=1)
    ps.x, ps.h = rng.uniform(0.0, 1.0, (3, n)), rng.uniform(0.2, 0.4, n)
    ps.inst_off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    off, idx = sph.neighbours(sph.Context(3, n, max_instances=8, max_neighbours=400), sph.DeviceState(ps), max_depth=20)
    off, idx = off.cpu().numpy(), idx.cpu().numpy()
    for k in range(8):
        s0, s1 = ps.inst_off[k], ps.inst_off[k + 1]
        roff, ridx = oracle.neighbours(ps.x[:, s0:s1], ps.h[s0:s1], 3)
        np.testing.assert_array_equal(off[s0:s1 + 1] - off[s0], roff)
        np.testing.assert_array_equal(idx[off[s0]:off[s1]] - s0, ridx)


@pytest.mark.parametrize("h", [0.05, 0.3])
def test_lists_of_a_state_in_tree_order(h):
    """Lists already ascending (short) or longer than the shared-memory form."""
    import oracle
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(7)
    ps = wl.lattice_block(nx=3000, ny=1, nz=1)
    ps.x, ps.h = rng.uniform(0.0, 1.0, (3, 3000)), np.full(3000, h)
    ctx = sph.Context(3, 3000, max_neighbours=600)
    ds = sph.DeviceState(ps)
    sph.build_tree(ctx, ds, reorder=True)
    off, idx = sph.neighbours(ctx, ds)
    roff, ridx = oracle.neighbours(ds.x.cpu().numpy(), ps.h, 3)
    assert (np.diff(roff).max() > 128) == (h > 0.1)
    np.testing.assert_array_equal(off.cpu().numpy(), roff)
    np.testing.assert_array_equal(idx.cpu().numpy(), ridx)

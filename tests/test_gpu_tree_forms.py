"""The tree build's one-pass sort and scans at the edges of their tiles (256
slots, 2048 pairs, 4096 counts), with repeated keys (stability), in 2D and 3D
and with instances: the permutation equals numpy's stable sort of the keys,
and the nodes partition every level's particles."""
import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _keys(x, off, depth):
    """Cell indices floor((x - min) / s0 2^depth) interleaved below the instance number."""
    dim, n = x.shape
    key = np.zeros(n, dtype=object if dim * depth + len(off).bit_length() > 62 else np.int64)
    for k in range(len(off) - 1):
        p = x[:, off[k]:off[k + 1]]
        if p.shape[1] == 0:
            continue
        lo = p.min(1, keepdims=True)
        ext = (p.max(1) - p.min(1)).max()
        s0 = ext * (1.0 + 2.0 ** -20) if ext > 0 else 1.0
        c = np.clip(np.floor(((p - lo) / s0) * 2.0 ** depth), 0, 2 ** depth - 1).astype(np.int64)
        v = np.zeros(p.shape[1], np.int64)
        for b in range(depth):
            for ax in range(dim):
                v |= ((c[ax] >> b) & 1) << (dim * b + ax)
        key[off[k]:off[k + 1]] = v + (k << (dim * depth))
    return key


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1023, 1025, 2047, 2048, 2049, 4095, 4097, 16383, 16385, 70001])
@pytest.mark.parametrize("dim,parts,depth", [(3, 1, 20), (2, 1, 21), (3, 5, 18)])
def test_permutation_is_the_stable_sort(n, dim, parts, depth):
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(n + dim)
    x = np.round(rng.uniform(0.0, 1.0, (dim, n)) * 40) / 40 if n % 2 else rng.uniform(0.0, 1.0, (dim, n))
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x = np.ascontiguousarray(x)
    cuts = np.sort(rng.integers(0, n + 1, parts - 1))  # empty instances among them
    off = np.concatenate([[0], cuts, [n]]).astype(np.int64)
    if parts > 1:
        ps.inst_off = off
    ctx = sph.Context(dim, n, max_instances=parts, max_neighbours=4)
    ds = sph.DeviceState(ps)
    perm = sph.build_tree(ctx, ds, leaf_size=8, max_depth=depth).cpu().numpy()
    want = np.argsort(_keys(x, off, depth), kind="stable")
    np.testing.assert_array_equal(perm, want)
    nodes = sph.tree_nodes(ctx, 4 * n + 4096)
    lev, cnt = nodes["level"].cpu().numpy(), nodes["count"].cpu().numpy()
    assert cnt[lev == 0].sum() == n
    # reordering the state gives the same particles in tree order
    sph.build_tree(ctx, ds, leaf_size=8, max_depth=depth, reorder=True)
    np.testing.assert_array_equal(ds.id.cpu().numpy(), want)
    np.testing.assert_array_equal(ds.x.cpu().numpy(), x[:, want])


def _nodes(key, dim, depth, leaf, off):
    """(level, count) of every node in pre-order, cell by cell from the sorted keys."""
    out = []

    def cell(a, b, level):
        out.append((level, b - a))
        if b - a <= leaf or level == depth:
            return
        pre = key[a:b] >> (dim * (depth - level - 1))
        cuts = [a] + [a + 1 + int(c) for c in np.nonzero(pre[1:] != pre[:-1])[0]] + [b]
        for lo, hi in zip(cuts[:-1], cuts[1:]):
            cell(lo, hi, level + 1)

    for lo, hi in zip(off[:-1], off[1:]):
        if hi > lo:
            cell(int(lo), int(hi), 0)
    return np.array(out).T


@pytest.mark.parametrize("n,dim,leaf,parts,kind", [
    (1, 3, 16, 1, "uniform"), (17, 3, 16, 1, "uniform"), (5000, 3, 1, 1, "uniform"), (5000, 2, 2, 1, "uniform"),
    (20000, 3, 16, 1, "uniform"), (20000, 3, 32, 7, "uniform"), (20000, 2, 8, 3, "grid"), (20000, 3, 16, 1, "clusters"),
    (3000, 3, 16, 2, "twins"), (40, 3, 16, 1, "twins")])
def test_nodes_are_the_cells_that_split(n, dim, leaf, parts, kind):
    from paper_1604_03290_gb300 import sph
    rng = np.random.default_rng(n + leaf)
    x = rng.uniform(0.0, 1.0, (dim, n))
    if kind == "grid":
        x = np.round(30 * x) / 30
    if kind == "clusters":  # a long tail of nested cells
        x = x * 0.5 ** rng.integers(0, 14, n)
    if kind == "twins":  # full-depth leaves with more than `leaf` members
        x[:, : n // 2] = x[:, :1]
    depth = 17
    ps = wl.lattice_block(nx=n, ny=1, nz=1, dim=dim)
    ps.x = np.ascontiguousarray(x)
    off = np.linspace(0, n, parts + 1).astype(np.int64)
    if parts > 1:
        ps.inst_off = off
    ctx = sph.Context(dim, n, max_instances=parts, max_neighbours=4, leaf_size=leaf)
    sph.build_tree(ctx, sph.DeviceState(ps), leaf_size=leaf, max_depth=depth)
    nodes = sph.tree_nodes(ctx, 8 * n + 8192)
    want = _nodes(np.sort(_keys(x, off, depth).astype(np.int64)), dim, depth, leaf, off)
    np.testing.assert_array_equal(nodes["level"].cpu().numpy(), want[0])
    np.testing.assert_array_equal(nodes["count"].cpu().numpy(), want[1])

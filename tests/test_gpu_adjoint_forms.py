"""The FP64 adjoint of the right-hand side at sizes whose partner lists are
shared by 8, 4, 2 and 1 lanes, in 2D and 3D, with and without XSPH, against
torch's automatic differentiation of a plain FP64 right-hand side
(perf/cases.py) on the same partners.  A cotangent is a sum over about 60
partners of terms of some 20 roundings each, at most about a hundred times the
field's largest value in magnitude: 1e-11 of that value."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1604_03290_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
FIELDS = ("dxdt", "dv", "drho", "du", "dS")


@pytest.mark.parametrize("dim,side,xsph", [(3, 6, 0.5), (3, 13, 0.0), (3, 24, 0.5), (3, 31, 0.5), (2, 20, 0.5),
                                           (2, 200, 0.0)])
def test_against_autograd(dim, side, xsph):
    import torch
    from paper_1604_03290_gb300 import sph
    from perf import cases
    rng = np.random.default_rng(side + dim)
    ps = wl.lattice_block(seed=side, nx=side, ny=side, nz=side, dim=dim, jitter=0.2)
    n = ps.n
    ps.v, ps.rho = rng.normal(0, 0.05, (dim, n)), 1.0 + rng.normal(0, 0.03, n)
    ps.u, ps.S = rng.uniform(0, 0.1, n), rng.normal(0, 0.02, (ps.nsym, n))
    ps.h = ps.h * rng.uniform(0.9, 1.1, n)
    M = replace(ps.materials[0], Y0=0.05)
    P = replace(ps.params, xsph=xsph, precision="fp64")
    ctx = sph.Context(dim, n, max_neighbours=160)
    ds = sph.DeviceState(ps)
    dbar = sph.alloc_derivs(ds)
    for k in FIELDS:
        dbar[k].copy_(torch.as_tensor(rng.normal(size=dbar[k].shape)))
    sbar = ds.zeros_like()
    pbar = torch.zeros((1, 1, 3), dtype=torch.float64, device="cuda")
    sph.rhs_adjoint(ctx, ds, [M], P, dbar, sbar, pbar)
    q = {k: getattr(ds, k) for k in ("x", "v", "rho", "u", "S", "m", "h")}
    leaf = {k: q[k].clone().requires_grad_(True) for k in ("x", "v", "rho", "u", "S")}
    par = torch.tensor([M.mu, M.Y0, 1.0], dtype=torch.float64, device="cuda", requires_grad=True)
    out = cases._rhs({**q, **leaf}, M, P, cases._pairs(q["x"], q["h"], torch.zeros(n, dtype=torch.long, device="cuda")),
                     par=par)
    want = torch.autograd.grad([out[k] for k in FIELDS], list(leaf.values()) + [par], [dbar[k] for k in FIELDS],
                               allow_unused=True)
    for k, w in zip(leaf, want):
        if w is None:  # u does not enter this material's right-hand side
            assert not getattr(sbar, k).any()
            continue
        assert float((getattr(sbar, k) - w).abs().max()) <= 1e-11 * float(w.abs().max()), k
    assert torch.allclose(pbar[0, 0, :2], want[-1][:2], rtol=1e-11, atol=0.0)

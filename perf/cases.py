"""Performance cases: what a user of this framework has it do, over the range of
sizes, precisions and options in use.

A case is a dict of plain values.  ``prepare`` builds what a program holds
before the call (the particle set from ``workloads``, its device state and
context), ``run`` is one pass through the public entry points of ``sph``,
``exact`` the same outputs from plain FP64 torch operations, written from the
method's equations without this package's kernels.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_1604_03290_gb300 import sph
from paper_1604_03290_gb300 import workloads as wl

F64 = torch.float64

# ---------------------------------------------------------------------------
# The cases.  `set` and `size` name the particle set: rings (size = lattice
# points per 10 cm, 44 size^2 / 100 particles), impact / measurement (size^3
# target particles), cloud (particles), pair (particles per body), batch
# (instances of 2k to 50k particles).
# ---------------------------------------------------------------------------
RINGS = {"call": "step", "set": "rings", "precision": "fp64", "steps": 10, "tree_reuse": 0}
RK3 = {"call": "rk3", "set": "measurement", "precision": "fp64", "steps": 2}
IMPACT = {"call": "step", "set": "impact", "precision": "mixed", "steps": 2, "tree_reuse": 0}
WINDOW = {"call": "step", "set": "measurement", "precision": "mixed", "steps": 5, "tree_reuse": 5}
RHS64 = {"call": "rhs", "set": "measurement", "precision": "fp64"}
CLOUD = {"call": "step", "set": "cloud", "precision": "mixed", "steps": 1, "tree_reuse": 0}
GRAV64 = {"call": "gravity", "set": "cloud", "precision": "fp64"}
PAIR = {"call": "step", "set": "pair", "precision": "mixed", "steps": 4, "tree_reuse": 4}
BATCH = {"call": "step", "set": "batch", "precision": "mixed", "steps": 4, "tree_reuse": 4}
ADJ32 = {"call": "adjoint", "set": "solid", "precision": "mixed"}
ADJ64 = {"call": "adjoint", "set": "solid", "precision": "fp64"}
LISTS = {"call": "neighbours", "set": "impact", "precision": "fp64"}


def listed():
    return [
        # the paper's rubber-ring bounce (2D, artificial stress, XSPH) in the default precision: the smallest
        # simulation there is, stepped ten steps a call
        {"name": "rings_step_fp64_4k", "size": 10, **RINGS},
        # two embedded Runge-Kutta attempts of a small damaged solid in the default precision
        {"name": "rk3_fp64_14k", "size": 24, **RK3},
        # the aluminium impact at its set-up's 64^3 target, a tree per step, as sph.step is called by default
        {"name": "impact_step_mixed_263k", "size": 64, **IMPACT},
        # the benchmark: the 1M-particle impact with damage, one tree per five steps
        {"name": "measurement_window_mixed_1m", "size": 100, **WINDOW},
        # one right-hand side in the default precision
        {"name": "measurement_rhs_fp64_263k", "size": 64, **RHS64},
        # the largest: the self-gravitating collapse with two million particles, a tree per evaluation
        {"name": "cloud_step_mixed_2m", "size": 2000000, **CLOUD},
        # Barnes-Hut accelerations alone in the default precision
        {"name": "gravity_fp64_50k", "size": 50000, **GRAV64},
        # two self-gravitating bodies with damage on a reused tree
        {"name": "pair_window_mixed_400k", "size": 200000, **PAIR},
        # many small uneven impacts in one state
        {"name": "batch_window_mixed_64", "size": 64, **BATCH},
        # reverse mode of the right-hand side, as a gradient run calls it at every evaluation
        {"name": "adjoint_mixed_1m", "size": 100, **ADJ32},
        {"name": "adjoint_fp64_33k", "size": 32, **ADJ64},
        # partner lists as CSR for a program of the user's own
        {"name": "neighbours_263k", "size": 64, **LISTS},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    base, lo, hi = rng.choice([(RINGS, 10, 40), (RK3, 11, 40), (IMPACT, 17, 64), (WINDOW, 21, 100), (RHS64, 17, 64),
                               (CLOUD, 20000, 2000000), (GRAV64, 5000, 100000), (PAIR, 5000, 200000), (BATCH, 4, 64),
                               (ADJ32, 17, 100), (ADJ64, 13, 40), (LISTS, 13, 72)])
    return {"size": size(lo, hi), **base}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _particles(case, seed):
    """The particle set of a case and the partners its lists must hold."""
    s, size = case["set"], case["size"]
    if s == "rings":
        dx = 1.0 / size
        return wl.rings_2d(seed=seed, dx=dx, h=2.5 * dx, artificial_stress=True), 96
    if s == "impact":
        ps = wl.al_impact(seed=seed, n_side=size)
        if case["call"] == "neighbours":  # the lattice fixes every list: the seed sets where the numbering starts
            return ps.subset_order(np.roll(np.arange(ps.n), np.random.default_rng(seed).integers(ps.n))), 128
        return ps, 256
    if s == "measurement":
        return wl.measurement_1m(seed=seed, n_side=size), 256
    if s == "cloud":
        # the jitter decides how many of the lattice points stay inside the sphere: thinned to `size` of them
        ps = wl.cloud_collapse(seed=seed, n=int(1.06 * size))
        ps = ps.subset_order(np.sort(np.random.default_rng(seed).permutation(ps.n)[:size]))
        ps.id = np.arange(ps.n, dtype=np.int32)
        return ps, 128
    if s == "pair":
        return wl.ceres_pair(seed=seed, n_each=size), 192
    if s == "batch":
        # one set of target sizes per batch size; the seed draws the impact speeds, the jitter and the flaws
        ps = wl.batched_impacts(seed=5, ninst=size)
        rng = np.random.default_rng(seed)
        ps.x += rng.uniform(-1e-5, 1e-5, ps.x.shape)
        ps.v *= np.repeat(rng.uniform(0.7, 1.0, ps.ninst), np.diff(ps.inst_off))
        ps.flaw_seed = seed + 2000
        return ps, 192
    # a strained solid without damage (compressed, cold and hot states, some yielding), as gradients are taken of
    ps = wl.measurement_1m(seed=seed, n_side=size, damage=False)
    rng = np.random.default_rng(seed)
    ps.u = rng.uniform(0.0, 6e6, ps.n)
    ps.S = rng.normal(0.0, 0.4 * ps.materials[0].Y0, (6, ps.n))
    ps.params = replace(ps.params, alpha=1.0, beta=2.0, xsph=0.5)
    return ps, 160


def prepare(case, seed):
    ps, kmax = _particles(case, seed)
    prm = replace(ps.params, precision=case["precision"], tree_reuse=case.get("tree_reuse", 0))
    ctx = sph.Context(ps.dim, ps.n, max_instances=ps.ninst, max_neighbours=kmax, leaf_size=prm.leaf_size)
    sph.fill_flaws(ctx, ps)
    ds = sph.DeviceState(ps)
    st = {"case": case, "ctx": ctx, "ds": ds, "mats": ps.materials, "prm": prm}
    if case["call"] == "rk3":
        st["dt"] = torch.zeros(ds.ninst, dtype=F64, device="cuda")
        st["t"] = torch.zeros(ds.ninst, dtype=F64, device="cuda")
    if case["call"] == "rhs":
        st["out"] = sph.alloc_derivs(ds)
    if case["call"] == "adjoint":
        g = torch.Generator(device="cuda").manual_seed(seed)
        # cotangents of the size the state's derivatives have in one step, per field
        scale = {"dxdt": 1e-3, "dv": 1e-6, "drho": 1.0, "du": 1e-6, "dS": 1e-9}
        st["dbar"] = sph.alloc_derivs(ds)
        for k, c in scale.items():
            st["dbar"][k].normal_(generator=g).mul_(c)
        st["sbar"] = ds.zeros_like()
        st["pbar"] = torch.zeros((1, len(ps.materials), 3), dtype=F64, device="cuda")
    return st


def _fields(ds):
    out = {k: getattr(ds, k) for k in ("x", "v", "rho", "u", "S", "dmg") if getattr(ds, k) is not None}
    out["id"] = ds.id
    return out


def run(st):
    case, ctx, ds, mats, prm = st["case"], st["ctx"], st["ds"], st["mats"], st["prm"]
    call = case["call"]
    if call == "step":
        dt = sph.step(ctx, ds, mats, prm, case["steps"])
        return {**_fields(ds), "dt": dt}
    if call == "rk3":
        dt, t, err, acc = sph.step_rk3(ctx, ds, mats, prm, 1e-3, case["steps"], dt=st["dt"], t=st["t"])
        return {**_fields(ds), "dt": dt, "t": t, "err": err, "acc": acc}
    if call == "rhs":
        return sph.rhs(ctx, ds, mats, prm, out=st["out"])
    if call == "gravity":
        return {"a": sph.gravity(ctx, ds, prm)}
    if call == "neighbours":
        off, idx = sph.neighbours(ctx, ds, prm.leaf_size, prm.max_depth)
        return {"off": off, "idx": idx}
    bar, pbar = st["sbar"], st["pbar"]
    for t in (bar.x, bar.v, bar.rho, bar.u, bar.S, pbar):
        t.zero_()
    sph.rhs_adjoint(ctx, ds, mats, prm, st["dbar"], bar, pbar)
    return {"x": bar.x, "v": bar.v, "rho": bar.rho, "u": bar.u, "S": bar.S, "param": pbar}


# ---------------------------------------------------------------------------
# Work of one pass: the state in and the result out once, and the pair and
# interaction arithmetic
# ---------------------------------------------------------------------------
def work(case):
    s, size, call = case["set"], case["size"], case["call"]
    solid = s in ("impact", "measurement", "solid")
    n = {"rings": 44.0 * size ** 2, "cloud": float(size), "pair": 2.0 * size,
         "batch": 16.5e3 * size}.get(s, 1.0042 * size ** 3)
    pairs = {"rings": 19.6, "cloud": 50.0}.get(s, 54.6 if solid else 53.0) * n
    nd = 10 if s == "rings" else (10 if s == "cloud" else 17)  # doubles of a particle's state
    state = n * (8.0 * nd + 8.0)
    # operations: pass A about 75 and pass B about 85 per pair, 300 per particle for the constitutive update;
    # a Barnes-Hut interaction 25 (877 nodes and 354 members a particle at 2M, fewer levels below)
    rhs = 160.0 * pairs + 300.0 * n
    inter = 1231.0 * n * (math.log2(max(n, 64.0)) - 5.0) / 16.0
    if call == "gravity":
        return {"bytes": n * (40.0 + 24.0), "flops": 25.0 * inter}
    if call == "neighbours":
        return {"bytes": n * 40.0 + 4.0 * pairs, "flops": 9.0 * pairs}
    if call == "rhs":
        return {"bytes": state + n * (8.0 * 16 + 8.0), "flops": rhs}
    if call == "adjoint":
        return {"bytes": state + n * 8.0 * (14 + 14), "flops": rhs + 560.0 * pairs}
    evals = (3 if call == "rk3" else 2) * case["steps"]
    return {"bytes": 2.0 * state, "flops": evals * (rhs + (25.0 * inter if s in ("cloud", "pair") else 0.0) + 100.0 * n)}


# ---------------------------------------------------------------------------
# FP64 reference in plain torch
# ---------------------------------------------------------------------------
def _sym(dim):
    return [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)] if dim == 3 else [(0, 0), (1, 1), (0, 1)]


def _spread(v, dim):
    """Bits of v moved dim places apart."""
    r = torch.zeros_like(v)
    for b in range(21):
        r |= ((v >> b) & 1) << (dim * b)
    return r


class _Cells:
    """Root cubes of the instances and the Morton keys in them (Sect. 3.5.1)."""

    def __init__(self, x, inst, ninst, depth):
        self.depth, self.dim = depth, x.shape[0]
        lo = torch.stack([torch.full((ninst,), math.inf, dtype=F64, device=x.device).scatter_reduce_(
            0, inst, c, "amin") for c in x])
        hi = torch.stack([torch.full((ninst,), -math.inf, dtype=F64, device=x.device).scatter_reduce_(
            0, inst, c, "amax") for c in x])
        s0 = (hi - lo).amax(0) * (1.0 + 2.0 ** -20)
        self.lo, self.s0 = lo, torch.where(s0 > 0, s0, torch.ones_like(s0))

    def keys(self, x, inst):
        top = 2 ** self.depth
        k = (((x - self.lo[:, inst]) / self.s0[inst]) * float(top)).floor().clamp(0, top - 1).long()
        key = inst << (self.dim * self.depth)
        for ax in range(self.dim):
            key = key | (_spread(k[ax], self.dim) << ax)
        return key


def _pairs(x, h, inst):
    """Partners (i, j) of every particle: r_ab^2 < h_ab^2 within an instance, sorted by i."""
    dim, n = x.shape
    edge = h.max() * (1.0 + 1e-9)
    c = ((x - x.amin(1, keepdim=True)) / edge).floor().long() + 1
    size = c.amax(1) + 2
    mul = [1, int(size[0]), int(size[0] * size[1])]
    key = inst * int(size.prod())
    for ax in range(dim):
        key = key + c[ax] * mul[ax]
    skey, order = torch.sort(key)
    out_i, out_j = [], []
    step = max(1, min(n, 4 << 20))
    side = range(-1, 2)
    for off in [(a, b, d) for d in (side if dim == 3 else (0,)) for b in side for a in side]:
        want = key + sum(off[ax] * mul[ax] for ax in range(dim))
        a0, a1 = torch.searchsorted(skey, want), torch.searchsorted(skey, want, right=True)
        for s in range(0, n, step):
            cnt = (a1 - a0)[s:s + step]
            i = torch.repeat_interleave(torch.arange(s, s + cnt.numel(), device=x.device), cnt)
            first = torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
            j = order[a0[i] + torch.arange(i.numel(), device=x.device) - first]
            r2 = torch.zeros_like(x[0, i])
            for ax in range(dim):
                d = x[ax, i] - x[ax, j]
                r2 = r2 + d * d
            hab = 0.5 * (h[i] + h[j])
            ok = (r2 < hab * hab) & (i != j)
            out_i.append(i[ok])
            out_j.append(j[ok])
    i, j = torch.cat(out_i), torch.cat(out_j)
    i, o = torch.sort(i, stable=True)
    return i, j[o]


def _kernel(q, hab, dim):
    """W and dW/dr of the cubic spline with support radius hab (Sect. 3.1.1)."""
    sig = (8.0 / math.pi if dim == 3 else 40.0 / (7.0 * math.pi)) / hab ** dim
    w = torch.where(q < 0.5, 6 * q ** 3 - 6 * q ** 2 + 1, 2 * (1 - q).clamp(min=0) ** 3)
    dw = torch.where(q < 0.5, 3 * q ** 2 - 2 * q, -(1 - q).clamp(min=0) ** 2)
    return sig * w, 6 * sig / hab * dw


def _eos(M, rho, u, scale):
    """Pressure and sound speed (Sect. 2.5); scale multiplies the bulk constants."""
    if M.eos == "isothermal":
        return M.cs ** 2 * rho, torch.full_like(rho, M.cs)
    if M.eos == "linear":
        p = M.cs ** 2 * (rho - M.rho0)
        return torch.where(rho / M.rho0 < M.rho_cut, torch.zeros_like(p), p), torch.full_like(rho, M.cs)
    A, B, a, b, E0, r0 = M.A_T * scale, M.B_T * scale, M.a_T, M.b_T, M.E0, M.rho0
    chi = (rho - r0) / r0
    eta = 1 + chi
    w = 1 + u / (E0 * eta ** 2)
    wr, wu = -2 * u / (E0 * eta ** 3 * r0), 1 / (E0 * eta ** 2)
    kc = a + b / w
    pc = kc * rho * u + A * chi + B * chi ** 2
    pcr = kc * u - b / w ** 2 * wr * rho * u + (A + 2 * B * chi) / r0
    pcu = kc * rho - b / w ** 2 * wu * rho * u
    low = rho <= 1e-3 * r0
    z = torch.where(low, torch.full_like(chi, 999.0), -chi / eta)
    dz = torch.where(low, torch.zeros_like(chi), -r0 / rho ** 2)
    eb, ea = torch.exp(-M.beta_T * z), torch.exp(-M.alpha_T * z * z)
    X = b * rho * u / w + A * chi * eb
    dX = b * u / w - b * rho * u / w ** 2 * wr + A / r0 * eb - A * chi * eb * M.beta_T * dz
    pe = a * rho * u + X * ea
    per = a * u + dX * ea - X * ea * 2 * M.alpha_T * z * dz
    peu = a * rho + (b * rho / w - b * rho * u / w ** 2 * wu) * ea
    f = ((u - M.E_iv) / (M.E_cv - M.E_iv)).clamp(0.0, 1.0)  # 0: cold branch, 1: fully expanded
    df = torch.where((u > M.E_iv) & (u < M.E_cv), (pe - pc) / (M.E_cv - M.E_iv), torch.zeros_like(u))
    cold = (chi >= 0) | (u <= M.E_iv)
    p = torch.where(cold, pc, f * pe + (1 - f) * pc)
    pr = torch.where(cold, pcr, f * per + (1 - f) * pcr)
    pu = torch.where(cold, pcu, f * peu + (1 - f) * pcu + df)
    c2 = pr + p / rho ** 2 * pu
    cmin = A / r0 + torch.zeros_like(c2)
    return p, torch.sqrt(torch.where(c2 > cmin, c2, cmin))


def _mat3(S, dim):
    """(n, D, D) from symmetric components."""
    M = [[None] * dim for _ in range(dim)]
    for k, (i, j) in enumerate(_sym(dim)):
        M[i][j] = M[j][i] = S[k]
    return torch.stack([torch.stack(r, -1) for r in M], -2)


def _eigen(S, dim):
    """Eigenvalues (D, n) and eigenvectors (D, D, n; columns) of symmetric components, by cyclic Jacobi rotations."""
    A = [[None] * dim for _ in range(dim)]
    for k, (i, j) in enumerate(_sym(dim)):
        A[i][j] = A[j][i] = S[k]
    one, zero = torch.ones_like(S[0]), torch.zeros_like(S[0])
    V = [[one if i == j else zero for j in range(dim)] for i in range(dim)]
    for _ in range(1 if dim == 2 else 7):
        for p, q in ((0, 1),) if dim == 2 else ((0, 1), (0, 2), (1, 2)):
            apq = A[p][q]
            tau = (A[q][q] - A[p][p]) / (2 * torch.where(apq == 0, one, apq))
            t = torch.where(tau >= 0, one, -one) / (tau.abs() + torch.sqrt(1 + tau * tau))
            t = torch.where(apq == 0, zero, t)
            c = 1 / torch.sqrt(1 + t * t)
            s = t * c
            A[p][p], A[q][q], A[p][q], A[q][p] = A[p][p] - t * apq, A[q][q] + t * apq, zero, zero
            for r in range(dim):
                if r not in (p, q):
                    A[r][p], A[r][q] = c * A[r][p] - s * A[r][q], s * A[r][p] + c * A[r][q]
                    A[p][r], A[q][r] = A[r][p], A[r][q]
                V[r][p], V[r][q] = c * V[r][p] - s * V[r][q], s * V[r][p] + c * V[r][q]
    return torch.stack([A[k][k] for k in range(dim)]), torch.stack([torch.stack(r) for r in V])


def _inverse(L):
    """Inverse and determinant of L[a][b] (rows of n-vectors), by cofactors."""
    if len(L) == 2:
        det = L[0][0] * L[1][1] - L[0][1] * L[1][0]
        return [[L[1][1] / det, -L[0][1] / det], [-L[1][0] / det, L[0][0] / det]], det
    cof = [[L[(a + 1) % 3][(b + 1) % 3] * L[(a + 2) % 3][(b + 2) % 3] -
            L[(a + 1) % 3][(b + 2) % 3] * L[(a + 2) % 3][(b + 1) % 3] for b in range(3)] for a in range(3)]
    det = sum(L[0][b] * cof[0][b] for b in range(3))
    return [[cof[b][a] / det for b in range(3)] for a in range(3)], det


def _yield(S, M, Y0):
    """f_Y of symmetric components S (Sect. 2.6)."""
    dim = 3 if S.shape[0] == 6 else 2
    J2 = 0.5 * (S[:dim] ** 2).sum(0) + (S[dim:] ** 2).sum(0)
    return torch.where(Y0 ** 2 < 3 * J2, Y0 ** 2 / (3 * J2).clamp(min=1e-300), torch.ones_like(J2))


def _rhs(q, M, P, pairs, par=None, ag=None):
    """The right-hand side (Sects. 2.4 to 3.2) of state q on the partners given."""
    i, j = pairs
    dim, n = q["x"].shape
    mu, Y0, scale = (M.mu, M.Y0, 1.0) if par is None else par
    gather = lambda t, k: t.index_select(-1, k)  # noqa: E731
    total = lambda t: torch.zeros(t.shape[:-1] + (n,), dtype=F64, device=t.device).index_add(-1, i, t)  # noqa: E731
    x, v, h, m, u = q["x"], q["v"], q["h"], q["m"], q["u"]
    d, w = gather(x, i) - gather(x, j), gather(v, i) - gather(v, j)
    hab = 0.5 * (h[i] + h[j])
    r = torch.sqrt((d * d).sum(0))
    W, dW = _kernel(r / hab, hab, dim)
    g = dW / r * d
    cnt = torch.bincount(i, minlength=n)
    rho = q["rho"]
    if P.density_sum:
        W0 = (8.0 / math.pi if dim == 3 else 40.0 / (7.0 * math.pi)) / h ** dim
        rho = total(m[j] * W) + m * W0
    vol = (m / rho)[j]
    srho = total(vol * (w * g).sum(0))
    out = {"drho": torch.zeros_like(rho) if P.density_sum else rho * srho, "rho": rho, "nnb": cnt.int()}
    G = torch.stack([-total(vol * w[a] * g) for a in range(dim)])  # G[a][b]
    if P.consistency:
        L = torch.stack([-total(vol * d[a] * g) for a in range(dim)])
        diag = torch.stack([L[a][a] for a in range(dim)]).abs().prod(0)
        ok = (_inverse(L)[1].abs() > 1e-8 * diag) & (diag > 0) & (cnt >= dim + 1)
        eye = torch.eye(dim, dtype=F64, device=x.device)[:, :, None]
        C = _inverse(torch.where(ok, L, eye))[0]
        gv = torch.stack([torch.stack([sum(G[a][b] * C[b][c] for b in range(dim)) for c in range(dim)], -1)
                          for a in range(dim)], -2)
    else:
        gv = G.permute(2, 0, 1)
    xs = 0.0
    if P.xsph:
        xs = P.xsph * total(-(2 * m[j] / (rho[i] + rho[j]) * W) * w)
    out["dxdt"] = v + xs
    p, cs = _eos(M, rho, u, scale)
    S = q.get("S")
    if S is not None:
        Se = S * _yield(S, M, Y0) if M.Y0 > 0 else S
        Sm = _mat3(Se, dim)
        sym = 0.5 * (gv + gv.transpose(1, 2))
        rot = 0.5 * (gv - gv.transpose(1, 2))
        tr = gv.diagonal(dim1=1, dim2=2).sum(1)
        dS = 2 * mu * (sym - (tr / dim)[:, None, None] * torch.eye(dim, dtype=F64, device=x.device))
        dS = dS + rot @ Sm - Sm @ rot
        out["dS"] = torch.stack([dS[:, a, b] for a, b in _sym(dim)])
    dd = q["dmg"] ** 3 if M.damage and q.get("dmg") is not None else torch.zeros_like(rho)
    phat = torch.where(p >= 0, p, (1 - dd) * p)
    sig = torch.zeros((len(_sym(dim)), n), dtype=F64, device=x.device) if S is None else (1 - dd) * Se
    sig = torch.cat([sig[:dim] - phat, sig[dim:]])
    T = sig / rho ** 2
    if M.damage or P.eps_s > 0:
        lam, vec = _eigen(sig, dim)
    if M.damage:
        E = 9 * M.K0 * mu / (3 * M.K0 + mu)
        eps = torch.where(dd < 1, lam.amax(0) / ((1 - dd) * E), torch.zeros_like(dd))
        off = q["flaw_off"]
        cnt_f = off[1:] - off[:-1]
        own = torch.repeat_interleave(torch.arange(n, device=x.device), cnt_f)
        by_id = torch.empty_like(eps).scatter_(0, q["id"].long(), eps)
        act = torch.zeros(n, dtype=F64, device=x.device).index_add_(0, own, (q["flaw_eps"].double() < by_id[own]).double())
        nact, ntot = act[q["id"].long()], cnt_f[q["id"].long()].double()
        cg = 0.4 * torch.sqrt((M.K0 + 4.0 / 3.0 * (1 - dd) * mu) / rho)
        grow = (nact > 0) & (dd * ntot < nact)
        out["ddmg"] = torch.where(grow, nact * cg / h, torch.zeros_like(cg))
        out["n_act"], out["_ntot"] = nact.int(), ntot
    out["p"], out["cs"] = p, cs
    # momentum and energy
    vx = (w * d).sum(0)
    nu = hab * vx / (r * r + P.eps_v * hab ** 2)
    Pi = (-P.alpha * 0.5 * (cs[i] + cs[j]) * nu + P.beta * nu ** 2) / (0.5 * (rho[i] + rho[j]))
    Pi = torch.where(vx < 0, Pi, torch.zeros_like(Pi))

    def dot(t, e):  # symmetric components times a vector
        o = [0.0] * dim
        for k, (a, b) in enumerate(_sym(dim)):
            o[a] = o[a] + t[k] * e[b]
            if a != b:
                o[b] = o[b] + t[k] * e[a]
        return torch.stack(o)

    su = dot(gather(T, i) + gather(T, j), g) - Pi * g
    sv = su
    if P.eps_s > 0:
        z = torch.where(lam > 0, -P.eps_s * lam / rho ** 2, torch.zeros_like(lam))
        Z = torch.stack([(vec[a] * z * vec[b]).sum(0) for a, b in _sym(dim)])
        f = W / _kernel(P.dmpd / hab, hab, dim)[0]
        sv = su + dot((gather(Z, i) + gather(Z, j)) * f ** P.n_as, g)
    out["dv"] = total(m[j] * sv)
    if ag is not None:
        out["dv"] = out["dv"] + ag
    out["du"] = total(-0.5 * m[j] * (w * su).sum(0))
    return out


class _Tree:
    """Barnes-Hut tree of one instance (Sects. 3.3, 3.5.1), level by level."""

    def __init__(self, q, leaf, depth):
        x, m = q["x"], q["m"]
        self.inst = torch.zeros(x.shape[1], dtype=torch.long, device=x.device)
        self.cells = _Cells(x, self.inst, 1, depth)
        key, self.order = torch.sort(self.cells.keys(x, self.inst), stable=True)
        xs, ms = x[:, self.order], m[self.order]
        dim, n = x.shape
        first, end = key.new_zeros(1), key.new_full((1,), n)
        self.levels = []
        for lev in range(depth + 1):
            k = first.numel()
            own = torch.repeat_interleave(torch.arange(k, device=x.device), end - first)
            slot = torch.arange(own.numel(), device=x.device) + torch.repeat_interleave(
                first - ((end - first).cumsum(0) - (end - first)), end - first)
            mass = torch.zeros(k, dtype=F64, device=x.device).index_add_(0, own, ms[slot])
            com = torch.zeros((dim, k), dtype=F64, device=x.device).index_add_(1, own, xs[:, slot] * ms[slot]) / mass
            shift = dim * (depth - lev)
            pre = key[first] >> shift
            node = {"first": first, "end": end, "mass": mass, "com": com, "pre": pre, "shift": shift,
                    "s": float(self.cells.s0[0]) * 2.0 ** -lev}
            node["leaf"] = (end - first <= leaf) if lev < depth else torch.ones_like(first, dtype=torch.bool)
            self.levels.append(node)
            split = torch.nonzero(~node["leaf"])[:, 0]
            if split.numel() == 0:
                break
            sub = (pre[split][:, None] << dim) + torch.arange(2 ** dim, device=x.device)
            f = torch.searchsorted(key, (sub << (shift - dim)).reshape(-1))
            last = (sub << (shift - dim)) + ((1 << (shift - dim)) - 1)
            e = torch.searchsorted(key, last.reshape(-1), right=True)
            keep = e > f
            child = torch.full((k, 2 ** dim), -1, dtype=torch.long, device=x.device)
            ids = torch.where(keep, keep.long().cumsum(0) - 1, torch.full_like(f, -1))
            child[split] = ids.view(-1, 2 ** dim)
            node["child"] = child
            first, end = f[keep], e[keep]

    def accel(self, q, P):
        x, m = q["x"], q["m"]
        dim, n = x.shape
        key = self.cells.keys(x, self.inst)
        eps2 = (P.eps_grav * q["h"]) ** 2
        acc = torch.zeros((dim, n), dtype=F64, device=x.device)

        def add(i, d, r2, mp):
            s = r2 + eps2[i]
            acc.index_add_(1, i, -P.G * mp / (s * torch.sqrt(s)) * d)

        chunk = 1 << 16
        for c in range(0, n, chunk):
            # along the sorted order, so that a chunk opens few nodes
            pi = self.order[c:c + chunk]
            nd = torch.zeros_like(pi)
            for node in self.levels:
                d = x[:, pi] - node["com"][:, nd]
                r2 = (d * d).sum(0)
                inside = (key[pi] >> node["shift"]) == node["pre"][nd]
                use = (node["s"] < P.theta * torch.sqrt(r2)) & ~inside
                add(pi[use], d[:, use], r2[use], node["mass"][nd[use]])
                near = ~use & node["leaf"][nd]
                li, ln = pi[near], nd[near]
                cnt = node["end"][ln] - node["first"][ln]
                i = torch.repeat_interleave(li, cnt)
                b = torch.repeat_interleave(node["first"][ln] - (cnt.cumsum(0) - cnt), cnt)
                b = self.order[b + torch.arange(b.numel(), device=x.device)]
                keep = i != b
                i, b = i[keep], b[keep]
                d = x[:, i] - x[:, b]
                add(i, d, (d * d).sum(0), m[b])
                go = ~use & ~node["leaf"][nd]
                if "child" not in node or not bool(go.any()):
                    break
                ch = node["child"][nd[go]]
                pi = pi[go][:, None].expand_as(ch)[ch >= 0]
                nd = ch[ch >= 0]
        return acc


_KEEP = ("m", "h", "mat", "id")


def _eval(q, M, P, tree=None):
    """Right-hand side on the exact partners; density-sum mode also sets q's density."""
    ag = tree.accel(q, P) if P.gravity else None
    out = _rhs(q, M, P, _pairs(q["x"], q["h"], q["inst"]), ag=ag)
    q["rho"] = out["rho"]
    return out


def _evolved(q, P):
    return {"x": "dxdt", "v": "dv", "u": "du", **({} if P.density_sum else {"rho": "drho"}),
            **({"S": "dS"} if q.get("S") is not None else {}), **({"dmg": "ddmg"} if q.get("dmg") is not None else {})}


def _update(q, M, P, dt, sets):
    """q + dt (c_0 d_0 + ...), then yield and the damage limits (Sect. 3.4.1)."""
    o = dict(q)
    for f, k in _evolved(q, P).items():
        o[f] = q[f] + dt[q["inst"]] * sum(c * d[k] for c, d in sets)
    if o.get("S") is not None and M.Y0 > 0:
        o["S"] = o["S"] * _yield(o["S"], M, M.Y0)
    if o.get("dmg") is not None:
        last = sets[-1][1]
        cap = (last["n_act"].double() / last["_ntot"]) ** (1.0 / 3.0)
        grow = sum(c * d["ddmg"] for c, d in sets) > 0
        o["dmg"] = torch.where(grow, torch.minimum(o["dmg"], cap), o["dmg"]).clamp(max=1.0)
    return o


def _limits(q, d, P, ninst):
    """Time step per instance (Sect. 3.4.1)."""
    if P.dt_fixed > 0:
        return torch.full((ninst,), P.dt_fixed, dtype=F64, device=q["x"].device)
    a = torch.sqrt((d["dv"] ** 2).sum(0))
    lim = [P.c_courant * q["h"] / d["cs"], P.c_accel * torch.sqrt(q["h"] / a)]

    def rate(f, k, floor):
        r = d[k] if f == "dmg" else d[k].abs()
        v = P.c_quantity * (q[f].abs() + floor) / r
        v = torch.where(r > 0, v, torch.full_like(v, math.inf))
        lim.append(v if v.dim() == 1 else v.amin(0))

    if not P.density_sum:
        rate("rho", "drho", 0.0)
    rate("u", "du", P.u_floor)
    if q.get("S") is not None:
        rate("S", "dS", P.S_floor)
    if q.get("dmg") is not None:
        rate("dmg", "ddmg", P.dmg_floor)
    dt = torch.full((ninst,), P.dt_max, dtype=F64, device=a.device)
    return dt.scatter_reduce_(0, q["inst"], torch.stack([v.nan_to_num(nan=math.inf) for v in lim]).amin(0), "amin")


def _reorder(q, P, ninst):
    o = torch.sort(_Cells(q["x"], q["inst"], ninst, P.max_depth).keys(q["x"], q["inst"]), stable=True)[1]
    for k in ("x", "v", "rho", "u", "S", "dmg") + _KEEP:
        if q.get(k) is not None:
            q[k] = q[k][..., o].contiguous()


def _build(q, P):
    return _Tree(q, P.leaf_size, P.max_depth) if P.gravity else None


def _exact_step(q, M, P, ninst, steps):
    tree = None
    for k in range(steps):
        if P.tree_reuse == 0 or k % P.tree_reuse == 0:
            _reorder(q, P, ninst)
            tree = _build(q, P)
        d0 = _eval(q, M, P, tree)
        dt = _limits(q, d0, P, ninst)
        qp = _update(q, M, P, dt, [(0.5, d0)])
        d1 = _eval(qp, M, P, tree if P.tree_reuse else _build(qp, P))
        q = _update(q, M, P, dt, [(1.0, d1)])
    return q, {"dt": dt}


def _exact_rk3(q, M, P, ninst, steps):
    dev = q["x"].device
    dt, t = torch.zeros(ninst, dtype=F64, device=dev), torch.zeros(ninst, dtype=F64, device=dev)
    errs, accs = [], []
    for _ in range(steps):
        _reorder(q, P, ninst)
        k1 = _eval(q, M, P, _build(q, P))
        dt = torch.where(dt > 0, dt, _limits(q, k1, P, ninst))
        q2 = _update(q, M, P, dt, [(0.5, k1)])
        k2 = _eval(q2, M, P, _build(q2, P))
        q3 = _update(q, M, P, dt, [(-1.0, k1), (2.0, k2)])
        k3 = _eval(q3, M, P, _build(q3, P))
        floor = {"x": q["h"], "v": k1["cs"], "rho": 0.0, "u": P.u_floor, "S": P.S_floor, "dmg": P.dmg_floor}
        e = torch.zeros_like(q["u"])
        for f, k in _evolved(q, P).items():
            r = dt[q["inst"]] / 6 * (2 * k2[k] - k1[k] - k3[k]).abs()
            r = r / ((q[f] + dt[q["inst"]] * k1[k]).abs() + floor[f])
            e = torch.maximum(e, r if r.dim() == 1 else r.amax(0))
        err = torch.zeros(ninst, dtype=F64, device=dev).scatter_reduce_(0, q["inst"], e, "amax")
        ok = err < 1e-3
        new = _update(q, M, P, dt, [(1 / 6, k1), (4 / 6, k2), (1 / 6, k3)])
        for f in _evolved(q, P):
            q[f] = torch.where(ok[q["inst"]], new[f], q[f])
        t = t + torch.where(ok, dt, torch.zeros_like(dt))
        dt = torch.where(ok, dt * (1e-3 / err) ** 0.3, 0.9 * dt * (1e-3 / err) ** 0.25).clamp(max=P.dt_max)
        errs.append(err)
        accs.append(ok)
    return q, {"dt": dt, "t": t, "err": torch.stack(errs), "acc": torch.stack(accs).int()}


def _exact_adjoint(q, M, P, dbar):
    leaf = {k: q[k].clone().requires_grad_(True) for k in ("x", "v", "rho", "u", "S")}
    kref = max(M.K0, M.A_T, M.B_T)
    par = torch.tensor([M.mu, M.Y0, 1.0], dtype=F64, device="cuda", requires_grad=True)
    out = _rhs({**q, **leaf}, M, P, _pairs(q["x"], q["h"], q["inst"]), par=par)
    names = ("dxdt", "dv", "drho", "du", "dS")
    g = torch.autograd.grad([out[k] for k in names], list(leaf.values()) + [par], [dbar[k] for k in names])
    res = dict(zip(leaf, g[:-1]))
    res["param"] = (g[-1] / torch.tensor([1.0, 1.0, kref], dtype=F64, device="cuda")).view(1, 1, 3)
    return res


def exact(case, seed):
    call = case["call"]
    if call == "neighbours":  # whole numbers
        return None
    st = prepare(case, seed)
    ds, M, P = st["ds"], st["mats"][0], st["prm"]
    off = ds.inst_off if ds.inst_off is not None else torch.tensor([0, ds.n], device="cuda")
    q = {k: getattr(ds, k) for k in ("x", "v", "rho", "u", "S", "dmg", "flaw_off", "flaw_eps") + _KEEP}
    q["inst"] = torch.repeat_interleave(torch.arange(ds.ninst, device="cuda"), off[1:] - off[:-1])
    dbar = st.get("dbar")
    st["ctx"].close()
    if call == "gravity":
        return {"a": _build(q, replace(P, gravity=True)).accel(q, P)}
    if call == "adjoint":
        return _exact_adjoint(q, M, P, dbar)
    if call == "rhs":
        o = _rhs(q, M, P, _pairs(q["x"], q["h"], q["inst"]))
        return {k: (None if k in ("n_act", "nnb") else o[k])
                for k in ("dxdt", "dv", "drho", "du", "dS", "ddmg", "cs", "p", "n_act", "nnb")}
    q, more = (_exact_step if call == "step" else _exact_rk3)(q, M, P, ds.ninst, case["steps"])
    more.pop("acc", None)
    out = {k: q[k] for k in ("x", "v", "rho", "u", "S", "dmg") if q.get(k) is not None}
    return {**out, "id": None, **more, **({"acc": None} if call == "rk3" else {})}

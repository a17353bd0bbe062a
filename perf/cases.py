"""Performance cases of the FMM gravity solve, through its public entry points.

A case is one call that a program using this framework makes again and again on a tree it keeps:
a whole solve step (eager or as a replayed CUDA graph), one pass of it, one iteration of the
self-consistent-field driver, or the time derivative of the field.  Trees are binaries of n = 1.5
polytropes on adaptive octrees, batches of such trees, and uniform octrees; the tree belongs to the
case, the density to the seed (centres, radii and densities of the stars are jittered within the
refined regions, as from one time step to the next).

`exact` solves the same problem in 64 bits with plain torch, written from the method's definitions.
"""

import functools
import itertools
import math

import numpy as np
import torch

import paper_1908_03121_gb300 as F
from paper_1908_03121_gb300 import scf

NCELL = 512
FLOOR = 1e-10
DEV = "cuda" if torch.cuda.is_available() else "cpu"
R1 = 0.12                       # radius of the first star of a binary, box widths
# operations per cell pair: multipole<-multipole, multipole<-monopole, monopole<-monopole,
# monopole<-multipole, at expansion orders 3 and 2 (derivative tensors in traceless bases)
FLOPS = {3: (240.0, 176.0, 8.0, 199.0), 2: (125.0, 107.0, 8.0, 102.0)}


def _case(kind, precision, tree, levels, theta=0.5, order=3, q=0.3, factor=1.0, contact=False, trees=1):
    return dict(kind=kind, precision=precision, tree=tree, levels=levels, theta=theta, order=order,
                q=q, factor=factor, contact=contact, trees=trees)


def listed():
    return [
        # the smallest solve: a root and 8 leaf sub-grids, FP64, launched eagerly (latency)
        dict(_case("step", "fp64", "uniform", 2), name="two_level_fp64_step"),
        # 64 leaf sub-grids, the default precision, launched eagerly
        dict(_case("step", "mixed", "uniform", 3), name="uniform3_mixed_step"),
        # one self-consistent-field iteration (solve, then density update with its host reads)
        dict(_case("scf", "mixed", "uniform", 4), name="uniform4_scf_mixed"),
        # the ordinary solve: an adaptive tree around a detached binary, as a captured graph
        dict(_case("replay", "mixed", "binary", 5, factor=1.5), name="adaptive5_mixed"),
        # the same method in plain FP64, the reference precision, on a contact binary to level 6
        dict(_case("replay", "fp64", "binary", 6, factor=1.2, contact=True), name="level6_fp64"),
        # ... and in the precision that conserves angular momentum to rounding
        dict(_case("replay", "dfloat", "binary", 6, factor=1.2, contact=True), name="level6_dfloat"),
        # the opening angle of production runs (1074-point stencil)
        dict(_case("replay", "mixed", "binary", 6, theta=0.35, factor=1.2, contact=True),
             name="level6_theta035_mixed"),
        # 16 independent trees of uneven depth in one solve
        dict(_case("replay", "mixed", "binary", 7, trees=16), name="batch16_mixed"),
        # the largest tree: a contact binary to level 7, 6 million leaf cells
        dict(_case("replay", "mixed", "binary", 7, factor=0.88, contact=True), name="level7_mixed"),
        # the passes one by one, as a program that overlaps them with its own work calls them
        dict(_case("upward", "mixed", "binary", 6, factor=1.2, contact=True), name="level6_upward_mixed"),
        dict(_case("m2l", "mixed", "binary", 6, factor=1.2, contact=True), name="level6_m2l_mixed"),
        dict(_case("downward", "mixed", "binary", 6, factor=1.2, contact=True),
             name="level6_downward_forces_mixed"),
    ]


def draw(rng):
    kind = rng.choice(("step", "step", "replay", "replay", "replay", "upward", "m2l", "downward", "scf",
                       "time_derivative"))
    precision = rng.choice(("mixed", "mixed", "mixed", "dfloat", "fp64"))
    theta = rng.choice((0.5, 0.5, 0.35, round(rng.uniform(0.3, 0.577), 3)))
    order = rng.choice((3, 3, 3, 2))
    q = round(rng.uniform(0.1, 1.0), 3)
    if kind == "scf":
        return _case(kind, precision, "uniform", rng.randint(3, 4), theta, 3, q)
    if kind == "time_derivative":
        return _case(kind, rng.choice(("fp64", "dfloat")), "binary", rng.randint(3, 4), 0.5, order, q,
                     round(rng.uniform(0.6, 1.4), 3))
    if rng.random() < 0.2:
        return _case(kind, precision, "uniform", rng.randint(2, 4), theta, order, q)
    if rng.random() < 0.2:
        return _case(kind, precision, "binary", 5 if precision == "fp64" else 6, theta, order, q,
                     trees=rng.randint(2, 6))
    # the number of sub-grids spreads over about 100 to 5000 (FP64: to 1700)
    return _case(kind, precision, "binary", rng.randint(3, 5 if precision == "fp64" else 6), theta, order,
                 q, round(math.exp(rng.uniform(math.log(0.5), math.log(1.3))), 3),
                 contact=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
def _binary(q, contact):
    """Two n = 1.5 polytropes of mass ratio q on the x axis: centres, radii, central densities."""
    r2 = R1 * q ** (-1.0 / 3.0)
    sep = R1 + r2 - 0.1 * R1 if contact else 0.4
    return ((0.5 - 0.5 * sep, 0.5, 0.5), (0.5 + 0.5 * sep, 0.5, 0.5)), (R1, r2), (1.0, q * q)


def _octree(want, levels, tree_id=0):
    """Descriptor rows (level, ix, iy, iz, parent, child[8], tree), breadth first.  want(level, xyz)
    says which nodes to refine; a refined node's in-domain neighbours all exist."""
    key = lambda a: (a[:, 2] * 4096 + a[:, 1]) * 4096 + a[:, 0]
    kids = np.array([(k & 1, (k >> 1) & 1, k >> 2) for k in range(8)])
    near = np.array(list(itertools.product((-1, 0, 1), repeat=3)))
    refined, front = {}, np.zeros((1, 3), np.int64)
    for lev in range(1, levels):
        refined[lev] = front[want(lev, front)]
        front = (2 * refined[lev][:, None] + kids).reshape(-1, 3)
    for lev in range(levels - 1, 1, -1):
        nb = (refined[lev][:, None] + near).reshape(-1, 3)
        nb = nb[((nb >= 0) & (nb < 2 ** (lev - 1))).all(1)]
        refined[lev - 1] = np.unique(np.concatenate([refined[lev - 1], nb // 2]), axis=0)
    rows, start, front, parent = [], 0, np.zeros((1, 3), np.int64), np.array([-1])
    for lev in range(1, levels + 1):
        o = np.argsort(key(front))
        front, parent = front[o], parent[o]
        r = np.full((len(front), 14), -1, np.int32)
        r[:, 0], r[:, 1:4], r[:, 4], r[:, 13] = lev, front, parent, tree_id
        rows.append(r)
        sub = np.isin(key(front), key(refined[lev])) if lev < levels else np.zeros(len(front), bool)
        parent = np.repeat(start + np.nonzero(sub)[0], 8)
        front = (2 * front[sub][:, None] + kids).reshape(-1, 3)
        start += len(r)
    d = np.concatenate(rows)
    has = d[:, 4] >= 0
    d[d[has, 4], 5 + (d[has, 1] & 1) + 2 * (d[has, 2] & 1) + 4 * (d[has, 3] & 1)] = np.nonzero(has)[0]
    return d


def _star_tree(q, contact, levels, factor, tree_id=0):
    centres, radii, _ = _binary(q, contact)

    def want(lev, xyz):
        w = 1.0 / 2 ** (lev - 1)
        hit = np.zeros(len(xyz), bool)
        for c, r in zip(centres, radii):
            d = np.clip(c, xyz * w, (xyz + 1) * w) - c
            hit |= (d * d).sum(1) <= (factor * r) ** 2
        return hit
    return _octree(want, levels, tree_id)


@functools.lru_cache(maxsize=None)
def _forest(tree, levels, factor, q, contact, trees):
    """The case's descriptors and each tree's mass ratio."""
    if tree == "uniform":
        return _octree(lambda lev, xyz: np.ones(len(xyz), bool), levels), (q,)
    if trees == 1:
        return _star_tree(q, contact, levels, factor), (q,)
    # uneven depths; each tree's refined region as large as leaves it at most 2000 leaf sub-grids
    qs, out, base = tuple(np.linspace(0.1, 1.0, trees)), [], 0
    for i, qi in enumerate(qs):
        for f in (1.6, 1.2, 0.85, 0.6, 0.42, 0.3, 0.2):
            d = _star_tree(qi, contact, levels - 3 + i % 4, f, i)
            if (d[:, 5] < 0).sum() <= 2000:
                break
        d[:, 4:13] += np.where(d[:, 4:13] >= 0, base, 0).astype(np.int32)
        out.append(d)
        base += len(d)
    return np.concatenate(out), qs


def _tree_of(case):
    return _forest(case["tree"], case["levels"], case["factor"], case["q"], case["contact"], case["trees"])


@functools.lru_cache(maxsize=None)
def _lane_emden(n=1.5, dxi=1e-3):
    """theta(xi) of the polytrope of index n to its first zero (RK4)."""
    f = lambda x, t, u: (u, -max(t, 0.0) ** n - 2.0 * u / x)
    x, t, u = dxi, 1.0 - dxi ** 2 / 6.0, -dxi / 3.0
    xs, ts = [0.0, x], [1.0, t]
    while t > 0.0:
        k1 = f(x, t, u)
        k2 = f(x + dxi / 2, t + dxi / 2 * k1[0], u + dxi / 2 * k1[1])
        k3 = f(x + dxi / 2, t + dxi / 2 * k2[0], u + dxi / 2 * k2[1])
        k4 = f(x + dxi, t + dxi * k3[0], u + dxi * k3[1])
        t, u = (t + dxi / 6 * (k1[0] + 2 * k2[0] + 2 * k3[0] + k4[0]),
                u + dxi / 6 * (k1[1] + 2 * k2[1] + 2 * k3[1] + k4[1]))
        x += dxi
        xs.append(x)
        ts.append(max(t, 0.0))
    return torch.tensor(xs, dtype=torch.float64, device=DEV), torch.tensor(ts, dtype=torch.float64, device=DEV)


def _polytrope(pos, c, radius, rho_c):
    xs, ts = _lane_emden()
    r = (pos - torch.as_tensor(c, dtype=torch.float64, device=DEV)).norm(dim=-1) * (float(xs[-1]) / radius)
    i = (r / float(xs[1])).long().clamp(0, len(xs) - 2)
    t = ts[i] + (ts[i + 1] - ts[i]) * (r - xs[i]) / (xs[i + 1] - xs[i])
    return rho_c * t.clamp(min=0.0) ** 1.5


def _cell_xyz():
    c = torch.arange(NCELL, device=DEV)
    return torch.stack([c & 7, (c >> 3) & 7, c >> 6], 1)


def _density(case, seed):
    """The leaf cells' density, (n_leaf, 512)."""
    desc, qs = _tree_of(case)
    rng = np.random.default_rng([seed, 1908])
    leaf = torch.as_tensor(desc[desc[:, 5] < 0].astype(np.int64), device=DEV)
    h = 0.125 * 0.5 ** (leaf[:, 0].double() - 1)
    rho = torch.empty((len(leaf), NCELL), dtype=torch.float64, device=DEV)
    for t, q in enumerate(qs):
        at = (leaf[:, 13] == t).nonzero()[:, 0]
        pos = (8 * leaf[at, None, 1:4] + _cell_xyz() + 0.5).double() * h[at, None, None]
        v = torch.full((len(at), NCELL), FLOOR, dtype=torch.float64, device=DEV)
        centres, radii, rho_c = _binary(q, case["contact"])
        for c, r, d in zip(centres, radii, rho_c):
            v += _polytrope(pos, np.array(c) + rng.uniform(-0.01, 0.01, 3), r * rng.uniform(0.95, 1.05),
                            d * rng.uniform(0.8, 1.2))
        rho[at] = v
    return rho


def _density_rate(rho, seed):
    """A density change of a few per cent a unit time, smooth within a sub-grid."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 77)
    k = torch.rand((len(rho), 3), generator=gen, dtype=torch.float64, device=DEV)
    return rho * 0.05 * torch.sin(k @ _cell_xyz().double().T * 0.4 + 6.0 * k[:, :1])


def _scf_params(case):
    h = 1.0 / (8 * 2 ** (case["levels"] - 1))
    return scf.binary_params((0.3, 0.5, 0.5), 0.15, (0.72, 0.5, 0.5), 0.13, (1.0, 0.5), h)


def _scf_density(case, seed):
    desc, _ = _tree_of(case)
    rng = np.random.default_rng([seed, 77])
    leaf = torch.as_tensor(desc[desc[:, 5] < 0].astype(np.int64), device=DEV)
    pos = (8 * leaf[:, None, 1:4] + _cell_xyz() + 0.5).double() / (8 * 2 ** (case["levels"] - 1))
    a, b = rng.uniform(0.9, 1.1, 2)
    return _polytrope(pos, (0.3, 0.5, 0.5), 0.15 * a, a) + _polytrope(pos, (0.72, 0.5, 0.5), 0.13 * b, 0.5 * b) + FLOOR


# -------------------------------------------------------------- the program
class State:
    pass


def prepare(case, seed):
    st = State()
    st.kind = case["kind"]
    desc, _ = _tree_of(case)
    st.s = F.Solver(desc, case["theta"], precision=case["precision"], order=case["order"])
    st.s.rho.copy_(_scf_density(case, seed) if st.kind == "scf" else _density(case, seed))
    if st.kind == "replay":
        st.s.capture()
    elif st.kind in ("m2l", "downward"):
        st.s.upward()
        if st.kind == "downward":
            st.s.m2l()
    elif st.kind == "scf":
        st.params = _scf_params(case)
        st.rho_out = torch.empty_like(st.s.rho)
    elif st.kind == "time_derivative":
        st.rho_dot = _density_rate(st.s.rho, seed)
        st.work = torch.empty_like(st.s.rho)
        st.phi_dot, st.g_dot = torch.empty_like(st.s.phi), torch.empty_like(st.s.g)
    return st


def run(st):
    s = st.s
    if st.kind == "replay":
        s.replay()
    elif st.kind == "step":
        s.step()
    elif st.kind == "upward":
        s.upward()
        return {"M": s.M, "com": s.com}
    elif st.kind == "m2l":
        s.m2l()
        out = {"L": s.L, "dL1": s.dL1}
        return out if s.Lc is None else dict(out, L_comp=s.Lc)
    elif st.kind == "downward":
        s.downward()
        s.forces()
        return {"L64": s.L64, "dL1_acc": s.dacc, "phi": s.phi, "g": s.g, "totals": s.totals}
    elif st.kind == "scf":
        s.step()
        r = F.fmm_scf_update(s.tree, st.params, s.phi, s.rho, st.rho_out)
        return {"phi": s.phi, "rho": st.rho_out, "omega2": r["omega2"], "C": r["C"], "H_max": r["H_max"],
                "com": r["com"], "mass": r["mass"]}
    else:
        s.time_derivative(st.rho_dot, 0.05, st.phi_dot, st.g_dot, rho_work=st.work)
        return {"phi_dot": st.phi_dot, "g_dot": st.g_dot}
    return {"phi": s.phi, "g": s.g, "totals": s.totals}


def work(case):
    desc, _ = _tree_of(case)
    tree = F.fmm_build_tree(desc, case["theta"], precision=case["precision"], host_only=True,
                            order=case["order"])
    pairs = sum(n * f for n, f in zip(tree.stats["interactions"], FLOPS[case["order"]]))
    n, leaves = len(desc), int((desc[:, 5] < 0).sum())
    refined = n - leaves
    cell = 8.0 * NCELL
    kind = case["kind"]
    # refined nodes: 17 moments and 3 coordinates, or 20 coefficients and 3 corrections; leaf nodes:
    # the mass, or 4 coefficients and 3 corrections
    moments, taylor = cell * (20 * refined + leaves), cell * (23 * refined + 7 * leaves)
    if kind == "upward":
        return {"bytes": cell * leaves + moments, "flops": NCELL * (leaves + 400.0 * refined)}
    if kind == "m2l":
        return {"bytes": moments + taylor, "flops": pairs}
    if kind == "downward":
        return {"bytes": 2 * taylor + 3 * cell * refined + 5 * cell * leaves,
                "flops": NCELL * (150.0 * leaves + 350.0 * refined)}
    solve = {"bytes": 5 * cell * leaves, "flops": pairs + NCELL * (151.0 * leaves + 750.0 * refined)}
    if kind == "time_derivative":          # value and derivative of the solve
        return {"bytes": 6 * cell * leaves, "flops": 2 * solve["flops"]}
    return {"bytes": solve["bytes"] + (2 * cell * leaves if kind == "scf" else 0), "flops": solve["flops"]}


# ------------------------------------------------------- the same in 64 bits
I2 = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
I3 = [(0, 0, 0), (0, 0, 1), (0, 0, 2), (0, 1, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2),
      (2, 2, 2)]


def _pairs(R, m, M2, M3, aA, order, high):
    """Taylor coefficients (level units) that sources (m, M2, M3) at separation R give a target, and
    the correction; aA: the target's M3 / M0 (order 3) or M2 / M0 (order 2), or None."""
    ri2 = 1.0 / (R * R).sum(-1)
    e1 = ri2.sqrt()
    e3, e5, e7 = e1 * ri2, e1 * ri2 ** 2, e1 * ri2 ** 3
    M2R = (M2 * R[..., None, :]).sum(-1)
    RMR, tr = (M2R * R).sum(-1), M2.diagonal(dim1=-2, dim2=-1).sum(-1)
    L0 = m * e1 + 0.5 * (3 * RMR * e5 - tr * e3)
    L1 = -(m * e3)[..., None] * R

    def d3(W):                                   # D3[i, jk] W_jk
        WR = (W * R[..., None, :]).sum(-1)
        t = W.diagonal(dim1=-2, dim2=-1).sum(-1)
        return ((3 * t * e5 - 15 * (WR * R).sum(-1) * e7)[..., None] * R + 6 * e5[..., None] * WR)

    if order == 3:
        M3RR = ((M3 * R[..., None, None, :]).sum(-1) * R[..., None, :]).sum(-1)
        v = M3.diagonal(dim1=-2, dim2=-1).sum(-1)
        L0 = L0 - (9 * (v * R).sum(-1) * e5 - 15 * (M3RR * R).sum(-1) * e7) / 6
        L1 = L1 + 0.5 * d3(M2)
        W = M3 if aA is None else M3 - m[..., None, None, None] * aA
        WRR = ((W * R[..., None, None, :]).sum(-1) * R[..., None, :]).sum(-1)
        w = W.diagonal(dim1=-2, dim2=-1).sum(-1)
        S = ((105 * (WRR * R).sum(-1) * e7 * ri2 - 45 * (w * R).sum(-1) * e7)[..., None] * R
             - 45 * e7[..., None] * WRR + 9 * e5[..., None] * w) / 6
    else:
        S = -0.5 * d3(M2 if aA is None else M2 + m[..., None, None] * aA)
    if not high:
        return [-L0, *(-L1[..., i] for i in range(3))], S
    x = [R[..., i] for i in range(3)]
    dl = lambda a, b: 1.0 if a == b else 0.0
    out = [-L0, *(-L1[..., i] for i in range(3))]
    out += [-m * (3 * e5 * x[a] * x[b] - dl(a, b) * e3) for a, b in I2]
    out += [-m * (3 * e5 * (dl(b, c) * x[a] + dl(a, c) * x[b] + dl(a, b) * x[c]) - 15 * e7 * x[a] * x[b] * x[c])
            if order == 3 else 0 * m for a, b, c in I3]
    return out, S


class _Exact:
    """The solve in 64 bits (or on complex numbers, for a derivative by complex step): moments summed
    from the children, every same-level pair of the opening rule, Taylor shifts down the tree.  Lengths
    in cell widths of a node's level until the downward pass."""

    def __init__(self, desc, rho, theta, order, solve=True):
        self.order, self.theta = order, theta
        dt = rho.dtype
        d = torch.as_tensor(desc.astype(np.int64), device=DEV)
        self.lev, self.xyz, self.parent, self.child = d[:, 0], d[:, 1:4], d[:, 4], d[:, 5:13]
        self.tree = d[:, 13]
        n = self.n = len(d)
        self.leaf = self.child[:, 0] < 0
        self.row = torch.cumsum(~self.leaf, 0) - 1
        nr = self.nr = int((~self.leaf).sum())
        self.row[self.leaf] = nr                        # the row of zeros after the refined nodes
        self.h = 0.125 * 0.5 ** (self.lev.double() - 1)
        self.c = _cell_xyz()
        # one more node and one more row for absent and leaf sources
        self.m = torch.zeros((n + 1, NCELL), dtype=dt, device=DEV)
        self.m[:n][self.leaf] = rho * self.h[self.leaf, None] ** 3
        self.off = torch.zeros((nr + 1, NCELL, 3), dtype=dt, device=DEV)
        self.M2 = torch.zeros((nr + 1, NCELL, 3, 3), dtype=dt, device=DEV)
        self.M3 = torch.zeros((nr + 1, NCELL, 3, 3, 3), dtype=dt, device=DEV)
        self.levels = range(1, int(self.lev.max()) + 1)
        self.up()
        if solve:
            self.same_level()

    def up(self):
        c = self.c
        k = (c[:, 0] >> 2) + 2 * (c[:, 1] >> 2) + 4 * (c[:, 2] >> 2)
        for lev in reversed(self.levels):
            nodes = ((self.lev == lev) & ~self.leaf).nonzero()[:, 0]
            if len(nodes) == 0:
                continue
            ch = self.child[nodes][:, k]                                      # (N, 512)
            ms, Xs, cells = [], [], []
            for j in range(8):
                b = torch.tensor([j & 1, (j >> 1) & 1, j >> 2], device=DEV)
                q = 2 * (c & 3) + b
                cc = (q[:, 0] + 8 * q[:, 1] + 64 * q[:, 2]).expand(len(nodes), -1)
                cells.append(cc)
                ms.append(self.m[ch, cc])
                Xs.append(0.5 * (b - 0.5) + 0.5 * self.off[self.row[ch], cc])
            m0 = sum(ms)
            X = sum(m[..., None] * x for m, x in zip(ms, Xs)) / m0[..., None]
            r = self.row[nodes]
            for m, x, cc in zip(ms, Xs, cells):
                s = x - X
                c2, c3 = 0.25 * self.M2[self.row[ch], cc], 0.125 * self.M3[self.row[ch], cc]
                ss = s[..., :, None] * s[..., None, :]
                t = c2[..., :, :, None] * s[..., None, None, :]
                self.M2[r] += c2 + m[..., None, None] * ss
                self.M3[r] += (c3 + t + t.transpose(-1, -2) + t.permute(*range(t.dim() - 3), -1, -3, -2)
                               + m[..., None, None, None] * ss[..., None] * s[..., None, None, :])
            self.m[nodes], self.off[r] = m0, X

    def neighbours(self):
        key = lambda lev, t, x: (((t * 32 + lev) * 4096 + x[:, 2]) * 4096 + x[:, 1]) * 4096 + x[:, 0]
        keys, at = torch.sort(key(self.lev, self.tree, self.xyz))
        nb = torch.full((self.n, 27), self.n, dtype=torch.int64, device=DEV)
        for s, (dz, dy, dx) in enumerate(itertools.product((-1, 0, 1), repeat=3)):
            x = self.xyz + torch.tensor([dx, dy, dz], device=DEV)
            ok = ((x >= 0) & (x < (1 << (self.lev - 1))[:, None])).all(1)
            want = key(self.lev, self.tree, x.clamp(min=0))
            i = torch.searchsorted(keys, want).clamp(max=self.n - 1)
            nb[:, s] = torch.where(ok & (keys[i] == want), at[i], nb[:, s])
        return nb

    def far(self, o):
        return self.theta ** 2 * float(sum(v * v for v in o)) > 1.0

    def source(self, node, cell, row):
        return self.m[node, cell], self.off[row, cell], self.M2[row, cell], self.M3[row, cell]

    def own(self, r, cells):
        """A refined target's offset and its share of the correction, (N, cells, ...)."""
        A = self.M3 if self.order == 3 else self.M2
        m = torch.zeros((self.nr + 1, NCELL), dtype=self.m.dtype, device=DEV)
        m[:self.nr] = self.m[:self.n][~self.leaf]
        m[self.nr] = 1.0
        a = A[r][:, cells]
        return self.off[r][:, cells], a / m[r][:, cells].reshape(a.shape[:2] + (1,) * (a.dim() - 2))

    def same_level(self):
        dt, dev = self.m.dtype, DEV
        self.L = torch.zeros((self.n, 20, NCELL), dtype=dt, device=dev)
        self.S = torch.zeros((self.n, 3, NCELL), dtype=dt, device=dev)
        row = torch.cat([self.row, torch.tensor([self.nr], device=dev)])
        nb = self.neighbours()
        inner = self.lev > 1
        ref = (inner & ~self.leaf).nonzero()[:, 0]
        lea = (inner & self.leaf).nonzero()[:, 0]
        refined_nb = (row[nb] < self.nr).any(1)
        mix = (inner & self.leaf & refined_nb).nonzero()[:, 0]
        mono = torch.where(row[:, None] == self.nr, self.m, torch.zeros_like(self.m))
        reach = 2 * int(math.floor(1.0 / self.theta)) + 1
        span = range(-reach, reach + 1)
        for p in range(8):
            pp = (p & 1, (p >> 1) & 1, p >> 2)
            cells = ((self.c & 1) == torch.tensor(pp, device=dev)).all(1).nonzero()[:, 0]
            ent = [o for o in itertools.product(span, repeat=3) if o != (0, 0, 0)
                   and not self.far([(pp[a] + o[a]) // 2 for a in range(3)])]
            for e0 in range(0, len(ent), 8):
                part = ent[e0:e0 + 8]
                o = torch.tensor(part, device=dev)
                b = self.c[cells][None] + o[:, None] + 8                      # (E, 64, 3)
                slot = (b[..., 0] >> 3) + 3 * (b[..., 1] >> 3) + 9 * (b[..., 2] >> 3)
                loc = (b[..., 0] & 7) + 8 * (b[..., 1] & 7) + 64 * (b[..., 2] & 7)
                od = o.to(dt)
                # leaf cells: point masses at offset o
                r = od.abs().square().sum(1).sqrt()
                w = torch.cat([-1 / r[:, None], -od / r[:, None] ** 3], 1)    # (E, 4)
                for g in lea.split(4096):
                    mass = mono[nb[g][:, slot], loc]
                    self.L[g[:, None, None], torch.arange(4, device=dev)[:, None], cells] += \
                        torch.einsum("nec,ek->nkc", mass, w)
                far = torch.tensor([self.far(v) for v in part], device=dev)[:, None]
                for nodes, high in ((ref, True), (mix, False)):
                    for g in nodes.split(512):
                        src = nb[g][:, slot]                                  # (N, E, 64)
                        rr = row[src]
                        m, d, M2, M3 = self.source(src, loc, rr)
                        if high:      # near sources: leaf cells only
                            keep = far | (rr == self.nr)
                            dA, aA = self.own(self.row[g], cells)
                            R, aA = dA[:, None] - d - od[:, None], aA[:, None]
                        else:         # leaf sources are above
                            keep = rr < self.nr
                            R, aA = -d - od[:, None], None
                        z = keep.to(dt)
                        L, S = _pairs(R, m * z, M2 * z[..., None, None], M3 * z[..., None, None, None], aA,
                                      self.order, high)
                        for k, v in enumerate(L):
                            self.L[g[:, None], k, cells] += v.sum(1)
                        for i in range(3):
                            self.S[g[:, None], i, cells] += S[..., i].sum(1)
        for node in (self.lev == 1).nonzero()[:, 0].tolist():                 # roots: all pairs
            lf, rt = bool(self.leaf[node]), int(self.row[node])
            cell = torch.arange(NCELL, device=dev)
            dA, aA = self.own(torch.tensor([rt], device=dev), cell)
            for t in cell.split(64):
                o = self.c[None] - self.c[t][:, None]                         # (t, 512, 3)
                o2 = (o * o).sum(-1)
                keep = (o2 > 0) & (lf | (self.theta ** 2 * o2.double() > 1.0))
                m, d, M2, M3 = self.source(node, cell, rt)
                R = dA[0, t][:, None] - d[None] - torch.where(keep[..., None], o, torch.ones_like(o)).to(dt)
                z = keep.to(dt)
                L, S = _pairs(R, m * z, M2 * z[..., None, None], M3 * z[..., None, None, None],
                              None if lf else aA[0, t][:, None], self.order, not lf)
                for k, v in enumerate(L):
                    self.L[node, k, t] = v.sum(1)
                self.S[node][:, t] = S.sum(1).T

    def down(self):
        dt = self.m.dtype
        n2 = [[I2.index(tuple(sorted((a, b)))) + 4 for b in range(3)] for a in range(3)]
        n3 = [[[I3.index(tuple(sorted((a, b, c)))) + 10 for c in range(3)] for b in range(3)] for a in range(3)]
        self.L64 = torch.zeros_like(self.L)
        self.dacc = torch.zeros_like(self.S)
        power = torch.tensor([1.0] + [2.0] * 3 + [3.0] * 6 + [4.0] * 10, dtype=torch.float64, device=DEV)
        c = self.c
        for lev in self.levels:
            for nodes in ((self.lev == lev).nonzero()[:, 0]).split(2048):
                h = self.h[nodes]
                L = self.L[nodes] * (h[:, None] ** -power)[..., None]
                S = self.S[nodes] * (h ** -2)[:, None, None]
                if lev > 1:
                    par = self.parent[nodes]
                    q = 4 * (self.xyz[nodes] & 1)[:, None] + (c >> 1)
                    pc = q[..., 0] + 8 * q[..., 1] + 64 * q[..., 2]           # (N, 512)
                    P = self.L64[par[:, None], :, pc]                         # (N, 512, 20)
                    d = (0.5 * ((c & 1) - 0.5) + 0.5 * self.off[self.row[nodes]] -
                         self.off[self.row[par][:, None], pc]) * (2 * h)[:, None, None]
                    g = lambda i: P[..., torch.tensor(i, device=DEV)]
                    P1, P2, P3 = P[..., 1:4], g(n2), g(n3)
                    P3d = (P3 * d[..., None, None, :]).sum(-1)
                    P2d, P3dd = (P2 * d[..., None, :]).sum(-1), (P3d * d[..., None, :]).sum(-1)
                    L[:, 0] += P[..., 0] + ((P1 + P2d / 2 + P3dd / 6) * d).sum(-1)
                    for i in range(3):
                        L[:, 1 + i] += P1[..., i] + P2d[..., i] + P3dd[..., i] / 2
                    for k, (a, b) in enumerate(I2):
                        L[:, 4 + k] += P2[..., a, b] + P3d[..., a, b]
                    for k in range(10):
                        L[:, 10 + k] += P[..., 10 + k]
                    S += self.dacc[par[:, None], :, pc].transpose(1, 2)
                self.L64[nodes], self.dacc[nodes] = L, S
        self.L64[self.leaf, 4:] = 0
        self.phi = self.L64[self.leaf, 0]
        self.g = -(self.L64[self.leaf, 1:4] + self.dacc[self.leaf])
        if dt.is_complex:
            return
        f = self.m[:self.n][self.leaf][:, None] * self.g
        x = ((8 * self.xyz[self.leaf][:, None] + c + 0.5).double() * self.h[self.leaf][:, None, None] - 0.5)
        x = x.transpose(1, 2)
        t = torch.linalg.cross(x, f, dim=1)
        v = torch.cat([f, t, f.norm(dim=1)[:, None], t.norm(dim=1)[:, None]], 1).sum(-1)
        self.totals = torch.zeros((int(self.tree.max()) + 1, 8), dtype=dt, device=DEV)
        self.totals.index_add_(0, self.tree[self.leaf], v)


def _exact_scf(case, e, rho):
    p = _scf_params(case)
    side = 8 * 2 ** (case["levels"] - 1)
    h = 1.0 / side
    pos = (8 * e.xyz[e.leaf][:, None] + e.c + 0.5).double() * h
    m = rho * h ** 3
    com = (m[..., None] * pos).sum((0, 1)) / m.sum()
    w2 = ((pos - com)[..., :2] ** 2).sum(-1)

    def at(point):                                   # the leaf cell that holds a point
        cell = [int(math.floor(v * side)) for v in point]
        hit = ((pos * side - 0.5).round().long() == torch.tensor(cell, device=DEV)).all(-1).nonzero()[0]
        return float(e.phi[tuple(hit)]), float(w2[tuple(hit)])
    (pa, wa), (pb, wb), (pc, wc) = at(p.point_a), at(p.point_b), at(p.point_c)
    om = 2 * (pa - pb) / (wa - wb)
    C = (pa - om * wa / 2, pc - om * wc / 2)
    out, hmax = torch.full_like(rho, p.rho_floor), []
    for i in range(2):
        ctr = torch.tensor(list(p.centre[i]), dtype=torch.float64, device=DEV)
        mine = ((pos - ctr).norm(dim=-1) <= p.r_lim[i]) & ((pos[..., 0] < p.x_split) == (i == 0))
        H = torch.where(mine, C[i] - e.phi + om * w2 / 2, torch.full_like(rho, -1.0))
        hmax.append(float(H.max()))
        new = (p.rho_max[i] * (H.clamp(min=0) / hmax[i]) ** p.n).clamp(min=p.rho_floor)
        out = torch.where(H > 0, new, out)
    return {"phi": e.phi, "rho": out, "omega2": om, "C": C, "H_max": tuple(hmax), "com": tuple(com.tolist()),
            "mass": float(m.sum())}


def exact(case, seed):
    desc, _ = _tree_of(case)
    kind = case["kind"]
    rho = _scf_density(case, seed) if kind == "scf" else _density(case, seed)
    if kind == "time_derivative":
        step = 1e-40
        e = _Exact(desc, torch.complex(rho, step * _density_rate(rho, seed)), case["theta"], case["order"])
        e.down()
        return {"phi_dot": e.phi.imag / step, "g_dot": e.g.imag / step}
    e = _Exact(desc, rho, case["theta"], case["order"], solve=kind != "upward")
    if kind == "upward":
        M = torch.zeros((e.n, 20, NCELL), dtype=torch.float64, device=DEV)
        com = torch.zeros((e.n, 3, NCELL), dtype=torch.float64, device=DEV)
        M[:, 0] = e.m[:e.n]
        ref = (~e.leaf).nonzero()[:, 0]
        h = e.h[ref][:, None]
        for k, (a, b) in enumerate(I2):
            M[ref, 4 + k] = e.M2[:-1, :, a, b] * h ** 2
        for k, (a, b, c) in enumerate(I3):
            M[ref, 10 + k] = e.M3[:-1, :, a, b, c] * h ** 3
        com[ref] = ((8 * e.xyz[ref][:, None] + e.c + 0.5 + e.off[:-1]) * h[..., None]).transpose(1, 2)
        return {"M": M, "com": com}
    if kind == "m2l":
        out = {"L": e.L, "dL1": e.S}
        return out if case["precision"] == "fp64" else dict(out, L_comp=None)
    e.down()
    if kind == "scf":
        return _exact_scf(case, e, rho)
    out = {"phi": e.phi, "g": e.g, "totals": e.totals}
    return dict(out, L64=e.L64, dL1_acc=e.dacc) if kind == "downward" else out

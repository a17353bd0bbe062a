"""fmm_scf_update's scalars and density against numpy on the solver's own
potential: polytropic indices that take products and a square root (2 n whole)
and one that takes pow, on uniform and adaptive trees."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from paper_1908_03121_gb300 import scf as D
from workloads import adaptive_tree, leaf_cell_centres, uniform_tree
from workloads.density import polytrope

pytestmark = pytest.mark.gpu

# FP64 throughout: sums of 4e4 cells in another order, and one power
TOL = 1e-12


def _tree(name):
    if name == "uniform3":
        return uniform_tree(3)
    c = np.array([0.3, 0.5, 0.5])

    def want(lo, hi):
        d = np.clip(c, lo, hi) - c
        return float(d @ d) < 0.12 ** 2
    return adaptive_tree(want, 4, min_level=2)


@pytest.mark.parametrize("name", ["uniform3", "adaptive4"])
@pytest.mark.parametrize("n", [0.5, 1.0, 1.25, 1.5, 3.0])
def test_update_matches_numpy(name, n):
    desc = _tree(name)
    pos = leaf_cell_centres(desc)                               # (leaves, 512, 3)
    lev = desc[desc[:, 5] < 0, 0]
    h = np.broadcast_to((1.0 / (8 * 2.0 ** (lev - 1)))[:, None], pos.shape[:2])
    c1, c2 = (0.3, 0.5, 0.5), (0.72, 0.5, 0.5)
    rho = polytrope(pos, np.array(c1), 0.15, 1.0) + polytrope(pos, np.array(c2), 0.13, 0.5) + 1e-10
    p = D.binary_params(c1, 0.15, c2, 0.13, (1.0, 0.5), 1.0 / 64, n=n)
    s = F.Solver(desc, 0.5, precision="fp64")
    s.rho.copy_(torch.from_numpy(rho.reshape(-1, 512)).cuda())
    out = torch.empty_like(s.rho)
    s.step()
    for _ in range(2):                                          # the second call finds the first's counters
        got = F.fmm_scf_update(s.tree, p, s.phi, s.rho, out)
    torch.cuda.synchronize()
    phi, m = s.phi.cpu().numpy(), rho.reshape(-1, 512) * h ** 3
    com = (m[..., None] * pos).sum((0, 1)) / m.sum()
    w2 = ((pos - com)[..., :2] ** 2).sum(-1)
    at = []
    for q in (p.point_a, p.point_b, p.point_c):
        inside = np.all(np.abs(pos - np.array(list(q))) <= 0.5 * h[..., None], axis=-1)
        at.append(tuple(np.argwhere(inside)[0]))
    np.testing.assert_allclose(got["phi_points"], [phi[a] for a in at], rtol=0)
    om = 2 * (phi[at[0]] - phi[at[1]]) / (w2[at[0]] - w2[at[1]])
    C = [phi[at[0]] - om * w2[at[0]] / 2, phi[at[2]] - om * w2[at[2]] / 2]
    np.testing.assert_allclose(got["com"], com, rtol=TOL)
    np.testing.assert_allclose([got["omega2"], *got["C"], got["mass"]], [om, *C, m.sum()], rtol=1e-10)
    want = np.full_like(phi, p.rho_floor)
    sure = np.ones(phi.shape, bool)          # H is not zero to rounding (u^n is steep there for n < 1)
    for i in range(2):
        mine = (((pos - np.array(list(p.centre[i]))) ** 2).sum(-1) < p.r_lim[i] ** 2) & \
            ((pos[..., 0] < p.x_split) == (i == 0))
        H = np.where(mine, got["C"][i] - phi + 0.5 * got["omega2"] * w2, -1.0)
        np.testing.assert_allclose(got["H_max"][i], H.max(), rtol=1e-10)
        sure &= ~mine | (np.abs(H) > 1e-9 * H.max())
        want = np.where(H > 0, np.maximum(p.rho_floor, p.rho_max[i] * (np.clip(H, 0, None) / H.max()) ** n), want)
    np.testing.assert_allclose(out.cpu().numpy()[sure], want[sure], rtol=1e-9, atol=1e-9)
    s.close()

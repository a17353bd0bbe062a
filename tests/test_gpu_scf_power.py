"""The density update's power u^n to a unit in the last place (pow's bound), for
the indices that take products and a square root and one that takes pow."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from paper_1908_03121_gb300 import scf as D
from workloads import leaf_cell_centres, uniform_tree
from workloads.density import polytrope

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0.5, 1.0, 1.25, 1.5, 2.0, 2.5, 3.0, 4.5, 6.0, 7.5, 8.0])
def test_power_to_one_ulp(n):
    desc, ctr = uniform_tree(3), (0.5, 0.5, 0.5)
    rho = polytrope(leaf_cell_centres(desc), np.array(ctr), 0.25, 1.0) + 1e-10
    s = F.Solver(desc, 0.5, precision="fp64")
    s.rho.copy_(torch.from_numpy(rho.reshape(-1, 512)).cuda())
    out = torch.empty_like(s.rho)
    s.step()
    got = F.fmm_scf_update(s.tree, D.single_star_params(ctr, 0.25, 1.0 / 32, n=n, rho_floor=1e-30), s.phi, s.rho, out)
    torch.cuda.synchronize()
    # no rotation: H = C - phi, u = H (1 / H_max), each rounded once as on the device
    u = (got["C"][0] - s.phi.cpu().numpy()) * (1.0 / got["H_max"][0])
    out = out.cpu().numpy()
    s.close()
    at = (out > 1e-30) & (u > 0)
    assert at.sum() > 1000
    v = u[at].astype(np.longdouble)
    want = v ** int(n) * (1 if n == int(n) else np.sqrt(v) if n % 1 == 0.5 else np.sqrt(np.sqrt(v)))
    assert (np.abs(out[at] - want) / np.spacing(out[at])).max() <= 1.0

"""The FP64 and double-float multipole and root kernels over the forms of
their dispatch: sixteenths of a sub-grid per item on small trees, quarters and
halves on larger ones, every stencil reach, both expansion orders."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from oracle import oracle as O
from workloads import adaptive_tree, leaf_cell_centres, uniform_tree
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu

# The oracle and the FP64 path agree to 1e-12 and double-float to 1e-12 on
# small trees (a few hundred terms of a hundred operations at 2^-48 each).
TOL = 1e-12


def _lopsided(max_level):
    c = np.array([0.3, 0.35, 0.3])

    def want(lo, hi):
        d = np.clip(c, lo, hi) - c
        return float(d @ d) < 0.16 ** 2
    return adaptive_tree(want, max_level)


def _case(name):
    # refined sub-grids below the root: 8 (sixteenths), 72 (quarters), and an
    # adaptive tree with leaf sources, absent ones and both mixed in a warp
    desc = {"uniform3": lambda: uniform_tree(3), "uniform4": lambda: uniform_tree(4),
            "adaptive5": lambda: _lopsided(5)}[name]()
    rng = np.random.default_rng(11)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.25, 0.6, (3, 3)), 0.07, 1.0)
    return desc, rho.reshape(-1, 512)


@pytest.mark.parametrize("precision", ["fp64", "dfloat"])
@pytest.mark.parametrize("name,theta,order", [("uniform3", 0.55, 3), ("uniform3", 0.35, 2),
                                              ("uniform4", 0.5, 3), ("adaptive5", 0.5, 3),
                                              ("adaptive5", 0.5, 2), ("adaptive5", 0.3, 3)])
def test_wide_kernels_match_oracle(name, theta, order, precision):
    desc, rho = _case(name)
    c = dict(desc=desc, theta=theta, G=1.0, box_lo=(0.0, 0.0, 0.0), box_size=1.0, order=order)
    ref = O.solve(O.Tree.from_config(c), rho)
    s = F.Solver(desc, theta, precision=precision, order=order)
    s.rho.copy_(torch.from_numpy(rho).cuda())
    bits = None
    for items in (0, 1, 2):                  # every item size gives the same bits
        F.fmm_set_tuning(s.tree, mp_items=items)
        s.step()
        torch.cuda.synchronize()
        g, phi = s.g.cpu().numpy(), s.phi.cpu().numpy()
        if bits is None:
            bits = g
        assert np.array_equal(g, bits)
    assert np.abs(g - ref["g"]).max() <= TOL * np.abs(ref["g"]).max()
    assert np.abs(phi - ref["phi"]).max() <= TOL * np.abs(ref["phi"]).max()
    tot = s.totals.cpu().numpy()[0]
    assert np.linalg.norm(tot[:3]) <= TOL * tot[6] and np.linalg.norm(tot[3:6]) <= TOL * tot[7]
    s.close()

"""Every order of the double-float Taylor coefficients against the oracle: sums
over a stencil whose terms cancel (L2, L3) as well as those whose terms do not."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from oracle import oracle as O
from workloads import leaf_cell_centres, uniform_tree
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu

# a term is some ten operations of 2^-48, whose roundings add up at random over
# the stencil: six units of 2^-48 of the order's size (2-norms)
TOL = 6 * 2.0 ** -48


@pytest.mark.parametrize("theta,order", [(0.5, 3), (0.35, 3), (0.5, 2)])
def test_orders_to_double_float_rounding(theta, order):
    desc = uniform_tree(4)
    rng = np.random.default_rng(11)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.25, 0.6, (3, 3)), 0.07, 1.0).reshape(-1, 512)
    c = dict(desc=desc, theta=theta, G=1.0, box_lo=(0.0, 0.0, 0.0), box_size=1.0, order=order)
    t = O.Tree.from_config(c)
    s = F.Solver(desc, theta, precision="dfloat", order=order)
    s.rho.copy_(torch.from_numpy(rho).cuda())
    s.upward()
    s.m2l()
    torch.cuda.synchronize()
    # (the oracle on the library's own moments: its upward pass sums one by one;
    # the library leaves a leaf cell's centre and moments implied)
    refined = desc[:, 5] >= 0
    M, com = s.M.cpu().numpy().copy(), s.com.cpu().numpy().copy()
    M[~refined, 1:] = 0.0
    com[~refined] = leaf_cell_centres(desc).transpose(0, 2, 1)
    ref, _, _ = O.m2l(t, M, com)
    L = s.L.double().cpu().numpy() + s.Lc.double().cpu().numpy()
    # the oracle's are physical, the library's in level units: G / h^(n+1)
    h = 1.0 / (8 * 2.0 ** (desc[:, 0] - 1))
    for n, sl in enumerate((slice(0, 1), slice(1, 4), slice(4, 10), slice(10, 20))):
        at = refined if n > 1 else slice(None)
        if n > order:
            continue
        a = L[:, sl][at]
        b = (np.asarray(ref).reshape(len(desc), 20, 512)[:, sl] * h[:, None, None] ** (n + 1))[at]
        assert np.linalg.norm(a - b) <= TOL * np.linalg.norm(b), n
    s.close()

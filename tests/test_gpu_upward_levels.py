"""The upward pass of the double-float precisions against moments combined child
by child in long double, over the kernels a level's nodes go through: only leaf
children, no leaf children, both in one launch (few nodes) and in two (many).
(The oracle sums thousands of leaf cells one after the other for a coarse cell,
to about 1e-12: too coarse a reference for this.)"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from workloads import make_config, uniform_tree, leaf_cell_centres
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu

# 48-bit arithmetic, about fifty operations per moment and level
TOL = 1e-12
I2 = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
I3 = [(0, 0, 0), (0, 0, 1), (0, 0, 2), (0, 1, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2),
      (2, 2, 2)]


def _case(name):
    if name == "cfg5_small":
        return make_config(name)
    desc = uniform_tree(3)
    rho = gaussian_blobs(leaf_cell_centres(desc), np.array([[0.4, 0.5, 0.6], [0.7, 0.3, 0.5]]), 0.08, 1.0)
    return dict(desc=desc, rho=rho.reshape(-1, 512), theta=0.5, G=1.0, box_lo=(0.0, 0.0, 0.0), box_size=1.0)


def _moments(desc, rho):
    """M [n][20][512] and com [n][3][512] of the refined nodes, child by child."""
    n = len(desc)
    c = np.arange(512)
    xyz = np.stack([c & 7, (c >> 3) & 7, c >> 6], 1)
    h = 1.0 / (8 * 2.0 ** (desc[:, 0] - 1))
    M = np.zeros((n, 20, 512), np.longdouble)
    X = ((8 * desc[:, None, 1:4] + xyz + 0.5) * h[:, None, None]).astype(np.longdouble)   # (n, 512, 3)
    leaf = desc[:, 5] < 0
    M[leaf, 0] = rho * h[leaf, None] ** 3
    kid = (xyz[:, 0] >> 2) + 2 * (xyz[:, 1] >> 2) + 4 * (xyz[:, 2] >> 2)
    for level in range(desc[:, 0].max(), 0, -1):
        at = np.nonzero(~leaf & (desc[:, 0] == level))[0]
        if len(at) == 0:
            continue
        ch = desc[at][:, 5 + kid]                                                         # (N, 512)
        cells = [((2 * (xyz & 3) + [j & 1, (j >> 1) & 1, j >> 2]) @ [1, 8, 64]) for j in range(8)]
        m = [M[ch, 0, cc] for cc in cells]
        x = [X[ch, cc] for cc in cells]
        m0 = sum(m)
        com = sum(a[..., None] * b for a, b in zip(m, x)) / m0[..., None]
        M[at, 0], X[at] = m0, com
        for a, b, cc in zip(m, x, cells):
            s = b - com
            c2 = {p: M[ch, 4 + k, cc] for k, p in enumerate(I2)}
            g = lambda i, j: c2[tuple(sorted((i, j)))]
            for k, (i, j) in enumerate(I2):
                M[at, 4 + k] += g(i, j) + a * s[..., i] * s[..., j]
            for k, (i, j, l) in enumerate(I3):
                M[at, 10 + k] += (M[ch, 10 + k, cc] + g(i, j) * s[..., l] + g(i, l) * s[..., j] +
                                  g(j, l) * s[..., i] + a * s[..., i] * s[..., j] * s[..., l])
    return M, X.transpose(0, 2, 1)


@pytest.mark.parametrize("precision", ["mixed", "dfloat"])
@pytest.mark.parametrize("name", ["uniform3", "cfg5_small"])
def test_moments_level_by_level(name, precision):
    c = _case(name)
    M_ref, com_ref = _moments(c["desc"], c["rho"])
    s = F.Solver(c["desc"], c["theta"], precision=precision)
    s.rho.copy_(torch.from_numpy(c["rho"]).cuda())
    s.upward()
    torch.cuda.synchronize()
    M, com = s.M.cpu().numpy(), s.com.cpu().numpy()
    refined = c["desc"][:, 5] >= 0
    for level in np.unique(c["desc"][refined, 0]):
        at = refined & (c["desc"][:, 0] == level)
        h = 1.0 / (8 * 2 ** (level - 1))
        assert np.abs(com[at] - com_ref[at]).max() <= TOL * h
        assert np.all(M[at][:, 1:4] == 0.0)
        for sl in (slice(0, 1), slice(4, 10), slice(10, 20)):
            assert np.abs(M[at][:, sl] - M_ref[at][:, sl]).max() <= TOL * np.abs(M_ref[at][:, sl]).max()
    s.close()

"""fmm_forces by its launch shapes (one, four or eight cells per thread) against
the fused leaf pass of fmm_step, bit for bit."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from workloads import adaptive_tree, leaf_cell_centres
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu


def _corner(max_level, radius):
    c = np.array([0.2, 0.25, 0.3])

    def want(lo, hi):
        d = np.clip(c, lo, hi) - c
        return float(d @ d) < radius ** 2
    return adaptive_tree(want, max_level)


# one cell per thread, four and eight
@pytest.mark.parametrize("precision", ["mixed", "dfloat", "fp64"])
@pytest.mark.parametrize("level,radius,leaves", [(5, 0.3, 876), (6, 0.15, 1653), (6, 0.18, 2115)])
def test_forces_shapes_agree(level, radius, leaves, precision):
    desc = _corner(level, radius)
    assert (desc[:, 5] < 0).sum() == leaves
    rng = np.random.default_rng(4)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.2, 0.5, (2, 3)), 0.06, 1.0).reshape(-1, 512)
    s = F.Solver(desc, 0.5, precision=precision)
    s.rho.copy_(torch.from_numpy(rho).cuda())
    out = []
    for run in (s.step, s.step_passes):
        for t in (s.phi, s.g, s.totals):
            t.zero_()
        run()
        torch.cuda.synchronize()
        out.append([t.cpu().numpy().copy() for t in (s.phi, s.g, s.totals)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    s.close()

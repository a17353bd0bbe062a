"""The mixed monopole kernel's form for trees with many leaf sub-grids (16-bit
window offsets) against its form for one sub-grid per pass, bit for bit, at
every reach and for an odd number of leaf sub-grids."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from workloads import adaptive_tree, leaf_cell_centres
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [0.57, 0.5, 0.35, 0.28])
def test_monopole_forms_agree(theta):
    # 4096 leaf sub-grids, 27 of them refined once more: 4285
    desc = adaptive_tree(lambda lo, hi: bool(np.all(lo < 0.55) and np.all(hi > 0.41)), 6, min_level=5)
    assert (desc[:, 5] < 0).sum() % 2 == 1 and (desc[:, 5] < 0).sum() > 2432
    rng = np.random.default_rng(11)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.3, 0.7, (3, 3)), 0.1, 1.0).reshape(-1, 512)
    s = F.Solver(desc, theta, precision="mixed")
    s.rho.copy_(torch.from_numpy(rho).cuda())
    out = []
    for subgrids in (2, 1):
        F.fmm_set_tuning(s.tree, mono_subgrids=subgrids)
        for run in (s.step, s.step_passes):
            for t in (s.L, s.Lc, s.phi, s.g):
                t.zero_()
            run()
            torch.cuda.synchronize()
            out.append([t.cpu().numpy().copy() for t in (s.L, s.Lc, s.phi, s.g, s.totals)])
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert np.array_equal(a, b)
    s.close()

"""The mixed precision's launch shapes for trees that do not fill the SMs (pairs
of warps, quarters, halves with the loads ahead, one thread per leaf cell) against
the shapes of large trees, bit for bit, and against the oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1908_03121_gb300 as F
from oracle import oracle as O
from workloads import adaptive_tree, leaf_cell_centres, uniform_tree
from workloads.density import gaussian_blobs

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-6                 # the mixed precision's bar


def _corner(max_level, radius=0.1):
    c = np.array([0.2, 0.25, 0.3])

    def want(lo, hi):
        d = np.clip(c, lo, hi) - c
        return float(d @ d) < radius ** 2
    return adaptive_tree(want, max_level)


# refined sub-grids below the root: 8 and 16 (pairs of warps), 44 and 72
# (quarters, four warps), 80 (halves with the loads ahead); leaf sub-grids: 64,
# 120 (a thread per cell), 316, 512 and 568
@pytest.mark.parametrize("tree,theta,order", [("uniform3", 0.5, 3), ("corner4", 0.5, 3),
                                              ("corner4", 0.35, 2), ("corner4", 0.28, 3),
                                              ("corner4", 0.57, 3), ("uniform4", 0.5, 3),
                                              ("corner5", 0.5, 2), ("corner5", 0.28, 3),
                                              ("corner5", 0.57, 3), ("wide5", 0.5, 3)])
def test_launch_shapes_agree(tree, theta, order):
    desc = {"uniform3": lambda: uniform_tree(3), "uniform4": lambda: uniform_tree(4),
            "corner4": lambda: _corner(4), "corner5": lambda: _corner(5, 0.13),
            "wide5": lambda: _corner(5, 0.2)}[tree]()
    rng = np.random.default_rng(3)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.2, 0.5, (2, 3)), 0.06, 1.0).reshape(-1, 512)
    c = dict(desc=desc, theta=theta, G=1.0, box_lo=(0.0, 0.0, 0.0), box_size=1.0, order=order)
    ref = O.solve(O.Tree.from_config(c), rho)
    s = F.Solver(desc, theta, precision="mixed", order=order)
    s.rho.copy_(torch.from_numpy(rho).cuda())
    out = []
    for items in (0, 1, 2):
        F.fmm_set_tuning(s.tree, mp_items=items)
        for run in (s.step, s.step_passes):
            run()
            torch.cuda.synchronize()
            out.append([t.cpu().numpy().copy() for t in (s.L64, s.dacc, s.phi, s.g, s.totals)])
    refined = desc[:, 5] >= 0
    written = np.broadcast_to(refined[:, None, None] | (np.arange(20) < 4)[None, :, None], out[0][0].shape)
    for o in out[1:]:
        assert np.array_equal(o[0][written], out[0][0][written])
        for a, b in zip(o[1:], out[0][1:]):
            assert np.array_equal(a, b)
    assert np.abs(out[0][3] - ref["g"]).max() <= FORCE_TOL * np.abs(ref["g"]).max()
    s.close()


# leaf sub-grids: 120, 260 (one cell per thread; FP64 four), 316, 568 (four)
@pytest.mark.parametrize("precision", ["mixed", "dfloat", "fp64"])
@pytest.mark.parametrize("radius,level", [(0.1, 4), (0.1, 5), (0.13, 5), (0.2, 5)])
def test_leaf_pass_shapes_agree(precision, radius, level):
    desc = _corner(level, radius)
    rng = np.random.default_rng(4)
    rho = gaussian_blobs(leaf_cell_centres(desc), rng.uniform(0.2, 0.5, (2, 3)), 0.06, 1.0).reshape(-1, 512)
    s = F.Solver(desc, 0.5, precision=precision)
    s.rho.copy_(torch.from_numpy(rho).cuda())
    out = []
    for run in (s.step, s.step_passes):      # the fused pass, and shifts and forces apart
        run()
        torch.cuda.synchronize()
        out.append([t.cpu().numpy().copy() for t in (s.phi, s.g, s.dacc, s.totals)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    s.close()

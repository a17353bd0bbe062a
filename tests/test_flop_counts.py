"""The operation counts behind the roofline figures: in FP64 and double-float a
monopole pair costs what the transformed kernel executes, not the direct form's
eight operations."""

import itertools

import pytest

import paper_1908_03121_gb300 as F
from workloads import uniform_tree


def _block_operations(theta):
    """Operations per pair of one block of eight target cells, counted from the
    near block offsets."""
    r = int(1.0 / theta)
    near = [d for d in itertools.product(range(-r, r + 1), repeat=3) if theta ** 2 * sum(x * x for x in d) <= 1.0]
    pairs = 8 * (8 * len(near) - 1)
    ops = 0.0
    for d in {tuple(abs(x) for x in d) for d in near} - {(0, 0, 0)}:
        k = sum(x > 0 for x in d)
        ops += 8 * 2 ** k * (2 * 4 + k)          # eight b: products with four components, sums over signs
    ops += (4 + 2 * r) ** 3 / 64 * 3 * 8         # sources' transform
    ops += 4 * (7 * 8 + 3 * 8)                   # sums over b, targets' transform
    own = sum(1 + sum(a != b for a, b in zip(p, s))
              for p, s in itertools.permutations(itertools.product((0, 1), repeat=3), 2))
    return (ops + 2 * own + 4 * 8) / pairs


@pytest.mark.parametrize("theta", [0.577, 0.5, 0.35, 0.28])
@pytest.mark.parametrize("precision", ["fp64", "dfloat"])
def test_wide_monopole_operations(theta, precision):
    t = F.fmm_build_tree(uniform_tree(2), theta, precision=precision, host_only=True)
    got = t.stats["flops_per_interaction"][2]
    assert got == pytest.approx(_block_operations(theta), rel=1e-12)
    assert got < 2.0
    t.close()


def test_mixed_monopole_operations():
    t = F.fmm_build_tree(uniform_tree(2), 0.5, precision="mixed", host_only=True)
    assert t.stats["flops_per_interaction"][2] == 8.0
    t.close()

"""Small point clouds run whole iterations in one launch of a cluster of 16 blocks (lamp_cluster.cu):
which problems do, and that the launch takes the decisions of the four-kernel iteration."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import gpu_solver

pytestmark = pytest.mark.gpu


def solver(n, m, d, cost="sqeuclid", **kw):
    w = W.points_problem(f"cl{n}", n, m, d, seed=3 * n + m, marg="random")
    w.kind = cost
    return gpu_solver(w, **kw)[0]


# at the limits: 1024 points a side, n m (2 d + 7) = 1.1e7 (d = 1: 1024 x 1024 is below it, d = 2 above)
@pytest.mark.parametrize("n,m,d,chip", [(1, 1, 1, True), (256, 256, 2, True), (1024, 1024, 1, True), (1024, 1024, 2, False),
                                        (1024, 976, 2, True), (1024, 977, 2, False), (1025, 16, 1, False),
                                        (16, 1025, 1, False), (1024, 467, 8, True), (1024, 468, 8, False)])
def test_which_problems_run_on_chip(n, m, d, chip):
    s = solver(n, m, d)
    assert s.on_chip() == chip
    s.close()


@pytest.mark.parametrize("n,m,d,cost", [(1, 1, 1, "sqeuclid"), (2, 1024, 2, "l1"), (256, 256, 2, "sqeuclid"),
                                        (1024, 1024, 1, "sqeuclid"), (1024, 976, 2, "linf"), (1024, 467, 8, "sqeuclid")])
def test_full_capacity_matches_four_kernels(n, m, d, cost):
    """The states of a launch are those of the four kernels (time_kernels) to the bit."""
    a, b = solver(n, m, d, cost), solver(n, m, d, cost)
    assert a.on_chip()
    a.iterate(23)
    b.time_kernels(22)
    sa, sb = a.get_state(), b.get_state()
    assert sa["t"] == sb["t"] == 23 and sa["kappa"] == sb["kappa"]
    for key in ("nu", "theta", "row_shifts"):
        assert np.array_equal(sa[key], sb[key]), key
    a.close()
    b.close()

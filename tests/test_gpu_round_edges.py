"""Round of l1 and l-inf costs at the edges of the packed pass that forms C delta_c (512 or 1024 rows per
block, tiles of 128 columns, pairs), against the oracle's dense Round.  Tolerance: OBJ_TOL of K for the
cost (float32 cost and sums, float64 results), RES_FLOOR for the masses."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from tests.gpu_util import OBJ_TOL, RES_FLOOR, gpu_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,d,cost", [(1, 1, 1, "l1"), (3, 1, 2, "linf"), (1, 129, 8, "l1"), (513, 127, 5, "linf"),
                                        (512, 128, 6, "l1"), (1025, 257, 3, "l1"), (1024, 384, 4, "linf"), (130, 2049, 1, "linf")])
def test_round_of_l1_and_linf(n, m, d, cost):
    w = W.points_problem(f"rd{n}", n, m, d, seed=n + m, marg="random")
    w.kind = cost
    sol, C, K = gpu_solver(w)
    sol.iterate(5)
    st = sol.get_state()
    got = sol.round()
    sol.close()
    X = w.r[:, None] * O.dual_to_primal(C, K, st["kappa"], st["nu"])[0]
    x, y, X2, dr, dc = O.round_factors(X, w.r, w.c)
    want = float((C * O.round_plan(X, w.r, w.c)).sum())
    assert abs(got["cost"] - want) <= OBJ_TOL * K
    assert abs(got["dr_l1"] - dr.sum()) <= RES_FLOOR and abs(got["dc_l1"] - dc.sum()) <= RES_FLOOR
    # the bilinear term alone: delta_r^T C delta_c / ||delta_r||
    if dr.sum() > 0.01:
        assert abs((got["cost"] - got["cost_scaled"]) - float(dr @ C @ dc) / dr.sum()) <= OBJ_TOL * K

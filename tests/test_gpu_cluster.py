"""Small point clouds run whole iterations in one launch of a cluster of 16 blocks (lamp_cluster.cu):
which problems do, and that the launch takes the decisions of the four-kernel iteration."""
import ctypes

import numpy as np
import pytest

import oracle as O

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


@pytest.mark.parametrize("n,chip", [(200, True), (1100, False)])
def test_an_earlier_numeric_failure_stops_the_iterations(n, chip):
    """A recorded LAMP_E_NUMERIC stops every later iteration until lamp_set_state, on either route."""
    import paper_2511_11359_gb300 as L

    w = W.points_problem("bad", n, n, 2, seed=n, marg="random", cost_scale=1.0)
    nu, bad = np.empty(n), w.r.copy()
    bad[n // 2] = np.nan  # column sums that are not numbers
    h = L.LampHost(w.r, w.c, x=w.x, y=w.y, cost_scale=w.cost_scale)
    assert bool(L.lib.lamp_on_chip(h._h)) == chip
    assert np.isfinite(h.step(3, nu_out=nu)) and np.abs(nu).max() > 0
    after, again = np.empty(n), np.empty(n)
    assert np.isnan(h.step(2, r=bad, nu_out=after))
    res = h.step(2, nu_out=again)  # good data again, but the failure stands
    assert np.isfinite(res)
    assert np.array_equal(after, nu) and np.array_equal(again, nu)
    assert L.lib.lamp_set_state(h._h, nu.ctypes.data, nu.ctypes.data, 1.0, 3, None) == 0
    h.step(2, nu_out=again)
    assert not np.array_equal(again, nu)
    h.close()


@pytest.mark.parametrize("n,chip", [(200, True), (1100, False)])
def test_row_sums_out_of_range(n, chip):
    """Row shifts far off leave row sums below the representable range: LAMP_E_NUMERIC, the state
    stays, and the reported infeasibility is that of the column sums (about 0 against c)."""
    import paper_2511_11359_gb300 as L

    s = solver(n, n, 2, tol=1e-9, max_iter=50)
    assert s.on_chip() == chip
    s.iterate(5)
    st = s.get_state()
    s.set_state(st["nu"], st["theta"], st["kappa"], st["t"], st["row_shifts"] + np.float32(300.0))
    out = L._Result()
    assert L.lib.lamp_solve(s._h, ctypes.byref(out)) == L.LAMP_E_NUMERIC
    assert out.status == L.LAMP_E_NUMERIC and out.iters == 5 and abs(out.infeas - 1.0) <= 1e-6
    assert np.array_equal(s.get_state()["nu"], st["nu"])
    s.close()


def test_stops_inside_a_launch():
    """A tolerance met, and max_iter reached, in the middle of a launch: the state is the one that four
    kernels reach at that iteration."""
    T = 85  # the first X^t below the geometric mean of its residual and the smallest one before
    w = W.points_problem("stop", 300, 260, 2, seed=9, marg="random")
    s, C, K = gpu_solver(w)
    s.close()
    P = O.LampParams(K=K)
    res = [O.objective_report(C, w.r, w.c, K, 0.0, O.lamp_run(C, w.r, w.c, P, t))["col_res"] for t in range(1, T + 1)]
    tol = float(np.sqrt(min(res[:-1]) * res[-1]))
    assert res[-1] < tol * (1 - 1e-3)
    b, _, _ = gpu_solver(w)
    b.time_kernels(T - 1)
    sb = b.get_state()
    for kw, conv in (({"tol": tol, "max_iter": 500}, True), ({"tol": 0.0, "max_iter": T}, False)):
        a, _, _ = gpu_solver(w, check_every=50, **kw)
        assert a.on_chip()
        info, sa = a.solve(), a.get_state()
        assert info["iters"] == T and info["converged"] == conv
        assert all(np.array_equal(sa[q], sb[q]) for q in ("nu", "theta", "row_shifts")) and sa["kappa"] == sb["kappa"]
        a.close()
    b.close()

"""The low-dimensional (d <= 8) and the stored-cost kernels at the edges of their tiles, against
the oracle: sweeps whose groups of 64 inner points are dealt to warps (a warp owns 32 outer
points, or 128), gradient, transport map and row maxima of the packed weighted-sum kernels, and
stored costs with rows that are not a multiple of 16 bytes apart (4 rows and 1024 columns, 256
columns and 16 rows per tile).  Tolerances: cost_slack (1e-5 plus 4 kappa times the float32 cost's
error) for potentials, the path's 1e-4 for gradients and maps, 1e-6 for the objective."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from tests.gpu_util import GRAD_TOL, OBJ_TOL, RES_FLOOR, cost_slack, gpu_solver, oracle_cost

pytestmark = pytest.mark.gpu

# (n, m, d, cost): one point; one past a warp, a group, a tile; several tiles per split; the wide form
POINTS = [(1, 3, 1, "sqeuclid"), (33, 65, 2, "sqeuclid"), (129, 127, 8, "l1"), (257, 1025, 5, "linf"),
          (700, 1000, 3, "sqeuclid"), (2100, 3333, 3, "sqeuclid"), (5000, 900, 7, "l1")]


@pytest.mark.parametrize("n,m,d,cost", POINTS)
def test_points_tile_edges(n, m, d, cost):
    import torch

    T = 12
    w = W.points_problem(f"dir{n}", n, m, d, seed=n + d, marg="random")
    w.kind = cost
    C, s, K = oracle_cost(w)
    ref = O.lamp_run(C, w.r, w.c, O.LampParams(K=K), T)
    sol, _, _ = gpu_solver(w, K=K, scale=s, check_every=5)
    sol.iterate(T)
    st = sol.get_state()
    tol = cost_slack(w, ref.kappa)
    assert np.abs(st["nu"] - ref.nu).max() <= tol and np.abs(st["theta"] - ref.theta).max() <= tol

    sol.set_state(ref.nu, ref.theta, ref.kappa, ref.t)
    ob, want = sol.objective(), O.objective_report(C, w.r, w.c, K, 0.0, ref)
    assert abs(ob["cost"] - want["cost"]) <= OBJ_TOL * want["cost"] + tol * RES_FLOOR
    dual = max(O.saddle_dual(C, w.r, w.c, K, ref.theta), O.saddle_dual(C, w.r, w.c, K, ref.nu))
    assert abs(ob["dual"] - dual) <= OBJ_TOL * K
    p = O.dual_to_primal(C, K, ref.kappa, ref.nu)[0]
    if cost == "sqeuclid":
        gx, gy = O.grad_envelope(w.x, w.y, w.r[:, None] * p, scale=s)
        dx, dy = (g.cpu().numpy().astype(np.float64) for g in sol.grad())
        assert np.abs(dx - gx).max() <= GRAD_TOL * np.abs(gx).max()
        assert np.abs(dy - gy).max() <= GRAD_TOL * np.abs(gy).max()
    rng = np.random.default_rng(n)
    for k in (1, 3, 6):
        V, U = (rng.standard_normal((q, k)).astype(np.float32) for q in (m, n))
        for side, val, out in ((0, V, p @ V), (1, U, p.T @ U)):
            got = sol.apply_map(torch.from_numpy(val).cuda(), side=side).cpu().numpy()
            assert np.abs(got - out).max() <= GRAD_TOL * max(1.0, np.abs(out).max())
    # log Z is the current state's after a map alone, too
    sol.set_state(ref.nu, ref.theta, ref.kappa, ref.t)
    assert np.isnan(sol.get_state()["logZ"]).all()
    sol.apply_map(torch.from_numpy(V).cuda(), side=0)
    lz = O.log_normalizers(C, K, ref.kappa, ref.nu)
    assert np.abs(sol.get_state()["logZ"] - lz).max() <= 1e-5 * (1.0 + np.abs(lz).max())
    sol.close()


@pytest.mark.parametrize("n,m", [(1, 1025), (5, 2047), (17, 257), (33, 1), (300, 1023), (1201, 1537)])
def test_stored_cost_unaligned_rows(n, m):
    w = W.dense_problem(f"odd{n}", n, m, seed=n + m)
    C, s, K = oracle_cost(w)
    T = 20
    ref = O.lamp_run(C, w.r, w.c, O.LampParams(K=K), T)
    sol, _, _ = gpu_solver(w, K=K, check_every=7)
    sol.iterate(T)
    st = sol.get_state()
    tol = cost_slack(w, ref.kappa)
    assert np.abs(st["nu"] - ref.nu).max() <= tol and np.abs(st["theta"] - ref.theta).max() <= tol
    sol.set_state(ref.nu, ref.theta, ref.kappa, ref.t)
    ob, want = sol.objective(), O.objective_report(C, w.r, w.c, K, 0.0, ref)
    assert abs(ob["cost"] - want["cost"]) <= OBJ_TOL * want["cost"]
    dual = max(O.saddle_dual(C, w.r, w.c, K, ref.theta), O.saddle_dual(C, w.r, w.c, K, ref.nu))
    assert abs(ob["dual"] - dual) <= 1e-9 * K
    sol.close()


@pytest.mark.parametrize("n,m", [(1, 4), (31, 260), (33, 1028), (300, 2052)])
def test_stored_cost_row_maxima(n, m):
    """Row maxima of stored costs read by tensor copies (32 x 256 tiles): the shifts of a run that
    resumes from a given state, and the dual bound's refined maxima."""
    w = W.dense_problem(f"mx{n}", n, m, seed=n + m)
    C, s, K = oracle_cost(w)
    P = O.LampParams(K=K)
    mid, ref = O.lamp_run(C, w.r, w.c, P, 20), O.lamp_run(C, w.r, w.c, P, 30)
    sol, _, _ = gpu_solver(w, K=K, check_every=7)
    sol.set_state(mid.nu, mid.theta, mid.kappa, mid.t)
    dual = max(O.saddle_dual(C, w.r, w.c, K, mid.theta), O.saddle_dual(C, w.r, w.c, K, mid.nu))
    assert abs(sol.objective()["dual"] - dual) <= 1e-9 * K
    sol.iterate(10)
    st = sol.get_state()
    tol = cost_slack(w, ref.kappa)
    assert np.abs(st["nu"] - ref.nu).max() <= tol and np.abs(st["theta"] - ref.theta).max() <= tol
    sol.close()


@pytest.mark.parametrize("n,m,d,cost,eta", [(1, 1, 1, "sqeuclid", 0.0), (2, 1024, 8, "sqeuclid", 0.0),
                                            (1024, 129, 3, "l1", 0.0), (97, 130, 2, "linf", 0.0),
                                            (256, 256, 2, "sqeuclid", 0.0), (500, 641, 4, "sqeuclid", 1e-2)])
def test_whole_iterations_in_one_launch(n, m, d, cost, eta):
    """Small problems run whole iterations in one launch; lamp_time_kernels runs the same
    iterations as four kernels each: the states are the same to the bit, whole and resumed."""
    T = 37
    w = W.points_problem(f"one{n}", n, m, d, seed=3 * n + m, marg="random", eta=eta)
    w.kind = cost
    a, _, K = gpu_solver(w, eta=eta)
    b, _, _ = gpu_solver(w, eta=eta)
    a.iterate(20)
    a.iterate(T - 20)
    b.time_kernels(T - 1)
    sa, sb = a.get_state(), b.get_state()
    assert sa["t"] == sb["t"] == T and sa["kappa"] == sb["kappa"]
    for key in ("nu", "theta", "row_shifts"):
        assert np.array_equal(sa[key], sb[key]), key
    oa, ob = a.objective(), b.objective()
    assert all(oa[q] == ob[q] or (np.isnan(oa[q]) and np.isnan(ob[q])) for q in oa)
    a.close()
    b.close()

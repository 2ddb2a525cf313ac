"""The float32 dot-form kernels (|x - y|^2 with d > 8: sweeps, gradient, transport map) at the
edges of their tiles (128 outer points, stages of 256 inner points, 16 value columns), against
the oracle.  Tolerances: potentials 1e-5 plus 4 kappa times the bound of the float32 dot
product's error, d 2^-24 s (max |x|^2 + max |y|^2); gradients and maps the path's 1e-4."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from tests.gpu_util import GRAD_TOL, POT_TOL, gpu_solver, oracle_cost

pytestmark = pytest.mark.gpu

SIZES = [(1, 3, 9), (127, 129, 9), (129, 257, 16), (256, 385, 33), (300, 128, 64), (1500, 2100, 17)]


@pytest.mark.parametrize("n,m,d", SIZES)
def test_dot_form_tile_edges(n, m, d):
    import torch

    T = 12
    w = W.points_problem(f"dot{n}", n, m, d, seed=n + d, dist="gauss_shift", marg="random", cost_scale=0.05)
    C, s, K = oracle_cost(w)
    ref = O.lamp_run(C, w.r, w.c, O.LampParams(K=K), T)
    sol, _, _ = gpu_solver(w, K=K, scale=s, check_every=5)
    sol.iterate(T)
    st = sol.get_state()
    nx, ny = (np.asarray(p, np.float64) ** 2 for p in (w.x, w.y))
    tol = POT_TOL + 4.0 * ref.kappa * d * 2.0 ** -24 * s * (nx.sum(1).max() + ny.sum(1).max())
    assert np.abs(st["nu"] - ref.nu).max() <= tol and np.abs(st["theta"] - ref.theta).max() <= tol

    sol.set_state(ref.nu, ref.theta, ref.kappa, ref.t)
    p = O.dual_to_primal(C, K, ref.kappa, ref.nu)[0]
    gx, gy = O.grad_envelope(w.x, w.y, w.r[:, None] * p, scale=s)
    dx, dy = (g.cpu().numpy().astype(np.float64) for g in sol.grad())
    assert np.abs(dx - gx).max() <= GRAD_TOL * np.abs(gx).max()
    assert np.abs(dy - gy).max() <= GRAD_TOL * np.abs(gy).max()
    rng = np.random.default_rng(d)
    V, U = (rng.standard_normal((q, 3)).astype(np.float32) for q in (m, n))
    for side, val, want in ((0, V, p @ V), (1, U, p.T @ U)):
        out = sol.apply_map(torch.from_numpy(val).cuda(), side=side).cpu().numpy()
        assert np.abs(out - want).max() <= GRAD_TOL * max(1.0, np.abs(want).max())
    sol.close()

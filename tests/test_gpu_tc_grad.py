"""The tensor-core gradient pass at the edges of its tiles (128 fixed points, 64 streamed points a
tile, three S / P buffers, five ring slots; four coordinates per thread in the finalize) against
the oracle's envelope gradient on the oracle's state.  Tolerance: the path's 1e-4 of the largest
gradient (P carries 16 significant bits, 2^-17 per entry)."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import workloads as W
from tests.gpu_util import GRAD_TOL, gpu_solver, oracle_cost

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,d", [(1, 1, 9), (2, 64, 64), (128, 65, 10), (129, 192, 11), (193, 257, 33), (321, 449, 62)])
def test_tc_gradient_tile_edges(n, m, d):
    w = W.points_problem(f"tce{n}", n, m, d, seed=n + d, dist="gauss_shift", marg="random", cost_scale=0.05)
    w = dataclasses.replace(w, x=W.bf16_round(w.x), y=W.bf16_round(w.y))
    C, s, K = oracle_cost(w)
    st = O.lamp_run(C, w.r, w.c, O.LampParams(K=K), 10)
    sol, _, _ = gpu_solver(w, K=K, scale=s, prec="bf16_tc", check_every=5)
    sol.set_state(st.nu, st.theta, st.kappa, st.t)
    X = w.r[:, None] * O.dual_to_primal(C, K, st.kappa, st.nu)[0]
    for got, want in zip(sol.grad(), O.grad_envelope(w.x, w.y, X, scale=s)):
        assert np.abs(got.cpu().numpy().astype(np.float64) - want).max() <= GRAD_TOL * np.abs(want).max()
    sol.close()

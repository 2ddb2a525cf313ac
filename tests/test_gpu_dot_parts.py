"""The float32 gradient with d > 8 of more points than its partial sums hold at a time (256 MiB): the
outer points go in parts of whole waves of tiles.  Against float64 at the same state; tolerance: the
path's 1e-4 of the largest gradient."""
import numpy as np
import pytest

from tests.gpu_util import GRAD_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(530001, 65), (33, 700000)])
def test_gradient_in_parts(n, m):
    import torch
    import paper_2511_11359_gb300 as L

    g = torch.Generator(device="cuda").manual_seed(n)
    d, s = 64, 1.0 / 64
    x = torch.randn(n, d, generator=g, device="cuda")
    y = torch.randn(m, d, generator=g, device="cuda") + 0.5
    r, c = (torch.rand(k, generator=g, device="cuda", dtype=torch.float64) + 0.1 for k in (n, m))
    r, c = r / r.sum(), c / c.sum()
    sol = L.Lamp(r, c, x=x, y=y, cost_scale=s)
    sol.iterate(6)
    st, K = sol.get_state(), sol.objective()["K"]
    dx, dy = sol.grad()
    sol.close()
    x, y, nu = x.double(), y.double(), torch.from_numpy(st["nu"]).cuda()
    C = s * ((x * x).sum(1)[:, None] + (y * y).sum(1)[None] - 2.0 * x @ y.T)
    X = r[:, None] * torch.softmax(-st["kappa"] * (C + 2.0 * K * nu[None]), 1)
    gx, gy = 2.0 * s * (r[:, None] * x - X @ y), 2.0 * s * (X.sum(0)[:, None] * y - X.T @ x)
    for got, want in ((dx, gx), (dy, gy)):
        # each part against its own largest gradient: points near the borders of the parts count as any other
        for a, b in zip(got.double().split(19456), want.split(19456)):
            assert (a - b).abs().max() <= GRAD_TOL * b.abs().max()

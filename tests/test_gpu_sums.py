"""Float32 partial sums of the gradient, the transport map and Round: how many terms are added before
they go into a wider sum.

At the start of Alg. 2 (kappa = 0) every weight is a power of two when n and m are, so the sums are
plain sums of the values.  Equal values c make the rounding errors of a chain of additions add up: a sum
of k equal terms is off by at most sum_{j <= k} j u / k = (k + 1) / 2 u of itself (u = 2^-24), 4.5 u for
the 8 terms that these passes add in float32; one more u for the float32 result.  For the values below
chains of 32 and 64 terms are off by 8 u and more."""
import numpy as np
import pytest

from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
VALUES = np.array([1.8835506439208984, 1.8873310089111328, 1.9065380096435547, 1.9167194366455078, 1.9315128326416016,
                   1.9315433502197266, 1.940958023071289, 1.9603939056396484], np.float32)
N, M = 512, 1024


def context(x, y, c=None, **kw):
    import paper_2511_11359_gb300 as L

    c = np.full(M, 1.0 / M) if c is None else c
    return L.Lamp(dev(np.full(N, 1.0 / N)), dev(c), x=dev(x), y=dev(y), **kw)


@pytest.mark.parametrize("d,prec,k", [(1, "fp32", 1), (3, "fp32", 3), (3, "fp32", 4), (8, "fp32", 8), (2, "fp32", 6),
                                      (12, "fp32", 3), (64, "fp32", 8), (64, "bf16_tc", 4)])
def test_transport_map(d, prec, k):
    rng = np.random.default_rng(d)
    s = context(rng.random((N, d), dtype=np.float32), rng.random((M, d), dtype=np.float32), prec=prec)
    for side, np_in, np_out in ((0, M, N), (1, N, M)):
        out = s.apply_map(dev(np.tile(VALUES[:k], (np_in, 1))), side).cpu().numpy().astype(np.float64)
        want = VALUES[:k].astype(np.float64) * (1.0 if side == 0 else N / M)  # row sums of p are 1, of p^T n / m
        assert out.shape == (np_out, k) and np.abs(out / want - 1.0).max() <= 5.5 * U
    s.close()


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8, 9, 17, 33, 64])
def test_gradient(d):
    v, z = np.resize(VALUES, d), np.zeros
    for x, y, which in ((z((N, d), np.float32), np.tile(v, (M, 1)), 0), (np.tile(v, (N, 1)), z((M, d), np.float32), 1)):
        s = context(x, y)
        g = s.grad()[which].cpu().numpy().astype(np.float64)  # 2 s (mass 0 - weight sum)
        want = -2.0 * v.astype(np.float64) / (N if which == 0 else M)
        assert np.abs(g / want - 1.0).max() <= 5.5 * U
        s.close()


@pytest.mark.parametrize("cost,d", [("l1", 1), ("linf", 8)])
def test_round(cost, d):
    """delta_r^T C delta_c / ||delta_r|| = c ||delta_c|| for a cost of equal entries c, with a power of
    two as delta_c of half the columns: 32 terms are added in float32, 16 to a lane of a pair, so the
    error is that of 16 additions (emulated here) and one more."""
    half = np.where(np.arange(M) < M // 2, 1.5, 0.5) / M
    for v in VALUES:
        s = context(np.zeros((N, d), np.float32), np.full((M, d), v, np.float32), half, cost=cost)
        o = s.round()
        s.close()
        assert o["dc_l1"] == 0.25
        a = np.float32(0.0)
        for _ in range(16):
            a += v
        err = (o["cost"] - o["cost_scaled"]) / (0.25 * float(v)) - 1.0
        assert abs(err) <= abs(float(a) / (16.0 * float(v)) - 1.0) + 1.0 * U

"""lamp_step_host on new points (float32 dot form and tensor cores): the copies that the kernels read
(transposed in tiles of 32 x 32, or bf16) are those of the new points, at the edges of their tiles.  The
points change sign, which keeps their norms, and K is given; the state is set after the upload, so that
its row shifts are those of the new points too (the start's are taken from the points of the creation)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,d", [(1, 3, 9), (31, 33, 31), (255, 257, 33), (256, 512, 64), (513, 130, 32)])
@pytest.mark.parametrize("prec", ["fp32", "bf16_tc"])
def test_steps_on_new_points(n, m, d, prec):
    import paper_2511_11359_gb300 as L

    w = W.points_problem(f"host{n}", n, m, d, seed=n + d, dist="gauss_shift", marg="random")
    K = 8.0 * float((w.x.astype(np.float64) ** 2).sum(1).max() + (w.y.astype(np.float64) ** 2).sum(1).max())
    kw = dict(prec=prec, K=K, cost_scale=0.5)
    h = L.LampHost(w.r, w.c, x=w.x, y=w.y, **kw)
    nu, zero = np.empty(m), np.zeros(m)
    for sign in (-1.0, 1.0):
        x = np.ascontiguousarray(np.float32(sign) * w.x)
        h.step(1, a=x, nu_out=nu)
        assert L.lib.lamp_set_state(h._h, zero.ctypes.data, zero.ctypes.data, 0.0, 0, None) == 0
        h.step(7, a=x, nu_out=nu)
        with L.Lamp(dev(w.r), dev(w.c), x=dev(x), y=dev(w.y), **kw) as s:
            s.iterate(7)
            assert np.array_equal(nu, s.get_state()["nu"])
    h.close()

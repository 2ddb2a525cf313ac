"""Points that start on a 4-byte boundary (a slice of a larger buffer): every cost and precision gives
what it gives for an aligned copy of them, to the bit."""
import ctypes

import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


def shifted(a):
    """The same values one float past a 16-byte boundary."""
    import torch

    buf = torch.empty(a.numel() + 4, dtype=a.dtype, device=a.device)
    v = buf[1:1 + a.numel()].view(a.shape)
    v.copy_(a)
    assert v.data_ptr() % 16 == 4 and v.is_contiguous()
    return v


@pytest.mark.parametrize("cost,d,prec", [("l1", 12, "fp32"), ("linf", 64, "fp32"), ("l1", 4, "fp32"), ("sqeuclid", 8, "fp32"),
                                         ("sqeuclid", 16, "fp32"), ("cosine", 12, "fp32"), ("sqeuclid", 64, "bf16_tc")])
def test_points_off_a_16_byte_boundary(cost, d, prec):
    import paper_2511_11359_gb300 as L

    w = W.points_problem("off", 150, 131, d, seed=d, marg="random")
    r, c, x, y = dev(w.r), dev(w.c), dev(w.x), dev(w.y)
    V = dev(np.random.default_rng(d).standard_normal((131, 3)).astype(np.float32))
    got = []
    for px, py, pv in ((x, y, V), (shifted(x), shifted(y), shifted(V))):
        with L.Lamp(r, c, x=px, y=py, cost=cost, prec=prec) as s:
            s.iterate(12)
            st = s.get_state()
            o = [st["nu"], st["theta"], np.array(list(s.objective().values())), np.array([s.round()["cost"]]),
                 s.apply_map(pv).cpu().numpy()]
            if cost == "sqeuclid":
                o += [g.cpu().numpy() for g in s.grad()]
            got.append(o)
    for a, b in zip(*got):
        assert np.array_equal(a, b, equal_nan=True)


def test_marginals_of_points_off_a_16_byte_boundary():
    import torch
    from tests.test_zz_no_alloc import _fn, _problem

    L, f = _fn()
    w = W.points_problem("off", 150, 131, 4, seed=4)
    t = {"r": dev(w.r), "c": dev(w.c), "x": dev(w.x), "y": dev(w.y)}
    nu = torch.linspace(-0.3, 0.3, 131, dtype=torch.float64, device="cuda")
    res = []
    for q in (t, {**t, "x": shifted(t["x"]), "y": shifted(t["y"])}):
        out = [torch.empty(k, dtype=torch.float64, device="cuda") for k in (150, 131, 1)]
        pr = _problem(L, w, q, 1.0)
        p = [ctypes.c_void_p(o.data_ptr()) for o in out]
        st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert f(ctypes.byref(pr), 3.0, 2.0, ctypes.c_void_p(nu.data_ptr()), *p, st) == 0
        torch.cuda.synchronize()
        res.append([o.cpu().numpy() for o in out])
    for a, b in zip(*res):
        assert np.isfinite(a).all() and np.array_equal(a, b)

"""Host code of the C ABI over a stand-in for the CUDA runtime (tests/fake_cudart.cpp): what a call
does on a second device and when an allocation or a runtime call fails.  The library's own object
files are linked with the stand-in; no kernel runs."""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2511_11359_gb300 import build as b
    import paper_2511_11359_gb300 as L

    b.build(force=not all((b.BUILD / (Path(s).stem + ".o")).exists() for s in b.SOURCES))
    so = tmp_path_factory.mktemp("fake") / "libfake.so"
    inc = Path(b.nvcc_path()).resolve().parents[1] / "include"
    objs = [str(b.BUILD / (Path(s).stem + ".o")) for s in b.SOURCES]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", str(inc),
                    str(ROOT / "tests" / "fake_cudart.cpp"), *objs, "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    vp, i64 = ctypes.c_void_p, ctypes.c_int64
    lib.lamp_create.argtypes = [ctypes.POINTER(vp), vp, vp, vp]
    lib.lamp_create_owned.argtypes = lib.lamp_create.argtypes
    lib.lamp_step_host.argtypes = [vp, vp, vp, vp, vp, i64, ctypes.POINTER(ctypes.c_double), vp]
    lib.lamp_iterate.argtypes = [vp, i64]
    lib.lamp_grad.argtypes = [vp, vp, vp]
    lib.lamp_apply_map.argtypes = [vp, vp, i64, vp, ctypes.c_int]
    lib.lamp_last_error.argtypes, lib.lamp_last_error.restype = [vp], ctypes.c_char_p
    lib.lamp_destroy.argtypes, lib.lamp_destroy.restype = [vp], None
    lib.fake_fail_alloc.argtypes = lib.fake_limit.argtypes = [ctypes.c_longlong]
    for f in ("bad", "reads", "launches", "graph_launches", "graphs", "bytes", "peak"):
        getattr(lib, "fake_" + f).restype = ctypes.c_longlong
    lib.L = L
    lib.fake_reset()
    yield lib


@pytest.fixture
def make(fake):
    """make(kind, n, m, d, prec) -> (code, handle); handles are destroyed afterwards."""
    L, made = fake.L, []

    def f(kind, n, m, d, prec=0, **params):
        buf = np.zeros(8)  # inputs are never read: no kernel runs
        p = L._Problem()
        p.n, p.m, p.d, p.kind, p.ldc, p.cost_scale = n, m, d, kind, m, 1.0
        p.C = p.x = p.y = p.r = p.c = buf.ctypes.data // 16 * 16
        h = ctypes.c_void_p()
        pa = L.default_params(prec=prec, K=1.0, **params)
        code = fake.lamp_create(ctypes.byref(h), ctypes.byref(p), ctypes.byref(pa), None)
        if h.value:
            made.append(h)
        return code, h

    fake.fake_reset()
    yield f
    for h in made:
        fake.lamp_destroy(h)
    fake.fake_reset()


BUF = ctypes.c_void_p(4096)  # an output that no kernel writes


@pytest.mark.parametrize("kind,d,prec", [("SQEUCLID", 64, 0), ("SQEUCLID", 64, 1), ("COSINE", 13, 0), ("L1", 64, 0),
                                         ("LINF", 48, 0), ("SQEUCLID", 8, 0), ("DENSE", 0, 0)])
def test_every_device_of_a_process(fake, make, kind, d, prec):
    """Shared-memory limits belong to a device: every kernel of a context launches on the second
    device that a process uses, too."""
    for device in (0, 1):
        fake.fake_set_device(device)
        code, h = make(getattr(fake.L, "COST_" + kind), 3000, 2048, d, prec)
        assert code == 0, fake.lamp_last_error(None)
        assert fake.lamp_iterate(h, 3) == 0, fake.lamp_last_error(h)
        for side in (0, 1):
            assert fake.lamp_apply_map(h, BUF, 3, BUF, side) == 0, fake.lamp_last_error(h)
        if kind == "SQEUCLID":
            assert fake.lamp_grad(h, BUF, BUF) == 0, fake.lamp_last_error(h)


@pytest.mark.parametrize("kind,d", [("SQEUCLID", 64), ("L1", 64)])
def test_failure_to_raise_a_limit_is_reported(fake, make, kind, d):
    fake.fake_fail_attr(1)
    code, h = make(getattr(fake.L, "COST_" + kind), 300, 200, d)
    assert code == fake.L.LAMP_E_CUDA and not h.value
    assert b"fake error" in fake.lamp_last_error(None)


def test_a_failed_allocation_is_reported_once(fake, make):
    code, h = make(fake.L.COST_SQEUCLID, 500, 400, 3)
    fake.fake_fail_alloc(0)
    assert code == 0 and fake.lamp_grad(h, BUF, BUF) == fake.L.LAMP_E_NOMEM
    fake.fake_fail_alloc(-1)
    assert fake.lamp_iterate(h, 2) == 0, fake.lamp_last_error(h)
    assert fake.lamp_grad(h, BUF, BUF) == 0


@pytest.mark.parametrize("kind,d,prec,call,watch,after", [
    # a tensor-core context's transposed points for the transport map, and those of its gradient
    ("SQEUCLID", 64, 1, "map", ("k_transpose_points", 3), 0), ("SQEUCLID", 64, 1, "map", ("k_transpose_points", 3), 1),
    ("SQEUCLID", 64, 1, "grad", ("k_transpose_bf16", 2), 0), ("SQEUCLID", 64, 1, "grad", ("k_transpose_bf16", 2), 1),
    # l1 with d > 8: wider partial sums, which the iteration's sweeps write too
    ("L1", 20, 0, "map", ("k_pts_sweep", 6), 0)])
def test_context_survives_a_failed_allocation(fake, make, kind, d, prec, call, watch, after):
    """LAMP_E_NOMEM leaves the context as it was: no later launch gets memory that was released or
    never allocated, and the call works once there is memory."""
    code, h = make(getattr(fake.L, "COST_" + kind), 500, 400, d, prec)
    assert code == 0
    if call == "map" and kind == "L1":
        assert fake.lamp_apply_map(h, BUF, 4, BUF, 0) == 0  # widened once already

    def run():
        return fake.lamp_grad(h, BUF, BUF) if call == "grad" else fake.lamp_apply_map(h, BUF, 8, BUF, 0)

    fake.fake_watch(watch[0].encode(), watch[1])
    before = fake.fake_bytes()
    fake.fake_fail_alloc(after)
    code = run()
    fake.fake_fail_alloc(-1)
    assert code == fake.L.LAMP_E_NOMEM
    assert fake.lamp_iterate(h, 2) == 0 and fake.fake_bad() == 0
    assert run() == 0 and fake.lamp_iterate(h, 2) == 0, fake.lamp_last_error(h)
    assert fake.fake_bad() == 0 and fake.fake_bytes() >= before


@pytest.mark.parametrize("n,m,d", [(1 << 18, 1 << 18, 64), (40001, 1 << 18, 33), (1 << 18, 100, 9), (3000, 3001, 64)])
@pytest.mark.parametrize("room", [256, 33])
def test_gradient_partials_are_bounded(fake, make, n, m, d, room):
    """The float32 gradient's partial sums stay within 256 MiB, whatever the number of points, and
    within 32 MiB where there is no more memory; they are allocated once, and every launch gets its
    part of them."""
    code, h = make(fake.L.COST_SQEUCLID, n, m, d)
    assert code == 0
    fake.fake_watch(b"k_dot_grad_fin", 0)
    before = fake.fake_bytes()
    fake.fake_limit(before + (room << 20))
    for _ in range(2):
        assert fake.lamp_grad(h, BUF, BUF) == 0, fake.lamp_last_error(h)
    assert 0 < fake.fake_bytes() - before <= room << 20
    assert fake.fake_bad() == 0


@pytest.mark.parametrize("d,prec", [(2, 0), (64, 0), (64, 1)])
def test_a_host_step_reads_the_control_block_once(fake, d, prec):
    """lamp_step_host reads back the control block, in one copy, and nu."""
    L, n, m = fake.L, 300, 200
    r, c, x, y, nu = (np.zeros(k) for k in (n, m, n * d, m * d, m))
    p = L._Problem()
    p.n, p.m, p.d, p.kind, p.cost_scale = n, m, d, L.COST_SQEUCLID, 1.0
    p.x, p.y, p.r, p.c = (a.ctypes.data for a in (x, y, r, c))
    h, inf = ctypes.c_void_p(), ctypes.c_double()
    fake.fake_reset()
    assert fake.lamp_create_owned(ctypes.byref(h), ctypes.byref(p), ctypes.byref(L.default_params(prec=prec, K=1.0)), None) == 0
    for out in (nu.ctypes.data, 0):
        before = fake.fake_reads()
        assert fake.lamp_step_host(h, p.x, p.y, p.r, p.c, 1, ctypes.byref(inf), out) == 0
        assert fake.fake_reads() - before == (2 if out else 1)
    fake.lamp_destroy(h)

"""The finalize step's table log2 (lamp_fin.cuh) against CUDA's over the range of the row sums, 1e-36 to
1e36, arguments near 1, near powers of two and near the table's boundaries: its result carries two
roundings of numbers of at most |v| + 1 and 2^-54 of the table's entry, CUDA's at most one unit in the
last place."""
import ctypes
import subprocess

import pytest

from paper_2511_11359_gb300 import build as b

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch

    torch.zeros(1, device="cuda")  # the primary context first
    so = tmp_path_factory.mktemp("probe") / "fin_probe.so"
    subprocess.run([b.nvcc_path(), *b.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
                    "-I", str(b.CSRC), str(b.ROOT / "tests" / "fin_probe.cu"), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def run(x):
        x = x.cuda().contiguous()
        got, want = torch.empty_like(x), torch.empty_like(x)
        torch.cuda.synchronize()
        p = [ctypes.c_void_p(t.data_ptr()) for t in (got, want)]
        assert lib.probe_log2(ctypes.c_void_p(x.data_ptr()), x.numel(), *p) == 0
        return got, want

    return run


def near(x, ulps):
    """x and its neighbours up to `ulps` units in the last place away."""
    import torch

    bits = x.view(torch.int64)
    return torch.cat([(bits + k).view(torch.float64) for k in range(-ulps, ulps + 1)])


def spread(gen, n, lo, hi):
    import torch

    return torch.exp2(lo + (hi - lo) * torch.rand(n, generator=gen, dtype=torch.float64))


def test_log2(probe):
    import torch

    g = torch.Generator().manual_seed(2)
    one = torch.ones(1, dtype=torch.float64)
    bounds = torch.cat([(1.0 + torch.arange(128, dtype=torch.float64) / 128) * s for s in (2.0 ** -119, 2.0 ** -1, 1.0, 2.0 ** 118)])
    x = torch.cat([spread(g, 1 << 20, -119.5, 119.5), spread(g, 1 << 18, -1.0, 1.0), near(one, 300), near(bounds, 8),
                   near(torch.exp2(torch.arange(-119, 120, dtype=torch.float64)), 8)]).clamp(1e-36, 1e36)
    got, want = probe(x)
    tol = 2.0 ** -52 * (want.abs().clamp(min=1.0) + 0.25) + 2.0 ** -53 * (want.abs() + 1.0)
    assert bool(((got - want).abs() <= tol).all()), float(((got - want).abs() / tol).max())

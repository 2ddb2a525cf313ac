"""What ptxas reports of the built kernels: the packed sweeps of low-dimensional point clouds keep
their state in registers.  Their unroll factors depend on d and on the sums, and a factor that is right
at one d spills at another."""
import re

import pytest

from paper_2511_11359_gb300 import build as b


def spills(unit):
    """{kernel: bytes of spill stores and loads} of a translation unit's kernels."""
    log = b.BUILD / (unit + ".log")
    b.build(force=not log.exists())
    out, name = {}, None
    for line in log.read_text().splitlines():
        m = re.search(r"Compiling entry function '(\w+)'", line)
        name = m.group(1) if m else name
        m = re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m:
            out[name] = int(m.group(1)) + int(m.group(2))
    return out


@pytest.mark.parametrize("unit,kernel,count", [("lamp_direct", "k_pts_direct", 96), ("lamp_direct_small", "k_direct_small", 192),
                                               ("lamp_cluster", "k_cluster_iterate", 24), ("lamp_wsum", "k_direct_max", 24)])
def test_packed_sweeps_do_not_spill(unit, kernel, count):
    got = {k: v for k, v in spills(unit).items() if kernel in k}
    assert len(got) == count
    assert not {k: v for k, v in got.items() if v}

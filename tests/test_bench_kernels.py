"""bench.py reports the kernels that a step launches: the four of an iteration, or the one launch of a
problem whose iterations run on chip."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


class Solver:
    def __init__(self, chip):
        self.chip, self.iterated = chip, 0

    def on_chip(self):
        return self.chip

    def iterate(self, k):
        self.iterated += k

    def time_kernels(self, iters):
        assert not self.chip
        return [4.0, 1.0, 5.0, 2.0]

    def launches_per_iteration(self):
        return 4


def test_kernels_of_a_step():
    s = Solver(False)
    kern, launches = bench.iteration_kernels(s, 5, None)
    assert kern == {"row_sweep": 4.0, "row_fin": 1.0, "col_sweep": 5.0, "col_fin": 2.0} and launches == 4
    assert bench.dominant_sweep(kern) == ("col_sweep", 5.0, "column")

    s = Solver(True)
    kern, launches = bench.iteration_kernels(s, 5, lambda f: f() or 40.0)
    assert s.iterated == 50 and kern == {"on_chip_iteration": 0.8} and launches == 1
    name, ms, what = bench.dominant_sweep(kern)
    assert name is None and ms == 0.4 and "on chip" in what


def test_no_traffic_record_names_an_on_chip_kernel():
    assert bench.ncu_traffic("plain_2d", "fp32", 256, 2, None) is None

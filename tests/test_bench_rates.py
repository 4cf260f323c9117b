"""Host-side helpers of bench.py (no GPU): the bytes that its rates are of, and which launch they name."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2102_04709_gb300 import workloads as W  # noqa: E402


class Sim:
    def __init__(self, rho):
        self.rho = rho

    def fields(self):
        return self.rho, None


def test_rates_are_of_the_emptier_end_of_a_run():
    """A droplet that has spread over more tiles: its bytes are not those of the run that led there."""
    w = W.pillars(nx=320, ny=120, count=3, r_lo=6.0, r_hi=9.0, x_lo=150.0, x_hi=260.0, gap=8.0, seed=5,
                  drop=(60.0, 60.0), r_core=8.0, r_shell=14.0, u_in=0.05)
    spread = w.rho.copy()
    spread[0, :, :200] += 1e-30
    before, after = (bench.bytes_moved(w, Sim(r), 72) for r in (w.rho, spread))
    assert after[0] > before[0] and after[1] > before[1] and after[2] < before[2]
    assert bench.fewer_bytes(before, after) == bench.fewer_bytes(after, before) == before


def test_rate_of_the_one_launch_of_small_grids():
    """No time of the pure tiles: all bytes over the time of the launch there is."""
    assert np.isclose(bench.pure_gbs((2e9, 3e9), 4.0, 7.0, 2), 1000.0)
    assert np.isclose(bench.pure_gbs((2e9, 3e9), 0.0, 6.0, 2), 1000.0)

"""bench.py reports measured DRAM traffic only for the kernel instance that was measured.

The persistent FP32 plane kernel is compiled per grid and disk bound, so a capture of one instance
says nothing about another on the same grid: such a system's line has no traffic figure.
"""

import types

import numpy as np

import bench
import synth


def traffic(n, L, variant):
    s = types.SimpleNamespace(grid=(n, n, n), miller=synth.half_sphere(L, 25.0))
    return bench.roofline_line(s, "mixed_df", variant, 3, 1.0, 3 * 32768, 1, 10.0)["traffic"], int(np.abs(s.miller[:, 0]).max())


def test_traffic_only_for_the_captured_instance():
    t, xmax = traffic(64, 20.0, 5)  # the medium system
    assert xmax == 15 and abs(t - (210.849e6 + 146.837e6)) < 1.0
    t, xmax = traffic(64, 64 * 28.0 / 96.0, 5)  # the batching family's cell on the same grid
    assert xmax == 14 and t is None
    t, xmax = traffic(96, 28.0, 5)
    assert xmax == 22 and t > 0
    assert traffic(64, 20.0, 8)[0] is None

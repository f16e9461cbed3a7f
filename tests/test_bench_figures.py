"""Figures of bench.py's JSON line that describe the present kernels: the bytes that they move
(the planes of the state by word, the cell counts) and how many of them are launched."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("pp_mat", [False, True])
def test_moved_bytes_follow_the_planes(pp_mat):
    N, bricks, nodes = 1 << 20, 64 ** 3, 3150 * 64
    plane, cell = 16, 4
    mb = bench.moved_bytes(N, bricks, nodes, pp_mat)
    assert mb["p2g"] == N * (4 + 6 * plane) + nodes * plane
    assert mb["g2p"] == N * (4 + 4 * plane + 8 * plane + 8 + (16 if pp_mat else 0)) + nodes * 2 * plane
    assert mb["grid"] == nodes * (2 * plane + cell)
    assert mb["sort"] == 4 * bricks + N * 16 + nodes * 2 * cell
    r = bench.roofline_fields(N, bricks, nodes, {"sort": 0.01, "p2g": 0.04, "grid": 0.005, "g2p": 0.06}, 0.12, 6790.7,
                              "measured", pp_mat)
    line = bench.published(r)
    assert line["moved_bytes_per_launch"] == mb["g2p"]
    assert line["moved_bytes_per_particle_substep"] == pytest.approx(sum(mb.values()) / N, abs=0.05)
    assert not [k for k in line if "implementation" in k]
    assert {k for k in r if k not in line} == {"implementation_bytes_per_launch", "implementation_bytes_per_particle_substep"}


def test_timed_launches():
    # scan, scatter, P2G, grid update, G2P; histogram reset and keys; with a restart the state write too
    assert bench.timed_launches(500, 0) == 5 * 500 + 2
    assert bench.timed_launches(525, 1) == 5 * 525 + 2 + 3

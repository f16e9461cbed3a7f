"""A mesh blade with one of its two reaches undefined (NaN): the faces, or the spine, touch
nothing, and the other one touches what it does with the first one's reach below zero."""
import numpy as np
import pytest

from paper_2502_18437_gb300 import mpm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lost", ["thickness", "spine_radius"])
def test_the_other_reach_of_a_mesh_blade_still_touches(lost):
    sc = W.elastic_cube()
    dx = 1.0 / sc["n"]
    mid = tuple(float(t) for t in 0.5 * (sc["x"].min(0) + sc["x"].max(0)) + np.array([0.31, 0.17, -0.23]) * dx)
    pts = np.linspace(-0.15, 0.15, 9)[:, None] * np.array([1.0, 0.2, -0.1])
    tris = [[k, k + 1, 9 + k] for k in range(8)] + [[k + 1, 10 + k, 9 + k] for k in range(8)]
    got = []
    for value in (-1.0, float("nan")):
        reach = {"thickness": 1.5 * dx, "spine_radius": 1.2 * dx, lost: value}
        tool = W.mesh_slicer(mid, (1, 0, 0, 0), np.concatenate([pts, pts + np.array([0.0, 0.1, 0.03])]), np.array(tris),
                             np.arange(9), vel=(0.3, -0.2, 0.1), mu_k=0.3, **reach)
        with mpm.from_workload(dict(sc, rigids=[tool])) as sim:
            sim.substep(sc["dt"], 2)
            got.append(sim.read_state(0, ("x", "v", "impulse")))
    assert np.abs(got[0]["impulse"][0, :3]).max() > 0
    for f in ("x", "v", "impulse"):
        assert np.abs(got[1][f] - got[0][f]).max() <= 1e-5 * np.abs(got[0][f]).max(), f

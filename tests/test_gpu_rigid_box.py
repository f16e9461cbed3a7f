"""Threads and mesh blades turned against the grid, with reaches from none to several
cells: the nodes that their bounding box leaves out are those that the oracle does not
touch.  The thread is straight and the blade flat, so that a node nearest to two
segments or triangles gets the same normal and tangent from either.  One substep against the FP64 oracle, with the tolerances of parity_util."""
import numpy as np
import pytest

from paper_2502_18437_gb300 import workloads as W
from tests.parity_util import Scales, assert_close, perturbed
from tests.test_gpu_parity import check_fields, check_grid, gpu_one_step, oracle_one_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", ["segments", "mesh_slicer"])
@pytest.mark.parametrize("margin", [0.0, 1.0, 3.5])
def test_bounding_box_leaves_out_no_contact(shape, margin):
    sc = W.elastic_cube()
    dx = 1.0 / sc["n"]
    x = sc["x"]
    mid = tuple(float(t) for t in 0.5 * (x.min(0) + x.max(0)) + np.array([0.31, 0.17, -0.23]) * dx)
    g = np.random.default_rng(23)
    q = g.normal(size=4)
    quat = tuple(q / np.linalg.norm(q))
    pts = np.linspace(-0.15, 0.15, 9)[:, None] * np.array([1.0, 0.2, -0.1])
    if shape == "segments":
        tool = W.segments(mid, quat, pts, radius=0.4 * dx, vel=(0.3, -0.2, 0.1), mu_k=0.3, c_d=0.9, margin=margin * dx)
    else:
        top = pts + np.array([0.0, 0.1, 0.03])
        tris = [[k, k + 1, 9 + k] for k in range(8)] + [[k + 1, 10 + k, 9 + k] for k in range(8)]
        tool = W.mesh_slicer(mid, quat, np.concatenate([pts, top]), np.array(tris), np.arange(9), thickness=0.5 * dx,
                             vel=(0.3, -0.2, 0.1), mu_k=0.3, c_d=0.9, margin=margin * dx)
    sc["rigids"] = [tool]
    v, C, F = perturbed(sc, seed=29, f_amp=0.01, c_amp=0.5)
    x, v, C, F, out = gpu_one_step(sc, v, C, F)
    st, gm, gv, err, imp = oracle_one_step(sc, x, v, C, F)
    assert err == 0
    check_fields(sc, out, st, Scales(sc, F))
    check_grid(sc, out, gm, gv, Scales(sc, F))
    assert np.abs(imp[:, :3]).max() > 0
    assert_close("impulse", out["impulse"][0], imp[0], rtol=1e-4, rel_scale=1e-4)

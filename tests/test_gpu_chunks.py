"""P2G and the cell sort where their chunks of slots are ragged: few particles, counts
around the 32 and 64 slots of a warp, runs longer than a chunk, rows of neighbouring
cells with gaps and across brick faces, and particles alone in their cell.  One substep
against the FP64 oracle, element by element, with the tolerances of parity_util."""
import numpy as np
import pytest

import oracle
from paper_2502_18437_gb300 import workloads as W
from tests.parity_util import Scales, assert_close, oracle_cfg, oracle_state, perturbed
from tests.test_gpu_parity import check_fields, check_grid, gpu_one_step, oracle_one_step
from tests.test_gpu_solvers import gpu_step

pytestmark = pytest.mark.gpu


def scene(kind, count):
    n = 32
    g = np.random.default_rng(17 + count)
    u = g.random((count, 3))
    if kind == "cell":
        cells = np.tile([10, 11, 12], (count, 1))
    elif kind == "rows":  # along z, through brick faces, every third cell empty
        z = g.choice([k for k in range(6, 26) if k % 3], size=count)
        cells = np.stack([np.full(count, 9), 11 + (np.arange(count) % 2), z], -1)
    else:  # one particle here and there
        cells = g.integers(5, 26, size=(count, 3))
    x = (cells + 0.5 + u) / n
    return W._scene(n, x, np.zeros_like(x), 1e4, 0.3, rho=1.0, V0=(0.5 / n) ** 3, model="fixed_corotated", dt=1e-4,
                    substeps=1, name=kind)


@pytest.mark.parametrize("kind", ["cell", "rows", "spread"])
@pytest.mark.parametrize("count", [1, 31, 32, 33, 65, 193, 1000])
def test_ragged_chunks_match_oracle(kind, count):
    sc = scene(kind, count)
    v, C, F = perturbed(sc, seed=count)
    x, v, C, F, out = gpu_one_step(sc, v, C, F)
    st, gm, gv, err, _ = oracle_one_step(sc, x, v, C, F)
    assert err == 0
    check_fields(sc, out, st, Scales(sc, F))
    check_grid(sc, out, gm, gv, Scales(sc, F))


@pytest.mark.parametrize("count", [1, 33, 193])
def test_ragged_chunks_standard_mpm(count):
    sc = scene("rows", count)
    v, C, F = perturbed(sc, seed=count, c_amp=0.0)
    st, out = gpu_step(sc, v, C, F, "standard")
    ost = oracle_state(sc, st["x"], st["v"], st["C"], st["F"])
    assert oracle.run_solver(oracle_cfg(sc), ost, sc["dt"], 1, "standard") == 0
    err = Scales(sc, st["F"])
    assert_close("x", out["x"], ost.x)
    assert_close("v", out["v"], ost.v, atol_floor=err.atol_v(ost.v))
    assert_close("L", out["C"], ost.C, atol_floor=err.atol_C(ost.v))
    assert_close("F", out["F"], ost.F)

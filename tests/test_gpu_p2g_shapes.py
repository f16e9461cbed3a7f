"""P2G with every number of slots that a warp stages (32, 48, 64), whatever the launch's size:
chunks of one batch, of one and a half and of two, ragged ones, runs longer than a batch or a
chunk, and several scenes in one chunk, for the three solvers.  Each scene against the FP64
oracle on that scene alone, from a state without the stored stress and from one with it, with
the tolerances of parity_util and test_gpu_solvers."""
import ctypes as ct

import numpy as np
import pytest

import oracle
from paper_2502_18437_gb300 import mpm
from tests.parity_util import EPS32, Scales, assert_close, oracle_cfg, oracle_state, perturbed
from tests.test_gpu_chunks import scene
from tests.test_gpu_parity import dense_bricks_scene

pytestmark = pytest.mark.gpu

COUNTS = [33, 0, 1, 47, 17, 48, 65, 5, 129, 700]  # scenes of one context
CYCLES = 2


def check(sc, solver, st, out):
    if len(sc["x"]) == 0:
        return
    ost = oracle_state(sc, st["x"], st["v"], st["C"], st["F"])
    if solver == "mls":
        assert oracle.run(oracle_cfg(sc), ost, sc["dt"], 1) == 0
    else:
        assert oracle.run_solver(oracle_cfg(sc), ost, sc["dt"], 1, solver, iters=CYCLES, beta=1.0) == 0
    err = Scales(sc, st["F"])
    vmax = np.abs(ost.v).max()
    c_floor = 8 * EPS32 / sc["dt"] * CYCLES  # the constraint's division by dt
    pb = solver == "pb"
    assert_close("x", out["x"], ost.x)
    assert_close("v", out["v"], ost.v, atol_floor=c_floor / sc["n"] + 2e-5 * vmax if pb else err.atol_v(ost.v))
    assert_close("C", out["C"], ost.C,
                 atol_floor=4 * c_floor + 27 * 4 * sc["n"] * EPS32 * vmax if pb else err.atol_C(ost.v))
    assert_close("F", out["F"], ost.F, atol_floor=c_floor * sc["dt"] if pb else 0.0)


@pytest.mark.parametrize("solver", ["mls", "standard", "pb"])
@pytest.mark.parametrize("kind", ["cell", "rows", "spread", "dense"])
@pytest.mark.parametrize("chunk", [384, 576, 768])
def test_chunks_match_oracle(chunk, kind, solver):
    scenes = [dense_bricks_scene()] if kind == "dense" else [scene(kind, c) for c in COUNTS]
    for sc in scenes:
        sc["dt"] = 0.02 if solver == "pb" else 1e-4
    with mpm.from_scenes(scenes, solver=solver, pb_iterations=CYCLES, pb_beta=1.0) as sim:
        sim.set_option("p2g_chunk", chunk)
        for s, sc in enumerate(scenes):
            if len(sc["x"]):
                v, C, F = perturbed(sc, seed=61 + s, c_amp=0.0 if solver == "standard" else 0.5, v_amp=0.05)
                sim.write_state(s, v=v, C=C, F=F)
        before = [sim.read_state(s) for s in range(len(scenes))]
        for _ in range(2):
            sim.substep(scenes[0]["dt"], 1)
            after = [sim.read_state(s) for s in range(len(scenes))]
            for sc, st, out in zip(scenes, before, after):
                check(sc, solver, st, out)
            before = after


def test_a_set_chunk_is_used_at_every_size():
    slots = getattr(mpm.lib(), "_ZN3mpm13p2g_slots_forEPK7mpm_ctxi")
    slots.restype, slots.argtypes = ct.c_int, [ct.c_void_p, ct.c_int]
    sc = dense_bricks_scene()
    with mpm.from_workload(sc) as sim:
        assert [slots(sim.h, n) for n in (1, 100000, 1 << 20)] == [32, 32, 64]
        assert sim.get_option("p2g_chunk") == 384  # of a launch over the scene's 2,200 particles
        for chunk in (384, 576, 768):
            sim.set_option("p2g_chunk", chunk)
            assert [slots(sim.h, n) for n in (1, 100000, 1 << 20)] == [chunk // 12] * 3
            assert sim.get_option("p2g_chunk") == chunk
        sim.autotune(sc["dt"], 2)
        assert slots(sim.h, 2200) == sim.get_option("p2g_chunk") // 12

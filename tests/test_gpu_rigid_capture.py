"""mpm_set_rigid while the context's stream is captured: refused, and nothing of the context or
of the capture changes."""
import numpy as np
import pytest

from paper_2502_18437_gb300 import mpm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refused", ["remove", "other kind", "another rigid"])
def test_a_refused_rigid_leaves_the_context_as_it_was(refused):
    torch = pytest.importorskip("torch")
    # a sphere inside the block pushes particles out and takes momentum from them
    sc = W.elastic_cube(n_side=10)
    mid = 0.5 * (sc["x"].min(0) + sc["x"].max(0))
    sc["rigids"] = [W.sphere(tuple(mid), 0.06, vel=(0.0, 0.3, 0.0), mu_k=0.2, margin=1 / 32)]
    thread = W.segments(tuple(mid), (1, 0, 0, 0), np.array([[-0.1, 0, 0], [0.1, 0, 0]]), radius=0.02)
    got = []
    for captured in (False, True):
        stream = torch.cuda.Stream()
        with mpm.from_workload(sc, stream=stream.cuda_stream) as sim:
            sim.substep(sc["dt"], 3)
            sim.read_state(0)
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                    with pytest.raises(mpm.MPMError) as e:
                        if refused == "remove":
                            sim.remove_rigid(0, 0)
                        else:
                            sim.set_rigid(0, 0 if refused == "other kind" else 1, thread)
                assert e.value.status == -3
            sim.impulse(0)
            sim.substep(sc["dt"], 5)
            got.append(sim.read_state(0, ("x", "v", "impulse")))
    assert np.abs(got[0]["impulse"][0, :3]).max() > 0
    for f in ("x", "v", "impulse"):
        scale = np.abs(got[0][f]).max()
        assert np.abs(got[1][f] - got[0][f]).max() <= 1e-5 * scale, f

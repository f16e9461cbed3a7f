"""State I/O next to ids that are not of the scene: a substep that a device error cut short
leaves slots of the buffer that becomes the state unwritten.  The I/O kernels are called on
buffers made here, with margins that take what a kernel without its bound would write, so
that nothing here can leave an allocation; then a context whose sort was made inconsistent
from the host reports the error and hands out its older positions."""
import ctypes as ct

import numpy as np
import pytest

from paper_2502_18437_gb300 import mpm, workloads as W

pytestmark = pytest.mark.gpu

COMPS = {"x": 3, "v": 3, "C": 9, "F": 9}
# float of each component in a particle's eight planes of four
AT = {"x": range(0, 3), "v": range(13, 16), "C": range(16, 25), "F": range(4, 13)}
MARGIN = 8  # entries before and after each array


class PState(ct.Structure):
    _fields_ = [("q", ct.c_void_p), ("mu", ct.c_void_p), ("lam", ct.c_void_p)]


class Fields(ct.Structure):
    _fields_ = [("f", ct.c_void_p * 4)]


def launch_fields():
    f = getattr(mpm.lib(), "_ZN3mpm13launch_fieldsERKNS_6PStateES2_iiiPiRKNS_6FieldsEbbP11CUstream_st")
    f.restype = ct.c_int
    f.argtypes = [ct.POINTER(PState), ct.POINTER(PState), ct.c_int, ct.c_int, ct.c_int, ct.c_void_p,
                  ct.POINTER(Fields), ct.c_bool, ct.c_bool, ct.c_void_p]
    return f


def spoil_sort(sim):
    """Zero the particle counts that the next substep's sort relies on."""
    f = getattr(mpm.lib(), "_ZN3mpm15reset_histogramEP7mpm_ctx")
    f.restype, f.argtypes = ct.c_int, [ct.c_void_p]
    assert f(sim.h) == 0


@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("by_id", [False, True])
@pytest.mark.parametrize("fields", ["x", "v", "C", "F", "xF", "vC", "xvCF"])
@pytest.mark.parametrize("np_,p0", [(1, 0), (33, 5), (128, 0), (300, 129)])
def test_fields_move_between_arrays_and_the_scenes_own_ids(np_, p0, fields, by_id, bad):
    torch = pytest.importorskip("torch")
    g = np.random.default_rng(np_ + p0)
    cap = p0 + np_ + 3
    stray = np.array([np_, -1, np_ + 5, -3])[: np_ // 8] if bad else np.zeros(0, int)
    ids = g.permutation(np_).astype(np.int32)
    lost = g.permutation(np_)[: len(stray)]  # slots whose id is not of the scene
    missing = ids[lost].copy()
    ids[lost] = stray
    own = np.setdiff1d(np.arange(np_), lost)
    state = g.normal(size=(8, cap, 4)).astype(np.float32)
    state[0, :, 3].view(np.int32)[...] = 0
    state[0, p0:p0 + np_, 3] = ids.view(np.float32)
    spare = g.normal(size=(8, cap, 4)).astype(np.float32)
    slots = p0 + np.arange(np_)
    by_slot = state.transpose(1, 0, 2).reshape(cap, 32)
    for out in (True, False):
        q, s = torch.tensor(state, device="cuda"), torch.tensor(spare, device="cuda")
        inv = torch.full((cap,), p0 + int(own[0]) if len(own) else p0, dtype=torch.int32, device="cuda")
        arrs, h = {}, Fields()
        for k, f in enumerate("xvCF"):
            if f in fields:
                host = g.normal(size=(np_ + 2 * MARGIN, COMPS[f])).astype(np.float32)
                arrs[f] = (torch.tensor(host, device="cuda"), host)
                h.f[k] = arrs[f][0].data_ptr() + 4 * MARGIN * COMPS[f]
        st, sp = PState(q.data_ptr(), None, None), PState(s.data_ptr(), None, None)
        stream = torch.cuda.current_stream().cuda_stream
        assert launch_fields()(ct.byref(st), ct.byref(sp), cap, p0, np_, inv.data_ptr(), ct.byref(h), out, by_id,
                               stream) == 0
        torch.cuda.synchronize()
        after = q.cpu().numpy()
        for f, (dev, host) in arrs.items():
            now = dev.cpu().numpy()
            want = host.copy()
            if out:
                want[MARGIN + ids[own]] = by_slot[p0 + own][:, list(AT[f])]
                if by_id:  # an id that no slot has: whatever its inverse's old entry points at
                    want[MARGIN + missing] = now[MARGIN + missing]
            assert np.array_equal(now.view(np.int32), want.view(np.int32)), f
        want = by_slot.copy()
        if not out:
            for f, (dev, host) in arrs.items():
                want[np.ix_(p0 + own, list(AT[f]))] = host[MARGIN + ids[own]]
            if "C" in fields:
                want[p0 + own, 25:28] = 0.0  # the stress beside C[8] is void after a write
        got = after.transpose(1, 0, 2).reshape(cap, 32)
        if by_id and not out and len(lost):
            # ids without a slot are written where their inverse's old entry points: leave that slot out
            got, want = np.delete(got, p0 + own[0], 0), np.delete(want, p0 + own[0], 0)
        assert np.array_equal(got.view(np.int32), want.view(np.int32))
        assert np.array_equal(s[0].cpu().numpy(), spare[0])  # plane 0 of the spare buffer is no scratch
        if not (out and by_id):
            assert np.array_equal(s.cpu().numpy(), spare)


def pinned_read(sim, n):
    """All fields into page-locked arrays: the way that packs records into the spare buffer."""
    torch = pytest.importorskip("torch")
    arrs = [torch.empty((n, k), dtype=torch.float32).pin_memory() for k in COMPS.values()]
    assert mpm.mpm_read_state(sim.h, 0, 15, [a.data_ptr() for a in arrs], mpm.MEM_HOST) == 0
    return arrs[0].numpy()


def test_state_after_a_skipped_substep_keeps_its_ids():
    sc = W.elastic_cube(n_side=9)
    with mpm.from_workload(sc) as sim:
        sim.substep(sc["dt"], 2)
        older = pinned_read(sim, len(sc["x"])).copy()
        sim.substep(sc["dt"], 1)
        pinned_read(sim, len(sc["x"]))
        spoil_sort(sim)
        sim.substep(sc["dt"], 1)
        for device in (True, False):
            out = sim.read_state(0, ("x", "order"), device=device, check=False)
            assert out["status"] == -10
            x, order = (np.asarray(out[f].cpu() if device else out[f]) for f in ("x", "order"))
            assert np.array_equal(np.sort(order), np.arange(len(order)))
            assert np.array_equal(x, older)


def test_backward_refuses_a_tape_with_a_skipped_substep():
    sc = W.elastic_cube(n_side=9)
    with mpm.from_workload(sc, tape_checkpoint_every=2, tape_max_substeps=4) as sim:
        sim.tape_begin()
        sim.substep(sc["dt"], 2)
        ones = np.ones((len(sc["x"]), 3), np.float32)
        dE, dnu, dv0 = sim.backward(ones, ones)
        assert np.abs(dv0).max() > 0
        sim.substep(sc["dt"], 1)  # (the counts are made anew after a reverse pass)
        spoil_sort(sim)
        sim.substep(sc["dt"], 1)
        for reverse in (lambda: sim.backward(ones, ones), lambda: sim.backward_state({"v": ones})):
            with pytest.raises(mpm.MPMError) as e:
                reverse()
            assert e.value.status == -10


@pytest.mark.parametrize("fields,count", [("xvCF", 1250000), ("xvCF", 1250113), ("xCF", 1428672), ("xvC", 2000001),
                                          ("CF", 1700000), ("x", 2000001)])
def test_large_reads_take_the_scenes_own_ids(fields, count):
    # the sizes from which three or more fields go through records, and fields that never do
    torch = pytest.importorskip("torch")
    p0, cap = 7, count + 9
    g = torch.Generator(device="cuda").manual_seed(count)
    state = torch.randn((8, cap, 4), generator=g, device="cuda")
    ids = torch.randperm(count, generator=g, device="cuda").int()
    state[0, p0:p0 + count, 3] = ids.view(torch.float32)
    by_slot = state.permute(1, 0, 2).reshape(cap, 32)[p0:p0 + count]
    spare = torch.randn((8, cap, 4), generator=g, device="cuda")
    first = spare[0].clone()
    inv = torch.empty(cap, dtype=torch.int32, device="cuda")
    arrs, h = {}, Fields()
    for k, f in enumerate("xvCF"):
        if f in fields:
            arrs[f] = torch.zeros((count + 2 * MARGIN, COMPS[f]), device="cuda")
            h.f[k] = arrs[f].data_ptr() + 4 * MARGIN * COMPS[f]
    st, sp = PState(state.data_ptr(), None, None), PState(spare.data_ptr(), None, None)
    assert launch_fields()(ct.byref(st), ct.byref(sp), cap, p0, count, inv.data_ptr(), ct.byref(h), True, False,
                           torch.cuda.current_stream().cuda_stream) == 0
    for f, a in arrs.items():
        want = torch.zeros_like(a)
        want[MARGIN + ids.long()] = by_slot[:, list(AT[f])]
        assert torch.equal(a, want), f
    assert torch.equal(spare[0].view(torch.int32), first.view(torch.int32))

"""Scratch memory of the sweeps: allocated and given back by lbps_set_sweeps
(and the calls that stand for it), never by a step."""
import time

import numpy as np
import pytest

from paper_2301_00228_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELDS = ("ux", "uy", "vx", "vy", "f_phi", "f_psi")
ET, EV = (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8)


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_00228_gb300 import lbps
    return lbps


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def rect(L, nx, ny, **kw):
    lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, ET, EV, a0_phi=0.99, **kw)
    return lat.init(*W.pulse_displacement(nx, ny, nx / 3, ny / 2, 30.0, 1e-3, "rotation"))


def copy_bytes(lat):
    """A state copy's size, from below: the populations and u."""
    return lat.nx * lat.ny * ((80 if lat.storage == "f64" else 40 if lat.storage == "f32" else 32) + 32)


def test_steps_allocate_nothing(L):
    """A lattice in the caller's block, through the C entry points alone, at a
    size that the binding's lattices take exact sweeps at."""
    nx, ny = 1030, 520
    nt, bv = L.lbps_rect_bc(nx, ny, False, False, 1.0, ET, EV)
    st = torch.cuda.Stream()
    p = L.lbps_params(nx, ny, 1.5, 1.0, 1.0, 1.0, 0.99, 0, 0, 0, 0, L.LBPS_STORAGE_F32, 0,
                      L.ctypes.c_void_p(st.cuda_stream))
    need = L.lbps_state_bytes(p)
    block = torch.empty(need, dtype=torch.uint8, device="cuda")
    h = L.lbps_create(p, nt, bv, block.data_ptr(), need)
    u = W.pulse_displacement(nx, ny, nx / 3, ny / 2, 30.0, 1e-3, "rotation")
    L.lbps_init(h, *u)
    assert L._lib.lbps_step(h, 1) == 0       # the module's own first-launch allocations
    a = torch.ones(8192, 8192, device="cuda")
    before = free()
    with torch.cuda.stream(st):
        for _ in range(1000):
            a.mul_(1.0)
    t = time.perf_counter()
    assert L._lib.lbps_step_async(h, 9) == 0
    t = time.perf_counter() - t
    busy = not st.query()
    assert L._lib.lbps_check(h) == 0
    assert busy and t < 0.05                 # it did not wait for the stream (the loop keeps it busy far longer)
    assert free() == before
    out = np.zeros((ny, nx))
    L.lbps_read(h, L.LBPS_UX, out)
    ref = rect(L, nx, ny, step_pairs=False).step(10)
    assert np.array_equal(out, ref.read("ux"))
    ref.close()
    L._lib.lbps_destroy(h)


def test_kinds_of_sweeps(L):
    lat, ref = rect(L, 500, 400, step_pairs=False), rect(L, 500, 400, step_pairs=False)
    assert L.lbps_sweeps(lat._h) == L.LBPS_SWEEPS_NONE
    start = free()
    for kind, exact in (("EXACT", True), ("NONE", True), ("TWO", False), ("FOUR", False), ("EXACT", False),
                        ("NONE", False)):
        kind = getattr(L, "LBPS_SWEEPS_" + kind)
        L.lbps_set_sweeps(lat._h, kind)
        assert L.lbps_sweeps(lat._h) == kind and L.lbps_step_pairs(lat._h) == int(kind >= L.LBPS_SWEEPS_TWO)
        copies = {L.LBPS_SWEEPS_NONE: 0, L.LBPS_SWEEPS_FOUR: 2}.get(kind, 1)
        assert copies * copy_bytes(lat) <= start - free() <= copies * lat.nbytes // 2 + (4 << 20)
        lat.step(9)
        ref.step(9)
        for k in ("f_phi", "f_psi") + (FIELDS if exact else ()):
            assert np.array_equal(lat.read(k), ref.read(k)), (kind, k)
    lat.close()
    ref.close()
    for nx, ny, kw, bad in ((500, 400, dict(storage="f64"), ("EXACT", "FOUR")), (500, 400, dict(storage="f16"), ("FOUR",)),
                            (500, 400, dict(periodic_x=True), ("EXACT", "TWO", "FOUR")), (500, 60, {}, ("FOUR",)),
                            (500, 15, {}, ("EXACT", "TWO", "FOUR"))):
        lat = rect(L, nx, ny, **kw)
        for kind in bad + (7,):
            with pytest.raises(L.LbpsError) as e:
                L.lbps_set_sweeps(lat._h, getattr(L, f"LBPS_SWEEPS_{kind}", kind))
            assert e.value.code == L.LBPS_ERR_INVALID and L.lbps_sweeps(lat._h) == L.LBPS_SWEEPS_NONE
        L.lbps_set_sweeps(lat._h, L.LBPS_SWEEPS_AUTO)
        assert L.lbps_sweeps(lat._h) == L.LBPS_SWEEPS_NONE
        lat.close()
    for size, want in (((1030, 520), "EXACT"), ((1733, 1741), "FOUR")):
        lat = L.Lattice.rectangle(*size, 1.5, 1.0, ET, EV)
        assert L.lbps_sweeps(lat._h) == getattr(L, "LBPS_SWEEPS_" + want)
        lat.close()


def test_batches_hold_one_copy_each(L):
    """FP32 lattices large enough for four steps a sweep hold one scratch copy
    in a batch; a batch whose lattice gave its copy up refuses to step."""
    lats = [rect(L, 1733, 1741, step_pairs=False) for _ in range(2)]
    start = free()
    b = L.Batch(lats)
    b.set_step_pairs(True)
    held = start - free()
    assert 2 * copy_bytes(lats[0]) <= held <= lats[0].nbytes + (16 << 20)
    b.step(4)
    assert b.check() == 0
    L.lbps_set_sweeps(lats[1]._h, L.LBPS_SWEEPS_NONE)
    with pytest.raises(L.LbpsError) as e:
        b.step(2)
    assert e.value.code == L.LBPS_ERR_STATE
    b.close()
    for lat in lats:
        lat.close()

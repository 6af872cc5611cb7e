"""Many single steps in one cooperative launch (the path of lattices up to
1.2 M points) against the same steps as separate launches (a lattice whose
launch shape was set takes those): the same bits in every storage, on sizes at
the edges of the strips and of the boundary tasks, periodic axes, a plate with
a hole, both readings of the boundary rules, ramped loads, synchronisation,
and odd and even step counts.  Two lattices on two streams at once each give
the bits they give alone."""
import numpy as np
import pytest

from paper_2301_00228_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELDS = ("ux", "uy", "vx", "vy", "f_phi", "f_psi")


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_00228_gb300 import lbps
    return lbps


def lattice(L, nx, ny, storage="f32", separate=False, hole=False, load=False, stream=None, **kw):
    et, ev = (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8)
    if hole:
        nt, bv, cell = L.lbps_disk_cells(nx, ny, 1.0, 0.5 * nx, 0.4 * ny, 0.2 * min(nx, ny), et, ev)
        lat = L.Lattice(nx, ny, 1.5, 1.0, a0_phi=0.99, node_type=nt, bc_value=bv, cell=cell, storage=storage,
                        stream=stream, **kw)
    else:
        lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, et, ev, a0_phi=0.99, storage=storage, stream=stream, **kw)
    if separate:
        L.lbps_set_tuning(lat._h, 2, 8)
    if load:
        lat.set_load(L.LBPS_NEUMANN, 20 * lat.dt, 45 * lat.dt)
        lat.set_load(L.LBPS_DIRICHLET, 15 * lat.dt)
    u = W.pulse_displacement(nx, ny, nx / 3, ny / 2, max(2.0, nx / 10), 1e-3, "rotation")
    v = 1e-4 * np.random.default_rng(nx + ny).standard_normal((ny, nx))
    return lat.init(*u, v, -v)


def both(L, steps, *a, **kw):
    got, want = (lattice(L, *a, separate=s, **kw) for s in (False, True))
    for n in steps:
        got.step(n)
        want.step(n)
    assert got.steps == want.steps == sum(steps) and got.check() == 0
    for k in FIELDS:
        assert np.array_equal(got.read(k), want.read(k)), (a, kw, k)
    got.close()
    want.close()


@pytest.mark.parametrize("storage", ["f32", "f64", "f16", "bf16", "bfp13"])
@pytest.mark.parametrize("size", [(4, 5), (30, 31), (32, 95), (61, 16), (257, 190), (1170, 389), (900, 820)])
def test_fused_equals_separate_launches(L, storage, size):
    both(L, (1, 2, 8), *size, storage=storage)


@pytest.mark.parametrize("kw", [dict(periodic_x=True), dict(periodic_y=True), dict(periodic_x=True, periodic_y=True),
                                dict(hole=True), dict(hole=True, storage="bfp13", load=True), dict(load=True),
                                dict(bc_feq_mode=1), dict(bc_j_mode=1), dict(sync_every=3),
                                dict(sync_every=4, hole=True)])
def test_fused_equals_separate_launches_options(L, kw):
    both(L, (5, 1, 4, 7), 93, 77, **kw)


def test_fused_smallest(L):
    both(L, (3, 4), 3, 3)
    both(L, (3, 4), 3, 40, storage="f64")


def test_fused_on_two_streams(L):
    def run(streams):
        lats = [lattice(L, 300 + 40 * q, 280, stream=s) for q, s in enumerate(streams)]
        for _ in range(6):
            for lat in lats:
                lat.step_async(50)
        out = []
        for lat in lats:
            assert lat.check() == 0
            out.append([lat.read(k) for k in FIELDS])
            lat.close()
        return out
    s = torch.cuda.current_stream()
    want = run([s, s])
    got = run([torch.cuda.Stream(), torch.cuda.Stream()])
    for a, b in zip(got, want):
        assert all(np.array_equal(x, y) for x, y in zip(a, b))


def test_nonfinite_is_seen_on_every_path(L):
    """The check after many-step launches alone reads host words instead of the
    device flag; it must see what a launch sets, keep it, forget it at the next
    initialisation, and see the flag of other paths (a batch, launches of a set
    shape, a loaded state's steps)."""
    u = W.pulse_displacement(64, 48, 20.0, 20.0, 4.0, 1e-3)
    bad = [a * 1e300 for a in u]

    def raises(lat, n=4):
        with pytest.raises(L.LbpsError) as e:
            lat.step(n)
        assert e.value.code == L.LBPS_ERR_NONFINITE
        assert lat.check() == L.LBPS_ERR_NONFINITE

    lat = lattice(L, 64, 48)
    lat.step(3)
    saved = lat.save_state()
    lat.init(*bad)
    raises(lat)
    lat.init(*u).step(5)                       # forgotten
    assert lat.check() == 0
    lat.init(*bad)
    b = L.Batch([lat])
    b.step(4)                                  # set by the batch, read by the lattice
    assert b.check() == L.LBPS_ERR_NONFINITE and lat.check() == L.LBPS_ERR_NONFINITE
    b.close()
    lat.init(*u).step(2)
    lat.load_state(saved).step(3)
    assert lat.check() == 0
    L.lbps_set_tuning(lat._h, 2, 8)
    lat.init(*bad)
    raises(lat)
    lat.close()

"""Two-step sweeps of batches, their rows fed by TMA through tensor maps in
device memory."""
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


def lattice(L, nx, ny, seed, storage):
    rng = np.random.default_rng(seed)
    lat = L.Lattice.rectangle(nx, ny, float(rng.uniform(0.5, 3.0)), 1.0, rng.integers(1, 3, 4),
                              rng.uniform(-2e-4, 2e-4, 8), a0_phi=0.99, storage=storage)
    return lat.init(*W.pulse_displacement(nx, ny, nx / 3, ny / 2, max(2.0, min(nx, ny) / 10), 1e-3, "rotation"))


@pytest.mark.parametrize("storage", ["f32", "bfp13"])
def test_remade_batches_read_their_own_lattices(L, storage):
    """Batches made one after the other of other lattices: their tensor maps
    may come to lie where those of the batch before lay.  Every member gets the
    bits of two steps per sweep on its own."""
    sizes = [(70, 45), (129, 64), (33, 200), (64, 91), (96, 96), (47, 31)]
    lats = [lattice(L, *s, q, storage) for q, s in enumerate(sizes)]
    alone = [lattice(L, *s, q, storage) for q, s in enumerate(sizes)]
    for lat in alone:
        L.lbps_set_step_pairs(lat._h, 1)
    for r in range(12):
        members = [(r + q) % len(lats) for q in range(3)]
        b = L.Batch([lats[m] for m in members])
        b.set_step_pairs(True)
        b.step(6)
        assert b.check() == 0
        b.close()
        for m in members:
            alone[m].step(6)
    for lat, ref in zip(lats, alone):
        assert lat.steps == ref.steps
        for k in FIELDS:
            assert np.array_equal(lat.read(k), ref.read(k)), k
        lat.close()
        ref.close()

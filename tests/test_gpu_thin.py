"""Narrow and flat rectangles: those with many boundary points take separate
launches instead of a many-step one, narrow ones no exact sweeps unless asked.
The same bits either way."""
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


@pytest.mark.parametrize("storage", ["f32", "f16", "bfp13", "f64"])
@pytest.mark.parametrize("nx,ny,exact", [
    (16, 8178, False), (16, 8179, False),         # 16384 and 16386 boundary points, 2^17 points and less
    (35, 4063, False), (4064, 35, False),         # 8192 and 8194, more than 2^17 points
    (64, 7900, True), (65, 300, True), (16, 40, True)])
def test_thin_lattices(L, storage, nx, ny, exact):
    if exact and storage == "f64":
        pytest.skip("no exact sweeps in FP64 storage")
    lats = []
    for single in (False, True):
        lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99,
                                  storage=storage)
        if single:
            L.lbps_set_tuning(lat._h, 2, 8)
        elif exact:
            L.lbps_set_sweeps(lat._h, L.LBPS_SWEEPS_EXACT)
        lat.init(*W.pulse_displacement(nx, ny, nx / 3, ny / 2, 4.0, 1e-3, "rotation"))
        lats.append(lat.step(1).step(12).step(5))
    assert lats[0].check() == 0
    for k in FIELDS:
        assert np.array_equal(lats[0].read(k), lats[1].read(k)), k
    for lat in lats:
        lat.close()

"""CUDA graphs of single steps, captured again when what they hold changes:
lattices whose launch shape is set from the start (others of this size take
many steps in one launch instead), and the change from one path to the other."""
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


@pytest.mark.parametrize("storage", ["f32", "f16", "bfp13"])
@pytest.mark.parametrize("k", [2, 4, 16])
def test_graphs_follow_every_change(L, storage, k):
    """Against per-kernel timing, which launches every kernel itself; every 7th
    step synchronises."""
    def run(timed):
        lat = L.Lattice.rectangle(71, 53, 1.4, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99,
                                  storage=storage, sync_every=7)
        L.lbps_profile(lat._h, int(timed))
        L.lbps_set_graph_steps(lat._h, k)
        lat.init(*W.pulse_displacement(71, 53, 20.0, 30.0, 6.0, 1e-3, "rotation"))
        lat.step(3)                              # many steps in one launch, unless timed
        L.lbps_set_tuning(lat._h, 2, 8)          # from here on graphs of this shape
        lat.step(10).step(5)
        L.lbps_set_tuning(lat._h, 5, 16)         # of another
        lat.step(9)
        lat.set_load(L.LBPS_NEUMANN, 20 * lat.dt, 40 * lat.dt)
        lat.step(30).step(2)
        L.lbps_set_graph_steps(lat._h, 2 if k > 2 else 4)
        lat.step(13)
        out = [lat.read(f) for f in FIELDS]
        assert lat.steps == 72
        lat.close()
        return out

    for a, b, f in zip(run(True), run(False), FIELDS):
        assert np.array_equal(a, b), f

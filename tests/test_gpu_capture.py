"""Steps captured by the caller into a CUDA graph and replayed."""
import numpy as np
import pytest

from paper_2301_00228_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_00228_gb300 import lbps
    return lbps


def lattice(L, nx, ny, stream, **kw):
    lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99, stream=stream,
                              **kw)
    return lat, W.pulse_displacement(nx, ny, nx / 3, ny / 2, max(2.0, min(nx, ny) / 10), 1e-3, "rotation")


def test_replayed_batch_steps_reach_the_lattice_check(L):
    """A lattice initialised after its batch's steps were captured: what a
    replay of them sets is seen by the lattice's own check."""
    s = torch.cuda.Stream()
    lats, us = zip(*(lattice(L, *size, s) for size in ((64, 48), (70, 45))))
    for lat, u in zip(lats, us):
        lat.init(*u)
    b = L.Batch(list(lats), stream=s)
    b.set_step_pairs(True)
    b.step(4)                        # two pairs: the same current copies after it
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        b.step(4)
    for lat, u in zip(lats, us):
        for _ in range(2):           # twice: the current copy is again the one the captured steps read
            lat.init(*u)
    g.replay()
    torch.cuda.synchronize()
    assert [lat.check() for lat in lats] == [0, 0]
    for _ in range(2):
        lats[1].init(*(1e300 * a for a in us[1]))
    g.replay()
    torch.cuda.synchronize()
    assert [lat.check() for lat in lats] == [0, L.LBPS_ERR_NONFINITE]
    assert b.check() == L.LBPS_ERR_NONFINITE
    b.close()
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("size,kw", [((300, 200), {}), ((1030, 520), {}), ((300, 200), dict(step_pairs=True)),
                                     ((1030, 520), dict(periodic_x=True, periodic_y=True))])
@pytest.mark.parametrize("warm", [0, 4])
def test_captured_steps_are_single_steps(L, size, kw, warm):
    """lbps_step_async into a capture, on lattices that otherwise take many
    steps a launch or sweeps: one step replayed once and four steps replayed
    three times give the bits of uncaptured single launches."""
    s = torch.cuda.Stream()

    def start(single):
        lat, u = lattice(L, *size, s, **({} if single else kw), **({k: v for k, v in kw.items() if single and
                                                                     k != "step_pairs"}))
        if single:
            L.lbps_set_tuning(lat._h, 2, 8)
        lat.set_load(L.LBPS_NEUMANN, 20 * lat.dt, 45 * lat.dt)
        return lat.init(*u).step(warm)

    for n, replays in ((1, 1), (4, 3)):
        lat, want = start(False), start(True)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.step_async(n)
        for _ in range(replays):
            g.replay()
        torch.cuda.synchronize()
        want.step(n * replays)
        assert lat.check() == 0
        for k in ("f_phi", "f_psi") + (() if "step_pairs" in kw and warm else ("ux", "uy", "vx", "vy")):
            assert np.array_equal(lat.read(k), want.read(k)), (n, k)
        lat.close()
        want.close()

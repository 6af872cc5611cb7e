"""Lattices on several streams at once: the bits each gets alone, whichever
launches they take beside one another, and no slower than separate launches."""
import time

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


def lattice(L, nx, ny, stream, storage="f32", separate=False):
    lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.9999,
                              storage=storage, stream=stream, step_pairs=False)
    if separate:
        L.lbps_set_tuning(lat._h, 0, 8)
    return lat.init(*W.pulse_displacement(nx, ny, nx / 3, ny / 2, max(2.0, nx / 10), 1e-3, "rotation"))


@pytest.mark.parametrize("storage", ["f32", "bfp13"])
def test_bits_beside_others(L, storage):
    """One stream, then two, then three, then a lattice that changes streams."""
    sizes = [(64, 48), (128, 96), (170, 130), (300, 280)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    lats = []
    for q, size in enumerate(sizes):
        lats.append(lattice(L, *size, streams[q % 3], storage))
        for n in (1, 20, 1, 7):
            for lat in lats:
                lat.step_async(n)
    torch.cuda.synchronize()
    L.lbps_set_stream(lats[1]._h, streams[0].cuda_stream)
    for _ in range(3):
        for lat in lats:
            lat.step_async(5)
    assert [lat.check() for lat in lats] == [0] * len(lats)
    got = [[lat.read(k) for k in FIELDS] for lat in lats]
    steps = [lat.steps for lat in lats]
    for lat in lats:
        lat.close()
    for size, n, fields in zip(sizes, steps, got):
        ref = lattice(L, *size, torch.cuda.current_stream(), storage, separate=True).step(n)
        for k, f in zip(FIELDS, fields):
            assert np.array_equal(f, ref.read(k)), (size, k)
        ref.close()


@pytest.mark.parametrize("size,count", [((300, 300), 4), ((700, 500), 4), ((64, 64), 4)])
def test_side_by_side_is_not_slower(L, size, count):
    """Lattices stepped on streams of their own, against the same with separate
    launches (as one after the other in many-step launches, 300 x 300 and 700 x
    500 took 2.1 and 1.4 times as long)."""
    def took(separate):
        lats = [lattice(L, *size, torch.cuda.Stream(), separate=separate) for _ in range(count)]
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(10):
                for lat in lats:
                    lat.step_async(20)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        for lat in lats:
            lat.close()
        return best

    assert took(False) < 1.25 * took(True)

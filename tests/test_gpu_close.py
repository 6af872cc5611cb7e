"""Closing a lattice does not wait for other work on the device."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2301_00228_gb300 import lbps
    return lbps


@pytest.mark.parametrize("steps", [0, 1, 8])
def test_close_beside_other_work(L, steps):
    def make():
        z = np.zeros((96, 128))
        lat = L.Lattice.rectangle(128, 96, 1.5, 1.0, (2, 1, 1, 2), np.zeros(8), stream=torch.cuda.Stream())
        lat.init(z, z)
        return lat.step(steps) if steps else lat

    make().close()
    lat = make()
    a = torch.ones(8192, 8192, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for _ in range(4000):      # some 300 ms
            a.mul_(1.0)
    lat.close()
    assert not s.query()
    s.synchronize()


def test_more_lattices_than_host_words(L):
    """2048 lattices hold host words at a time; further ones, and those made
    after some were given back, report what theirs and only theirs did."""
    z = np.zeros((8, 8))
    lats = [L.Lattice(8, 8, 1.0, 1.0, periodic_x=True, periodic_y=True) for _ in range(2100)]
    rng = np.random.default_rng(1)

    def go(lat, bad):
        u = rng.uniform(-1.0, 1.0, (8, 8))
        lat.init((1e300 if bad else 1e-3) * u, z).step_async(6)

    for q, lat in enumerate(lats):
        go(lat, q % 7 == 3)
    assert [lat.check() for lat in lats] == [L.LBPS_ERR_NONFINITE if q % 7 == 3 else 0 for q in range(len(lats))]
    for lat in lats[::2]:
        lat.close()
    more = [L.Lattice(8, 8, 1.0, 1.0, periodic_x=True, periodic_y=True) for _ in range(40)]
    for q, lat in enumerate(more):
        go(lat, q % 3 == 1)
    assert [lat.check() for lat in more] == [L.LBPS_ERR_NONFINITE if q % 3 == 1 else 0 for q in range(len(more))]
    for lat in more + lats[1::2]:
        lat.close()


def test_lattices_after_a_device_reset():
    """The page of host words goes with its context; lattices made after a reset
    get one of their own.  In a child process, the library's own memory."""
    import subprocess
    import sys
    from pathlib import Path

    root = Path(__file__).resolve().parents[1]
    code = f"import sys; sys.path.insert(0, {str(root)!r})" + r"""
import ctypes
import numpy as np
from paper_2301_00228_gb300 import lbps as L

def run():
    nt, bv = L.lbps_rect_bc(32, 24, False, False, 1.0, (2, 1, 1, 2), np.zeros(8))
    h = L.lbps_create(L.lbps_params(32, 24, 1.5, 1.0, 1.0, 1.0, 0.99, 0, 0, 0, 0, 0, 0, None), nt, bv, 0, 0)
    u = 1e-3 * np.random.default_rng(1).standard_normal((24, 32))
    L.lbps_init(h, u, u)
    assert L._lib.lbps_step(h, 20) == 0
    out = np.zeros((24, 32))
    L.lbps_read(h, L.LBPS_UX, out)
    L.lbps_destroy(h)
    return out

a = run()
assert ctypes.CDLL("libcuda.so.1").cuDevicePrimaryCtxReset_v2(0) == 0
assert np.array_equal(a, run()) and np.array_equal(a, run())
print("OK")
"""
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip().endswith("OK"), out.stdout + out.stderr

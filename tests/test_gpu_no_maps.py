"""A driver that makes no tensor maps (the library is built as if it made none):
every call that takes sweeps works with what is left, two composed steps per
sweep whose rows come through registers, or single steps."""
import pytest

import variant

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = r"""
import numpy as np, torch
from paper_2301_00228_gb300 import lbps as L

def rect(size, storage, single=False, **kw):
    lat = L.Lattice.rectangle(*size, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99, storage=storage,
                              **kw)
    if single:
        L.lbps_set_sweeps(lat._h, L.LBPS_SWEEPS_NONE)
        L.lbps_set_tuning(lat._h, 2, 8)
    y, x = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (size[1], size[0]))
    return lat.init(*(1e-3 * torch.sin(a * x)[None, :] * torch.cos(b * y)[:, None] for a, b in ((.05, .03), (.02, .07))))

def same(a, b, what, exact=False):
    for k in ("f_phi", "f_psi") + (("ux", "vy") if exact else ()):
        assert torch.equal(a.read_device(k), b.read_device(k)), (what, k)
    a.close()
    b.close()

for storage in ("f32", "f16", "bf16", "bfp13"):
    for size, kw, kind in (((1003, 517), {}, "NONE"), ((517, 1003), dict(periodic_x=True, periodic_y=True), "NONE"),
                           ((1733, 1741), {}, "TWO"), ((67, 45), dict(step_pairs=True), "TWO")):
        a = rect(size, storage, **kw)
        assert a.sweeps == getattr(L, "LBPS_SWEEPS_" + kind)
        if kind == "TWO":
            assert L.lbps_step_pairs(a._h) == 1
        for bad in (L.LBPS_SWEEPS_EXACT, L.LBPS_SWEEPS_FOUR):
            assert L._lib.lbps_set_sweeps(a._h, bad) == L.LBPS_ERR_INVALID
        same(a.step(7), rect(size, storage, True, **{k: v for k, v in kw.items() if k != "step_pairs"}).step(7),
             (storage, size), kind == "NONE")
    lats = [rect(s, storage) for s in ((70, 45), (33, 129), (64, 91), (16, 16))]
    b = L.Batch(lats)
    b.set_step_pairs(True)
    b.step(6)
    assert b.check() == 0
    b.close()
    for lat in lats:
        same(lat, rect((lat.nx, lat.ny), storage, True).step(6), (storage, "batch"))
print("OK")
"""


def test_without_tensor_maps(tmp_path):
    assert variant.run(variant.package(tmp_path, "lbps_sweep", "LBPS_NO_TENSOR_MAPS"), CODE).strip().endswith("OK")

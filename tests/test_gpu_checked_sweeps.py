"""The sweeps of several steps under the range-checked build: two exact steps,
two and four of the caller's, periodic ones and a batch's, on sides that leave
remainders.  No access may be refused, and the fields are those of single
launches, whose kernels are another translation unit's (the populations are
the same bits; a refused store would leave them stale)."""
import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parents[1]

CHILD = r"""
import os, sys
sys.path.insert(0, ROOT)
from paper_2301_00228_gb300 import build
build.build(checked=True)
os.environ["LBPS_CHECKED"] = "1"
import numpy as np, torch
from paper_2301_00228_gb300 import lbps as L

def rect(size, storage, single=False, **kw):
    lat = L.Lattice.rectangle(*size, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99, storage=storage,
                              step_pairs=False, **kw)
    if single:
        L.lbps_set_tuning(lat._h, 2, 8)
    y, x = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (size[1], size[0]))
    return lat.init(*(1e-3 * torch.sin(a * x)[None, :] * torch.cos(b * y)[:, None] for a, b in ((.05, .03), (.02, .07))))

def same(a, b, what):
    for k in ("f_phi", "f_psi"):
        assert torch.equal(a.read_device(k), b.read_device(k)), (what, k)
    a.close()
    b.close()

runs = 0
for storage in ("f32", "f16", "bfp13"):
    for size, kw in (((1003, 517), {}), ((517, 1003), dict(periodic_x=True, periodic_y=True))):   # exact
        a = rect(size, storage, **kw)
        if not kw:
            L.lbps_set_sweeps(a._h, L.LBPS_SWEEPS_EXACT)
        same(a.step(5), rect(size, storage, True, **kw).step(5), (storage, size))
        runs += 1
    pairs = [((67, 45), storage), ((16, 16), storage)] + ([((1733, 1741), "f32")] if storage == "f32" else [])
    for size, st in pairs:                                                                        # the caller's
        a = rect(size, st)
        L.lbps_set_step_pairs(a._h, 1)
        same(a.step(7), rect(size, st, True).step(7), (st, size))
        runs += 1
    lats = [rect(s, storage) for s in ((70, 45), (33, 129), (64, 91))]
    b = L.Batch(lats)
    b.set_step_pairs(True)
    b.step(6)
    assert b.check() == 0
    b.close()
    for lat in lats:
        same(lat, rect((lat.nx, lat.ny), storage, True).step(6), (storage, "batch"))
        runs += 1
rc, line, addr = L.lbps_check_report()
print("REPORT", rc, line, addr, runs)
"""


def test_checked_sweeps():
    env = dict(os.environ)
    env.pop("LBPS_CHECKED", None)
    out = subprocess.run([sys.executable, "-c", f"ROOT = {str(ROOT)!r}\n" + CHILD],
                         capture_output=True, text=True, timeout=1200, env=env, cwd=str(ROOT))
    report = [ln for ln in out.stdout.splitlines() if ln.startswith("REPORT")]
    assert out.returncode == 0 and report, out.stdout[-2000:] + out.stderr[-3000:]
    rc, line, addr, runs = (int(x) for x in report[-1].split()[1:])
    assert rc == 1, "the checked build was not loaded"
    assert (line, addr) == (0, 0), f"first violation at source line {line}, address {addr:#x}"
    assert runs == 22

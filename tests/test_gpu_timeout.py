"""A sweep whose wait for its rows runs out: the library is built with a limit
of no polls, so that every wait does (the copies arrive all the same, and each
warp sees them land before it returns).  The check reports the timeout, the
lattice has no state until the next initialisation, and the context stays
usable: a lattice of another path then runs to the oracle's fields."""
import pytest

import variant

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = r"""
import numpy as np, torch
from paper_2301_00228_gb300 import lbps as L, workloads as W
assert "liblbps" in L._lib._name and "paper_2301" in L._lib._name
ET, EV = (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8)
u = {s: W.pulse_displacement(*s, s[0] / 3, s[1] / 2, 6.0, 1e-3, "rotation") for s in ((150, 90), (1030, 520), (45, 38))}

def rect(size, storage="f32", **kw):
    return L.Lattice.rectangle(*size, 1.5, 1.0, ET, EV, a0_phi=0.9, storage=storage, **kw).init(*u[size])

def runs_out(lat, n):
    assert L._lib.lbps_step(lat._h, n) == L.LBPS_ERR_TIMEOUT
    assert L._lib.lbps_step(lat._h, 1) == L.LBPS_ERR_STATE
    lat.close()

for storage in ("f32", "bfp13"):
    runs_out(rect((150, 90), storage, step_pairs=True), 2)      # two steps, caller's
    runs_out(rect((1030, 520), storage, periodic_x=True, periodic_y=True), 2)
    a, b = rect((150, 90), storage), rect((45, 38), storage)
    batch = L.Batch([a, b])
    batch.set_step_pairs(True)
    batch.step(2)
    assert batch.check() == L.LBPS_ERR_TIMEOUT
    batch.close()
import oracle as O
nt, bv = O.rect_bc(45, 38, ET, EV)
ref = O.OracleLattice(45, 38, 1.5, 1.0, a0_phi=0.9, node_type=nt, bc_value=bv).init(*u[(45, 38)]).step(60).fields()
got = b.init(*u[(45, 38)])
L.lbps_set_step_pairs(b._h, 0)
got = got.step(60).fields()
for k in ("ux", "uy", "phi", "psi"):
    err = np.linalg.norm(got[k] - ref[k]) / np.linalg.norm(ref[k])
    assert err <= 1e-3, (k, err)      # b is in BFP13
print("OK")
"""


def test_a_sweep_that_gives_up(tmp_path):
    where = variant.package(tmp_path, "lbps_sweep", "LBPS_SWEEP_POLLS=0")
    code = f"import sys; sys.path.append({str(variant.B.ROOT)!r})\n" + CODE
    assert variant.run(where, code).strip().endswith("OK")

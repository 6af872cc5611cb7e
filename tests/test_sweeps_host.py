"""Which sweeps a lattice takes by default (lbps_default_sweeps), on the host."""
import pytest


@pytest.fixture(scope="module")
def L():
    from paper_2301_00228_gb300 import build as B
    B.build()
    from paper_2301_00228_gb300 import lbps
    return lbps


@pytest.mark.parametrize("nx,ny,storage,kw,want", [
    (706, 708, "f32", {}, "NONE"), (708, 708, "f32", {}, "EXACT"), (1733, 1731, "bf16", {}, "EXACT"),
    (708, 708, "f64", {}, "NONE"), (708, 708, "f32", dict(sync_every=1), "NONE"),
    (708, 708, "f32", dict(sync_every=2), "EXACT"), (708, 708, "f32", dict(periodic_x=1), "NONE"),
    (9000, 63, "f32", {}, "NONE"), (9000, 64, "f32", {}, "EXACT"),
    (127, 9000, "f16", {}, "NONE"), (128, 9000, "f16", {}, "EXACT"), (64, 46874, "f32", {}, "NONE"),
    (1733, 1732, "f32", {}, "FOUR"), (1733, 1732, "bfp13", {}, "TWO"), (1733, 1732, "f64", {}, "NONE"),
    (60000, 63, "f32", {}, "TWO"), (200000, 15, "f32", {}, "NONE"), (1733, 1732, "f32", dict(periodic_y=1), "NONE")])
def test_default_sweeps(L, nx, ny, storage, kw, want):
    p = L.lbps_params(nx, ny, 1.0, 1.0, 1.0, 1.0, 0.99, kw.get("periodic_x", 0), kw.get("periodic_y", 0), 0,
                      kw.get("sync_every", 0), L.STORAGES[storage], 0, None)
    assert L.lbps_default_sweeps(p) == getattr(L, "LBPS_SWEEPS_" + want)


def test_default_sweeps_refuses_bad_parameters(L):
    with pytest.raises(L.LbpsError):
        L.lbps_default_sweeps(L.lbps_params(2, 5, 1.0, 1.0, 1.0, 1.0, 0.99, 0, 0, 0, 0, 0, 0, None))

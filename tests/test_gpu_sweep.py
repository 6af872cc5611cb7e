"""Sweeps of several steps.  Exact sweeps of two (mid-size lattices) against
single launches (a lattice whose launch shape was set takes those): the same
bits.  Four time steps per sweep (FP32 lattices of 3 M points and more) against
single steps: the populations and step counts are the same bits, u and du/dt
agree up to the rounding of the composed Newmark update (one FP32 rounding of
the acceleration sums per pair of steps: 1e-7 of the field's largest magnitude
over some tens of steps), on sides that leave every remainder of the 24-column
strips and of the row chunks, at the smallest side, with step counts that leave
0 to 3 steps over and synchronisation points that cut sweeps short."""
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


def run(L, nx, ny, pairs, chunks, sync=0, load=False):
    lat = L.Lattice.rectangle(nx, ny, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99,
                              sync_every=sync, step_pairs=pairs)
    if load:
        lat.set_load(L.LBPS_NEUMANN, 20 * lat.dt, 45 * lat.dt)
    y, x = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (ny, nx))
    u = [1e-3 * torch.sin(a * x)[None, :] * torch.cos(b * y)[:, None] for a, b in ((0.05, 0.03), (0.02, 0.07))]
    v = [1e-2 * q.flip(0).contiguous() for q in u]
    lat.init(*u, *v)
    for n in chunks:
        lat.step(n)
    assert lat.check() == 0
    out = {k: lat.read_device(k) for k in FIELDS}
    steps = lat.steps
    lat.close()
    return out, steps


@pytest.mark.parametrize("size", [(2003, 1501), (64, 46900), (46877, 65), (1733, 1741)])
@pytest.mark.parametrize("chunks,sync", [((4, 7, 34, 1), 0), ((41,), 7)])
def test_four_steps_per_sweep_equal_single_steps(L, size, chunks, sync):
    want, n0 = run(L, *size, False, chunks, sync, load=True)
    got, n1 = run(L, *size, True, chunks, sync, load=True)
    assert n0 == n1 == sum(chunks)
    for k in FIELDS:
        if k.startswith("f_") and not sync:
            assert torch.equal(got[k], want[k]), (size, k)
        else:
            err = float((got[k] - want[k]).abs().max()) / float(want[k].abs().max())
            assert err <= 1e-7, (size, k, err)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "bfp13"])
@pytest.mark.parametrize("size", [(64, 7900), (7843, 65), (740, 701), (1003, 997)])
@pytest.mark.parametrize("kw", [dict(), dict(periodic_x=True, periodic_y=True), dict(sync_every=5),
                                dict(sync_every=5, periodic_x=True, periodic_y=True)])
def test_exact_sweeps_equal_single_launches(L, storage, size, kw):
    """500000 points and more, strips of 28 columns and chunks of 16 .. 32 rows
    with every kind of remainder, seams of periodic axes, odd step counts,
    synchronisation points inside pairs."""
    lats = []
    for separate in (False, True):
        lat = L.Lattice.rectangle(*size, 1.5, 1.0, (2, 1, 1, 2), np.linspace(-2e-4, 2e-4, 8), a0_phi=0.99,
                                  storage=storage, **kw)
        if separate:
            L.lbps_set_tuning(lat._h, 2, 8)
        y, x = (torch.arange(n, dtype=torch.float64, device="cuda") for n in (size[1], size[0]))
        u = [1e-3 * torch.sin(a * x)[None, :] * torch.cos(b * y)[:, None] for a, b in ((0.05, 0.03), (0.02, 0.07))]
        lat.init(*u, *(1e-2 * q.flip(0).contiguous() for q in u))
        lats.append(lat.step(1).step(9).step(34))
    assert lats[0].check() == 0 and lats[0].steps == lats[1].steps == 44
    for k in FIELDS:
        assert torch.equal(lats[0].read_device(k), lats[1].read_device(k)), k
    for lat in lats:
        lat.close()


def test_exact_sweeps_and_the_switch(L):
    """Turning sweeps off frees the scratch copy and keeps the bits; turning
    them on takes over from exact ones."""
    out = []
    for switch in ((), (0,), (1, 0)):
        lat = L.Lattice.rectangle(800, 700, 1.5, 1.0, (2, 1, 1, 2), np.zeros(8), a0_phi=0.99)
        u = W.pulse_displacement(800, 700, 300.0, 400.0, 40.0, 1e-3, "rotation")
        lat.init(*u).step(6)
        for on in switch:
            L.lbps_set_step_pairs(lat._h, on)
            assert L.lbps_step_pairs(lat._h) == on
        lat.step(7)
        out.append([lat.read(k) for k in FIELDS])
        lat.close()
    for other in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], other))


@pytest.mark.parametrize("pairs", [False, True])
def test_scratch_is_cleared_before_the_first_sweep(L, pairs):
    """The first sweeps of a lattice on its own stream, the default stream busy
    for longer than they take: clearing the scratch copy does not wait for it."""
    out = []
    a = torch.ones(8192, 8192, device="cuda")
    for busy in (False, True):
        lat = L.Lattice.rectangle(1200, 1100, 1.5, 1.0, (2, 1, 1, 2), np.zeros(8), a0_phi=0.99,
                                  stream=torch.cuda.Stream())
        lat.init(*W.pulse_displacement(1200, 1100, 300.0, 400.0, 40.0, 1e-3, "rotation"))
        torch.cuda.synchronize()
        if busy:
            for _ in range(400):
                a.mul_(1.0)
        if pairs:
            L.lbps_set_step_pairs(lat._h, 1)
        lat.step(200)
        torch.cuda.synchronize()
        out.append([lat.read(k) for k in FIELDS])
        lat.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))

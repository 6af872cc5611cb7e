"""The server's memory budget with the sweeps' scratch copies, on the CPU:
lattices and batches are replaced by fakes that know what the real ones would
hold, and every step of any of them checks the sum against the budget."""
import pytest

from paper_2301_00228_gb300 import serve as S
from paper_2301_00228_gb300 import workloads as W

pytestmark = pytest.mark.timeout(60)
L = S.lbps


class FakeLattice:
    live = set()

    def __init__(self, d, storage):
        self.d, self.done, self._h, self.kind = d, 0, self, L.LBPS_SWEEPS_NONE
        self.block = L.lbps_state_bytes(S._params(d, storage))
        self.kinds = []
        FakeLattice.live.add(self)

    def set_sweeps(self, kind):
        assert self in FakeLattice.live
        self.kind = kind
        self.kinds.append(kind)
        return self

    def held(self):
        return self.block + S.SCRATCH_COPIES[self.kind] * (self.block // 2)

    def norms(self, name):
        return None

    def close(self):
        FakeLattice.live.discard(self)


class FakeBatch:
    def __init__(self, lats, stream=None):
        self.lats = lats
        self.made_of = [lat.d for lat in lats]

    def set_step_pairs(self, on):
        for lat in self.lats:
            if lat.kind < L.LBPS_SWEEPS_TWO:
                lat.set_sweeps(L.LBPS_SWEEPS_TWO)

    def step(self, k):
        assert all(lat.d is d for lat, d in zip(self.lats, self.made_of)), "a batch of closed lattices"
        for lat in self.lats:
            step(lat, k)

    def check(self):
        return 0

    def close(self):
        pass


BUDGET, PEAK = [0], [0]


def step(lat, k):
    held = sum(x.held() for x in FakeLattice.live)
    PEAK[0] = max(PEAK[0], held)
    assert held <= BUDGET[0]
    lat.done += k
    return 0


class StepClock:
    def __init__(self):
        self.t = 0.0

    def __call__(self):
        self.t += 1.0
        return self.t


@pytest.fixture
def serve(monkeypatch):
    made = []

    def make(d, storage, u0=None, stream=None):
        made.append(FakeLattice(d, storage))
        return made[-1]

    FakeLattice.live = set()
    PEAK[0] = 0
    monkeypatch.setattr(S, "_lattice", make)
    monkeypatch.setattr(S.lbps, "Batch", FakeBatch)
    monkeypatch.setattr(S.lbps, "lbps_step_async", step)
    monkeypatch.setattr(S.lbps, "lbps_check", lambda h: 0)

    def run(sizes, budget, arrivals=None, steps=None, cancel=None, **kw):
        BUDGET[0] = budget
        reqs = [S.Request(q, arrivals[q] if arrivals else 0.0, W.Domain(*s, 1.0, 1.0), steps[q] if steps else 400,
                          cancel[q] if cancel else None) for q, s in enumerate(sizes)]
        rep = S.serve_batched(reqs, budget, max_chunk=100, keep_fields=False, clock=StepClock(), **kw)
        for r in rep.results:
            assert made[r.rid].done == reqs[r.rid].steps
        assert not FakeLattice.live and PEAK[0] <= rep.peak_bytes <= budget
        return rep, made
    return run


def block(nx, ny, storage="f32"):
    return L.lbps_state_bytes(S._params(W.Domain(nx, ny, 1.0, 1.0), storage))


SMALL, MID, LARGE = (300, 200), (1030, 520), (1733, 1741)
NONE, EXACT, TWO, FOUR = L.LBPS_SWEEPS_NONE, L.LBPS_SWEEPS_EXACT, L.LBPS_SWEEPS_TWO, L.LBPS_SWEEPS_FOUR


@pytest.mark.parametrize("size,halves,pairs,storage,want", [
    (SMALL, 4, False, "f32", NONE), (SMALL, 4, True, "f32", NONE),
    (MID, 2, False, "f32", NONE), (MID, 3, False, "f32", EXACT), (MID, 3, True, "f32", EXACT),
    (MID, 4, False, "f64", NONE),
    (LARGE, 2, False, "f32", NONE), (LARGE, 3, False, "f32", TWO), (LARGE, 4, False, "f32", FOUR),
    (LARGE, 3, True, "f32", TWO), (LARGE, 4, True, "f32", FOUR), (LARGE, 4, True, "f16", TWO)])
def test_a_lone_solve_takes_the_sweeps_that_fit(serve, size, halves, pairs, storage, want):
    b = block(*size, storage)
    rep, made = serve([size], b // 2 * halves + b % 2 * 4, storage=storage, pairs=pairs)
    assert made[0].kinds[0] == want and made[0].kinds[-1] == NONE
    assert len(rep.results) == 1 and rep.memory_waits == 0


def test_scratch_goes_back_when_others_need_the_memory(serve):
    """A request that fits only without the lone solve's scratch is admitted at
    the next boundary; one that fits beside it at once."""
    for budget, kind in ((2 * block(*MID), EXACT), (4 * block(*MID), EXACT)):
        rep, made = serve([MID, MID], budget, arrivals=[0.0, 4.0], steps=[2000, 300])
        assert made[-2].kinds[0] == kind and rep.max_active == 2
        assert len(rep.results) == 2
        made.clear()


def test_members_of_a_batch_hold_what_they_are_charged(serve):
    for pairs in (False, True):
        charge = 3 * block(*LARGE) // 2 if pairs else block(*LARGE)
        rep, made = serve([LARGE, LARGE, MID], 2 * charge + 2 * block(*MID), steps=[500, 700, 300], pairs=pairs)
        assert rep.max_active == 3 and rep.memory_waits == 0
        made.clear()


def test_a_withdrawn_lone_solve_gives_everything_back(serve):
    rep, made = serve([MID, SMALL], 2 * block(*MID), arrivals=[0.0, 40.0], steps=[4000, 50], cancel=[5.0, None])
    assert rep.cancelled == [0] and [r.rid for r in rep.results] == [1]


@pytest.mark.parametrize("arrival", range(1, 14))
def test_new_members_get_a_batch_of_their_own(serve, monkeypatch, arrival):
    """Two requests that arrive as a batch of two ends, their lattices made where
    the closed ones lay (here: the same objects)."""
    pool = []

    def recycle(d, storage, u0=None, stream=None):
        free = [x for x in pool if x not in FakeLattice.live]
        if not free:
            pool.append(FakeLattice(d, storage))
            return pool[-1]
        free[0].__init__(d, storage)
        return free[0]

    monkeypatch.setattr(S, "_lattice", recycle)
    BUDGET[0] = 10 * block(*MID)
    reqs = [S.Request(q, 0.0 if q < 2 else arrival + 0.5, W.Domain(*SMALL, 1.0, 1.0), 100) for q in range(4)]
    rep = S.serve_batched(reqs, BUDGET[0], max_chunk=100, keep_fields=False, clock=StepClock())
    assert len(rep.results) == 4

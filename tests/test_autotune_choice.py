"""What the autotuner hands out when the timings are known (no GPU: the simulations, the batches and
the clock are stand-ins).  The library's own default must be among the timed choices and must come
out as itself when it is the fastest."""
import pytest

from paper_1903_01168_gb300 import autotune as A
from paper_1903_01168_gb300 import lbm as L


class Sim:
    def __init__(self, nx, ny, choice):
        self.nx, self.ny, self.choice = nx, ny, choice
        self.params = L.lbm_params()

    def step(self, n):
        Clock.choice = (self.choice["kernel"], self.choice["plan_rows"])

    def close(self):
        pass


class Batch:
    def __init__(self, sims, row_overhead=None, plan=L.LBM_PLAN_AUTO, member_plan_rows=None):
        self.choice = (plan, row_overhead, tuple(member_plan_rows or [0] * len(sims)))

    def step(self, n, use_graph=True):
        Clock.choice = self.choice

    def close(self):
        pass


class Clock:
    choice = None


@pytest.fixture
def clock(monkeypatch):
    """Give it ms(choice): that is what every run takes."""
    def use(ms):
        def event_ms(run, steps):
            run(steps)
            return ms(Clock.choice)
        monkeypatch.setattr(A, "_event_ms", event_ms)
        monkeypatch.setattr(A, "_start", lambda nx, ny, params, choice: Sim(nx, ny, choice))
        monkeypatch.setattr(A.L, "Batch", Batch)
    return use


def test_single_lattice_keeps_the_default_where_it_is_fastest(clock):
    clock(lambda c: {(L.LBM_KERNEL_FUSED, 0): 4.4, (L.LBM_KERNEL_TWOPASS, 0): 12.4}.get(c, 15.0))
    t = A.Autotuner()
    assert t.tune_single(64, 64)["plan_rows"] == 0
    assert t.params_for(64, 64, False, gamma=1.0) == {"gamma": 1.0, "kernel": L.LBM_KERNEL_FUSED, "plan_rows": 0}


def rows_ms(best):
    """A batch whose two classes are fastest with these plan_rows."""
    return lambda c: 10.0 + sum(0.0 if r == b else 1.0 for r, b in zip(c[2], best)) + abs(c[1] or 0.0) * 0.01


SIMS = [Sim(300, 200, None), Sim(64, 64, None)]


@pytest.mark.parametrize("best", [(0, 0), (8, 0), (0, 16), (64, 8)])
def test_batch_rows_come_out_as_timed(clock, best):
    clock(rows_ms(best))
    t = A.Autotuner()
    got = t.tune_batch(SIMS)
    assert tuple(got["member_plan_rows"]) == best
    for s, r in zip(SIMS, best):
        assert t.params_for(s.nx, s.ny, True) == {"plan_rows": r}


def test_one_slow_timing_of_the_default_does_not_decide(clock):
    calls = []

    def ms(c):
        calls.append(c)
        return 100.0 if len(calls) == 1 else rows_ms((0, 0))(c)

    clock(ms)
    assert A.Autotuner().tune_batch(SIMS)["member_plan_rows"] == [0, 0]


def test_the_default_plan_is_a_candidate(clock):
    clock(lambda c: 5.0 if c[:2] == (L.LBM_PLAN_AUTO, -1.0) else 6.0)
    best, timings = A.tune_plan(SIMS)
    assert best == (L.LBM_PLAN_AUTO, -1.0) and len(timings) == len(A.PLAN_OPTION_CANDIDATES)
    assert {(L.LBM_PLAN_SPLIT, 8.0), (L.LBM_PLAN_BALANCED, 8.0)} <= set(timings)   # the default's row cost

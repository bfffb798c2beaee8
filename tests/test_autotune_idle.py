"""Options that shape no launch at a precision are not searched: the binding
names them, and the search holds them at their defaults.  The shared-memory
copy of the fused coarse V-cycle is a choice at every precision."""
from paper_1703_06606_gb300 import autotune, qnsch
from paper_1703_06606_gb300 import workloads as W


def search(idle):
    calls, t = [], [0.0]

    class Solver:
        IDLE_OPTIONS = idle

        def __init__(self, **kw):
            self.kw = kw
            calls.append(kw)

        def set_fields(self, f):
            pass

        def step(self, dt):  # noise that favours whatever is tried with 8192
            t[0] += 0.9 if self.kw["vanka_team_max32"] == 8192 else 1.0
            return 5, 1e-10
    best, _, _ = autotune.tune(W.small_case(32, 32, False), precision=1, steps=2, warmup=0,
                               solver_cls=Solver, clock=lambda: t[0])
    return best, {c["vanka_team_max32"] for c in calls}


def test_idle_options_keep_their_defaults():
    best, tried = search(qnsch.Solver.IDLE_OPTIONS)
    assert best["vanka_team_max32"] == 65536 and tried == {65536}
    assert best["ch_team_max32"] == 0
    best, tried = search({})
    assert best["vanka_team_max32"] == 8192 and len(tried) > 1


def test_the_copy_is_searched_at_every_precision():
    assert all("coarse_smem" in knobs for knobs in autotune.KNOBS.values())

"""The autotuner spends no search over norm estimates on a knob that changes nothing."""
from paper_1808_00128_gb300 import autotune


def test_norm_folds_are_not_searched():
    assert autotune.CANDIDATES["norm_max_folds"] == [12]


def test_values_of_one_candidate_are_timed_once():
    class Sim:
        n, chi, device = 40, 1 << 16, 0
        tuning = dict(mc_chains_per_block=64, mc_stages=1, mc_lookahead=2)

        def set_tuning(self, name, value):
            self.tuning[name] = value

        def get_tuning(self, name):
            return self.tuning[name]

        def metropolis(self, steps, seed):
            pass

    calls = []

    def timer(fn):
        calls.append(dict(Sim.tuning))
        return 1.0

    keep = autotune.CANDIDATES["mc_lookahead"]
    try:
        autotune.CANDIDATES["mc_lookahead"] = [2]
        chosen = autotune.tune(Sim(), chains=64, timer=timer)
    finally:
        autotune.CANDIDATES["mc_lookahead"] = keep
    assert chosen["mc_lookahead"] == (2, 1.0)
    assert len(calls) == 2 + 4 + 1

"""The tuner's timing of one candidate: a disturbed repetition, which can only be slower, does not count."""
import pytest

from paper_0704_1672_gb300 import autotune


class FakeCtx:
    def __init__(self, times):
        self.times, self.profiling = list(times), False

    def tcm_ctx_set_profiling(self, on):
        self.profiling = on

    def tcm_ctx_read_profile(self):
        return {"moments": self.times.pop(0)}, {}


@pytest.mark.parametrize("times, want", [((1.0, 1.4), 1.0), ((1.4, 1.0), 1.0), ((1.1, 1.0, 3.0), 1.0), ((2.0,), 2.0)])
def test_a_slow_repetition_does_not_count(times, want):
    ctx, runs = FakeCtx((0.0,) + times), []  # the read before the repetitions clears the profile
    assert autotune.moment_phase_ms(ctx, lambda: runs.append(1), len(times)) == want
    assert len(runs) == len(times) + 1 and ctx.profiling is False


class SettingsCtx:
    """Records tunings; the moment phase's time is given by the test."""

    def __init__(self):
        self.tiling, self.km = {}, {}

    def tcm_ctx_set_tiling_l(self, precision, L, apl, cps):
        self.tiling[L] = (apl, cps)

    def tcm_ctx_get_tiling_l(self, precision, L):
        return self.tiling.get(L, (64, 2))

    def tcm_ctx_set_chunking_l(self, L, km):
        self.km[L] = km

    def tcm_ctx_get_chunking_l(self, L):
        return self.km.get(L, 160), 1

    def tcm_energy_batch_packed(self, pb, precision):
        pass


@pytest.mark.parametrize("ms96, ms64, sampled, want", [
    (1.00, 1.015, True, 64),   # within 2 % of the fastest: the setting in force stays
    (1.015, 1.00, True, 64),
    (1.00, 1.03, True, 96),    # a gain beyond 2 %: taken
    (1.00, 1.015, False, 96)])  # the whole batch was timed: the fastest
def test_a_sampled_degree_leaves_its_setting_only_for_a_gain(ms96, ms64, sampled, want):
    import numpy as np
    from paper_0704_1672_gb300 import tcm
    ctx, k = SettingsCtx(), 10
    system = tcm.tcm_system()
    times = {(96, 2, 160): ms96, (64, 2, 160): ms64}
    res = autotune.tune(ctx, [system, system], np.zeros(k, int), np.ones(k, int), np.full(k, 16), np.ones((k, 3)),
                        precision=tcm.TCM_MIXED, max_items_per_l=4 if sampled else 64, atoms_per_lane=(32, 64, 96),
                        measure=lambda L, run: times.get(autotune.get_setting(ctx, tcm.TCM_MIXED, L), 9.0))
    assert res.best[16] == (want, 2, 160) == autotune.get_setting(ctx, tcm.TCM_MIXED, 16)

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

"""The autotuner compiles and times every kernel once (no GPU: the search against a cost table)."""
import pytest

from paper_1504_00353_gb300 import autotune

# what changes the generated kernel or its launch; local_leaves is accepted in a shape and
# changes nothing
KERNEL_KEYS = [k for k in autotune.SHAPE_KEYS if k != "local_leaves"]


class CountingTuner(autotune.CodeTuner):
    def __init__(self, latency):  # no device: only the search logic
        self.N, self.K, self.dtype, self.latency = 32768, 29492, "i8", latency
        self.seen, self.log, self.timed = {}, None, []

    def measure(self, shapes):
        for s in map(self.clamp, shapes):
            k = autotune._shape_key(s)
            if k not in self.seen:
                self.seen[k] = 1.0 + len(self.seen) * 1e-6  # the first stays the best
                self.timed.append(tuple(s[k] for k in KERNEL_KEYS))


@pytest.mark.parametrize("latency", [False, True])
def test_no_kernel_is_timed_twice(latency):
    t = CountingTuner(latency)
    best, _ = t.tune_latency() if latency else t.tune()
    assert len(t.timed) == len(set(t.timed)), [s for s in t.timed if t.timed.count(s) > 1]
    assert best["local_leaves"] == 0

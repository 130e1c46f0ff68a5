"""The chain's kernels against themselves: what a pass may not cost beside a pass that does the
same work or more. Least of several means over many launches, so other work on the machine
does not decide."""
import pytest

torch = pytest.importorskip("torch")

from paper_1504_00353_gb300 import polar, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def us(fn, launches=100, repeats=9):
    for _ in range(10):
        fn()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(repeats):
        torch.cuda._sleep(1_000_000)  # the launches queue up behind it
        a.record()
        for _ in range(launches):
            fn()
        b.record()
        b.synchronize()
        best = min(best, 1e3 * a.elapsed_time(b) / launches)
    return best


@pytest.mark.parametrize("N,K,n", [(32, 23, 5000), (64, 47, 5000)])
def test_counting_errors_costs_no_more_than_none(N, K, n):
    """Every frame in error (a simulation at low Eb/N0) against no frame in error: the same
    bytes are read, only the sums differ (equal times; five times as long with an atomic per
    lane)."""
    code = polar.polar_code_create(N, K, synth.frozen_mask(N, K, 3.0))
    sent = torch.zeros((n, (K + 7) // 8), dtype=torch.uint8, device="cuda")
    wrong = torch.full_like(sent, 1)
    cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
    none = us(lambda: polar.polar_count_errors(code, sent, sent, cnt))
    every = us(lambda: polar.polar_count_errors(code, wrong, sent, cnt))
    assert every < 2.5 * none, (every, none)


def test_encoding_few_long_frames_keeps_their_chain_short():
    """Few frames: a frame of twice the length gets twice the warps, so it takes hardly longer
    (6.2 us both; 10.3 with the words of N = 8192 on one warp)."""
    t = {}
    for N in (4096, 8192):
        K = 3 * N // 4
        code = polar.polar_code_create(N, K, synth.frozen_mask(N, K, 3.0))
        info = torch.zeros((100, K // 8), dtype=torch.uint8, device="cuda")
        cw = torch.zeros((100, N // 8), dtype=torch.uint8, device="cuda")
        t[N] = us(lambda: polar.polar_encode_systematic_device(code, info, cw))
    assert t[8192] < 1.4 * t[4096], t

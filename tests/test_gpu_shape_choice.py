"""Which decoder a handle runs for a batch size: what a program asked for stays what it gets,
and every choice gives the oracle's bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_00353_gb300 import autotune, polar
from tests import _cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def make(N, K, n, i8, seed=3):
    rng = np.random.default_rng(seed)
    mask = _cases.random_mask(rng, N, K)
    y = rng.integers(-127, 128, (n, N)).astype(np.int8) if i8 else \
        (rng.standard_normal((n, N)) * 3).astype(np.float32)
    return mask, y, torch.from_numpy(y).cuda()


def check_bits(code, mask, y, t, i8, n):
    got = (polar.polar_decode_i8 if i8 else polar.polar_decode)(code, t[:n]).cpu().numpy()
    polar.polar_code_check(code)
    sample = np.unique(np.concatenate([np.arange(min(3, n)), [n // 2, n - 1]]))
    assert np.array_equal(got[sample], oracle.decode_batch(mask, y, frames=sample))


@pytest.mark.parametrize("i8", [False, True])
@pytest.mark.parametrize("frames", [0, 1])
def test_zero_or_one_is_one_frame_per_cta(frames, i8):
    """polar_code_set_frames_per_cta(0) and (1) both mean one frame per CTA, also for batches
    for which the library would choose several."""
    n = 12 * sms() + 3
    mask, y, t = make(256, 100, n, i8)
    code = polar.polar_code_create(256, 100, mask)
    polar.polar_code_set_frames_per_cta(code, i8, frames)
    polar.polar_code_compile(code, i8, n)
    launch = polar.polar_code_get_launch(code, i8, n)
    assert launch["unrolled"] and launch["frames_per_cta"] == 1
    check_bits(code, mask, y, t, i8, n)
    autotune.configure(code, "i8" if i8 else "f32", {}, n)  # an empty shape does not undo it
    assert polar.polar_code_get_launch(code, i8, n)["frames_per_cta"] == 1


def test_empty_shape_leaves_the_choice_to_the_library():
    n = 12 * sms() + 3
    mask, _, _ = make(256, 100, 1, True)
    code = polar.polar_code_create(256, 100, mask)
    autotune.configure(code, "i8", {}, n)
    assert polar.polar_code_get_launch(code, True, n)["frames_per_cta"] == 4


@pytest.mark.parametrize("i8", [False, True])
def test_narrow_warp_stage_is_kept(i8):
    """warp_stage_max = 32 with 32-leaf register subtrees: nodes of 64 run on the whole CTA. The
    interpreter, whose subtrees have 64 leaves, takes 64."""
    n = 200
    mask, y, t = make(512, 200, n, i8)
    code = polar.polar_code_create(512, 200, mask)
    polar.polar_code_set_launch(code, i8, threads=64, warp_stage_max=32)
    assert polar.polar_code_get_launch(code, i8, n)["warp_stage_max"] == 64
    check_bits(code, mask, y, t, i8, n)
    polar.polar_code_compile(code, i8, n, 32)
    launch = polar.polar_code_get_launch(code, i8, n)
    assert launch["unrolled"] == 32 and launch["warp_stage_max"] == 32
    check_bits(code, mask, y, t, i8, n)


def short_list(N):
    """A mask with a short operation list."""
    mask = np.ones(N, np.uint8)
    mask[N // 2:] = 0
    mask[N // 2::4096] = 1
    return mask


@pytest.mark.parametrize("i8", [False, True])
@pytest.mark.parametrize("N,frames", [(1 << 16, 4), (1 << 18, 1)])
def test_long_codes_keep_frames_in_flight(N, frames, i8):
    """The library's own shape takes several frames per CTA only where shared memory then still
    holds eight frames per SM: not for N = 2^18, whose bits alone are 32 KB a frame."""
    mask = short_list(N)
    K, n = int((mask == 0).sum()), 12 * sms()
    code = polar.polar_code_create(N, K, mask)
    polar.polar_code_compile(code, i8, n)
    launch = polar.polar_code_get_launch(code, i8, n)
    assert launch["unrolled"] and launch["frames_per_cta"] == frames
    rng = np.random.default_rng(5)
    y = rng.integers(-127, 128, (80, N)).astype(np.int8 if i8 else np.float32)
    t = torch.from_numpy(y).cuda()
    check_bits(code, mask, y, t, i8, 80)


@pytest.mark.parametrize("i8", [False, True])
def test_full_batch_handle_decodes_smaller_batches_one_per_cta(i8):
    """A handle compiled for a full batch of a long code runs batches that one CTA per frame
    holds at once with one frame per CTA, larger ones with four; the decoder of an earlier
    compile is kept beside them."""
    N, full = 1 << 14, 12 * sms() + 3
    mask = short_list(N)
    K = int((mask == 0).sum())
    rng = np.random.default_rng(6)
    y = rng.integers(-9, 10, (full, N)).astype(np.int8 if i8 else np.float32)
    t = torch.from_numpy(y).cuda()
    code = polar.polar_code_create(N, K, mask)
    for first in (full, 1):  # alone, then beside the batch-1 decoder
        if first == 1:
            polar.polar_code_compile(code, i8, 0)
            polar.polar_code_compile(code, i8, 1)
        polar.polar_code_compile(code, i8, full)
        for n, frames in ((full, 4), (12 * sms() - 1, 4), (8 * sms(), 1), (sms() + 1, 1), (1, 1)):
            launch = polar.polar_code_get_launch(code, i8, n)
            assert launch["frames_per_cta"] == frames, n
            assert bool(launch["unrolled"]) == (n > 1 or first == 1)
            check_bits(code, mask, y, t, i8, n)
    host = polar.polar_decode_host(code, t[:sms() * 8].cpu()).numpy()  # eight chunks
    assert np.array_equal(host[:2], oracle.decode_batch(mask, y, frames=np.arange(2)))
    assert np.array_equal(host, (polar.polar_decode_i8 if i8 else polar.polar_decode)(code, t[:sms() * 8]).cpu().numpy())

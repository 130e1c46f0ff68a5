"""Register subtrees and output packing of the specialised decoders at the sizes
where they can go wrong, bit for bit against the CPU oracle: subtree sizes on both
sides of a warp's lanes, LLRs with zeros and ties, and rows whose length is no
multiple of a word. Every comparison is exact (integers and IEEE operations in the
oracle's order), so no tolerance enters."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_00353_gb300 import polar
from tests import _cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def decode(code, y, i8, out=None):
    t = torch.from_numpy(np.ascontiguousarray(y)).cuda()
    got = (polar.polar_decode_i8 if i8 else polar.polar_decode)(code, t, out)
    torch.cuda.synchronize()
    polar.polar_code_check(code)
    return got


def llrs(rng, n, N, i8):
    """Small integers: many zeros and equal magnitudes, and int8 sums that saturate."""
    y = np.where(rng.random((n, N)) < 0.2, rng.integers(-127, 128, (n, N)), rng.integers(-3, 4, (n, N)))
    return y.astype(np.int8) if i8 else y.astype(np.float32)


@pytest.mark.parametrize("N,K", [(2, 1), (32, 9), (64, 33), (128, 31), (256, 97), (1024, 1000),
                                 (2048, 40), (4096, 3687)])
@pytest.mark.parametrize("compiled", [False, True])
def test_packed_rows(N, K, compiled):
    """Rows of every length mod 4 at every alignment, sparse and dense information sets."""
    rng = np.random.default_rng(N + K)
    mask = _cases.random_mask(rng, N, K)
    code = polar.polar_code_create(N, K, mask)
    n, row = 37, (K + 7) // 8
    y = rng.integers(-127, 128, (n, N)).astype(np.int8)
    want = oracle.decode_batch(mask, y)
    if compiled:
        polar.polar_code_compile(code, True, n)
    buf = torch.full((n * row + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    for shift in range(4):  # the row's address mod 4; nothing outside the rows is written
        buf.fill_(0xA5)
        decode(code, y, True, buf[shift:shift + n * row])
        got = buf.cpu().numpy()
        assert np.array_equal(got[shift:shift + n * row].reshape(n, row), want)
        assert (got[:shift] == 0xA5).all() and (got[shift + n * row:] == 0xA5).all()


@pytest.mark.parametrize("i8", [False, True])
@pytest.mark.parametrize("N,reg", [(4, 32), (16, 32), (32, 32), (64, 32), (64, 64), (64, 128),
                                   (512, 512)])
def test_one_frame_subtrees(N, reg, i8):
    """One frame per warp, subtrees of fewer, as many and more leaves than lanes."""
    rng = np.random.default_rng(7 * N + reg)
    for K in sorted({1, N // 4 + 1, N // 2, N - 1}):
        mask = _cases.random_mask(rng, N, K)
        code = polar.polar_code_create(N, K, mask)
        y = llrs(rng, 65, N, i8)
        polar.polar_code_compile(code, i8, 65, reg)
        assert np.array_equal(decode(code, y, i8).cpu().numpy(), oracle.decode_batch(mask, y))


@pytest.mark.parametrize("compiled", [False, True])
def test_negative_zero_decides_zero(compiled):
    """F of a zero and a negative LLR is -0.0, which is not negative: a wide Rate-1 node in
    memory decides 0 for it."""
    mask = np.concatenate([np.zeros(512, np.uint8), np.ones(511, np.uint8), [0]]).astype(np.uint8)
    rng = np.random.default_rng(5)
    y = rng.integers(-2, 3, (40, 1024)).astype(np.float32)
    code = polar.polar_code_create(1024, 513, mask)
    if compiled:
        polar.polar_code_compile(code, False, 40)
    assert np.array_equal(decode(code, y, False).cpu().numpy(), oracle.decode_batch(mask, y))


@pytest.mark.parametrize("i8", [False, True])
@pytest.mark.parametrize("N,K", [(2, 1), (8, 3), (64, 33), (512, 257), (2048, 1707), (8192, 4501)])
def test_library_shape(N, K, i8):
    """The library's own shape: one frame per CTA for few frames, four for many, and whichever
    was compiled for decodes of the other size."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few, many = 4 * sms + 1, 12 * sms + 3
    rng = np.random.default_rng(N + i8)
    mask = _cases.random_mask(rng, N, K)
    y = llrs(rng, many, N, i8)
    sample = np.unique(np.concatenate([np.arange(3), rng.integers(0, few, 20), [few - 1, many - 1]]))
    want = oracle.decode_batch(mask, y, frames=sample)
    for compiled, frames in ((few, 1), (many, 4)):
        code = polar.polar_code_create(N, K, mask)
        polar.polar_code_compile(code, i8, compiled)
        for n in (few, many):
            assert polar.polar_code_get_launch(code, i8, n)["frames_per_cta"] == frames
            got = decode(code, y[:n], i8).cpu().numpy()
            assert np.array_equal(got[sample[sample < n]], want[sample < n]), (compiled, n)
    both = polar.polar_code_create(N, K, mask)
    polar.polar_code_compile(both, i8, few)
    polar.polar_code_compile(both, i8, many)
    assert polar.polar_code_get_launch(both, i8, few)["frames_per_cta"] == 1
    assert polar.polar_code_get_launch(both, i8, many)["frames_per_cta"] == 4


@pytest.mark.parametrize("i8", [False, True])
@pytest.mark.parametrize("N", [2, 4, 16, 64, 128, 1024])
def test_interpreter_subtrees(N, i8):
    """The interpreter's register subtrees, all node kinds and sides, against the oracle."""
    rng = np.random.default_rng(3 * N + i8)
    for K in sorted({1, N // 3 + 1, N // 2, N - N // 8, N - 1}):
        mask = _cases.random_mask(rng, N, K)
        y = llrs(rng, 65, N, i8)
        code = polar.polar_code_create(N, K, mask)
        assert polar.polar_code_get_launch(code, i8, 65)["unrolled"] == 0
        assert np.array_equal(decode(code, y, i8).cpu().numpy(), oracle.decode_batch(mask, y))


@pytest.mark.parametrize("threads,F", [(32, 1), (32, 4), (128, 1)])
@pytest.mark.parametrize("n", [512, 1024, 4096])
def test_wide_int8_nodes(n, threads, F):
    """int8 SPC and Rate-1 nodes in memory, the latter right after their G, on one warp and on a
    CTA: ties of the least magnitude in several vectors, all-zero nodes, odd and even parity."""
    spc = np.zeros(n, np.uint8)
    spc[0] = 1
    for mask in (np.concatenate([spc, np.zeros(n, np.uint8)]), np.concatenate([spc, spc])):
        N, K = 2 * n, int((mask == 0).sum())
        rng = np.random.default_rng(n + threads)
        y = llrs(rng, 150, N, True)
        y[0] = 0
        y[1] = 127
        y[2] = -127
        y[3:40] = np.where(y[3:40] == 0, 5, y[3:40])
        code = polar.polar_code_create(N, K, mask)
        polar.polar_code_set_launch(code, True, threads=threads, smem_stage_max=64 if n < 4096 else 1024,
                                    warp_stage_max=256 if threads > 32 else 0, stage_channel=2)
        polar.polar_code_set_frames_per_cta(code, True, F)
        polar.polar_code_compile(code, True, 150, 256)
        assert polar.polar_code_get_launch(code, True, 150)["frames_per_cta"] == F
        want = oracle.decode_batch(mask, y)
        assert np.array_equal(decode(code, y, True).cpu().numpy(), want)
        polar.polar_code_compile(code, True, 0)  # and the interpreter
        assert np.array_equal(decode(code, y, True).cpu().numpy(), want)

"""The chain's kernels at sizes on both sides of their splits (words per lane, warps
per frame, draws per warp, lanes per frame) and at every row alignment, against the
oracle's encoder, Philox from its definition and plain counting: all bits, compared
exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1504_00353_gb300 import polar, synth
from tests import _philox

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def rows(n, row, shift):
    """A device buffer of n rows that starts `shift` bytes off, and all of its bytes."""
    buf = torch.full((n * row + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    return buf[shift:shift + n * row], buf


@pytest.mark.parametrize("N,K", [(2, 1), (4, 3), (32, 16), (64, 40), (128, 71), (256, 128), (512, 300),
                                 (4096, 3001), (8192, 7000), (16384, 9001), (65536, 50001),
                                 (131072, 100003), (262144, 200001), (524288, 300007)])
@pytest.mark.parametrize("shift", [0, 1])
def test_encoder_sizes(N, K, shift):
    mask = synth.frozen_mask(N, K, 3.0)
    code = polar.polar_code_create(N, K, mask)
    n, row, out_row = 5, (K + 7) // 8, (N + 7) // 8
    d = synth.info_bits(np.random.default_rng(N + shift), n, K)
    info, _ = rows(n, row, shift)
    info.copy_(torch.from_numpy(synth.pack_bits(d).reshape(-1)))
    cw, whole = rows(n, out_row, shift)
    polar.polar_encode_systematic_device(code, info, cw, n_frames=n)
    got = synth.unpack_bits(cw.cpu().numpy().reshape(n, out_row), N)
    for f in range(n):
        assert np.array_equal(got[f], oracle.encode_systematic(mask, d[f])), f
    w = whole.cpu().numpy()
    assert (w[:shift] == 0xA5).all() and (w[shift + n * out_row:] == 0xA5).all()


@pytest.mark.parametrize("K", [1, 125, 129, 4093, 4096, 4101, 8200])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_random_info_rows(K, shift):
    N = 1 << max(1, int(np.ceil(np.log2(K + 1))))
    code = polar.polar_code_create(N, K, synth.frozen_mask(N, K, 3.0))
    n, row = 3, (K + 7) // 8
    out, whole = rows(n, row, shift)
    polar.polar_random_info(code, out, 0x5EED_0000_0007, 11, n_frames=n)
    got = out.cpu().numpy().reshape(n, row)
    for f in range(n):
        assert np.array_equal(got[f], _philox.info_bytes(K, 0x5EED_0000_0007, 11 + f)), f
    w = whole.cpu().numpy()
    assert (w[:shift] == 0xA5).all() and (w[shift + n * row:] == 0xA5).all()


@pytest.mark.parametrize("K", [3, 128, 130, 1000, 4099])
@pytest.mark.parametrize("shift", [(0, 0), (1, 1), (0, 5)])
def test_count_errors_rows(K, shift):
    N = 1 << int(np.ceil(np.log2(K + 1)))
    code = polar.polar_code_create(N, K, synth.frozen_mask(N, K, 3.0))
    n, row = 1003, (K + 7) // 8
    rng = np.random.default_rng(K)
    x = rng.integers(0, 256, (n, row), dtype=np.uint8)
    y = x ^ np.where(rng.random((n, row)) < 0.3 / row, rng.integers(0, 256, (n, row)), 0).astype(np.uint8)
    a, _ = rows(n, row, shift[0])
    b, _ = rows(n, row, shift[1])
    a.copy_(torch.from_numpy(x.reshape(-1)))
    b.copy_(torch.from_numpy(y.reshape(-1)))
    cnt = torch.tensor([5, 7], dtype=torch.int64, device="cuda")
    polar.polar_count_errors(code, a, b, cnt, n_frames=n)
    diff = np.unpackbits(x ^ y, axis=1).sum(1)
    assert cnt.tolist() == [5 + int((diff > 0).sum()), 7 + int(diff.sum())]

"""The int8 clamp as one f16 operation (``hsat2`` in ``polar_ops.cuh``): Eq. 1 with the constant
127 is min(|v|, 127) with the sign of v, which is clamp(v, -127, 127) for every sum v of two int8
LLRs. Checked on the host for all 509 sums and both zeros."""
import numpy as np


def test_eq1_with_127_is_the_clamp():
    c = np.array(0x57F0, np.uint16).view(np.float16)
    assert c == 127
    v = np.concatenate([np.arange(-254, 255), [-0.0]]).astype(np.float16)
    neg = np.signbit(v) ^ np.signbit(c)
    r = np.where(neg, -np.minimum(np.abs(v), np.abs(c)), np.minimum(np.abs(v), np.abs(c)))
    assert np.array_equal(r.astype(np.float64), np.clip(v.astype(np.float64), -127, 127))

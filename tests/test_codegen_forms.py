"""Which form of an operation a generated decoder uses for which launch shape, read off the
program (polar_codegen.cpp) on the host."""
import subprocess

import pytest

from paper_1504_00353_gb300 import synth
from tests.test_codegen_store_policies import emitter  # noqa: F401


def emit(emitter, tmp_path, *, N=8192, K=6000, i8=1, T=32, S=512, F=1, reg=256, outline=0):  # noqa: F811
    (tmp_path / "mask.bin").write_bytes(synth.frozen_mask(N, K, 3.0).astype("uint8").tobytes())
    out = tmp_path / "code.cu"
    r = subprocess.run([str(a) for a in (emitter, "code", out, tmp_path / "mask.bin", N, K, i8, T, S,
                                         1024, F, 0, reg, outline, 0)],
                       capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout
    return out.read_text()


@pytest.mark.parametrize("T,F,outline,fused", [(32, 1, 0, False), (64, 1, 0, False), (256, 1, 1, False),
                                               (128, 4, 0, True), (64, 2, 1, True), (128, 4, 3, False)])
def test_g_with_rate1_in_one_pass_only_for_several_frames(emitter, tmp_path, T, F, outline, fused):  # noqa: F811
    """The G / Rate-1 pass holds eight vectors and pays only where frames share a CTA's code."""
    assert ("op_g_r1<" in emit(emitter, tmp_path, T=T, F=F, outline=outline)) == fused
    assert "op_g_r1<" not in emit(emitter, tmp_path, i8=0, T=T, F=F, outline=outline)

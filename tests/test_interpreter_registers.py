"""The operation-list interpreter keeps its state in registers: compiled for sm_103a with the
build's flags, its decoding kernels spill nothing to local memory (ptxas -v, no GPU), so a
subtree's registers do not live on across the memory-level operations."""
import os
import re
import shutil
import subprocess

import pytest

from paper_1504_00353_gb300 import build


def test_interpreter_kernels_do_not_spill(tmp_path):
    nvcc = build.nvcc()
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    build.build()  # also writes the generated include
    r = subprocess.run([nvcc, "-O3", "-std=c++17", *build.ARCH, "-lineinfo", "-Xptxas", "-v",
                        "-I" + os.path.join(build.ROOT, "include"), "-I" + build.CSRC, "-I" + build.GEN,
                        "-c", os.path.join(build.CSRC, "polar_kernels.cu"), "-o", str(tmp_path / "k.o")],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    found = {}
    for name, spill in re.findall(r"entry function '([^']*fastssc_decode_kernel[^']*)'.*?"
                                  r"(\d+) bytes spill stores", r.stderr, re.S):
        # template arguments: LLR type, trace, staged channel
        typ, trace, stage = re.search(r"kernelI([af])Lb([01])ELb([01])E", name).groups()
        found[typ, trace == "1", stage] = int(spill)
    assert len(found) == 8, found
    assert all(v == 0 for (_, trace, _), v in found.items() if not trace), found
    assert all(v <= 32 for v in found.values()), found

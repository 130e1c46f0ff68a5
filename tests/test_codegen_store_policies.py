"""Scratch stages that a specialised decoder stores with the L2 evict-last policy are
discarded after their last read, so no line keeps that priority when the launch is over.
Read off the generated program (polar_codegen.cpp) on the host, in program order."""
import os
import re
import shutil
import subprocess

import pytest

from paper_1504_00353_gb300 import build, synth

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1504_00353_gb300", "csrc")
NEAR = 2  # ST_NEAR of polar_ops.cuh

STAGE = re.compile(r"gen_out<T, S, (\d+)u>\(fr\)")


@pytest.fixture(scope="module")
def emitter(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    lib = build.build()
    exe = tmp_path_factory.mktemp("emit") / "codegen_source"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", "/usr/local/cuda/include", os.path.join(HERE, "cpp", "codegen_source.cpp"),
                    "-L", os.path.dirname(lib), "-lpolar_gb300",
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True)
    return exe


def near_stores(line):
    """Stages that an operation of the generated program stores evict-last."""
    m = re.search(r"(op|mem)_(fg|chain)<T, \w+, ([^>]*)>\(", line)
    if not m:
        return []
    args, outs = m.group(3).split(", "), [int(n) for n in STAGE.findall(line)]
    if m.group(2) == "fg":
        wr = int(args[2].rstrip("u")) if len(args) > 2 else 0
        return outs if wr == NEAR else []
    length, store = int(args[0].rstrip("u")), int(args[4].rstrip("u"))
    wr = int(args[6].rstrip("u")) if len(args) > 6 else 0
    assert len(outs) == length
    stored = [k for k in range(length) if k == length - 1 or store >> k & 1]
    return [outs[k] for k in stored if wr >> (2 * k) & 3 == NEAR]


@pytest.mark.parametrize("i8", [0, 1])
@pytest.mark.parametrize("T,S,F,reg,outline", [(32, 64, 1, 256, 0), (128, 64, 1, 512, 1), (128, 256, 4, 512, 1),
                                               (128, 512, 1, 1024, 3), (128, 1024, 4, 256, 1)])
def test_evict_last_stages_are_discarded(emitter, tmp_path, i8, T, S, F, reg, outline):
    N, K = 8192, 6000
    (tmp_path / "mask.bin").write_bytes(synth.frozen_mask(N, K, 3.0).astype("uint8").tobytes())
    out = tmp_path / "code.cu"
    r = subprocess.run([str(a) for a in (emitter, "code", out, tmp_path / "mask.bin", N, K, i8, T, S,
                                         2048, F, 0, reg, outline, 0)],
                       capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout
    held, seen = {}, 0  # stage -> line of its evict-last store, not yet discarded
    for line in out.read_text().splitlines():
        for n in re.findall(r"discard_l2<\w+>\(gen_in<T, N, S, (\d+)u>", line):
            held.pop(int(n), None)
        for n in near_stores(line):
            assert n not in held, f"stage {n} stored again before it was discarded: {held[n]}"
            held[n] = line.strip()
            seen += 1
    assert not held, held
    assert seen  # the shape has such stages

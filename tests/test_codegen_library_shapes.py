"""The programs that the library builds by its own choice compile for sm_103a with nvcc
(no GPU): the int8 mixed batch with its 512-leaf register subtrees, and the four-frames-per-CTA
shape of a handle whose launch shape is left to the library, both LLR types. The tuned shapes of
the benchmark are compiled by test_codegen_compiles.py."""
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

from paper_1504_00353_gb300 import build, synth
from tests.test_codegen_compiles import CSRC, CUDA_INC, HERE, ROOT, _mask_file, _tools

# (name, (N, K, design dB), is_i8, S): 128 threads, four frames per CTA, W = 512, 256-leaf
# register subtrees, CTAs per SM as for a few thousand frames
LIBRARY = [("i8_library", (2048, 1707, 3.5), 1, 1024), ("f32_library", (8192, 6000, 3.0), 0, 512)]
MIXED_S, MIXED_W, MIXED_R = [128, 512, 1024, 1024, 1024], [512, 1024, 2048, 2048, 2048], 512


def test_library_shapes_compile_for_sm103a(tmp_path):
    cxx, nvcc = _tools()
    lib = build.build()
    exe = tmp_path / "codegen_source"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", CUDA_INC, os.path.join(HERE, "cpp", "codegen_source.cpp"),
                    "-L", os.path.dirname(lib), "-lpolar_gb300",
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True)
    jobs = [(tmp_path / f"{name}.cu", "polar_unrolled(",
             ["code", tmp_path / f"{name}.cu", _mask_file(tmp_path, N, K, db), N, K, i8, 128, S, 512,
              4, 0, 256, 0, 7]) for name, (N, K, db), i8, S in LIBRARY]
    args = ["batch", tmp_path / "i8_mixed.cu", 1, 128, 7, 1, 1]
    for (N, K), S, W in zip(synth.MIXED_CODES, MIXED_S, MIXED_W):
        args += [_mask_file(tmp_path, N, K, synth.MIXED_DESIGN_DB), N, K, S, W, MIXED_R]
    jobs.append((tmp_path / "i8_mixed.cu", "polar_batch(", args))
    for src, entry, a in jobs:
        r = subprocess.run([str(exe), *map(str, a)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0 and r.stdout.startswith("OK"), r.stdout
        assert entry in src.read_text()

    def compile_one(src):
        return subprocess.run([nvcc, "-std=c++17", "-cubin", *build.ARCH, "-I", CSRC,
                               "-o", str(src.with_suffix(".cubin")), str(src)],
                              capture_output=True, text=True, timeout=900)

    with ThreadPoolExecutor(max_workers=len(jobs)) as ex:
        for (src, _, _), r in zip(jobs, ex.map(compile_one, [j[0] for j in jobs])):
            assert r.returncode == 0, f"{src.name}:\n{r.stderr[-3000:]}"

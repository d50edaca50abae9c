"""What the assembler reports for kernels that no benchmark runs: the observing and calibrating instantiations of the fused
kernel do not spill more than their row pointers."""
import os
import re
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

import pytest

from paper_2508_13478_b200 import build

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
# width, then PER_TOKEN, ROT, SPREAD, AHEAD, DUMP, BOTH, CALIB, GABOR, MIXED: the worst of each kind when the warp's number
# was a uniform value in all of them (488 to 816 bytes)
KERNELS = [(512, 0, 0, 1, 0, 0, 0, 1, 0, 0), (512, 1, 0, 0, 0, 1, 0, 0, 0, 1), (256, 0, 1, 0, 1, 1, 0, 0, 0, 0), (128, 1, 1, 0, 0, 1, 1, 0, 0, 0),
           (128, 1, 0, 0, 0, 1, 0, 0, 1, 0), (128, 1, 0, 0, 1, 1, 0, 0, 0, 1)]


def spilled_bytes(kernel, folder):
    width, *flags = kernel
    flags = [str(bool(f)).lower() for f in flags]
    src = os.path.join(folder, "k" + "_".join(map(str, kernel)) + ".cu")
    with open(src, "w") as f:
        f.write('#include "dhq_fused.cuh"\nnamespace dhq {\ntemplate __global__ void fused_kernel<%d, %s>(const __grid_constant__ ParamsOf<%s, %s> p);\n}\n'
                % (width, ", ".join(flags), flags[4], flags[6]))
    r = subprocess.run([NVCC, *build.NVCC_FLAGS, "-Xptxas", "-v", "-I", build.CSRC, "-c", "-o", src[:-2] + "o", src], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    after = r.stderr[r.stderr.index("Compiling entry function"):]
    return int(re.search(r"(\d+) bytes spill stores", after[after.index("fused_kernel"):]).group(1))


@pytest.mark.skipif(not shutil.which(NVCC), reason="needs nvcc")
def test_observing_and_calibrating_kernels_spill_little(tmp_path):
    with ThreadPoolExecutor(len(KERNELS)) as pool:
        spills = dict(zip(KERNELS, pool.map(lambda k: spilled_bytes(k, str(tmp_path)), KERNELS)))
    print(spills)
    assert max(spills.values()) <= 240   # bytes a thread stores; 176 when this was written

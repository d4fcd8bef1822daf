"""What the compiler gives the kernels whose speed hangs on how many of them an SM holds (nvcc -Xptxas -v; no GPU)."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2110_00256_gb300 import build

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")


def resources(source, folder):
    """{demangled kernel name: (registers, bytes of spill loads)} of one source file."""
    out = subprocess.run([NVCC] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o",
                                                              str(folder / "x.o")], capture_output=True, text=True, check=True).stderr
    found, name = {}, None
    for line in out.splitlines():
        if m := re.search(r"Compiling entry function '(\S+)'", line):
            name, spill = m.group(1), 0
        elif m := re.search(r"(\d+) bytes spill loads", line):
            spill = int(m.group(1))
        elif (m := re.search(r"Used (\d+) registers", line)) and name:
            found[name], name = (int(m.group(1)), spill), None
    plain = subprocess.run(["c++filt"], input="\n".join(found), capture_output=True, text=True, check=True).stdout.split("\n")
    return dict(zip(plain, found.values()))


def test_event_kernels_with_the_learned_sampler_fit_twice(tmp_path):
    """Two CTAs of 256 threads per SM: at most 128 registers."""
    r = {k: v for k, v in resources("events.cu", tmp_path).items() if re.search(r"(qs|bw)_event_kernel<(float|double), true>", k)}
    assert len(r) == 4
    assert all(v[0] <= 128 for v in r.values()), r


def test_direct_segment_evolution_reloads_no_more(tmp_path):
    """FP32, four particles per thread at 80 registers: bound by its memory streams, and slower by 3 to 7 % with 64 bytes
    of reloads per thread than with 44."""
    r = {k: v for k, v in resources("evolve.cu", tmp_path).items() if re.search(r"evolve_seg_kernel<float, 4, (128|256)>", k)}
    assert len(r) == 2
    assert all(v[0] <= 80 and v[1] <= 44 for v in r.values()), r

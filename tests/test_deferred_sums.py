"""The deferred sums of the clique count (NeCount, clique_nonedge.cuh) are
folded before a lane's can wrap, however many sets one root has: the device
code itself, on the CPU (simt.h)."""
from __future__ import annotations

import os
import re
import subprocess

import pytest

from paper_2212_04551_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def wide_set(tmp_path_factory):
    folder = tmp_path_factory.mktemp("simt")
    for name in ("common.cuh", "clique_nonedge.cuh", "clique_nonedge.cu"):
        src = open(os.path.join(build.CSRC, name)).read()
        src = src.split("// ------------------------------------------------------------------- host")[0]
        src = re.sub(r'asm volatile\("mov.u64 %0, %%globaltimer;" : "=l"\(t\)\);', "t = 0;", src)
        src = re.sub(r'asm\("mov.u32 %0, %%lanemask_lt;" : "=r"\(m\)\);', "m = (1u << (threadIdx.x & 31)) - 1;", src)
        src = src.replace("extern __shared__ __align__(16) uint32_t smem[];", "uint32_t* smem = simt_smem;")
        if name.endswith(".cu"):
            name, src = "device_part.h", src + "\n}\n"
        (folder / name).write_text(src)
    exe = str(folder / "wide_set")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", str(folder), "-I", HERE, "-I", build.INCLUDE, "-I",
                    os.path.join(cuda, "include"), os.path.join(HERE, "simt_wide_set.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("before", [0, 24 << 53])
def test_sets_of_three_sizes_to_go_are_folded(wide_set, before):
    """acc[0] is 24 times what a lane has counted; 24 x 2^53 is above the line
    (2^57) that asks for a fold."""
    out = subprocess.run([wide_set, str(before)], check=True, capture_output=True, text=True).stdout.split()
    most, counted, want = map(int, out)
    assert counted == want + 32 * before // 24
    assert most < 1 << 57

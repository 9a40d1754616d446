"""Device code that no GPU test can bring to its limits, run on the CPU
(simt.h): one block of the kernels' own source."""
from __future__ import annotations

import os
import re
import subprocess

import numpy as np
import pytest

from paper_2212_04551_gb300 import build
from paper_2212_04551_gb300 import graphs as G

HERE = os.path.dirname(os.path.abspath(__file__))


def compile_on_host(folder, program, kernels, host_functions=()):
    """tests/<program>.cpp with the device part of csrc/<kernels> as device_part.h."""
    for name in os.listdir(build.CSRC):
        if not name.endswith(".cuh") and name != kernels:
            continue
        src, _, host = open(os.path.join(build.CSRC, name)).read().partition(
            "// ------------------------------------------------------------------- host")
        src = re.sub(r'asm volatile\("mov.u64 %0, %%globaltimer;" : "=l"\(t\)\);', "t = 0;", src)
        src = re.sub(r'asm\("mov.u32 %0, %%lanemask_lt;" : "=r"\(m\)\);', "m = (1u << (threadIdx.x & 31)) - 1;", src)
        src = src.replace("extern __shared__ __align__(16) uint32_t smem[];", "uint32_t* smem = simt_smem;")
        if name == kernels:
            for f in host_functions:
                src += re.search(r"^\w+ %s\(.*?^}\n" % f, host, flags=re.S | re.M).group(0)
            name, src = "device_part.h", src + "\n}\n"
        (folder / name).write_text(src)
    exe = str(folder / program)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", str(folder), "-I", HERE, "-I", build.INCLUDE, "-I",
                    os.path.join(cuda, "include"), os.path.join(HERE, program + ".cpp"), "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def wide_set(tmp_path_factory):
    return compile_on_host(tmp_path_factory.mktemp("simt"), "simt_wide_set", "clique_nonedge.cu")


@pytest.mark.parametrize("before", [0, 24 << 53])
def test_sets_of_three_sizes_to_go_are_folded(wide_set, before):
    """The deferred sums of the clique count are folded before a lane's can
    wrap, however many sets one root has.  acc[0] is 24 times what a lane has
    counted; 24 x 2^53 is above the line (2^57) that asks for a fold."""
    out = subprocess.run([wide_set, str(before)], check=True, capture_output=True, text=True).stdout.split()
    most, counted, want = map(int, out)
    assert counted == want + 32 * before // 24
    assert most < 1 << 57


@pytest.fixture(scope="module")
def hom5(tmp_path_factory):
    return compile_on_host(tmp_path_factory.mktemp("simt"), "simt_hom", "motif_hom.cu", ("hom_m_words", "hom_warp_words"))


@pytest.mark.parametrize("order", ["sorted", "shuffled"])
def test_unsorted_lists_stay_in_shared_memory(hom5, tmp_path, order):
    """GPM_SKIP_VALIDATE takes lists in any order: the counts are not defined
    then, every access is in bounds."""
    n, hub = 2000, 110
    rng = np.random.default_rng(1)
    around = rng.choice(np.arange(1, n), hub, replace=False)
    g = G.from_edges(n, np.r_[np.zeros(hub, int), around, around[:-1], np.arange(n - 1)],
                     np.r_[around, rng.permutation(around), around[1:], np.arange(1, n)])
    indices = g.indices.copy()
    if order == "shuffled":
        for v in range(n):
            rng.shuffle(indices[g.indptr[v]:g.indptr[v + 1]])
    path = tmp_path / "graph"
    np.r_[[n], g.indptr, indices].astype(np.int32).tofile(path)
    out = subprocess.run([hom5, str(path)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    sums = [int(x) for x in out.stdout.split()]
    assert sums[:2] == [n, len(indices)]

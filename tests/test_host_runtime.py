"""The library's host code on a stand-in CUDA runtime (fake_gpu.py): the order
of copies and launches, failing calls, limits.  CPU only."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from fake_gpu import link
from paper_2212_04551_gb300 import gpm


@pytest.fixture(scope="module")
def _linked(tmp_path_factory):
    # a library of its own per test module: tables are uploaded once per process
    return link(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def gpu(_linked):
    _linked.lib.fake_reset()
    return _linked


def _path(n):
    """A path's CSR, n >= 2."""
    indptr = np.r_[0, 1, np.arange(3, 2 * n - 2, 2), 2 * n - 2]
    indices = np.ravel(np.c_[np.arange(n) - 1, np.arange(n) + 1])[1:-1]
    return indptr, indices


def _two_paths(n):
    ip, ix = _path(n)
    return [0, n, 2 * n], np.r_[ip, ip[-1] + ip[1:]], np.r_[ix, ix + n]


@pytest.mark.parametrize("what", ["binomials", "patterns", "batch"])
def test_tables_have_landed_before_a_launch_on_another_stream(gpu, what):
    """The tables come from pageable memory, whose copy may still be in flight
    when the call returns, and a non-blocking stream waits for no other."""
    if what == "batch":
        b = gpu.batch(*_two_paths(20))            # on a non-blocking stream of its own
        assert gpu.batch_count(b, 0, 5, 2) == gpm.GPM_OK, gpu.error()     # homomorphism table
        assert gpu.batch_count(b, 0, 6, 2) == gpm.GPM_OK, gpu.error()     # pattern table
        gpu.lib.gpm_batch_destroy(b)
    else:
        n, k = (20000, 4) if what == "binomials" else (40, 7)
        g = gpu.graph(*_path(n), stream=gpu.lib.fake_stream(1))
        assert gpu.motifs(g, k) == gpm.GPM_OK, gpu.error()
        gpu.lib.gpm_graph_destroy(g)
    assert gpu.log()
    assert gpu.lib.fake_violations() == 0


@pytest.mark.parametrize("kc,km", [(4, 5), (5, 4), (4, 6), (3, 0)])
def test_a_failed_first_batch_call_leaves_nothing_behind(gpu, kc, km):
    """Whatever allocation (or step of the capture) fails in a batch's first
    call, the next one tries again and succeeds, and nothing is leaked."""
    warm = gpu.batch(*_two_paths(20))                       # the tables of the process
    assert gpu.batch_count(warm, kc, km, 2) == gpm.GPM_OK, gpu.error()
    gpu.lib.gpm_batch_destroy(warm)
    before = gpu.lib.fake_memory_in_use()
    for at in range(1, 100):
        b = gpu.batch(*_two_paths(20))
        gpu.lib.fake_fail(b"alloc", at)
        st = gpu.batch_count(b, kc, km, 2)
        failed = gpu.lib.fake_failed()
        assert st == (gpm.GPM_ENOMEM if failed else gpm.GPM_OK), (at, gpu.error())
        gpu.lib.fake_fail(b"", 0)
        assert gpu.batch_count(b, kc, km, 2) == gpm.GPM_OK, (at, gpu.error())
        gpu.lib.gpm_batch_destroy(b)
        assert gpu.lib.fake_memory_in_use() == before, at
        if not failed:
            break
    assert at > 3 and not failed


@pytest.mark.parametrize("k", [5, 6])
def test_a_smaller_graph_counted_meanwhile_takes_no_shared_memory_away(gpu, k):
    """Between one call's plan and its launch, another (another thread's) counts
    a small graph with the same kernel."""
    n = {5: 9000, 6: 11000}[k]                              # more than 48 KB a block
    big, small = gpu.graph(*_path(n)), gpu.graph(*_path(20))
    seen = []
    meanwhile = ctypes.CFUNCTYPE(None)(lambda: seen.append(gpu.motifs(small, k)))
    gpu.log()
    gpu.lib.fake_on_event_record(ctypes.cast(meanwhile, ctypes.c_void_p))
    assert gpu.motifs(big, k) == gpm.GPM_OK, gpu.error()
    assert seen == [gpm.GPM_OK]
    assert max(x[3] for x in gpu.log()) > 48 * 1024
    for g in (big, small):
        gpu.lib.gpm_graph_destroy(g)

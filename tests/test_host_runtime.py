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
    for agg in (16, 0):
        gpu.configure(warm, batch=True, motif_agg_min=agg)
        assert gpu.batch_count(warm, kc, km, 2) == gpm.GPM_OK, gpu.error()
    gpu.lib.gpm_batch_destroy(warm)
    before = gpu.lib.fake_memory_in_use()
    for at in range(1, 100):
        b = gpu.batch(*_two_paths(20))
        gpu.lib.fake_fail(b"alloc", at)
        st = gpu.batch_count(b, kc, km, 2)
        failed = gpu.lib.fake_failed()
        # (what only the homomorphism counts need is not missed: the walk counts)
        assert st == gpm.GPM_OK or (failed and st == gpm.GPM_ENOMEM), (at, gpu.error())
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


@pytest.mark.parametrize("n,k", [(300, 3), (300, 5), (20000, 3), (20000, 4), (200000, 4)])
def test_motifs_are_counted_without_the_memory_for_the_homomorphism_sums(gpu, n, k):
    """Whichever allocation of the sums' route fails, the walk counts, and what
    the attempt took is given back."""
    warm = gpu.graph(*_path(n))
    for agg in (16, 0):
        gpu.configure(warm, motif_agg_min=agg)
        assert gpu.motifs(warm, k) == gpm.GPM_OK, gpu.error()
    gpu.lib.gpm_graph_destroy(warm)
    walk = gpu.graph(*_path(n))
    gpu.configure(walk, motif_agg_min=0)
    before = gpu.lib.fake_memory_in_use()
    assert gpu.motifs(walk, k) == gpm.GPM_OK, gpu.error()
    walked = gpu.lib.fake_memory_in_use() - before
    gpu.lib.gpm_graph_destroy(walk)
    for at in range(1, 100):
        g = gpu.graph(*_path(n))
        before = gpu.lib.fake_memory_in_use()
        gpu.log()
        gpu.lib.fake_fail(b"cudaMalloc", at)
        assert gpu.motifs(g, k) == gpm.GPM_OK, (at, gpu.error())
        failed = gpu.lib.fake_failed()
        gpu.lib.fake_fail(b"", 0)
        assert failed == any("k_motif" in x[0] for x in gpu.log())
        if failed:
            # (besides the walk's: small scratch only)
            assert gpu.lib.fake_memory_in_use() - before <= walked + 4 * n + 4096
        gpu.lib.gpm_graph_destroy(g)
        if not failed:
            break
    assert at > 1 and not failed


@pytest.mark.parametrize("tail", [dict(clique_cpl=0), dict(clique_cpl=1), dict(clique_cpl=50), dict(clique_tail=2),
                                  dict(clique_tail=3), dict(clique_compact=1), dict(clique_compact=2),
                                  dict(clique_compact3=0), dict(clique_compact3=2), {}])
def test_a_chosen_tail_of_the_clique_walk_is_walked(gpu, tail):
    g = gpu.graph(*_path(30))
    gpu.configure(g, **tail)
    gpu.log()
    assert gpu.cliques(g, 7) == gpm.GPM_OK and gpu.cliques(g, 4, 8) == gpm.GPM_OK, gpu.error()
    assert sum("8k_cliqueE" in x[0] for x in gpu.log()) == (2 if tail else 0)
    gpu.lib.gpm_graph_destroy(g)


@pytest.mark.parametrize("n,k,kernel", [(9000, 5, "5k_homILi5"), (400, 4, "5k_homILi4"), (200000, 3, "11k_edge_sums"),
                                        (9000, 6, "7k_motif")])
def test_launch_shapes_follow_the_configuration(gpu, n, k, kernel):
    """blocks_per_sm bounds every launch over the vertices; warps_per_block is
    the kernel's, where it has a choice."""
    g = gpu.graph(*_path(n))
    for wpb, bps in ((0, 0), (0, 1), (1, 1), (2, 1), (16, 2)):
        gpu.configure(g, warps_per_block=wpb, blocks_per_sm=bps)
        gpu.log()
        assert gpu.motifs(g, k) == gpm.GPM_OK, gpu.error()
        (_, blocks, threads, _), = [x for x in gpu.log() if kernel in x[0]]
        assert blocks <= 152 * (bps or 32)
        if "k_hom" in kernel:
            assert threads <= 128 and (not wpb or threads <= 32 * wpb)
    gpu.lib.gpm_graph_destroy(g)
    b = gpu.batch(*_two_paths(2000))
    for wpb, bps in ((1, 1), (2, 2), (16, 1)):
        gpu.configure(b, batch=True, warps_per_block=wpb, blocks_per_sm=bps)
        gpu.log()
        assert gpu.batch_count(b, 0, 5, 2) == gpm.GPM_OK, gpu.error()
        (_, blocks, threads, _), = [x for x in gpu.log() if "k_homILi5" in x[0]]
        assert blocks <= 152 * bps and threads <= 32 * wpb
    gpu.lib.gpm_batch_destroy(b)


def test_autotune_keeps_the_callers_split_a_candidate(gpu):
    """Every replay takes the same time here, so that the first candidate is
    kept: the caller's split, where roots are split at all."""
    b = gpu.batch(*_two_paths(30))
    gpu.configure(b, batch=True, batch_split=64)
    assert gpu.autotune(b, 6, 4).batch_split == 64
    gpu.lib.gpm_batch_destroy(b)


def test_one_capture_for_settings_that_a_launch_does_not_look_at(gpu):
    """Cliques no larger than the motifs: one homomorphism launch, whatever the
    order, the threshold and the split."""
    b = gpu.batch(*_two_paths(31))
    captures = lambda: gpu.lib.fake_calls(b"cudaGraphInstantiate")
    for cfg in (dict(), dict(batch_split=16), dict(motif_agg_min=4), dict(motif_agg_min=64, batch_split=4),
                dict(warps_per_block=4), dict(warps_per_block=16)):
        gpu.configure(b, batch=True, **cfg)
        assert gpu.batch_count(b, 4, 5, 2) == gpm.GPM_OK, gpu.error()
        assert captures() == 1
    gpu.configure(b, batch=True, batch_split=64)
    before = captures()
    best = gpu.autotune(b, 4, 5)
    # shapes of 2 and 4 warps at 0, 1 and 2 blocks per SM (one is there already), and the walk
    assert captures() - before <= 6
    assert best.batch_split == 1 and best.warps_per_block in (2, 4)
    gpu.lib.gpm_batch_destroy(b)


def test_noalloc_checks_the_longest_list_of_entries_with_a_full_grid(gpu):
    indptr = np.array([0, 2 ** 31 - 2], np.int32)           # (2^31 - 2) + 255 does not fit in 32 bits
    indices, counts = np.zeros(1, np.int32), np.zeros(2, np.uint64)
    gpu.log()
    gpu.lib.gpm_motif_count_noalloc(indptr.ctypes.data, indices.ctypes.data, 1, 3, counts.ctypes.data_as(gpm._u64p), 2, None)
    (_, blocks, threads, _), = [x for x in gpu.log() if "k_validate" in x[0]]
    assert (blocks, threads) == (152 * 8, 256)


def _ring_of_cliques(n, degree):
    """n vertices of the given even degree (a circulant)."""
    steps = np.arange(1, degree // 2 + 1)
    v = np.arange(n)[:, None]
    return np.arange(n + 1) * degree, np.sort(np.c_[(v + steps) % n, (v - steps) % n], axis=1).ravel()


@pytest.mark.parametrize("n,degree,k,hom", [
    (2048, 64, 3, True), (2100, 64, 3, False), (2100, 32, 3, True), (16384, 32, 3, True), (16384, 34, 3, False),
    (3000, 2, 4, True), (3002, 2, 4, False), (3002, 4, 4, True), (12290, 4, 4, False), (12290, 6, 4, True),
    (3000, 2, 5, True), (3002, 2, 5, False), (16384, 4, 5, True), (300, 4, 6, False)])
def test_route_of_a_batchs_motifs(gpu, n, degree, k, hom):
    """Size and average degree choose between the homomorphism launch and the walk."""
    ip, ix = _ring_of_cliques(n, degree)
    b = gpu.batch([0, n], ip, ix)
    gpu.log()
    assert gpu.batch_count(b, 0, k, 1) == gpm.GPM_OK, gpu.error()
    names = [x[0] for x in gpu.log()]
    assert any("5k_hom" in x for x in names) == hom and any("7k_batch" in x for x in names) != hom
    gpu.lib.gpm_batch_destroy(b)


@pytest.mark.parametrize("n,k,hom", [(8192, 3, True), (8194, 3, False), (6144, 4, True), (6146, 4, False), (16384, 5, True)])
def test_route_of_a_graphs_motifs(gpu, n, k, hom):
    g = gpu.graph(*_ring_of_cliques(n, 4))
    gpu.log()
    assert gpu.motifs(g, k) == gpm.GPM_OK, gpu.error()
    names = [x[0] for x in gpu.log()]
    assert any("5k_hom" in x for x in names) == hom and any("11k_edge_sums" in x for x in names) != hom
    gpu.lib.gpm_graph_destroy(g)

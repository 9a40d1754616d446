"""The walks over cliques and sets, which whole-graph calls at the default
settings no longer take, under every setting: over all roots
(gpm_count_roots) and in batches with motifs too large for the homomorphism
counts.  Counts are integers: they equal the oracle's and closed forms."""
from __future__ import annotations

import functools
from math import comb

import numpy as np
import pytest

from oracle import oracle as O
from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


def _by_code(counts, k):
    return {gpm.gpm_motif_pattern(k, p): int(c) for p, c in enumerate(counts) if c}


@functools.lru_cache(maxsize=1)
def _blocks():
    g = G.sbm(600, 60, 0.4, 0.02, 5)
    return g, [O.clique_count(g, k) for k in (4, 6)], O.motif_count(g, 4)


@pytest.mark.parametrize("cfg", [
    dict(), dict(donate=0), dict(donate_min=2, donate_after_us=0), dict(warps_per_block=4),
    dict(warps_per_block=16, blocks_per_sm=1), dict(warps_per_block=1, blocks_per_sm=1), dict(clique_tail=3),
    dict(clique_compact=2), dict(motif_agg_min=0), dict(motif_agg_min=1),
    dict(motif_agg_min=1, donate_min=2, donate_after_us=0), dict(donate=0, motif_agg_min=1)])
def test_settings_over_all_roots(cfg):
    g, cliques, motifs = _blocks()
    dg = gpm.graph_from_csr(g)
    gpm.gpm_set_config(dg, **cfg)
    assert [int(gpm.gpm_count_roots(dg, gpm.GPM_APP_CLIQUE, k)[0][0]) for k in (4, 6)] == cliques
    assert _by_code(gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, 4)[0], 4) == motifs


@pytest.mark.parametrize("compact3", [0, 1, 2])
@pytest.mark.parametrize("cpl", [0, 1, 85])
def test_three_level_clique_tails_over_all_roots(compact3, cpl):
    def count(g, k):
        dg = gpm.graph_from_csr(g)
        gpm.gpm_set_config(dg, clique_compact3=compact3, clique_cpl=cpl, donate_after_us=0, donate_min=2)
        return int(gpm.gpm_count_roots(dg, gpm.GPM_APP_CLIQUE, k)[0][0])

    for n, k in ((40, 8), (70, 8), (97, 7)):
        assert count(G.complete(n), k) == comb(n, k)
    g = G.gnp(90, 0.8, 3)
    want = O.clique_count_bits(g, 8)
    assert [count(g, k) for k in (7, 8)] == [int(want[k]) for k in (7, 8)]


@pytest.mark.parametrize("agg_min", [1, 16])
@pytest.mark.parametrize("k", [3, 4, 5])
def test_motif_tails_over_all_roots(agg_min, k):
    for g in (G.gnp(60, 0.15, 41), G.star(70), G.disjoint_union(G.complete(9), G.path(6)), G.gnp(40, 0.6, 5)):
        dg = gpm.graph_from_csr(g)
        gpm.gpm_set_config(dg, motif_agg_min=agg_min, donate_after_us=0, donate_min=2)
        assert _by_code(gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, k)[0], k) == O.motif_count(g, k)


def test_batch_units_under_every_knob():
    """6-vertex motifs are walked: shapes, thresholds and splits act on units."""
    gs = [G.gnp(n, p, n) for n, p in ((5, 0.5), (17, 0.3), (24, 0.25), (33, 0.15), (40, 0.1))] + [G.empty(3), G.star(25)]
    cliques, motifs = [O.clique_count(g, 4) for g in gs], [O.motif_count(g, 6) for g in gs]
    b = gpm.batch_from_graphs(gs)
    for cfg in (dict(), dict(warps_per_block=2), dict(warps_per_block=1, blocks_per_sm=1),
                dict(warps_per_block=4, motif_agg_min=0), dict(motif_agg_min=1, batch_split=16),
                dict(motif_agg_min=4, batch_split=64), dict(motif_agg_min=64, batch_split=4)):
        gpm.gpm_batch_set_config(b, **cfg)
        c, m = gpm.gpm_batch_count(b, 4, 6)
        assert [int(x) for x in c] == cliques and [_by_code(row, 6) for row in m] == motifs, cfg
    gpm.gpm_batch_autotune(b, 4, 6, reps=1)
    c, m = gpm.gpm_batch_count(b, 4, 6)
    assert [int(x) for x in c] == cliques and [_by_code(row, 6) for row in m] == motifs


def _padded(n):
    parts = [G.gnp(60, 0.5, 2), G.turan(50, 2), G.star(90), G.cycle(40), G.complete(34)]
    return G.disjoint_union(*parts, G.empty(n - sum(p.n for p in parts)))


def _hub(n, d):
    """A vertex of degree d whose neighbours form a path with chords, and isolated vertices."""
    around = np.arange(1, d + 1)
    return G.from_edges(n, np.r_[np.zeros(d, int), around[:-1], around[:-7]], np.r_[around, around[1:], around[7:]])


def _edges(n, m, seed):
    rng = np.random.default_rng(seed)
    return G.from_edges(n, rng.integers(0, n, m), rng.integers(0, n, m))


@pytest.mark.parametrize("make,ks", [
    (lambda: _padded(1 << 14), (3, 4, 5)), (lambda: _padded((1 << 14) + 1), (3, 4, 5)),
    # one warp's arrays just below and just above 220 KB
    (lambda: _hub(1 << 14, 800), (5,)), (lambda: _hub(1 << 14, 820), (5,)),
    # the 16-bit counters of the cycles of four: all of shared memory, and one vertex more
    (lambda: _edges(110 * 1024, 250000, 7), (3, 4)), (lambda: _edges(110 * 1024 + 1, 250000, 8), (3, 4))],
    ids=["n16384", "n16385", "hub800", "hub820", "n112640", "n112641"])
def test_whole_graph_motifs_at_the_routes_limits_equal_the_walk(make, ks):
    dg = gpm.graph_from_csr(make())
    for k in ks:
        assert np.array_equal(gpm.gpm_motif_count(dg, k), gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, k)[0])

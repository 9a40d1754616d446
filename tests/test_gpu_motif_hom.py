"""Whole-graph motif counts of 3 .. 5 vertices from homomorphism counts
(motif_hom.cu): degrees and orders at the edges of the 32-bit rows and of the
eight-lane groups, graphs without triangles, isolated vertices, hubs, the
largest degree the rule takes and the first it does not.  Counts are integers:
they equal the oracle's, and the walk's (motif_agg_min = 0)."""
from __future__ import annotations

from math import comb

import numpy as np
import pytest

from oracle import oracle as O
from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu

GRAPHS = {
    "edgeless": lambda: G.empty(5), "edge": lambda: G.path(2), "path": lambda: G.path(9), "cycle5": lambda: G.cycle(5),
    "petersen": G.petersen, "star33": lambda: G.star(33), "k7": lambda: G.complete(7), "k34": lambda: G.complete(34),
    "bipartite": lambda: G.turan(40, 2), "turan": lambda: G.turan(37, 5), "gnp33": lambda: G.gnp(33, 0.5, 1),
    "gnp66": lambda: G.gnp(66, 0.3, 2), "sparse300": lambda: G.erdos_renyi_m(300, 500, 3),
    "ba": lambda: G.barabasi_albert_batch(1, 350, 350, 5, 5, seed=4)[0],
    "parts": lambda: G.disjoint_union(G.complete(6), G.empty(3), G.star(9), G.cycle(4), G.gnp(20, 0.4, 5)),
}


def _by_code(dg, k):
    return {gpm.gpm_motif_pattern(k, p): int(c) for p, c in enumerate(gpm.gpm_motif_count(dg, k)) if c}


@pytest.mark.parametrize("name", GRAPHS)
@pytest.mark.parametrize("k", [3, 4, 5])
def test_against_the_oracle(name, k):
    g = GRAPHS[name]()
    assert _by_code(gpm.graph_from_csr(g), k) == O.motif_count(g, k)


@pytest.mark.parametrize("name,k", [("sbm", 5), ("sbm", 4), ("rmat", 4), ("rmat", 5)])
def test_against_the_walk(name, k):
    g = G.sbm(500, 100, 0.5, 0.01, 3) if name == "sbm" else G.rmat(10, 8, 0.57, 0.19, 0.19, 6)
    dg = gpm.graph_from_csr(g)
    ours = gpm.gpm_motif_count(dg, k)
    assert np.array_equal(ours, gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, k)[0])
    gpm.gpm_set_config(dg, motif_agg_min=0)
    assert np.array_equal(ours, gpm.gpm_motif_count(dg, k))


@pytest.mark.parametrize("leaves", [1023, 1024, 1025])
def test_degree_limit(leaves):
    """A star with one edge between two leaves, on both sides of the limit."""
    g = G.from_edges(leaves + 1, np.r_[np.zeros(leaves, int), 1], np.r_[np.arange(1, leaves + 1), 2])
    dg = gpm.graph_from_csr(g)
    for k in (3, 4, 5):
        got = _by_code(dg, k)
        assert sum(got.values()) == comb(leaves, k - 1) and len(got) == 2
        assert max(got.values()) == comb(leaves, k - 1) - comb(leaves - 2, k - 3)


def _random_edges(n, m, seed):
    rng = np.random.default_rng(seed)
    return G.from_edges(n, rng.integers(0, n, m), rng.integers(0, n, m))


SPARSE = {
    "rmat15": lambda: G.rmat(15, 8, 0.57, 0.19, 0.19, 3),
    "rmat15_any_order": lambda: G.relabel(G.rmat(15, 4, 0.57, 0.19, 0.19, 4), np.random.default_rng(1).permutation(1 << 15)),
    "hub": lambda: G.disjoint_union(G.star(1500), G.gnp(60, 0.5, 2), G.turan(50, 2), G.empty(7)),
    "above_16_bit_ids": lambda: _random_edges(70001, 200000, 5),
    "global_counters": lambda: G.disjoint_union(_random_edges(115001, 250000, 6), G.complete(40), G.turan(90, 3)),
}


@pytest.mark.parametrize("name", SPARSE)
@pytest.mark.parametrize("k", [3, 4])
def test_larger_graphs_against_the_walk(name, k):
    """Graphs beyond the per-vertex arrays (motif_sparse.cu)."""
    g = SPARSE[name]()
    dg = gpm.graph_from_csr(g)
    ours = gpm.gpm_motif_count(dg, k)
    assert gpm.gpm_get_stats(dg)["kernel_launches"] >= 2
    assert np.array_equal(ours, gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, k)[0])
    gpm.gpm_set_config(dg, motif_agg_min=0)
    assert np.array_equal(ours, gpm.gpm_motif_count(dg, k))


@pytest.mark.parametrize("kc,km", [(3, 3), (3, 5), (4, 4), (4, 5), (5, 5), (5, 4), (6, 5)])
def test_batched_cliques_from_the_same_sums(kc, km):
    """Cliques no larger than the motifs share their sums; the others, and the
    walk's form of the call, keep units of their own."""
    gs = [make() for make in GRAPHS.values()] + [G.empty(0), G.empty(1), G.complete(40)]
    b = gpm.batch_from_graphs(gs)
    cliques, motifs = gpm.gpm_batch_count(b, kc, km)
    assert [int(c) for c in cliques] == [O.clique_count(g, kc) for g in gs]
    gpm.gpm_batch_set_config(b, motif_agg_min=0)
    walked = gpm.gpm_batch_count(b, kc, km)
    assert np.array_equal(cliques, walked[0]) and np.array_equal(motifs, walked[1])

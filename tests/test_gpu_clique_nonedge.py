"""Whole-graph clique counts by branching on non-edges (clique_nonedge.cu):
sets at the edges of the row words and of the re-indexed universe, members
without non-edges, disjoint non-edges, dense and sparse complements, every
number of sizes to go.  Counts are integers: they equal the closed form or the
oracle's bitset route, and the walk that visits the cliques (clique_cpl = 0)."""
from __future__ import annotations

from math import comb

import numpy as np
import pytest

from oracle import oracle as O
from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu

RANGES = [(3, 3), (3, 4), (4, 4), (3, 5), (5, 5), (4, 6), (6, 6), (5, 7), (7, 8)]


def _cocktail(pairs):
    """Every vertex misses exactly one other: 2^k C(pairs, k) k-cliques."""
    return G.turan(2 * pairs, pairs)


def _elem_sym(parts, k):
    e = [1] + [0] * k
    for s in parts:
        for j in range(k, 0, -1):
            e[j] += s * e[j - 1]
    return e[k]


@pytest.mark.parametrize("pairs", [2, 16, 17, 33, 65, 129, 200])
def test_disjoint_non_edges(pairs):
    dg = gpm.graph_from_csr(_cocktail(pairs))
    for lo, hi in RANGES + [(9, 9), (9, 11)]:
        want = [2 ** k * comb(pairs, k) for k in range(lo, hi + 1)]
        if max(want) >= 2 ** 64:
            continue
        assert gpm.gpm_clique_count_range(dg, lo, hi) == want, (lo, hi)


@pytest.mark.parametrize("n,r", [(33, 3), (66, 33), (97, 7), (130, 2), (260, 4), (300, 12), (700, 3)])
def test_complete_multipartite(n, r):
    g = G.turan(n, r)
    parts = np.bincount(np.arange(n) % r).tolist()
    dg = gpm.graph_from_csr(g)
    for lo, hi in RANGES:
        assert gpm.gpm_clique_count_range(dg, lo, hi) == [_elem_sym(parts, k) for k in range(lo, hi + 1)], (lo, hi)


@pytest.mark.parametrize("n,p,hi", [(33, 0.5, 9), (34, 0.97, 8), (65, 0.3, 7), (66, 0.9, 7), (100, 0.95, 6),
                                    (140, 0.6, 7), (200, 0.2, 7), (320, 0.12, 6), (300, 0.6, 6), (160, 0.9, 5)])
def test_random_graphs_against_the_oracle(n, p, hi):
    g = G.gnp(n, p, 7 * n)
    want = O.clique_count_bits(g, hi)
    dg = gpm.graph_from_csr(g)
    for lo, up in [(lo, up) for lo, up in RANGES + [(8, 9)] if up <= hi]:
        assert gpm.gpm_clique_count_range(dg, lo, up) == [int(want[k]) for k in range(lo, up + 1)], (lo, up)
    ref = gpm.gpm_clique_count_range(dg, 3, hi)
    gpm.gpm_set_config(dg, clique_cpl=0)
    assert gpm.gpm_clique_count_range(dg, 3, hi) == ref


def test_complete_graphs_up_to_the_last_bit():
    dg = gpm.graph_from_csr(G.complete(100))
    assert gpm.gpm_clique_count_range(dg, 13, 16) == [comb(100, k) for k in range(13, 17)]
    assert comb(150, 16) >= 2 ** 64 > comb(150, 10)
    dg = gpm.graph_from_csr(G.complete(150))
    with pytest.raises(gpm.GpmError) as e:
        gpm.gpm_clique_count(dg, 16)
    assert e.value.status == gpm.GPM_EOVERFLOW
    assert gpm.gpm_clique_count(dg, 10) == comb(150, 10)

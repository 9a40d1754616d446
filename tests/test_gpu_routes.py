"""Batches on both sides of the rule that chooses the homomorphism launch or the
walk: every graph's motifs equal those of the graph alone, and the walk's."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


def _edges(n, m, seed):
    rng = np.random.default_rng(seed)
    return G.from_edges(n, rng.integers(0, n, m), rng.integers(0, n, m))


@pytest.mark.parametrize("make", [
    lambda: [_edges(2000, 40000, 1), _edges(1999, 60000, 2)], lambda: [_edges(2100, 40000, 3), _edges(50, 300, 4)],
    lambda: [G.path(3000), G.cycle(7)], lambda: [G.path(3001), G.cycle(8), _edges(60, 200, 5)],
    lambda: [_edges(12400, 24000, 6), G.star(40)], lambda: [_edges(12400, 40000, 7), G.empty(1)],
    lambda: [_edges(16384, 30000, 8), G.complete(12), G.empty(0)]],
    ids=["n2000", "n2100", "path3000", "path3001", "n12400sparse", "n12400", "n16384"])
def test_batches_on_both_sides_of_the_route(make):
    gs = make()
    b = gpm.batch_from_graphs(gs)
    for k in (3, 4, 5):
        _, motifs = gpm.gpm_batch_count(b, 0, k)
        for row, g in zip(motifs, gs):
            dg = gpm.graph_from_csr(g)
            assert np.array_equal(row, gpm.gpm_count_roots(dg, gpm.GPM_APP_MOTIF, k)[0]), (g.n, k)
            assert np.array_equal(row, gpm.gpm_motif_count(dg, k)), (g.n, k)

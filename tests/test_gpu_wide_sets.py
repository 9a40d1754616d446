"""Clique counts whose candidate sets have hundreds of members with non-edges."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


def _partite(n, parts, p, seed):
    """A complete multipartite graph with every edge kept with probability p."""
    rng = np.random.default_rng(seed)
    u, v = np.triu_indices(n, 1)
    keep = (u % parts != v % parts) & (rng.random(u.size) < p)
    return G.from_edges(n, u[keep], v[keep])


@pytest.mark.parametrize("make", [
    lambda: G.turan(330, 3), lambda: G.turan(240, 3), lambda: G.turan(420, 60), lambda: G.turan(450, 90), lambda: G.gnp(320, 0.85, 4),
    lambda: G.gnp(260, 0.97, 5), lambda: _partite(450, 5, 0.8, 6)],
    ids=["turan330_3", "turan240_3", "turan420_60", "turan450_90", "gnp320", "gnp260", "partite450"])
def test_wide_candidate_sets_against_the_walk(make):
    """Sets of more than 160 members with non-edges and three sizes to go, on both
    sides of the rule that counts their triangles directly."""
    dg = gpm.graph_from_csr(make())
    ranges = [(5, 5), (3, 5), (6, 6)]
    got = [gpm.gpm_clique_count_range(dg, lo, hi) for lo, hi in ranges]
    gpm.gpm_set_config(dg, clique_cpl=0)
    assert got == [gpm.gpm_clique_count_range(dg, lo, hi) for lo, hi in ranges]

"""Core numbers (root feature 6) against a sequential peeling, where the
launch's forms meet: one removed vertex per round up to more than there are
threads, lists at and above a block's width, one cluster and the whole grid."""
import numpy as np
import pytest

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


def peel(g):
    """Core numbers by removing a vertex of the smallest remaining degree at a time."""
    deg = np.diff(g.indptr).astype(int).tolist()
    indptr, indices = g.indptr.tolist(), g.indices.tolist()
    buckets = [[] for _ in range(max(deg, default=0) + 1)]
    for v, d in enumerate(deg):
        buckets[d].append(v)
    core = [-1] * g.n
    c = d = 0
    while d < len(buckets):
        if not buckets[d]:
            d += 1
            continue
        v = buckets[d].pop()
        if core[v] >= 0 or deg[v] != d:
            continue
        c = max(c, d)
        core[v] = c
        for u in indices[indptr[v]:indptr[v + 1]]:
            if core[u] < 0:
                deg[u] -= 1
                buckets[deg[u]].append(u)
        d = max(d - 1, 0)
    return np.array(core)


@pytest.mark.parametrize("name", ["one", "edgeless", "star", "path", "hub_lists", "rmat12", "cluster_edge", "grid"])
def test_core_numbers(name):
    g = {
        "one": lambda: G.complete(1),
        "edgeless": lambda: G.erdos_renyi_m(5000, 0, 1),
        "star": lambda: G.star(4200),                                # a round of more than 4,096 vertices
        "path": lambda: G.path(3000),                                # 1,500 rounds of two
        "hub_lists": lambda: G.disjoint_union(*(G.complete(d + 1) for d in (7, 8, 31, 32, 127, 511, 512, 513))),
        "rmat12": lambda: G.rmat(12, 8, 0.57, 0.19, 0.19, 5),
        "cluster_edge": lambda: G.disjoint_union(G.complete(40), G.erdos_renyi_m((1 << 17) - 40, 300000, 2)),
        "grid": lambda: G.disjoint_union(G.complete(40), G.star(600), G.erdos_renyi_m(1 << 17, 300000, 3)),
    }[name]()
    f = gpm.gpm_root_features(gpm.graph_from_csr(g), 4)
    assert np.array_equal(np.rint(np.expm1(f[:, 6].astype(np.float64))).astype(int), peel(g))

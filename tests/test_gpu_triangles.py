"""Triangles rooted at a vertex, by the length of its list."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [255, 257, 258, 600, 1024, 1025, 1026, 1100])
def test_triangles_of_a_root_by_list_length(n):
    """Root feature 5 on K_n: the vertex with d later ones has C(d, 2) triangles,
    d = n - 1, n - 2, ..; log1p in fp32 is within a few units of its last place."""
    f = gpm.gpm_root_features(gpm.graph_from_csr(G.complete(n)), 4)
    d = np.arange(n - 1, -1, -1, dtype=np.float64)
    assert np.abs(np.sort(f[:, 5].astype(np.float64))[::-1] - np.log1p(d * (d - 1) / 2)).max() <= 1e-5

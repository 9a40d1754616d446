"""Statistics of calls that make several launches, and the launch shapes of
the whole-graph counts."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2212_04551_gb300 import gpm
from paper_2212_04551_gb300 import graphs as G

pytestmark = pytest.mark.gpu


def _bicliques(parts, side):
    return G.disjoint_union(*[G.turan(2 * side, 2)] * parts)


def _communities(count):
    """Out-degrees on both sides of 32: a heavy and a light launch of comparable length."""
    return G.disjoint_union(*[G.gnp(90, 0.6, s) for s in range(count)], *[G.gnp(30, 0.6, s) for s in range(count * 10)])


def _one_heavy():
    """A single root above 32 out-neighbours: the first launch has one block."""
    return G.disjoint_union(G.complete(34), *[G.gnp(30, 0.6, s) for s in range(2500)])


@pytest.mark.parametrize("graph,call", [
    (_one_heavy, lambda g: gpm.gpm_clique_count(g, 4)),
    (_one_heavy, lambda g: gpm.gpm_motif_count(g, 4)),
    (lambda: _bicliques(12, 700), lambda g: gpm.gpm_motif_count(g, 4)),         # the cycles of four take the time
    (lambda: _communities(200), lambda g: gpm.gpm_clique_count(g, 4)),
    (lambda: _communities(200), lambda g: gpm.gpm_clique_count_range(g, 3, 8))])
def test_busy_time_of_several_launches(graph, call):
    """All launches hand out their work by tickets and none waits: the slots
    are busy for most of the time and (but for the timer's steps) never for
    more than all of it."""
    dg = gpm.graph_from_csr(graph())
    for _ in range(3):
        call(dg)
    st = gpm.gpm_get_stats(dg)
    slots = st["grid_blocks"] * st["warps_per_block"] * st["kernel_ms"] * 1e6
    assert st["kernel_launches"] >= 2
    assert 0.3 * slots <= st["busy_warp_ns"] <= 1.02 * slots


def test_busy_time_of_a_batch():
    """Clique units and the homomorphism launch in one call."""
    b = gpm.batch_from_graphs([G.gnp(90, 0.3, s) for s in range(800)])
    for _ in range(3):
        gpm.gpm_batch_count(b, 6, 4)
    st = gpm.gpm_batch_get_stats(b)
    slots = st["grid_blocks"] * st["warps_per_block"] * st["kernel_ms"] * 1e6
    assert 0.3 * slots <= st["busy_warp_ns"] <= 1.02 * slots


def test_blocks_per_sm_bounds_the_clique_launches():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    a = 400
    i = np.arange(a * a).reshape(a, a)
    light = G.from_edges(a * a, np.r_[i[:, :-1].ravel(), i[:-1].ravel()], np.r_[i[:, 1:].ravel(), i[1:].ravel()])
    for g in (light, _communities(60)):
        dg = gpm.graph_from_csr(g)
        want = gpm.gpm_clique_count(dg, 3)
        for bps in (1, 2):
            gpm.gpm_set_config(dg, blocks_per_sm=bps)
            assert gpm.gpm_clique_count(dg, 3) == want
            assert gpm.gpm_get_stats(dg)["grid_blocks"] <= bps * sms

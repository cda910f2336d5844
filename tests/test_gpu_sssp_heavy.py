"""SSSP's plain offsets where they come from the heavy-vertex schedule: in
degree order the tiles of 512 labels that hold none but heavy vertices are
filled from it.  511 to 1,024 heavy vertices, with nothing after them (the last
offset then belongs to no tile) or with light vertices.  Distances equal
Dijkstra's.
"""
import numpy as np
import pytest

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


def graph(heavy, light):
    """`heavy` vertices, all joined to one another, then a chain of `light` ones."""
    u, v = np.triu_indices(heavy, 1)
    chain = np.arange(heavy - 1, heavy + light - 1)
    edges = np.r_[np.stack([u, v], 1), np.stack([chain, chain + 1], 1)]
    labels = np.random.default_rng(heavy + light).permutation(heavy + light)
    return gen.from_edges(heavy + light, labels[edges], weighted=True, seed=heavy)


@pytest.mark.parametrize("off_mode", [lg.LG_OFF_PACKED, lg.LG_OFF_EF])
@pytest.mark.parametrize("light", [0, 1, 700])
@pytest.mark.parametrize("heavy", [511, 512, 513, 1024])
def test_distances(heavy, light, off_mode):
    lg.load(auto_build=True)
    h = graph(heavy, light)
    n = heavy + light
    g = lg.lg_encode(h.row_ptr, h.col, h.weights, off_mode=off_mode, relabel=lg.LG_RELABEL_DM)
    for s in (0, n // 2, n - 1):
        want = oracle.sssp(n, h.row_ptr, h.col, h.weights, s)
        assert np.array_equal(lg.lg_sssp(g, s).cpu().numpy().view(np.uint64), want), s


@pytest.mark.parametrize("id_mode", [lg.LG_ID_GLOBAL, lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("heavy, light", [(512, 0), (1024, 0), (1024, 700), (1500, 1)])
def test_ranks(heavy, light, id_mode):
    """PageRank's first contributions come from the schedule in the same way,
    by more blocks than there are tiles left."""
    lg.load(auto_build=True)
    h = graph(heavy, light)
    g = lg.lg_encode(h.row_ptr, h.col, id_mode=id_mode, off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM)
    want = oracle.pagerank(heavy + light, h.row_ptr, h.col, 0.85, 5)
    got = lg.lg_pagerank(g, 0.85, 5).cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-4

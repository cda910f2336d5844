"""Tiles of the degree-ordered vertices of more than 32 arcs in bottom-up BFS
and personalized PageRank: 64 vertices on a small or skewed graph, up to 512 on
one of even degrees.  Depths equal a plain search's.
"""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


def even(n, half):
    rng = np.random.default_rng(n)
    u = np.repeat(np.arange(n), half)
    return gen.from_edges(n, np.stack([u, rng.integers(0, n, n * half)], 1))


# tiles of 64, 128, 256 and 512 vertices; 100,001 and 200,003 end in a part of one
@pytest.mark.parametrize("n, half", [(20000, 20), (100001, 40), (200003, 60), (400000, 100)])
@pytest.mark.parametrize("id_mode", [lg.LG_ID_GLOBAL, lg.LG_ID_LOCAL_GAP])
def test_depths(n, half, id_mode):
    lg.load(auto_build=True)
    h = even(n, half)
    g = lg.lg_encode(h.row_ptr, h.col, id_mode=id_mode, off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM)
    sources = np.array([0, n // 3, n - 1], dtype=np.uint32)
    got = lg.lg_bfs(g, torch.from_numpy(sources.view(np.int32)).cuda()).cpu().numpy().view(np.uint32)
    for d, s in zip(got, sources):
        assert np.array_equal(d, oracle.bfs(n, h.row_ptr, h.col, int(s)))
    got = lg.lg_pagerank(g, 0.85, 2, personalize=5).cpu().numpy()
    want = oracle.pagerank(n, h.row_ptr, h.col, 0.85, 2, personalize=5)
    assert np.all(np.abs(got - want) <= 1e-4 * want)

"""SSSP's relaxation windows of 256 arc slots at their edges: hubs over many
windows, windows of nothing but single arcs, vertices that begin exactly at a
window's start, vertices without outgoing arcs in between, queues of more than
2,048 vertices, more than 64 rounds.  Distances equal Dijkstra's.
"""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


def directed(n, u, v):
    key = np.unique(u.astype(np.uint64) * np.uint64(n) + v.astype(np.uint64))
    rp = np.searchsorted(key, np.arange(n + 1, dtype=np.uint64) * np.uint64(n)).astype(np.uint64)
    col = (key % np.uint64(n)).astype(np.uint32)
    return rp, col, (col * 37 % 200 + 1).astype(np.uint32)


def graphs():
    rng = np.random.default_rng(6)
    n = 6000
    # levels 0 -> 1..255 or 256 -> the rest, half of which have no outgoing arcs
    for first in (255, 256, 257):
        u = np.r_[np.zeros(first, np.int64), np.repeat(np.arange(1, first + 1), 40)]
        v = np.r_[np.arange(1, first + 1), rng.integers(first + 1, n, 40 * first)]
        more = rng.integers(first + 1, n, 3000)
        yield directed(n, np.r_[u, more[more % 2 == 0]], np.r_[v, rng.integers(0, n, int((more % 2 == 0).sum()))])
    # every window exactly one vertex: degree 256
    m = 300
    yield directed(m, np.repeat(np.arange(m), 256), (np.repeat(np.arange(m), 256) + 1 + np.tile(np.arange(256), m)) % m)
    h = gen.from_edges(30000, np.r_[np.stack([np.zeros(29999, np.int64), np.arange(1, 30000)], 1),
                                    rng.integers(0, 30000, (20000, 2))], weighted=True, seed=3)
    yield h.row_ptr, h.col, h.weights
    h = gen.from_edges(1500, [(i, i + 1) for i in range(1499)], weighted=True, seed=4)  # 1,499 rounds
    yield h.row_ptr, h.col, h.weights


@pytest.mark.parametrize("case", range(6))
@pytest.mark.parametrize("opts", [dict(id_mode=lg.LG_ID_GLOBAL, off_mode=lg.LG_OFF_EF, relabel=True),
                                  dict(id_mode=lg.LG_ID_GLOBAL, off_mode=lg.LG_OFF_PACKED),
                                  dict(id_mode=lg.LG_ID_CSR32)])
def test_distances(case, opts):
    lg.load(auto_build=True)
    rp, col, w = list(graphs())[case]
    g = lg.lg_encode(rp, col, w, **opts)
    for s in (0, 1, rp.size - 2):
        want = oracle.sssp(rp.size - 1, rp, col, w, s)
        for delta in (0, 1, 7, 1 << 20):
            got = lg.lg_sssp(g, s, delta).cpu().numpy().view(np.uint64)
            assert np.array_equal(got, want), (s, delta)

"""The two paths of a batch run at their edges: graphs of up to 65,536 vertices
keep their state in shared memory (one CTA that fits twice, one that does not,
teams; tables that cover the graph or a part of it), larger ones do not.
Checked against the oracle graph by graph.
"""
import numpy as np
import pytest
import torch

import gen
import paper_2010_15879_gb300 as lg
from test_gpu_batch import concat, create, host_batch_arrays, run_and_check

pytestmark = pytest.mark.gpu


def graph(n, m, seed, hubs=()):
    rng = np.random.default_rng(seed)
    e = rng.integers(0, n, (m, 2))
    for h, d in hubs:
        e = np.concatenate([e, np.stack([np.full(d, h), rng.permutation(n)[:d]], 1)])
    return gen.from_edges(n, e)


@pytest.fixture(scope="module")
def edges():
    lg.load(auto_build=True)
    graphs = [graph(n, 6 * n, n) for n in (2, 31, 32, 33, 63, 64, 65, 127, 257)]
    graphs += [
        graph(20000, 60000, 1, [(0, 300), (5, 15000)]),   # fits the table twice; a hub over many windows
        graph(23000, 400000, 2),
        graph(45000, 90000, 3, [(7, 256), (8, 257)]),     # fits, or is larger than the table by a part
        graph(65535, 200000, 4),
        graph(65536, 500000, 5, [(65535, 40000)]),        # 16-bit IDs, the largest of the path
        graph(65537, 200000, 6, [(1, 9000)]),             # 17-bit IDs: the other path
        graph(90000, 300000, 7),
        gen.from_edges(3000, [(i, i + 1) for i in range(2999)]),  # 2,999 levels
    ]
    return host_batch_arrays(concat(graphs))


@pytest.mark.parametrize("tile", [1 << 22, 1 << 17, 1 << 12])
@pytest.mark.parametrize("lanes", [1, 8, 32])
def test_paths(edges, tile, lanes):
    b = create(edges, autotune=False, lanes=lanes, tile_arcs=tile)
    assert (b.info()["max_team"] > 1) == (tile < 1 << 22)
    run_and_check(b, edges)
    b.free()


def test_paths_autotuned_and_repeated(edges):
    b = create(edges, autotune=True)
    d1, r1 = lg.lg_batch_run(b, 0.85, 3)
    d1, r1 = d1.clone(), r1.clone()
    d2, r2 = lg.lg_batch_run(b, 0.85, 3)
    lg.lg_batch_status(b)
    assert torch.equal(d1, d2) and torch.equal(r1, r2)
    run_and_check(b, edges, iters=3)
    b.free()

"""PageRank sweeps of graphs without degrees far above the mean: tiles of 4 to
128 vertices by the graph's size, heavy items after them, several to a ticket
where there are many.  Ranks against the FP64 oracle, and the same bits from
run to run.
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


def check(h, n, iters=3, **opts):
    g = lg.lg_encode(h.row_ptr, h.col, **opts)
    got = lg.lg_pagerank(g, 0.85, iters)
    assert torch.equal(got, lg.lg_pagerank(g, 0.85, iters))
    want = oracle.pagerank(n, h.row_ptr, h.col, 0.85, iters)
    assert np.max(np.abs(got.cpu().numpy() - want) / want) <= 1e-4
    if n <= 1 << 20:
        out = torch.empty(n, device="cuda")
        assert torch.equal(got, lg.lg_pagerank_noalloc(g, 0.85, iters, out))


MODES = [dict(), dict(id_mode=lg.LG_ID_LOCAL_GAP, off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM),
         dict(id_mode=lg.LG_ID_LOCAL, relabel=lg.LG_RELABEL_DM)]


@pytest.mark.parametrize("n", [100, 7297, 14593, 29185, 58369, 116737, 233473, 300001])
@pytest.mark.parametrize("opts", MODES)
def test_tiles(n, opts):
    lg.load(auto_build=True)
    check(even(n, 12), n, **opts)


# every vertex an item or two, a part of them, and next to none
@pytest.mark.parametrize("heavy_min, seg", [("4", "4096"), ("12", "32"), ("24", "4096"), ("30", "32")])
@pytest.mark.parametrize("opts", MODES)
def test_tickets(monkeypatch, heavy_min, seg, opts):
    lg.load(auto_build=True)
    monkeypatch.setenv("LG_HEAVY_MIN", heavy_min)
    monkeypatch.setenv("LG_HEAVY_SEG", seg)
    check(even(200003, 12), 200003, **opts)


# tiles start right after the vertices that are all in the schedule
@pytest.mark.parametrize("hubs", [1, 10, 127, 128, 129, 200])
@pytest.mark.parametrize("opts", MODES + [dict(off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM)])
def test_hubs(hubs, opts):
    lg.load(auto_build=True)
    n, rng = 50001, np.random.default_rng(hubs)
    e = [np.stack([np.full(3000, v), rng.integers(0, n, 3000)], 1) for v in range(hubs)]
    h = gen.from_edges(n, np.concatenate(e + [rng.integers(0, n, (n, 2))]))
    check(h, n, **opts)

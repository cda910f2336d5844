"""Rows of neighbor lookups at the sizes where their sort changes (1, 2, 4 and 8
keys a lane, the CTA's network, the caller's sort), with and without weights,
one to eight queries per CTA.  Offsets, IDs and weights equal the input rows.
"""
import numpy as np
import pytest
import torch

import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu

SIZES = [0, 1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 160, 255, 256, 257, 511, 512, 513, 2000, 4095, 4096, 4097, 5000]
N = 40000


def rows(seed):
    """Row v of the first vertices has SIZES[v] neighbors, the others at most 40;
    directed, spread over all labels."""
    rng = np.random.default_rng(seed)
    d = rng.integers(0, 41, N)
    at = rng.permutation(N)[:6 * len(SIZES)]
    d[at] = SIZES * 6
    rp = np.zeros(N + 1, dtype=np.int64)
    np.cumsum(d, out=rp[1:])
    col = np.concatenate([np.sort(rng.choice(N, k, replace=False)) for k in d]).astype(np.int32)
    w = rng.integers(0, 256, col.size).astype(np.int32)
    return rp, col, w, at


@pytest.fixture(scope="module")
def graph():
    lg.load(auto_build=True)
    return rows(3)


@pytest.mark.parametrize("k", [1, 150, 607, 1300, 5000])
@pytest.mark.parametrize("relabel", [lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM, lg.LG_RELABEL_GREEDY])
@pytest.mark.parametrize("ids, weighted", [(lg.LG_ID_GLOBAL, True), (lg.LG_ID_GLOBAL, False), (lg.LG_ID_LOCAL, False),
                                           (lg.LG_ID_LOCAL_GAP, False), (lg.LG_ID_CSR32, True)])
def test_rows(graph, k, relabel, ids, weighted):
    rp, col, w, at = graph
    g = lg.lg_encode(rp, col, w if weighted else None, id_mode=ids, off_mode=lg.LG_OFF_EF, relabel=relabel)
    rng = np.random.default_rng(k)
    q = np.r_[rng.permutation(at)[:k], rng.integers(0, N, max(0, k - at.size))].astype(np.int32)
    got = lg.lg_neighbors(g, torch.from_numpy(q).cuda(), with_weights=weighted)
    off = np.concatenate([[0], np.cumsum(rp[q + 1] - rp[q])])
    src = np.concatenate([np.arange(rp[v], rp[v + 1]) for v in q])
    assert np.array_equal(got[0].cpu().numpy(), off)
    assert np.array_equal(got[1].cpu().numpy(), col[src])
    if weighted:
        assert np.array_equal(got[2].cpu().numpy(), w[src])


@pytest.mark.parametrize("n", [1 << 24, (1 << 24) + 1])
def test_weights_of_large_ids(n):
    """Up to 2^24 vertices an ID shares its word with the field of its weight."""
    lg.load(auto_build=True)
    rng = np.random.default_rng(n)
    d = np.zeros(n, dtype=np.int64)
    at = np.r_[0, n - 1, rng.integers(1, n - 1, 60)]
    d[at] = np.resize([1, 32, 33, 64, 100, 128, 200, 255, 256], at.size)
    at = np.flatnonzero(d)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(d, out=rp[1:])
    # every row ends at the largest ID
    col = np.concatenate([np.r_[np.sort(rng.choice(n - 1, d[v] - 1, replace=False)), n - 1] for v in at]).astype(np.int32)
    w = rng.integers(0, 256, col.size).astype(np.int32)
    g = lg.lg_encode(rp, col, w, off_mode=lg.LG_OFF_PACKED, relabel=lg.LG_RELABEL_DM)
    got = lg.lg_neighbors(g, torch.from_numpy(at.astype(np.int32)).cuda(), with_weights=True)
    assert np.array_equal(got[1].cpu().numpy(), col) and np.array_equal(got[2].cpu().numpy(), w)


@pytest.mark.parametrize("k", [1, 608, 609, 2000, 5000])
def test_long_rows(k):
    """Rows of 257 and more on the average: one to eight queries per CTA."""
    lg.load(auto_build=True)
    n, rng = 3000, np.random.default_rng(4)
    d = rng.integers(200, 500, n)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(d, out=rp[1:])
    col = np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in d]).astype(np.int32)
    w = rng.integers(0, 256, col.size).astype(np.int32)
    g = lg.lg_encode(rp, col, w, off_mode=lg.LG_OFF_EF, relabel=lg.LG_RELABEL_DM)
    q = rng.integers(0, n, k).astype(np.int32)
    got = lg.lg_neighbors(g, torch.from_numpy(q).cuda(), with_weights=True)
    src = np.concatenate([np.arange(rp[v], rp[v + 1]) for v in q])
    assert np.array_equal(got[1].cpu().numpy(), col[src]) and np.array_equal(got[2].cpu().numpy(), w[src])

"""PageRank's warp tiles at the sizes where they can go wrong: tile edges,
degrees around the light limit, heavy vertices between light ones (which break
the run of stream bits), neighborhoods that cross windows of 256 fields, records
wider than 40 bits (half windows), every tile size, and the shared-memory table
on and off.  Reference: the same sums in 64 bits (torch).
"""
import numpy as np
import pytest
import torch

import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu

DAMPING, ITERS = 0.85, 3
# A sweep adds a vertex's FP32 terms in at most 8 (lane) + 5 (scan) + 17 (windows
# of a light vertex; Kahan and a tree for heavy ones) roundings of 2^-24, plus a
# division, a product and a sum: under 40 * 2^-24 = 2.4e-6 a sweep, all terms >= 0.
RTOL = ITERS * 2.4e-6
MODES = [(i, o, r) for i in (lg.LG_ID_GLOBAL, lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP, lg.LG_ID_CSR32)
         for o in (lg.LG_OFF_PACKED, lg.LG_OFF_EF) for r in (lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM)]


def csr(n, u, v):
    keep = u != v
    u, v = u[keep].long(), v[keep].long()
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    rp = torch.searchsorted(key, torch.arange(n + 1, device=key.device) * n)
    return rp, (key % n).int()


def ranks64(rp, col, source=None):
    n = rp.numel() - 1
    deg = (rp[1:] - rp[:-1]).double()
    inv = torch.where(deg > 0, 1 / deg.clamp(min=1), 0 * deg)
    row = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
    base = torch.zeros(n, dtype=torch.float64, device=rp.device)
    if source is None:
        base += 1 / n
    else:
        base[source] = 1
    r = base
    for _ in range(ITERS):
        r = (1 - DAMPING) * base + DAMPING * torch.zeros_like(r).index_add_(0, row, (r * inv)[col.long()])
    return r


def check(rp, col, w=None, source=None, **opts):
    g = lg.lg_encode(rp, col, w, **opts)
    got = lg.lg_pagerank(g, DAMPING, ITERS, personalize=source).double()
    want = ranks64(rp, col, source)
    assert torch.all((got - want).abs() <= RTOL * want), float(((got - want).abs() / want.clamp(min=1e-30)).max())
    again = lg.lg_pagerank(g, DAMPING, ITERS, personalize=source).double()
    assert torch.equal(got, again)
    return g


def random_edges(n, m, seed):
    rng = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randint(n, (m,), generator=rng, device="cuda"), torch.randint(n, (m,), generator=rng, device="cuda"))


@pytest.mark.parametrize("ids,off,relabel", MODES)
def test_tile_edges(ids, off, relabel):
    for n in (2, 3, 4, 5, 31, 33, 127, 128, 129, 511, 513, 1000):
        rp, col = csr(n, *random_edges(n, 5 * n, n))
        check(rp, col, id_mode=ids, off_mode=off, relabel=relabel, source=n // 2 if n % 2 else None)


@pytest.mark.parametrize("ids,off,relabel", MODES)
def test_heavy_between_light(ids, off, relabel):
    # hubs of 255, 256, 257, 512, 4096, 4097 and 9000 arcs among vertices of few, some adjacent to each other
    n, hubs = 20000, {100: 255, 101: 256, 102: 257, 127: 512, 128: 4096, 129: 4097, 5000: 9000, 5001: 300, 19999: 257}
    u, v = random_edges(n, 2 * n, 7)
    rng = torch.Generator(device="cuda").manual_seed(9)
    for h, d in hubs.items():
        u = torch.cat([u, torch.full((d,), h, device="cuda")])
        v = torch.cat([v, torch.randperm(n, generator=rng, device="cuda")[:d]])
    rp, col = csr(n, u, v)
    check(rp, col, id_mode=ids, off_mode=off, relabel=relabel, select_sample=4096 if off else 512)


@pytest.mark.parametrize("bits", [1, 12, 13, 24, 25, 26, 32])
def test_wide_records(bits):
    # 15-bit IDs: records of 16 .. 47 bits, windows of 256 fields up to 40 bits, 128 above
    n = 30000
    rp, col = csr(n, *random_edges(n, 30 * n, 3))
    w = (col & ((1 << min(bits, 31)) - 1)).clamp(min=1).int()
    for relabel in (lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM):
        check(rp, col, w, id_mode=lg.LG_ID_GLOBAL, off_mode=lg.LG_OFF_EF, weight_bits=bits, relabel=relabel)


@pytest.mark.parametrize("ids,off,relabel", MODES)
def test_large_tiles(ids, off, relabel):
    # tiles of 128 vertices (n above 2 x 3648 x 128); degrees 0 .. a few, no heavy vertex
    n = 1_000_003
    rp, col = csr(n, *random_edges(n, n, 5))
    check(rp, col, id_mode=ids, off_mode=off, relabel=relabel)


@pytest.mark.parametrize("ids", [lg.LG_ID_GLOBAL, lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("n", [700_001, 1_100_003])
def test_shared_memory_table(ids, n):
    # more than 2^24 arcs, over a twelfth of them on the first labels in DM order
    u, v = random_edges(n, 9_000_000, 11)
    u = torch.where(torch.arange(u.numel(), device="cuda") % 3 == 0, u % 3000, u)
    rp, col = csr(n, u, v)
    assert int(rp[-1]) > 1 << 24
    for relabel in (lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM):
        check(rp, col, id_mode=ids, off_mode=lg.LG_OFF_EF, relabel=relabel)

"""Whole-graph decode of local IDs: warp tiles of 32, 64 and 128 vertices (graphs
below 155,648, below 622,592 and from there on), smaller ones for the long rows
of degree-mapped graphs, last tiles of one vertex, hubs
alone, next to each other and at a tile's edges, vertices without neighbors,
windows of 256 fields with one vertex or many.  The decoded CSR is the encoded one.
"""
import pytest
import torch

import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 257, 20000, 155647, 155649, 622591, 622593])
@pytest.mark.parametrize("ids", [lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("off", [lg.LG_OFF_PACKED, lg.LG_OFF_EF])
def test_round_trip(n, ids, off):
    lg.load(auto_build=True)
    rng = torch.Generator(device="cuda").manual_seed(n)
    d = torch.randint(0, 9, (n,), generator=rng, device="cuda") * (torch.rand(n, generator=rng, device="cuda") < 0.8)
    for v, k in ((0, 256), (5, 257), (6, 512), (127, 5000), (128, 9001), (129, 4096), (130, 4097), (300, 70), (1023, 6000),
                 (1024, 20000), (1025, 5000), (9000, 255), (n - 1, 12000)):
        if v < n:
            d[v] = k
    d.clamp_(max=n)
    # row v holds d[v] of the n vertices: a random stride from a random start, in order
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(d, 0)
    at = torch.arange(row.numel(), device="cuda") - rp[row]
    step = torch.div(n, d.clamp(min=1), rounding_mode="floor")
    step = (torch.rand(n, generator=rng, device="cuda") * step).long() + 1
    step = torch.minimum(step, torch.div(n - 1, d.clamp(min=2) - 1, rounding_mode="floor").clamp(min=1))
    room = n - 1 - (d.clamp(min=1) - 1) * step
    start = (torch.rand(n, generator=rng, device="cuda") * (room + 1)).long().clamp_(max=n - 1)
    col = (start[row] + at * step[row]).int()
    assert int(col.max()) < n if col.numel() else True
    g = lg.lg_encode(rp, col, id_mode=ids, off_mode=off)
    got = lg.lg_decode(g)
    assert torch.equal(got[0], rp) and torch.equal(got[1], col)
    # in DM order smaller tiles hold the rows of more than 32 arcs: the same decode
    # as that of plain rows
    g = lg.lg_encode(rp, col, id_mode=ids, off_mode=off, relabel=True)
    want = lg.lg_decode(lg.lg_encode(rp, col, id_mode=lg.LG_ID_CSR32, relabel=True))
    got = lg.lg_decode(g)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])

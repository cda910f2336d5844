"""Whole-graph decode of local IDs on graphs of even degrees: tiles of one size
in degree order too, and the heavy items in a launch of their own where the
schedule has most arcs.
"""
import pytest
import torch

import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, half", [(300, 70), (1000, 130), (1000, 300), (5000, 700), (30000, 3), (100001, 20), (700000, 18)])
@pytest.mark.parametrize("ids", [lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("off", [lg.LG_OFF_PACKED, lg.LG_OFF_EF])
def test_round_trip(n, half, ids, off):
    lg.load(auto_build=True)
    rng = torch.Generator(device="cuda").manual_seed(n)
    u = torch.arange(n, device="cuda").repeat_interleave(half)
    v = torch.randint(n, (n * half,), generator=rng, device="cuda")
    if n == 30000:  # most arcs on forty hubs, some vertices without any
        u, v = u[u < 12000], v[u < 12000]
        u = torch.cat([u, torch.arange(40, device="cuda").repeat_interleave(20000)])
        v = torch.cat([v, torch.randint(n // 2, (800000,), generator=rng, device="cuda")])
    if n == 5000:  # neighborhoods of no arc and of one between them
        keep = (u % 7 != 0) & (v % 7 != 0)
        u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n)
    col = (key % n).int()
    got = lg.lg_decode(lg.lg_encode(rp, col, id_mode=ids, off_mode=off))
    assert torch.equal(got[0], rp) and torch.equal(got[1], col)
    want = lg.lg_decode(lg.lg_encode(rp, col, id_mode=lg.LG_ID_CSR32, relabel=True))
    got = lg.lg_decode(lg.lg_encode(rp, col, id_mode=ids, off_mode=off, relabel=True))
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])

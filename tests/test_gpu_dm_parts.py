"""The degree-mapped rows of more than 32 arcs: their IDs are mapped in one
phase or in several (a phase per 2^23 vertices), rows of up to 4,096 arcs by
groups, longer ones by tiles of 4,096, and sorted by size class.  Row sizes lie
at the edges of the classes.  The relabeled CSR equals one built by a plain
sort of (new row, new ID).
"""
import pytest
import torch

import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu

SIZES = [33, 64, 65, 128, 129, 143, 144, 256, 257, 512, 513, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 8192, 8193,
         16383, 16384, 16385,
         70000]


def relabeled(n, rp, col, w):
    d = rp[1:] - rp[:-1]
    inv = torch.argsort(d, descending=True, stable=True)
    perm = torch.empty_like(inv)
    perm[inv] = torch.arange(n, device="cuda")
    row = perm[torch.repeat_interleave(torch.arange(n, device="cuda"), d)]
    key, at = torch.sort(row * n + perm[col.long()])
    nrp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    nrp[1:] = torch.cumsum(d[inv], 0)
    return nrp, (key % n).int(), w[at]


@pytest.mark.parametrize("n", [80001, 1 << 23, (1 << 23) + 1, 40000003])
@pytest.mark.parametrize("spread", [1.0, 3.0])
def test_relabeled_rows(n, spread):
    lg.load(auto_build=True)
    rng = torch.Generator(device="cuda").manual_seed(n)
    d = torch.zeros(n, dtype=torch.int64, device="cuda")
    at = torch.randperm(n, generator=rng, device="cuda")
    sizes = torch.tensor(SIZES * 5 + [40] * 333 + [200] * 99 + [700] * 17 + [1500] * 9, device="cuda")
    d[at[:sizes.numel()]] = sizes
    d[at[sizes.numel():40000]] = torch.randint(0, 33, (40000 - sizes.numel(),), generator=rng, device="cuda")
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    col = (torch.rand(row.numel(), generator=rng, device="cuda", dtype=torch.float64) ** spread * n).long().clamp_(max=n - 1)
    # half of the targets among 3,000 vertices whose degrees differ
    pick = torch.rand(row.numel(), generator=rng, device="cuda") < 0.5
    col = torch.where(pick, at[(torch.rand(row.numel(), generator=rng, device="cuda") * 3000).long()], col)
    key = torch.unique(row * n + col)  # sorted; rows that lost arcs to duplicates get new ones below
    short = d - torch.bincount(key // n, minlength=n)
    while int(short.sum()):
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), short)
        key = torch.unique(torch.cat([key, row * n + torch.randint(0, n, (row.numel(),), generator=rng, device="cuda")]))
        short = d - torch.bincount(key // n, minlength=n)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(d, 0)
    col = (key % n).int()
    w = torch.randint(1, 256, (col.numel(),), generator=rng, device="cuda", dtype=torch.int32)
    want = relabeled(n, rp, col, w)
    g = lg.lg_encode(rp, col, w, id_mode=lg.LG_ID_CSR32, relabel=True)
    got = lg.lg_decode(g, with_weights=True)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    g = lg.lg_encode(rp, col, id_mode=lg.LG_ID_CSR32, relabel=True)
    assert torch.equal(lg.lg_decode(g)[1], want[1])

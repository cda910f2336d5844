"""Random vertex access (lookups, SSSP) where the offsets are uneven: hubs whose
Elias-Fano gaps span thousands of words, at the front (DM order, looked up in
the heavy schedule) and in between (no relabeling, long scans), at the smallest
and the largest sample rate, with and without vertices in the schedule.
"""
import numpy as np
import pytest
import torch

import gen
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


def hub_graph(n, hubs, seed):
    rng = np.random.default_rng(seed)
    e = [rng.integers(0, n, (2 * n, 2))]
    e += [np.stack([np.full(d, h), rng.permutation(n)[:d]], 1) for h, d in hubs]
    return gen.from_edges(n, np.concatenate(e))


@pytest.mark.parametrize("sample", [64, 512, 65536])
@pytest.mark.parametrize("relabel", [lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM])
@pytest.mark.parametrize("ids", [lg.LG_ID_GLOBAL, lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("hubs", [[], [(0, 39000), (1, 257), (511, 9000), (512, 8000), (513, 4097), (39999, 300)]])
def test_lookup_every_vertex(sample, relabel, ids, hubs):
    lg.load(auto_build=True)
    g = hub_graph(40000, hubs, 4)
    rp, col = torch.from_numpy(g.row_ptr.view(np.int64)).cuda(), torch.from_numpy(g.col.view(np.int32)).cuda()
    e = lg.lg_encode(rp, col, id_mode=ids, off_mode=lg.LG_OFF_EF, relabel=relabel, select_sample=sample)
    vs = torch.from_numpy(np.random.default_rng(1).permutation(g.n).astype(np.int32)).cuda()
    off, out = lg.lg_neighbors(e, vs)
    deg = (rp[1:] - rp[:-1])[vs.long()]
    assert torch.equal(off[1:] - off[:-1], deg)
    at = torch.arange(out.numel(), device="cuda") - torch.repeat_interleave(off[:-1], deg)
    assert torch.equal(out, col[torch.repeat_interleave(rp[:-1][vs.long()], deg) + at])


@pytest.mark.parametrize("relabel", [lg.LG_RELABEL_NONE, lg.LG_RELABEL_DM, lg.LG_RELABEL_GREEDY])
@pytest.mark.parametrize("ids,weighted", [(lg.LG_ID_GLOBAL, True), (lg.LG_ID_GLOBAL, False), (lg.LG_ID_CSR32, True),
                                          (lg.LG_ID_LOCAL, False), (lg.LG_ID_LOCAL_GAP, False)])
def test_lookup_row_lengths(relabel, ids, weighted):
    """Rows at the edges of the warp's (256) and the CTA's (4,096) part, with
    repeats, in batches whose offsets one block scans and in one above that."""
    lg.load(auto_build=True)
    degrees = [0, 1, 31, 32, 33, 255, 256, 257, 300, 511, 512, 513, 1025, 4095, 4096, 4097, 20000]
    n, rng = 60000, np.random.default_rng(2)
    lo = len(degrees)
    u = np.concatenate([np.full(d, i) for i, d in enumerate(degrees)])
    v = np.concatenate([lo + rng.permutation(n - lo)[:d] for d in degrees])
    g = gen.from_edges(n, np.stack([u, v], 1))
    rp, col = torch.from_numpy(g.row_ptr.view(np.int64)).cuda(), torch.from_numpy(g.col.view(np.int32)).cuda()
    assert [int(x) for x in (rp[1:] - rp[:-1])[:lo]] == degrees
    w = (col * 7 % 251 + 1).int() if weighted else None
    e = lg.lg_encode(rp, col, w, id_mode=ids, off_mode=lg.LG_OFF_EF, relabel=relabel)
    for vs in (np.arange(lo), np.r_[lo - 1, np.arange(lo)[::-1], 5, 5], np.arange(n) % 9000, np.array([n - 1]),
               np.r_[np.arange(lo), np.arange(40000)]):
        vs = torch.from_numpy(vs.astype(np.int32)).cuda()
        got = lg.lg_neighbors(e, vs, with_weights=weighted)
        deg = (rp[1:] - rp[:-1])[vs.long()]
        assert torch.equal(got[0][1:] - got[0][:-1], deg) and int(got[0][0]) == 0
        at = torch.repeat_interleave(rp[:-1][vs.long()] - got[0][:-1], deg) + torch.arange(got[1].numel(), device="cuda")
        assert torch.equal(got[1], col[at])
        if weighted:
            assert torch.equal(got[2], w[at])

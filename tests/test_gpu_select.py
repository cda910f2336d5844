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

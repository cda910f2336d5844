"""Local widths and packing of rows around 256 arcs (listed above) and around the
window of 1,024: one and several windows, a last window of one field, long rows beside short ones in one
group of 32, gaps whose largest lies on either side of a window's edge.  The
streams must equal the oracle's bit for bit.
"""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ids", [lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("relabel", [False, True])
@pytest.mark.parametrize("big", [255, 256, 257, 1023, 1024, 1025, 1026, 2048, 2049, 2050, 9000])
def test_streams(ids, relabel, big):
    lg.load(auto_build=True)
    n, rng = 12000, np.random.default_rng(big)
    e = [rng.integers(0, n, (n, 2))]
    for h, d in ((40, big), (41, 5), (42, 1030), (63, big + 1), (9000, big)):
        e.append(np.stack([np.full(d, h), np.sort(rng.permutation(n)[:d])], 1))
    # a dense run with one wide gap at its 1,024th or 1,025th neighbor
    e.append(np.stack([np.full(2000, 7), np.r_[np.arange(100, 1123 + big % 2), np.arange(4000, 4977 - big % 2)]], 1))
    g = gen.from_edges(n, np.concatenate(e))
    x = lg.lg_encode(torch.from_numpy(g.row_ptr.view(np.int64)).cuda(), torch.from_numpy(g.col.view(np.int32)).cuda(),
                     id_mode=ids, off_mode=lg.LG_OFF_EF, relabel=relabel)
    want = oracle.encode(n, g.row_ptr, g.col, id_mode=ids, off_mode=oracle.OFF_EF, relabel=relabel)
    got = lg.lg_arrays_get(x)
    for name, ref in (("A", want.A), ("ef_low", want.ef_low), ("ef_high", want.ef_high), ("ef_samples", want.samples)):
        assert np.array_equal(got[name], ref), name

"""Local widths and packing of graphs whose rows are all alike and no longer than
a window of 1,024 arcs: nothing is listed, from 77,824 vertices on.  The streams
must equal the oracle's bit for bit.
"""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ids", [lg.LG_ID_LOCAL, lg.LG_ID_LOCAL_GAP])
@pytest.mark.parametrize("n, half, most", [(77823, 130, 0), (77824, 130, 0), (80001, 130, 1024), (80001, 130, 1025)])
def test_streams_of_even_graphs(ids, n, half, most):
    """Rows all alike and no longer than a window stay with their warps."""
    lg.load(auto_build=True)
    rng = np.random.default_rng(n)
    u = np.repeat(np.arange(n), half)
    e = [np.stack([u, rng.integers(0, n, n * half)], 1)]
    if most:  # one row of exactly that many arcs
        v = np.arange(5, 5 + most)
        keep = (e[0][:, 0] != 0) & (e[0][:, 1] != 0)
        e = [e[0][keep], np.stack([np.zeros(most, np.int64), v], 1)]
    g = gen.from_edges(n, np.concatenate(e))
    assert not most or int(np.diff(g.row_ptr.astype(np.int64)).max()) == most
    x = lg.lg_encode(torch.from_numpy(g.row_ptr.view(np.int64)).cuda(), torch.from_numpy(g.col.view(np.int32)).cuda(),
                     id_mode=ids, off_mode=lg.LG_OFF_PACKED)
    want = oracle.encode(n, g.row_ptr, g.col, id_mode=ids, off_mode=oracle.OFF_PACKED)
    got = lg.lg_arrays_get(x)
    assert np.array_equal(got["A"], want.A) and np.array_equal(got["O"], want.O)

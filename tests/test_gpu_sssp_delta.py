"""SSSP's bucket width when the caller names none: it follows the weights, so
weights multiplied by 257 take about as many rounds; narrow, wide and zero
weights give Dijkstra's distances.
"""
import numpy as np
import pytest

import gen
import oracle
import paper_2010_15879_gb300 as lg

pytestmark = pytest.mark.gpu


def graph():
    lg.load(auto_build=True)
    return gen.rmat(12, 8, seed=5, weighted=True)


def dist(g, s):
    l0 = lg.lg_kernel_launches()
    d = lg.lg_sssp(g, s).cpu().numpy().view(np.uint64)
    return d, lg.lg_kernel_launches() - l0


@pytest.mark.parametrize("opts", [dict(), dict(id_mode=lg.LG_ID_CSR32), dict(weight_bits=32)])
def test_width_follows_the_weights(opts):
    h = graph()
    s = int(np.argmax(np.diff(h.row_ptr.astype(np.int64))))
    narrow, few = dist(lg.lg_encode(h.row_ptr, h.col, h.weights, **opts), s)
    wide, many = dist(lg.lg_encode(h.row_ptr, h.col, h.weights * np.uint32(257), **opts), s)
    reached = narrow != np.uint64(2 ** 64 - 1)
    assert np.array_equal(wide[reached], narrow[reached] * np.uint64(257)) and np.array_equal(wide[~reached], narrow[~reached])
    assert many <= 2 * few, (few, many)


@pytest.mark.parametrize("factor, modulus", [(0, 1), (1, 2), (1, 16), (1 << 23, 256)])
@pytest.mark.parametrize("opts", [dict(), dict(relabel=lg.LG_RELABEL_DM, off_mode=lg.LG_OFF_EF), dict(id_mode=lg.LG_ID_CSR32)])
def test_distances(factor, modulus, opts):
    h = graph()
    w = (h.weights % modulus * factor).astype(np.uint32)
    g = lg.lg_encode(h.row_ptr, h.col, w, **opts)
    for s in (0, 1000):
        assert np.array_equal(dist(g, s)[0], oracle.sssp(h.n, h.row_ptr, h.col, w, s))


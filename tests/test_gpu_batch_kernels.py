"""Which kernels a batch runs: graphs of more than 65,536 vertices go to a
kernel of small CTAs with a team limit of its own, the others to the
shared-memory kernel, and a batch of one kind launches one of them only.
"""
import numpy as np
import pytest

import gen
import paper_2010_15879_gb300 as lg
from test_gpu_batch import concat, create, host_batch_arrays, run_and_check

pytestmark = pytest.mark.gpu

LARGE = [65537, 140000]
SMALL = [65536, 300, 2]


def batch(sizes):
    graphs = []
    for n in sizes:
        e = np.random.default_rng(n).integers(0, n, (2 * n, 2))
        graphs.append(gen.from_edges(n, e))
    return host_batch_arrays(concat(graphs))


@pytest.mark.parametrize("tile", [1 << 10, 1 << 17, 0])  # more items than SMs, fewer, by rule
@pytest.mark.parametrize("sizes, kernels", [(SMALL, 1), (LARGE, 1), (LARGE + SMALL, 2)])
def test_kernels(sizes, kernels, tile):
    lg.load(auto_build=True)
    hb = batch(sizes)
    b = create(hb, autotune=False, tile_arcs=tile)
    info = b.info()
    if tile == 1 << 10:  # a team of the larger graphs may take more members than half the SMs
        assert (info["max_team"] > 76) == (len(set(sizes) & set(LARGE)) > 0)
    l0 = lg.lg_kernel_launches()
    run_and_check(b, hb)
    assert lg.lg_kernel_launches() - l0 == kernels
    b.free()

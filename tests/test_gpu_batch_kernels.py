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


def test_parts_of_a_cta():
    """Many small graphs: those of up to 856 vertices go to one warp, those of up
    to 6,868 to eight, if a few thousand others share the chip; every size class
    has its edges in the batch, beside long paths, stars and empty graphs."""
    lg.load(auto_build=True)
    rng = np.random.default_rng(9)
    sizes = [1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 129, 855, 856, 857, 858, 4000, 6867, 6868, 6869, 6870]
    graphs = [gen.from_edges(n, rng.integers(0, n, (k * n, 2))) for n in sizes for k in (1, 5)]
    graphs += [gen.from_edges(n, [(i, i + 1) for i in range(n - 1)]) for n in (856, 2000)]  # a level per vertex
    graphs += [gen.from_edges(n, np.stack([np.full(n - 1, n // 2), np.delete(np.arange(n), n // 2)], 1)) for n in (800, 6000)]
    graphs += [gen.from_edges(500, np.zeros((0, 2)))]
    graphs += [gen.from_edges(200, rng.integers(0, 200, (4000, 2)))]  # 256 fields and more to a vertex's tile
    pool = [gen.from_edges(n, rng.integers(0, n, (12 * n, 2))) for n in (64, 200, 5000)]
    graphs += [pool[i % 3] for i in range(3000)]
    hb = host_batch_arrays(concat(graphs))
    b = create(hb, autotune=False)
    run_and_check(b, hb, graphs=range(60))
    d1, r1 = (x.clone() for x in lg.lg_batch_run(b, 0.85, 4))
    d2, r2 = lg.lg_batch_run(b, 0.85, 4)
    lg.lg_batch_status(b)
    assert bool((d1 == d2).all()) and bool((r1 == r2).all())
    b.free()
    b = create(hb, autotune=True)
    run_and_check(b, hb, graphs=range(60))
    b.free()

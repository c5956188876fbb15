"""The tile sweep in every lane class, against the oracle (integers: equal): the
whole of a small graph in tiles (no core: more upward labels in a tile than it has
rows for, tiers of one tile), arbitrary multigraphs, and a graph of many tiles
under the default core, with distances, lists, vertices in range and a second
batch on the same workspace."""

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

LANES = (1, 3, 7, 16, 21, 64)  # one batch of every lane class (1, 4, 8, 16, 32, 64 lanes)


def check(g, dg, k, tmax, seed, **opts):
    ws = P.Workspace(dg, k, **opts)
    assert ws.sweep_info()["chunks"] > 0
    for s in (seed, seed + 1):
        srcs = synth.draw_sources(g, k, s)
        taus = synth.draw_taus_uniform(k, 0, tmax, s + 100)
        ws.submit(srcs, taus, want_dist=True)
        off, arcs, dist = ws.collect(want_dist=True)
        bits = ws.collect_range()
        o_off, o_arcs, o_dist = oracle.query_batch(g.n, g.tail, g.head, g.weight, srcs, taus, want_dist=True, threads=8)
        assert np.array_equal(off, o_off) and np.array_equal(arcs, o_arcs) and np.array_equal(dist, o_dist)
        got = np.unpackbits(bits.view(np.uint8), axis=1, bitorder="little")[:, :g.n].astype(bool)
        assert np.array_equal(got, o_dist != P.INF)
    ws.free()


@pytest.mark.parametrize("k", LANES)
def test_small_graph_all_in_tiles(k):
    g = synth.grid_road_graph(61, 47, seed=11)
    dg = P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))
    check(g, dg, k, 2500, 300 + k, core_vertices=-1)
    check(g, dg, k, 2500, 400 + k, core_vertices=40, use_cuda_graph=1)
    dg.free()


@pytest.mark.parametrize("k", LANES)
@pytest.mark.parametrize("n,m", [(2, 3), (70, 200), (900, 2000)])
def test_multigraphs_all_in_tiles(k, n, m):
    g = synth.random_graph(n, m, seed=n + k)
    dg = P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))
    check(g, dg, k, 60, 500 + k, core_vertices=-1)
    dg.free()


@pytest.fixture(scope="module")
def region():
    g = synth.grid_road_graph(401, 307, highways=((32, 4),), seed=12)
    return g, P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))


@pytest.mark.parametrize("k", LANES)
def test_many_tiles_below_the_core(region, k):
    check(*region, k, 20000, 600 + k, use_cuda_graph=1)

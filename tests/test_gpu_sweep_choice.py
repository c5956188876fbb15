"""Which sweep a workspace runs (iso_sweep_info.sweep): tiles in every lane class
where the options leave the choice to the library, the chunk schedule where a vertex
below the core has more sources than a tile has rows, and the kernels that options
name; results against the oracle (integers: equal)."""

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROWS = {1: 2500, 4: 1000, 8: 400, 16: 300, 32: 200, 64: 100}  # label rows of a tile, by lane class


class Sink:
    """A road graph and a vertex that 310 roads lead into: it is contracted early, with
    310 sources, more than a tile holds at 16 lanes and above."""

    def __init__(self, rows, cols):
        g = synth.grid_road_graph(rows, cols, highways=((32, 4),), seed=5)
        into = np.linspace(0, g.n - 1, 310).astype(np.int32)
        self.n = g.n + 1
        self.tail = np.concatenate([g.tail, into])
        self.head = np.concatenate([g.head, np.full(310, g.n, np.int32)])
        self.weight = np.concatenate([g.weight, (np.arange(310) % 90 + 1).astype(np.int32)])


@pytest.fixture(scope="module")
def sink():
    g = Sink(250, 200)
    dg = P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))
    yield g, dg
    dg.free()


def check(g, ws, k, seed):
    srcs = synth.draw_sources(g, k, seed)
    taus = synth.draw_taus_uniform(k, 0, 9000, seed + 1)
    ws.submit(srcs, taus, want_dist=True)
    off, arcs, dist = ws.collect(want_dist=True)
    o_off, o_arcs, o_dist = oracle.query_batch(g.n, g.tail, g.head, g.weight, srcs, taus, want_dist=True, threads=8)
    assert np.array_equal(off, o_off) and np.array_equal(arcs, o_arcs) and np.array_equal(dist, o_dist)


@pytest.mark.parametrize("k", sorted(ROWS))
def test_tiles_unless_a_vertex_has_more_sources_than_rows(sink, k):
    g, dg = sink
    ws = P.Workspace(dg, k, use_cuda_graph=1)
    info = ws.sweep_info()
    assert info["sweep"] == (2 if ROWS[k] > 310 else 1)
    if info["sweep"] == 2:
        assert info["dep_cap"] == ROWS[k] and info["core_vertices"] <= 20000 and info["chunks"] > 0
    for seed in (10, 20):
        check(g, ws, k, seed + k)
    ws.free()


@pytest.mark.parametrize("core", [0, -1, 3000])
@pytest.mark.parametrize("k", sorted(ROWS))
def test_tiles_on_a_road_graph(k, core):
    g = synth.grid_road_graph(150, 130, seed=6)
    dg = P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))
    ws = P.Workspace(dg, k, core_vertices=core)
    info = ws.sweep_info()
    assert info["sweep"] == 2 and info["dep_cap"] == ROWS[k]
    check(g, ws, k, 30 + k)
    for kernel, sweep in ((1, 1), (2, 0)):
        other = P.Workspace(dg, k, sweep_kernel=kernel, core_vertices=core)
        assert other.sweep_info()["sweep"] == sweep
        other.free()
    ws.free()
    dg.free()

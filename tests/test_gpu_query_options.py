"""iso_query keeps a workspace per lane class while the options stay what they were,
and makes another when an option with an effect changes: the default core above the
tiles is not the core of 53,248 vertices that may be asked for by number."""

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import synth

from counting_alloc import upload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("k", [1, 16, 64])
def test_core_vertices_by_number_is_not_the_default(k, monkeypatch):
    g = synth.grid_road_graph(401, 307, highways=((32, 4),), seed=12)
    dg, mem = upload(P.iso_build_ch(g.n, g.tail, g.head, g.weight), monkeypatch)
    srcs, taus = synth.draw_sources(g, k, 1), synth.draw_taus_uniform(k, 0, 9000, 2)
    want = oracle.query_batch(g.n, g.tail, g.head, g.weight, srcs, taus, threads=8)
    for core in (0, 53248, 0):
        for call in range(2):
            before = len(mem.log)
            off, arcs, _ = P.iso_query(dg, srcs, taus, core_vertices=core, use_cuda_graph=1)
            assert np.array_equal(off, want[0]) and np.array_equal(arcs, want[1])
            assert (len(mem.log) > before) == (call == 0), (core, call)
        ws = P.Workspace(dg, k, core_vertices=core)
        n_core = ws.sweep_info()["core_vertices"]
        assert (n_core > 20000) == (core > 0)
        ws.free()
    dg.free()

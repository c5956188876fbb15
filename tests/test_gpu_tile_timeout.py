"""The tile sweep stops early and the call reports it.  Its bounded waits run out (a
barrier that expects an arrival that never comes): behind the per-lane core with no
tiles (64 x 64 vertices lie in the core), between tiers with and without a core, with
a tile's record still on its way.  Or another lane's source is invalid, found by the
upward search: the sweep then leaves upward labels unused, and the same workspace's
next batch must not see them.  Results against the oracle (integers: equal)."""

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import synth

from helpers import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

LIMIT_NS = 20_000_000


def equal(g, srcs, taus, off, arcs, dist):
    o_off, o_arcs, o_dist = oracle.query_batch(g.n, g.tail, g.head, g.weight, srcs, taus, want_dist=True, threads=8)
    assert np.array_equal(off, o_off) and np.array_equal(arcs, o_arcs) and np.array_equal(dist, o_dist)


@pytest.mark.parametrize("k", [1, 16, 64])
@pytest.mark.parametrize("name,core", [("grid64", 0), ("grid64", -1), ("grid1k", 0), ("grid1k", -1)])
def test_tile_sweep_gives_up_and_the_next_call_is_right(name, core, k):
    g, ch = workload(name)
    dg = P.iso_upload_graph(ch)
    srcs = synth.draw_sources(g, k, 2 + k)
    taus = synth.draw_taus_uniform(k, 500, 6000, 3 + k)
    for graph in (0, 1):
        ws = P.Workspace(dg, k, core_vertices=core, debug_barrier_extra=1, barrier_timeout_ns=LIMIT_NS,
                         use_cuda_graph=graph)
        assert ws.sweep_info()["sweep"] == 2
        for _ in range(2):  # the second batch starts on what the first one left
            ws.submit(srcs, taus)
            with pytest.raises(P.IsoError) as e:
                ws.collect()
            assert e.value.code == P.ISO_E_TIMEOUT
        ws.free()
        torch.cuda.synchronize()
    equal(g, srcs, taus, *P.iso_query(dg, srcs, taus, want_dist=True, core_vertices=core))
    dg.free()


@pytest.mark.parametrize("k", [4, 64])
@pytest.mark.parametrize("name,core", [("grid64", 0), ("grid64", -1), ("grid1k", 0), ("grid1k", -1)])
def test_workspace_after_a_stopped_sweep(name, core, k):
    g, ch = workload(name)
    dg = P.iso_upload_graph(ch)
    ws = P.Workspace(dg, k, core_vertices=core, use_cuda_graph=1)
    assert ws.sweep_info()["sweep"] == 2
    for seed in (5, 6):
        srcs = synth.draw_sources(g, k, seed)
        bad = srcs.copy()
        bad[k // 2] = g.n + 7
        ws.submit(*(torch.from_numpy(x).cuda() for x in (bad, np.full(k, 9000, np.int32))))
        with pytest.raises(P.IsoError) as e:
            ws.collect()
        assert e.value.code == P.ISO_E_INVAL
        srcs = synth.draw_sources(g, k, seed + 10)
        taus = synth.draw_taus_uniform(k, 500, 6000, seed + 20)
        ws.submit(srcs, taus, want_dist=True)
        equal(g, srcs, taus, *ws.collect(want_dist=True))
    ws.free()
    dg.free()

"""A tile plan that cannot be made (a vertex with more sources than a tile has rows) is
tried once per graph, lane class and core: the next workspace goes to the chunk schedule,
which the graph keeps, at once.  The first one takes the attempt (over all of the
graph's vertices) and the schedule; a later one allocates and copies, a small part of that."""

import time

import numpy as np
import pytest

import paper_1512_09090_gb300 as P

from test_gpu_sweep_choice import Sink, check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def test_refused_plan_is_remembered():
    g = Sink(1000, 1000)
    dg = P.iso_upload_graph(P.iso_build_ch(g.n, g.tail, g.head, g.weight))
    P.Workspace(dg, 64, sweep_kernel=1).free()  # the chunk schedule, and the allocator's first blocks
    took = []
    for _ in range(4):
        t0 = time.perf_counter()
        ws = P.Workspace(dg, 64)
        took.append(time.perf_counter() - t0)
        assert ws.sweep_info()["sweep"] == 1
        if len(took) == 4:
            check(g, ws, 64, 40)
        ws.free()
    print("seconds:", np.round(took, 4))
    assert min(took[1:]) < took[0] / 4
    dg.free()

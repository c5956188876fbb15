"""Tile plans and device memory, with an allocator that hands out a set number of bytes:
a workspace for which there is room only without a plan takes the chunk schedule, and
plans that no workspace uses make room for what is asked for later."""

import numpy as np
import pytest

import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import synth

from counting_alloc import upload
from helpers import workload
from test_gpu_sweep_choice import check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def needs(ch, monkeypatch, **opts):
    """Bytes that a 64-lane workspace of these options takes at most, its plan included."""
    dg, mem = upload(ch, monkeypatch)
    base = mem.peak = mem.live
    P.Workspace(dg, 64, **opts).free()
    dg.free()
    assert mem.live == 0
    return mem.peak - base


def test_chunk_schedule_where_a_plan_has_no_room(monkeypatch):
    g, ch = workload("grid1k")
    room = needs(ch, monkeypatch, sweep_kernel=1)
    assert needs(ch, monkeypatch) > room
    dg, mem = upload(ch, monkeypatch)
    mem.limit = mem.live + room
    ws = P.Workspace(dg, 64)
    assert ws.sweep_info()["sweep"] == 1
    mem.limit = None
    check(g, ws, 64, 50)
    ws.free()
    before = mem.live
    mem.limit = before + room // 2  # not enough for either: refused, and nothing is lost
    with pytest.raises(P.IsoError) as e:
        P.Workspace(dg, 64)
    assert e.value.code == P.ISO_E_NOMEM and mem.live == before
    mem.limit = None
    ws = P.Workspace(dg, 64)
    assert ws.sweep_info()["sweep"] == 2
    check(g, ws, 64, 60)
    ws.free()
    dg.free()
    assert mem.live == 0


def test_idle_plans_make_room(monkeypatch):
    g, ch = workload("grid1k")
    room = needs(ch, monkeypatch)
    dg, mem = upload(ch, monkeypatch)
    base = mem.live
    P.Workspace(dg, 1).free()
    assert mem.live > base  # (its plan)
    mem.limit = base + room
    ws = P.Workspace(dg, 64)
    assert ws.sweep_info()["sweep"] == 2
    ws.free()
    # a buffer that an existing workspace asks for later
    ws = P.Workspace(dg, 64)
    ws.submit(synth.draw_sources(g, 64, 70), np.full(64, 900, np.int32))
    ws.collect()
    mem.limit = None
    P.Workspace(dg, 4).free()
    mem.limit = mem.live
    ws.collect_range()
    mem.limit = None
    check(g, ws, 64, 80)
    ws.free()
    dg.free()
    assert mem.live == 0


def test_a_plan_is_reported_by_the_workspace_that_made_it(monkeypatch):
    g = synth.grid_road_graph(250, 200, seed=9)
    dg, mem = upload(P.iso_build_ch(g.n, g.tail, g.head, g.weight), monkeypatch)
    took = []
    for k in (16, 16, 64):
        before = mem.live
        ws = P.Workspace(dg, k)
        took.append((ws.sweep_info()["plan_kib"], mem.live - before))
        ws.free()
    assert took[0][0] > 0 and took[1][0] == 0 and took[2][0] > 0
    # (allocations are rounded up to 256 bytes each)
    assert 0 <= took[0][1] - took[1][1] - (took[0][0] << 10) < 2048
    P.Workspace(dg, 64, sweep_kernel=1).free()
    dg.free()

"""The server's growth by device memory where workspaces share a tile plan: the plan is
made with the first workspace and counted apart, so that the pool grows as soon as
there is room for what another workspace takes by itself (fake device memory, CPU)."""

import pytest

from paper_1512_09090_gb300 import serving

from test_serving_host import FakeDevWorkspace, _flood, fake_device  # noqa: F401

PLAN = 3 << 30


class SharedPlanWorkspace(FakeDevWorkspace):
    def __init__(self, g, lanes, **opts):
        super().__init__(g, lanes, **opts)
        pool = FakeDevWorkspace.pool
        self.plan_kib = 0 if "plan" in pool else PLAN >> 10
        if self.plan_kib:
            pool["plan"] = True
            pool["free"] -= PLAN

    def sweep_info(self):
        return {"plan_kib": self.plan_kib}


@pytest.mark.parametrize("there", [False, True])  # the plan is made by the server, or was there before it
def test_plan_is_not_counted_with_every_workspace(fake_device, monkeypatch, there):  # noqa: F811
    monkeypatch.setattr(serving._lib, "Workspace", SharedPlanWorkspace)
    # after the plan and the first workspace (1 GB) 4 GB are free: half of that covers
    # another workspace, not another workspace and a plan
    fake_device["free"] = 5 << 30
    if there:
        fake_device["plan"] = True
    else:
        fake_device["free"] += PLAN
    with serving.IsoServer(object(), lanes=4, workspaces=1, max_workspaces=2, memory_fraction=0.5) as srv:
        assert srv.bytes_per_workspace == 1 << 30
        _flood(srv, 200)
        assert srv.grown == 1 and srv.refused_growth == 0

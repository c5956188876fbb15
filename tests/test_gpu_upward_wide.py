"""Upward searches that are wide from the start, against the oracle (integers: equal): a
depot with one-way roads to many yards, which lead to a few gates.  The depot is
contracted first, so that its search has all the yards in its first rounds: below the
shared-memory table's limit, about it, and above it (then redone in global memory, and
the batch run again with larger tables); with other sources in the same batch."""

import time

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

GATES = 7


def depot(yards):
    """0 -> yards -> gates -> the next gate; returns (n, tail, head, weight)."""
    y = np.arange(1, yards + 1, dtype=np.int32)
    g = yards + 1 + np.arange(GATES, dtype=np.int32)
    tail = np.concatenate([np.zeros(yards, np.int32), y, g[:-1]])
    head = np.concatenate([y, g[y % GATES], g[1:]])
    return yards + 1 + GATES, tail, head, (np.arange(tail.size) * 7919 % 97 + 1).astype(np.int32)


def hubs(yards):
    """The same with three roads from each gate to other gates, which keeps the gates above
    the yards: every yard is in the frontier of the second round."""
    n, tail, head, weight = depot(yards)
    g = yards + 1 + np.arange(GATES, dtype=np.int32)
    more = 3 * GATES
    return (n, np.concatenate([tail, g, g, g]), np.concatenate([head, np.roll(g, -1), np.roll(g, -2), np.roll(g, -3)]),
            np.concatenate([weight, (np.arange(more) * 31 % 89 + 1).astype(np.int32)]))


def run(dg, graph, k, yards, **opts):
    srcs = (np.arange(k) % 3 * (yards // 2)).astype(np.int32)  # the depot and two yards
    taus = (200 - np.arange(k)).astype(np.int32)
    off, arcs, dist = P.iso_query(dg, srcs, taus, want_dist=True, **opts)
    want = oracle.query_batch(*graph, srcs, taus, want_dist=True, threads=8)
    assert np.array_equal(off, want[0]) and np.array_equal(arcs, want[1]) and np.array_equal(dist, want[2])


@pytest.mark.parametrize("yards", [15, 16, 17, 100, 3000, 6200, 8150, 8184, 8185, 9000, 20_000])
def test_wide_searches(yards):
    graph = depot(yards)
    dg = P.iso_upload_graph(P.iso_build_ch(*graph))
    for k, opts in ((1, {}), (5, dict(core_vertices=-1)), (64, dict(use_cuda_graph=1)), (4, dict(sweep_kernel=2))):
        run(dg, graph, k, yards, **opts)
    dg.free()


# a frontier of shared memory's 3,072 entries, and one, two and three times as many to
# come from global memory; the last ones about the table's limit
@pytest.mark.parametrize("yards", [33, 3071, 3072, 3073, 3100, 6143, 6144, 6145, 7000, 8180, 8183, 8184, 8190, 8200])
def test_wide_frontiers(yards):
    graph = hubs(yards)
    dg = P.iso_upload_graph(P.iso_build_ch(*graph))
    for k, opts in ((1, {}), (64, dict(use_cuda_graph=1)), (4, dict(sweep_kernel=2))):
        run(dg, graph, k, yards, **opts)
    # the allocation-free call (tables of 8,192 vertices; 93% of the yards are within 90)
    srcs, taus = np.zeros(3, np.int32), np.array([90, 40, 0], np.int32)
    off, arcs, _ = P.iso_query(dg, srcs, taus)
    d_off = torch.zeros(4, dtype=torch.int64, device="cuda")
    d_arcs = torch.zeros(int(off[-1]), dtype=torch.int32, device="cuda")
    P._lib.iso_query_noalloc(dg, torch.from_numpy(srcs).cuda(), torch.from_numpy(taus).cuda(), d_off, d_arcs)
    assert np.array_equal(d_off.cpu().numpy(), off) and np.array_equal(d_arcs.cpu().numpy(), arcs)
    dg.free()


def test_a_search_far_above_the_tables_stops_early():
    # a round that overflows a table frees what it puts in: filled to the last slot, the table
    # was walked whole for every further yard (9 s a batch, now 20 ms)
    graph = depot(40_000)
    dg = P.iso_upload_graph(P.iso_build_ch(*graph))
    run(dg, graph, 1, 100)
    t0 = time.perf_counter()
    ws = P.Workspace(dg, 64)
    ws.submit(np.zeros(64, np.int32), np.full(64, 200, np.int32))
    ws.collect()
    took = time.perf_counter() - t0
    ws.free()
    print(f"seconds: {took:.3f}")
    assert took < 2.0
    dg.free()

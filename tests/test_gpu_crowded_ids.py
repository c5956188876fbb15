"""Lists whose ids all lie close together among many (every id in one sorting CTA's part
and in few of its buckets), at the sizes where the number of buckets changes, in every
number of CTAs per list: hubs with arcs of consecutive ids, beside a long road that
takes up most ids.  With limit 0 a hub's list is its arcs' ids."""

import numpy as np
import pytest

import paper_1512_09090_gb300 as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SIZES = (1, 3, 4, 5, 8, 9, 64, 65, 256, 257, 1024, 1025, 4096, 4097, 8000)
ROAD = 600_000


@pytest.fixture(scope="module", params=["before", "between", "after"])
def hubs(request):
    """(device graph, hub vertices, first id of each hub's arcs); hubs' arcs shuffled in heads"""
    a = np.arange(ROAD - 1, dtype=np.int32)
    road = (np.concatenate([a, a + 1]), np.concatenate([a + 1, a]))
    rng, n, hub, star = np.random.default_rng(1), ROAD, [], [[], []]
    for size in SIZES:
        hub.append(n)
        star[0].append(np.full(size, n, np.int32))
        star[1].append(rng.permutation(np.arange(n + 1, n + 1 + size, dtype=np.int32)))
        n += 1 + size
    star = tuple(np.concatenate(x) for x in star)
    half = road[0].size // 2
    parts = {"before": [star, road], "after": [road, star],
             "between": [tuple(x[:half] for x in road), star, tuple(x[half:] for x in road)]}[request.param]
    tail, head = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    first = {"before": 0, "after": road[0].size, "between": half}[request.param] + np.cumsum((0,) + SIZES)[:-1]
    dg = P.iso_upload_graph(P.iso_build_ch(n, tail, head, (np.arange(tail.size) % 7 + 1).astype(np.int32)))
    yield dg, np.array(hub, np.int32), first
    dg.free()


@pytest.mark.parametrize("k", [1, 4, 8, 16, 32, 64])
def test_neighbouring_ids(hubs, k):
    dg, hub, first = hubs
    for start in range(0, len(SIZES), k):
        which = (start + np.arange(k)) % len(SIZES)
        off, arcs, _ = P.iso_query(dg, hub[which], np.zeros(k, np.int32))
        want = [np.arange(first[i], first[i] + SIZES[i]) for i in which]
        assert np.array_equal(np.diff(off), [w.size for w in want]) and np.array_equal(arcs, np.concatenate(want))

"""Emission where most of a CTA's rounds leave its edge buffer past the mark at which
the CTA empties it, over several rounds and repeated batches.

A CTA decides between two rounds whether to empty the buffer; a decision that is not
the same in all of its threads loses or doubles edges.  The graph is a road of
unit-length segments with a far-off vertex at every fourth place: all of these arcs
cross for a query that covers the road, and what crosses is known without a search."""

import numpy as np
import pytest

import paper_1512_09090_gb300 as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROAD, EVERY, FAR = 800_000, 4, 1_000_000


@pytest.fixture(scope="module")
def road():
    a = np.arange(ROAD - 1, dtype=np.int32)
    r = np.arange(0, ROAD, EVERY, dtype=np.int32)
    b = (ROAD + np.arange(r.size)).astype(np.int32)
    tail, head = np.concatenate([a, a + 1, r, b]), np.concatenate([a + 1, a, b, r])
    weight = np.concatenate([np.ones(2 * a.size, np.int32), np.full(2 * r.size, FAR, np.int32)])
    dg = P.iso_upload_graph(P.iso_build_ch(ROAD + r.size, tail, head, weight))
    yield dg
    dg.free()


def crossing(s, tau):
    """Ids of the arcs with exactly one endpoint within tau < FAR of road vertex s."""
    lo, hi = max(0, s - tau), min(ROAD - 1, s + tau)
    ends = [i for i in (s - tau - 1, s + tau) if 0 <= i < ROAD - 1]
    far = np.arange(-(-lo // EVERY), hi // EVERY + 1)
    base = 2 * (ROAD - 1)
    return np.sort(np.concatenate([ends, [ROAD - 1 + i for i in ends], base + far, base + -(-ROAD // EVERY) + far]))


@pytest.mark.parametrize("k", [1, 4, 16, 64])  # 100 to 6,500 edges a round, of 2,048 that the buffer holds
def test_buffer_emptied_in_most_rounds(road, k):
    rng = np.random.default_rng(k)
    ws = P.Workspace(road, k, use_cuda_graph=1)
    for _ in range(4):
        srcs = rng.integers(0, ROAD, k).astype(np.int32)
        taus = rng.integers(0, ROAD // 2, k).astype(np.int32)
        taus[0] = ROAD - 1  # (everything)
        ws.submit(srcs, taus)
        off, arcs, _ = ws.collect()
        for i in range(k):
            assert np.array_equal(arcs[off[i]:off[i + 1]], crossing(int(srcs[i]), int(taus[i]))), i
    ws.free()

"""Emission and sort at the sizes where they change course, against the oracle
(integers: equal): more isochrone edges at one vertex than a CTA's buffer holds,
ids crowded into a few buckets, into one sorting CTA's part, and a list that no
part's shared memory holds; few ids (below the bucket resolution); no edges."""

import numpy as np
import pytest

import oracle
import paper_1512_09090_gb300 as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def star_and_road(leaves, road, star_first):
    """A star (its arcs leave vertex 0, consecutive ids) and a two-way road apart
    from it, which adds ids that never cross for a source in the star."""
    t0, h0 = np.zeros(leaves, np.int32), np.arange(1, leaves + 1, dtype=np.int32)
    a = np.arange(leaves + 1, leaves + road, dtype=np.int32)
    t1, h1 = np.concatenate([a, a + 1]), np.concatenate([a + 1, a])
    parts = [(t0, h0), (t1, h1)] if star_first else [(t1, h1), (t0, h0)]
    tail, head = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    weight = (np.arange(tail.size) % 7 + 1).astype(np.int32)
    return leaves + 1 + road, tail, head, weight


@pytest.mark.parametrize("leaves,road,star_first", [
    (90, 5, True),            # fewer ids than buckets
    (3000, 4, True),          # one vertex fills a CTA's edge buffer
    (3000, 100_000, False),   # 3,000 ids in a few of the buckets
    (40_000, 200_000, True),  # 40,000 ids in one or two of the parts: sorted in global memory
])
def test_crowded_lists(leaves, road, star_first):
    n, tail, head, weight = star_and_road(leaves, road, star_first)
    dg = P.iso_upload_graph(P.iso_build_ch(n, tail, head, weight))
    for k in (1, 20, 64):  # every number of sorting CTAs per list
        srcs = np.where(np.arange(k) % 8 < 7, 0, leaves // 2).astype(np.int32)  # the hub, or a leaf (no edges)
        taus = (np.arange(k) % 9).astype(np.int32)
        off, arcs, _ = P.iso_query(dg, srcs, taus)
        same = sorted({(int(s), int(t)) for s, t in zip(srcs, taus)})
        o_off, o_arcs, _ = oracle.query_batch(n, tail, head, weight, np.array([s for s, _ in same], np.int32),
                                              np.array([t for _, t in same], np.int32), threads=8)
        for i in range(k):
            j = same.index((int(srcs[i]), int(taus[i])))
            assert np.array_equal(arcs[off[i]:off[i + 1]], o_arcs[o_off[j]:o_off[j + 1]]), (k, i)
    dg.free()

"""VT rows of every length class against the CPU oracle, bit for bit: stars
sorted two to a thread (up to 16, 24 and 32 tets), one to a thread (33 to
64) and by a warp (more), rows padded and compact, more than 255 neighbours
(rank prefixes modulo 256), 16-bit positions (more than 256 tets), tets too
many to carry the vertex's slot (more than 16,383) and stars counted in two
words (more than 21,845 tets)."""
import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk

pytestmark = pytest.mark.gpu


def fans(sizes, seg_of, seed):
    """One fan of k tets around an edge per k: its two end vertices have
    stars of k tets.  They get the largest ids, so that no vertex has many
    neighbours above it; the other ids are drawn."""
    tv, n = [], 0
    for k in sizes:
        ring = n + np.arange(k + 1)
        n += k + 1
        tv += [[-1, -2, ring[i], ring[i + 1]] for i in range(k)]
    tv = np.array(tv, np.int64)
    fan = np.repeat(np.arange(len(sizes)), sizes)
    tv[:, 0], tv[:, 1] = n + 2 * fan, n + 2 * fan + 1
    nv = n + 2 * len(sizes)
    rng = np.random.default_rng(seed)
    p = np.concatenate([rng.permutation(n), n + rng.permutation(2 * len(sizes))])
    tv = p[tv][rng.permutation(len(tv))]
    tv = np.take_along_axis(tv, rng.random(tv.shape).argsort(1), 1)
    seg = seg_of(rng, nv)
    return gen.Mesh(rng.random((nv, 3)).astype(np.float32), tv.astype(np.int32), seg.astype(np.int32), int(seg.max()) + 1)


ONE = lambda rng, nv: np.zeros(nv, np.int64)  # noqa: E731
TWO = lambda rng, nv: np.concatenate([[0, 1], rng.integers(0, 2, nv - 2)])  # noqa: E731


@pytest.mark.parametrize("sizes,seg_of", [
    ((1,), ONE), ((2, 3), TWO), ((16,), ONE), ((15, 16, 17), TWO), ((23, 24, 25), ONE), ((31, 32), TWO),
    ((33,), ONE), ((32, 33, 34), TWO), ((63, 64, 65), ONE), ((64, 64, 1), TWO), ((66, 127, 128, 129), ONE),
    ((254, 255), TWO), ((256, 257, 300), ONE), ((300, 20), TWO), ((22000,), ONE)], ids=str)
def test_star_sizes(sizes, seg_of):
    m = fans(sizes, seg_of, seed=len(sizes) + sizes[0])
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    with gale.Context.load(m, device=0, part_vertices=-1) as ctx:
        for mask in (gale.ALL, gale.VT, gale.VT | gale.VV, gale.TT):
            ctx.build(None, mask, gale.MODE_BATCHED)
            ctx.synchronize()
            assert_bulk_equal(ctx.export(mask), expected_bulk(rel, canon, range(m.nclusters), mask))

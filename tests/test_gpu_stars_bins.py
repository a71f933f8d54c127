"""Stars of every length class under plans made for several clusters at once:
test_gpu_stars' meshes have one or two clusters, which one launch builds under
their own plans, while a large mesh runs size bins of unequal clusters at one
block size.  A block size set by the caller keeps the bins' launches.  Also
vertices with more than 255 neighbours of which many are on each side, whose
edge ranks count modulo 256 from minus the lower ones."""
import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk
from test_gpu_stars import fans

pytestmark = pytest.mark.gpu


def spread(K):
    return lambda rng, nv: np.concatenate([np.arange(K), rng.integers(0, K, nv - K)])


def hub(k, above, K, seed=9):
    """A fan of k tets whose first end vertex has `above` ring vertices above
    it (and the second end vertex, the last of all) and the rest below."""
    ring = np.delete(np.arange(k + 2), k + 1 - above)
    h = k + 1 - above
    rng = np.random.default_rng(seed)
    ring = rng.permutation(ring)
    tv = np.array([[h, k + 2, ring[i], ring[i + 1]] for i in range(k)])
    tv = np.take_along_axis(tv, rng.random(tv.shape).argsort(1), 1)[rng.permutation(k)]
    # input order is canonical order within a cluster, clusters one after another
    seg = np.sort(np.concatenate([np.arange(K), rng.integers(0, K, k + 3 - K)]))
    return gen.Mesh(rng.random((k + 3, 3)).astype(np.float32), tv.astype(np.int32), seg.astype(np.int32), K)


MESHES = {
    "short": lambda: fans((1, 2, 3, 5, 7, 8, 12, 15, 16, 16, 17), spread(4), 1),
    "to-24": lambda: fans((17, 20, 23, 24, 24, 25, 9, 4), spread(5), 2),
    "to-32": lambda: fans((24, 25, 28, 31, 32, 32, 33, 2), spread(4), 3),
    "to-64": lambda: fans((33, 40, 48, 63, 64, 64, 20, 1), spread(6), 4),
    "long": lambda: fans((65, 66, 90, 127, 128, 129, 7), spread(3), 5),
    "wide-positions": lambda: fans((255, 256, 257, 300, 12), spread(3), 6),
    "hub-254-up": lambda: hub(400, 254, 1),
    "hub-128-up": lambda: hub(600, 128, 2),
    "hub-3-up": lambda: hub(300, 3, 3),
}


@pytest.mark.parametrize("threads", [64, 128, 512])
@pytest.mark.parametrize("kind", MESHES)
def test_bins_of_unequal_clusters(kind, threads):
    import torch
    m = MESHES[kind]()
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    every = np.arange(m.nclusters, dtype=np.int32)
    with gale.Context.load(m, device=0, part_vertices=-1) as ctx:
        ctx.set_tuning(threads)
        bins = ctx.bins()
        assert not any(b["spill"] for b in bins)
        if kind in ("short", "to-24", "to-32", "to-64"):
            assert any(b["clusters"] > 1 and not b["per_item"] for b in bins), bins
        for mask in (gale.ALL, gale.VT, gale.VV | gale.ET, gale.TT):
            want = expected_bulk(rel, canon, every, mask)
            ctx.build(None, mask, gale.MODE_BATCHED)
            ctx.synchronize()
            assert ctx.last_launch_count() == 1 + len(bins)
            assert_bulk_equal(ctx.export(mask), want)
            lens = ctx.output_lengths(every, mask)
            out = {n: torch.empty(lens[n], dtype=torch.int32, device="cuda") for n in want}
            ctx.build_noalloc(every, mask, out)
            assert_bulk_equal({n: t.cpu().numpy() for n, t in out.items()}, want)


def test_full_builds_under_alternating_masks_read_by_views():
    """A full build's placement is kept while its mask stays the same."""
    m = gen.freudenthal_mesh(10, 64, with_field=False)
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)

    def check(ctx, ids, mask):
        ctx.synchronize()
        for i in (0, len(ids) // 2, len(ids) - 1):
            got = gale.view_to_numpy(ctx.bulk_view(i))
            for name, a in expected_bulk(rel, canon, [ids[i]], mask).items():
                assert np.array_equal(got[name], a), (ids[i], mask, name)

    every = np.arange(m.nclusters, dtype=np.int32)
    some = every[::-2].copy()
    with gale.Context.load(m, device=0) as ctx:
        def full(mask):
            ctx.build(None, mask, gale.MODE_BATCHED)
            check(ctx, every, mask)

        for mask in (gale.VT, gale.ALL, gale.ALL, gale.TT | gale.VV, gale.VT, gale.VT):
            full(mask)
        ctx.build(some, gale.VT, gale.MODE_BATCHED)
        check(ctx, some, gale.VT)
        full(gale.VT)
        ctx.build_export(some, gale.VT, chunks=2)
        full(gale.VT)
        ctx.autotune(gale.ALL, reps=1)
        full(gale.VT)
        ctx.build(None, gale.VT, gale.MODE_PER_CLUSTER)
        check(ctx, every, gale.VT)
        full(gale.VT)
        ctx.set_tuning(64)
        full(gale.VT)

"""What gale_autotune keeps is what runs: either the bins' launches as tuned,
or one launch of all of them, whose block size the bins then report."""
import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk

pytestmark = pytest.mark.gpu


def launches(ctx):
    return ctx.last_launch_count()


@pytest.mark.parametrize("kind", ["grid16", "grid24", "delaunay4000", "delaunay12000"])
def test_the_reported_choice_runs(kind):
    n = int(kind.lstrip("abcdefghijklmnopqrstuvwxyz"))
    m = (gen.freudenthal_mesh(n, 64 if n == 16 else 256, with_field=False) if kind[0] == "g"
         else gen.delaunay_mesh(n, seed=5, with_field=False))
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    with gale.Context.load(m, device=0) as ctx:
        best = ctx.autotune(gale.ALL, reps=2)
        bins = [b for b in ctx.bins() if b["parts"] != -1]
        assert len(bins) > 1
        every = np.arange(m.nclusters, dtype=np.int32)
        for ids in (None, every[::3].copy()):
            ctx.build(ids, gale.ALL, gale.MODE_BATCHED)
            ctx.synchronize()
            assert_bulk_equal(ctx.export(gale.ALL), expected_bulk(rel, canon, every if ids is None else ids))
            if launches(ctx) == 2:  # placement and one build
                assert all(b["threads"] == 512 for b in bins), bins
                assert len({round(x, 6) for x in best if x > 0}) == 1
            elif ids is None:
                assert launches(ctx) == 1 + len(bins)
        ctx.set_tuning(0)  # back to the rule
        ctx.build(None, gale.ALL, gale.MODE_BATCHED)
        ctx.synchronize()
        assert launches(ctx) == 2
        assert_bulk_equal(ctx.export(gale.ALL), expected_bulk(rel, canon, every))

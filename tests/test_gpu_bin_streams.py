"""The streams that several size bins' launches fork to are made when the
mesh is loaded, so that the first build of a context does not pay for them."""
import numpy as np
import pytest

import gen
import paper_2507_15230_gb300 as gale
from plan_util import probe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["grid", "delaunay"])
def test_no_stream_is_made_by_the_first_builds(kind):
    m = (gen.freudenthal_mesh(80, 512, with_field=False) if kind == "grid"
         else gen.delaunay_mesh(60000, 5, with_field=False))
    with gale.Context.load(m, device=0) as ctx:
        nb = sum(b["parts"] != -1 for b in ctx.bins())
        made = probe().probe_bin_streams(ctx._h)
        assert nb > 1 and made == min(nb - 1, 5)
        ids = np.random.default_rng(1).permutation(ctx.K).astype(np.int32)
        ctx.build(ids[: ctx.K - 1], gale.ALL, gale.MODE_BATCHED)
        ctx.build(None, gale.ALL, gale.MODE_BATCHED)
        ctx.synchronize()
        assert probe().probe_bin_streams(ctx._h) == made

"""Registers do not halve the team CTAs an SM holds: 512 threads leave 128
registers a thread for one CTA, and a second one fits with 64.  `ctas` is what
fits at 64 registers."""
import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,teams,ctas", [(128, 4, 2), (128, 2, 4), (64, 4, 4), (64, 8, 2), (32, 8, 4)])
def test_teams_an_sm_holds(threads, teams, ctas):
    m = gen.small_grid(with_field=False)
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    with gale.Context.load(m, device=0) as ctx:
        ctx.set_teams(threads, teams)
        bins = ctx.bins()
        assert all(b["teams"] == teams for b in bins)
        for b in bins:
            by_memory = 233_472 // (b["bytes"] * teams + 1024 + 1632)
            assert min(ctas, by_memory) / 2 < b["ctas_per_sm"] <= min(ctas, by_memory)
        ctx.build(None, gale.ALL, gale.MODE_BATCHED)
        ctx.synchronize()
        assert_bulk_equal(ctx.export(gale.ALL), expected_bulk(rel, canon, np.arange(m.nclusters)))

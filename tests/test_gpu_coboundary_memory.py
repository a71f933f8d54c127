"""Device memory a coboundary call takes: the relations it was asked for (VF
with the sorted numbering is made from VE and EF), the counters and lookups
these need, and the index of the enumeration, no more.  The relations are
also equal to the oracle's when one context is asked for different ones in
turn, so that its scratch grows and is laid out again."""
import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale

pytestmark = pytest.mark.gpu

VE, VF, EF, FT = gale.CB_VE, gale.CB_VF, gale.CB_EF, gale.CB_FT
ORDERS = {"sorted": gale.ENUM_SORTED, "first": gale.ENUM_FIRST_APPEARANCE}


def words(which, order, nv, nt, nE, nF, K):
    """int32 words of a first call."""
    if which & VF and order == "sorted":
        which |= VE | EF
    index = 2 * (nv + 1) + 3 * nE + 1 + 2 * nF
    if order == "first":  # the mesh rows and the lists come from the host
        index += 4 * nt + nv + 3 * nE + 4 * nF + 4 * (K + 1)
    w = {VE: 2 * nv + nE, VF: 2 * nv, EF: 2 * nE + 4 * nF, FT: 2 * nF}
    if which & EF and which & FT:  # FT's slots take the place of EF's lookups
        w[FT] = 0
    if which & VF:
        w[VF] += 2 * nE if order == "sorted" else 3 * nv
    scratch = sum(x for rel, x in w.items() if which & rel)
    counts = max(nv if which & (VE | VF) else 0, nE if which & EF else 0)
    rows = {VE: nv + 2 * nE, VF: nv + 3 * nF, EF: nE + 3 * nF, FT: nF + 4 * nt}
    return index + 1.125 * (scratch + counts + sum(x for rel, x in rows.items() if which & rel)), which


@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("which", [VE, VF, EF, FT, VE | VF, EF | FT, VE | VF | EF | FT])
def test_bytes_of_a_first_call(which, order, monkeypatch):
    import torch
    m = gen.freudenthal_mesh(24, 128, with_field=False)
    with gale.Context.load(m, device=0) as ctx:
        en = ctx.enumerate(ORDERS[order])
        torch.cuda.synchronize()
        taken, alloc = [], torch.cuda.caching_allocator_alloc
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc",
                            lambda n, *a: (taken.append(int(n)), alloc(n, *a))[1])
        ctx.coboundary(which)
        monkeypatch.undo()
        limit, _ = words(which, order, m.nv, len(m.tv), len(en["E"]), len(en["F"]), ctx.K)
        assert 0 < sum(taken) <= 4 * limit + 64 * 1024


@pytest.mark.parametrize("order", ORDERS)
def test_relations_in_turn(order):
    m = gen.freudenthal_mesh(9, 64, jitter=0.3, with_field=False)
    canon = oracle.canonicalize(m.nv, m.tv, m.seg, m.nclusters)
    want = oracle.coboundary(canon, oracle.enumerate_simplices(canon, order))
    with gale.Context.load(m, device=0) as ctx:
        ctx.enumerate(ORDERS[order])
        for which in (FT, VE, EF, EF | FT, VF, VF | FT, VE | VF | EF | FT, FT, VF | EF):
            for name, (off, val) in ctx.coboundary(which).items():
                rows = want[name]
                assert np.array_equal(np.diff(off), [len(r) for r in rows]), (which, name)
                assert np.array_equal(val, np.concatenate(rows)), (which, name)

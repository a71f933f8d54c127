"""The size class draws the lines callers see, so whatever it lets into a
CTA's shared memory must have a build plan that fits there: where the rows
in arrival order would pass the limit, the tight layout takes over."""
import ctypes

import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk
from plan_util import item_plans, probe

TIGHT = 4  # SmemPlan mode bit
COMPACT_FIT, CTA_BYTES = 227 * 1024 - 1664, 227 * 1024
MESHES = ["plate", "plate-fan40", "plate-fan70", "slab"]


def relabel(xyz, tv, seg):
    """Cluster ids without gaps, vertices in random order."""
    seg = np.unique(seg, return_inverse=True)[1]
    p = np.random.default_rng(4).permutation(len(seg))
    return gen.Mesh(xyz[p].astype(np.float32), np.argsort(p)[tv].astype(np.int32), seg[p].astype(np.int32),
                    int(seg.max()) + 1)


def mesh(kind):
    """A mesh whose last cluster has few or no internal tets for its
    vertices: a plate of one layer in a grid, with or without a fan of tets
    around two more vertices (stars over 32 and over 64), or the end slab of
    a Delaunay mesh."""
    if kind == "slab":
        m = gen.delaunay_mesh(60000, 5, with_field=False)
        rank = np.argsort(np.argsort(m.xyz[:, 0], kind="stable"))
        return gen.Mesh(m.xyz, m.tv, (rank * 200 // m.nv).astype(np.int32), 200)
    fan = int(kind[9:] or 0)
    xyz, tv = gen.freudenthal_grid(23, permute=False)
    ijk = np.rint(xyz).astype(int)
    g = ijk // 4
    seg = (g[:, 0] * 6 + g[:, 1]) * 6 + g[:, 2]
    seg[((ijk >= 1) & (ijk <= [20, 20 if fan == 70 else 21, 1])).all(1)] = 1000
    if fan:
        h, ring = len(xyz), len(xyz) + 2 + np.arange(fan + 1)
        tv = np.concatenate([tv, [[h, h + 1, ring[i], ring[i + 1]] for i in range(fan)]])
        xyz = np.concatenate([xyz, np.random.default_rng(1).random((fan + 3, 3))])
        seg = np.concatenate([seg, [1000] * 2, np.arange(fan + 1) // 60])
    return relabel(xyz, tv, seg)


def test_any_class_that_fits_has_a_plan_that_fits():
    rng = np.random.default_rng(7)
    words = probe().probe_caps_words()
    fields = ("blk_words", "nv_own", "n_vt", "n_own", "nv_loc", "nv_nb", "max_deg", "max_vv", "max_e", "max_etv",
              "max_tt", "hcap", "n_tot", "n_star")
    assert words == len(fields)
    for threads in (64, 512, 1024):
        n = 200_000
        nvo = rng.integers(1, 1500, n)
        star = (nvo * rng.uniform(0, 24, n)).astype(int)
        own = (star * rng.random(n) ** 2).astype(int)
        vt = (star * rng.uniform(1, 4, n)).astype(int)
        e = (nvo * rng.uniform(0, 12, n)).astype(int)
        deg = rng.choice([8, 24, 30, 32, 33, 60, 62, 63, 64, 90, 130, 256, 257, 300, 22000], n)
        nb = nvo + (nvo * rng.uniform(0, 3, n)).astype(int)
        c = {"blk_words": rng.integers(12, 20000, n), "nv_own": nvo, "n_vt": vt, "n_own": own, "nv_loc": nb,
             "nv_nb": nb, "max_deg": deg, "max_vv": (nvo * rng.uniform(0, 20, n)).astype(int), "max_e": e,
             "max_etv": (vt * rng.uniform(0, 2, n)).astype(int), "max_tt": 4 * own,
             "hcap": 1 << rng.integers(6, 12, n), "n_tot": star, "n_star": star}
        caps = np.stack([np.asarray(c[f]) for f in fields], 1).astype(np.int32)
        out = np.zeros((n, 3), np.int64)
        probe().probe_caps(caps.ctypes.data_as(ctypes.c_void_p), n, threads, out.ctypes.data_as(ctypes.c_void_p))
        cls, total, mode = out.T
        fits = cls <= CTA_BYTES
        assert (total[fits] <= np.maximum(cls[fits], COMPACT_FIT)).all()
        tight = (mode & TIGHT) != 0
        assert (tight & fits).sum() > 20  # the rule was reached
        assert (total[tight] <= CTA_BYTES).all()


@pytest.mark.parametrize("kind", MESHES)
def test_meshes_at_the_limit(kind):
    with gale.Context.load(mesh(kind), device=-1, part_vertices=-1) as ctx:
        p = item_plans(ctx, 512)
        last = ctx.K - 1
        assert p["class"][last] <= COMPACT_FIT and p["total"][last] <= p["class"][last]
        assert p["mode"][last] & TIGHT
        over = p["total"] > np.maximum(p["class"], COMPACT_FIT)
        assert not (over & (p["class"] <= CTA_BYTES)).any()


@pytest.mark.gpu
def test_the_limit_lies_between_the_constants():
    out = (ctypes.c_int64 * 3)()
    probe().probe_limits(out)
    assert (out[0], out[1]) == (COMPACT_FIT, CTA_BYTES)
    assert COMPACT_FIT <= out[2] <= CTA_BYTES


def bin_of(ctx, k):
    ends = np.cumsum([b["clusters"] for b in ctx.bins()])
    return ctx.bins()[int(np.searchsorted(ends, ctx.bin_members().tolist().index(k), "right"))]


@pytest.mark.gpu
@pytest.mark.parametrize("kind", MESHES)
def test_cluster_at_the_limit_is_built_in_every_form(kind):
    import torch
    m = mesh(kind)
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    last = m.nclusters - 1
    with gale.Context.load(m, device=0, part_vertices=-1, cache_budget_bytes=64 << 20) as ctx:
        others = [k for k in range(last) if not bin_of(ctx, k)["spill"]]
        ids = np.array(others[:1] + [last] + others[1:3], np.int32)
        for threads in (0, 64, 512, 1024):
            ctx.set_tuning(threads)
            assert not bin_of(ctx, last)["spill"] and bin_of(ctx, last)["per_item"]
            for mask in (gale.ALL, gale.VT, gale.VV | gale.TT, gale.ET):
                want = expected_bulk(rel, canon, ids, mask)
                lens = ctx.output_lengths(ids, mask)
                out = {n: torch.empty(lens[n], dtype=torch.int32, device="cuda") for n in want}
                ctx.build_noalloc(ids, mask, out)
                assert_bulk_equal({n: t.cpu().numpy() for n, t in out.items()}, want)
                for mode in (gale.MODE_BATCHED, gale.MODE_PER_CLUSTER):
                    ctx.build(ids, mask, mode)
                    ctx.synchronize()
                    assert_bulk_equal(ctx.export(mask), want)
        ctx.set_tuning(0)
        ctx.autotune(gale.ALL, reps=1)
        ctx.build(None, gale.ALL, gale.MODE_BATCHED)
        ctx.synchronize()
        assert_bulk_equal(ctx.export(gale.ALL), expected_bulk(rel, canon, range(m.nclusters)))
        v = ctx.request(last, gale.ALL, timeout_ns=20_000_000_000)
        got = gale.view_to_numpy(v)
        ctx.release(v)
        for name, a in expected_bulk(rel, canon, [last]).items():
            assert np.array_equal(got[name], a), name

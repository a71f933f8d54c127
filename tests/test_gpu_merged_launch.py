"""Short lists built by one launch, each item under its own plan.

A size bin's plan is made from the maxima over its members, and that plan
can be smaller than a member's own: one longer star takes the padded rows
away from the whole bin.  The launch of a short list asks for the largest
member's plan, so that is what the kernels' limit has to allow."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import gen
import oracle
import paper_2507_15230_gb300 as gale
from parity_util import assert_bulk_equal, expected_bulk
from plan_util import item_plans, merged_total, probe

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def two_boxes(split=4):
    """A 16^3 Freudenthal grid with two large flat clusters inside it, 5 x 9
    x 9 and 4 x 9 x 9 vertices, among blocks of up to 4 x 4 x 4.  Four of
    the tets at one vertex of the smaller cluster are split at their
    centres, which lengthens its star from 24 to 32.  The two have the
    highest ids, and so few internal tets for their vertices."""
    xyz, tv = gen.freudenthal_grid(16, permute=False)
    ijk = np.rint(xyz).astype(int)
    b = ijk // 4
    seg = (b[:, 0] * 5 + b[:, 1]) * 5 + b[:, 2]
    seg[((ijk >= 1) & (ijk <= [5, 9, 9])).all(1)] = 500
    seg[((ijk >= [7, 1, 1]) & (ijk <= [10, 9, 9])).all(1)] = 501
    mid = np.flatnonzero((ijk == [9, 4, 4]).all(1))[0]
    add, new = [], []
    for t in np.flatnonzero((tv == mid).any(1))[:split]:
        v, c = tv[t].copy(), len(xyz) + len(add)
        add.append(xyz[v].mean(0))
        rows = [np.where(np.arange(4) == s, c, v) for s in range(4)]
        tv[t] = rows[0]
        new += rows[1:]
    xyz = np.concatenate([xyz, np.array(add, np.float32)])
    tv = np.concatenate([tv, np.array(new, np.int32)])
    seg = np.unique(np.concatenate([seg, np.full(split, 501)]), return_inverse=True)[1]
    p = np.random.default_rng(2).permutation(len(xyz))
    q = np.argsort(p)
    return gen.Mesh(xyz[p], q[tv].astype(np.int32), seg[p].astype(np.int32), int(seg.max()) + 1)


def test_a_bin_can_take_less_than_its_member():
    with gale.Context.load(two_boxes(), device=-1, part_vertices=-1) as ctx:
        p, big, starred = item_plans(ctx, 512), ctx.K - 2, ctx.K - 1
        assert p["max_deg"][[big, starred]].tolist() == [24, 32]
        assert merged_total(ctx, [big, starred], 512) < p["total"][big]
        assert p["total"][:big].max() < p["total"][starred] < p["total"][big]


def build_all_ways():
    m = two_boxes()
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    big = m.nclusters - 2
    ids = np.array([big, 5, 40], np.int32)
    with gale.Context.load(m, device=0, part_vertices=-1) as ctx:
        ends = np.cumsum([b["clusters"] for b in ctx.bins()])
        top = ctx.bins()[int(np.searchsorted(ends, ctx.bin_members().tolist().index(big), "right"))]
        assert top["clusters"] == 2 and not top["per_item"], top
        import torch
        want = expected_bulk(rel, canon, ids)
        lens = ctx.output_lengths(ids, gale.ALL)
        out = {n: torch.empty(lens[n], dtype=torch.int32, device="cuda") for n in gale.ARRAYS}
        ctx.build_noalloc(ids, gale.ALL, out)
        assert_bulk_equal({n: t.cpu().numpy() for n, t in out.items()}, want)
        ctx.build(ids, gale.ALL, gale.MODE_BATCHED)
        ctx.synchronize()
        assert_bulk_equal(ctx.export(gale.ALL), want)
        assert_bulk_equal(ctx.build_export(ids, gale.ALL, chunks=1), want)


@pytest.mark.gpu
def test_list_with_the_largest_member_in_a_fresh_process():
    """The limit belongs to the process and only grows, so nothing larger
    may have been loaded before."""
    r = subprocess.run([sys.executable, "-c", "import test_gpu_merged_launch as t; t.build_all_ways()"], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")])),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]


def with_third_tets(m, clusters):
    """m with one more vertex per listed cluster, on a triangle between two of
    its internal tets: the triangle then lies in three tets."""
    tv, seg, xyz = [m.tv], [m.seg], [m.xyz]
    own = (m.seg[m.tv] == np.arange(m.nclusters)[:, None, None]).all(2)
    for i, k in enumerate(clusters):
        inside = m.tv[own[k]]
        faces = np.sort(inside[:, [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]].reshape(-1, 3), 1)
        f, n = np.unique(faces, axis=0, return_counts=True)
        tv.append([[*f[np.argmax(n == 2)], m.nv + i]])
        seg.append([k])
        xyz.append(m.xyz[f[np.argmax(n == 2)]].mean(0, keepdims=True))
    return gen.Mesh(np.concatenate(xyz), np.concatenate(tv).astype(np.int32), np.concatenate(seg).astype(np.int32),
                    m.nclusters)


def test_non_manifold_members_can_take_more_than_their_bin():
    m = two_boxes()
    with gale.Context.load(with_third_tets(m, [m.nclusters - 2, m.nclusters - 1]), device=-1, part_vertices=-1) as ctx:
        p, big, starred = item_plans(ctx, 512), ctx.K - 2, ctx.K - 1
        assert merged_total(ctx, [big, starred], 512) < p["total"][big]


@pytest.mark.gpu
def test_per_item_launches_hold_their_largest_member():
    """Non-manifold clusters share a per-item bin, whose launch has to take
    the largest member's own plan."""
    m = two_boxes()
    m = with_third_tets(m, [m.nclusters - 2, m.nclusters - 1])
    canon, rel = oracle.build_all(m.nv, m.tv, m.seg, m.nclusters)
    out = (ctypes.c_int64 * 2)()
    with gale.Context.load(m, device=0, part_vertices=-1) as ctx:
        for threads in (0, 256, 1024):
            ctx.set_tuning(threads)
            probe().probe_per_item(ctx._h, out)
            assert out[0] >= 1 and out[1] == 0
            ctx.build(None, gale.ALL, gale.MODE_BATCHED)
            ctx.synchronize()
            assert_bulk_equal(ctx.export(gale.ALL), expected_bulk(rel, canon, range(m.nclusters)))


@pytest.mark.gpu
def test_planned_occupancy_is_the_devices():
    """The kernel's static shared memory counts: two CTAs of 115,200 bytes
    each do not fit an SM beside it."""
    out = (ctypes.c_int32 * 2)()
    with gale.Context.load(gen.small_grid(with_field=False), device=0) as ctx:
        for total in (0, 16, 57_344, 74_000, 113_000, *range(114_000, 116_000, 16), 150_000, 230_000, 230_816):
            probe().probe_merged_ctas(ctx._h, total, out)
            assert out[0] == out[1] >= 1, total
        probe().probe_merged_ctas(ctx._h, 115_200, out)
        assert out[0] == 1

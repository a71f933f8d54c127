"""The work a user of the producer has it do, as measured cases.

Every relation array is whole numbers, so no case has a floating output.  A
case is a mesh (a jittered Freudenthal grid or a Delaunay mesh of a Gaussian
mixture, from the seeded generator the tests and the benchmark use) and one
way of asking for its relations:

  build      every cluster's relations, batched, left on the device
  list       the same for a list of clusters
  noalloc    a leader's batch of clusters into the caller's own device arrays
  export     every cluster's relations in the caller's pinned host memory
  serve      one consumer walking over clusters through the request loop,
             copying each view to the host, under a budget the walk exceeds
  coboundary VE, VF, EF, FT of the whole mesh
  gradient   what the discrete gradient reads: the enumeration, VE, VF and VT
"""
import ctypes

import numpy as np
import torch

import gen
import paper_2507_15230_gb300 as gale

CP = gale.VT | gale.VV | gale.TT  # what the critical-point consumer asks for
BITS = (gale.VT, gale.VV, gale.ET, gale.TT)


def listed():
    return [
        # one segment on demand: the smallest call, all latency
        dict(name="noalloc-1", kind="noalloc", mesh="grid", n=32, cap=512, mask=CP, count=1),
        # a leader's batch of queued requests on an unstructured mesh with uneven leaves
        dict(name="noalloc-batch", kind="noalloc", mesh="delaunay", n=20000, cap=2048, mask=gale.ALL, count=37),
        # the smallest whole mesh (24,576 tets in 128 leaves of <= 64 vertices)
        dict(name="grid16", kind="build", mesh="grid", n=16, cap=64, mask=gale.ALL, tune=False),
        # a medium grid under the critical-point consumer's mask
        dict(name="grid64-cp", kind="build", mesh="grid", n=64, cap=512, mask=CP, tune=False),
        # an ordinary mesh with a ragged size, untuned
        dict(name="grid101", kind="build", mesh="grid", n=101, cap=512, mask=gale.ALL, tune=False),
        # the at-scale, Stent-shaped grid (100.7M tets), tuned as the benchmark does
        dict(name="grid256", kind="build", mesh="grid", n=256, cap=512, mask=gale.ALL, tune=True),
        # an unstructured mesh with uneven leaves, some cut into parts
        dict(name="delaunay200k", kind="build", mesh="delaunay", n=200000, cap=2048, mask=gale.ALL, tune=True),
        # a quarter of a mesh's clusters in arbitrary order
        dict(name="list80", kind="list", mesh="grid", n=80, cap=512, mask=gale.ALL, share=0.25),
        # end to end into host memory
        dict(name="export96", kind="export", mesh="grid", n=96, cap=512, mask=gale.ALL),
        # a single consumer (kd-order walk with jumps) through the request loop
        dict(name="serve64", kind="serve", mesh="grid", n=64, cap=512, mask=CP, count=96),
        # the coboundary relations of an ordinary mesh
        dict(name="coboundary128", kind="coboundary", mesh="grid", n=128, cap=512, which=15),
        # the relations of the discrete gradient, from a loaded mesh
        dict(name="gradient48", kind="gradient", mesh="grid", n=48, cap=512),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "list", "list", "noalloc", "noalloc", "export", "serve",
                       "coboundary", "coboundary", "gradient"])
    top = {"build": 200, "list": 128, "noalloc": 64, "export": 96, "serve": 64, "coboundary": 128, "gradient": 64}[kind]
    c = dict(kind=kind)
    if kind != "serve" and rng.random() < 0.35:
        c.update(mesh="delaunay", n=_log(rng, 3000, 20000 if kind == "noalloc" else 200000), cap=2048)
    else:
        c.update(mesh="grid", n=_log(rng, 32 if kind == "serve" else 12, top), cap=rng.choice([64, 128, 256, 512, 512]))
    if kind in ("build", "list", "noalloc", "export"):
        c["mask"] = rng.choice([gale.ALL, gale.ALL, CP, gale.VT | gale.VV, gale.ET, gale.TT, gale.VT | gale.ET])
    if kind == "serve":
        c["mask"] = rng.choice([CP, gale.ALL])
    if kind == "build":
        c["tune"] = rng.random() < 0.3
    if kind == "list":
        c["share"] = round(0.02 * 50 ** rng.random(), 4)
    if kind in ("noalloc", "serve"):
        c["count"] = _log(rng, 1, 200) if kind == "noalloc" else _log(rng, 12, 48)
    if kind == "coboundary":
        c["which"] = rng.choice([15, 15, gale.CB_VE | gale.CB_VF, gale.CB_FT, gale.CB_EF | gale.CB_FT])
    return c


_made = {}  # the last generated mesh: its vertex ids are drawn again for every seed


def _mesh(case, seed):
    """A grid of the seed's jitter and vertex ids where a whole mesh is asked
    for (its totals do not depend on them); otherwise one mesh of the case's
    size under vertex ids drawn from the seed, so that the lengths of the
    listed clusters' arrays are the case's own."""
    if case["mesh"] == "grid" and "share" not in case and "count" not in case:
        return gen.freudenthal_mesh(case["n"], case["cap"], seed=1 + seed, jitter=0.3, with_field=False)
    key = (case["mesh"], case["n"], case["cap"])
    if key not in _made:
        _made.clear()
        if case["mesh"] == "grid":
            _made[key] = gen.freudenthal_mesh(case["n"], case["cap"], seed=3, jitter=0.3, with_field=False)
        else:
            _made[key] = gen.delaunay_mesh(case["n"], 5, kd_cap=case["cap"], with_field=False)
    m = _made[key]
    p = np.random.default_rng(seed).permutation(m.nv).astype(np.int32)
    seg = np.empty_like(m.seg)
    seg[p] = m.seg
    return gale.Mesh(None, p[m.tv], seg, m.nclusters)


class _State:
    """What a user's program holds between calls: the context, its lists and
    buffers, and tensors over the library's device arrays (made again only
    when the library hands out other ones)."""

    def __init__(self, case, seed):
        kind = case["kind"]
        rng = np.random.default_rng(case["n"])  # which clusters are asked for: the case's, for any seed
        mesh = _mesh(case, seed)
        self.kind, self.mask, self.case = kind, case.get("mask", gale.ALL), case
        budget = 3 << 19 if kind == "serve" else 0
        if kind == "serve" and self.mask == gale.ALL:
            budget *= 2
        precond = {"coboundary": gale.ALL, "gradient": gale.VT | gale.ET}.get(kind, self.mask)
        self.ctx = ctx = gale.Context.load(mesh, precondition_mask=precond, cache_budget_bytes=budget)
        self.held = {}
        if kind == "build" and case["tune"]:
            ctx.autotune(self.mask)
        elif kind == "list":
            n = max(1, int(round(case["share"] * ctx.K)))
            self.ids = rng.permutation(ctx.K)[:n].astype(np.int32)
        elif kind == "noalloc":
            ok = np.ones(ctx.K, bool)
            at, members = 0, ctx.bin_members()
            for b in ctx.bins():  # clusters of global-scratch bins are refused
                m = members[at:at + b["clusters"]]
                at += b["clusters"]
                if b["spill"]:
                    ok[m[m < ctx.K]] = False
            self.ids = rng.permutation(np.flatnonzero(ok))[:case["count"]].astype(np.int32)
            lens = ctx.output_lengths(self.ids, self.mask)
            self.out = {n: torch.empty(lens[n], dtype=torch.int32, device="cuda")
                        for n, r in zip(gale.ARRAYS, gale.ARRAY_REL) if self.mask & r}
        elif kind == "export":
            lens = ctx.output_lengths(None, self.mask)
            self.out = {n: torch.empty(lens[n], dtype=torch.int32, pin_memory=True).numpy()
                        for n, r in zip(gale.ARRAYS, gale.ARRAY_REL) if self.mask & r}
        elif kind == "serve":
            # a walk in kd order with jumps, over distinct clusters
            todo, walk, k = set(range(ctx.K)), [], int(rng.integers(ctx.K))
            while todo and len(walk) < case["count"]:
                if k not in todo or rng.random() < 0.1:
                    k = sorted(todo)[int(rng.integers(len(todo)))]
                todo.remove(k)
                walk.append(k)
                k += 1
            ctx.serve_configure(gale.SERVE_LOOP, idle_us=200, loop_ctas=16)
            I_V, I_T, sizes = ctx.intervals()
            self.walk, self.out = walk, {}
            for k in walk:  # the consumer's own row buffers
                nvo, nown = int(I_V[k + 1] - I_V[k]), int(I_T[k + 1] - I_T[k])
                vt, vv, e, et, tt = (int(x) for x in sizes[k])
                n = dict(zip(gale.ARRAYS, (nvo + 1, vt, nvo + 1, vv, nvo + 1, e, e + 1, et, nown + 1, tt)))
                self.out[k] = {a: np.empty(n[a], np.int32) for a, r in zip(gale.ARRAYS, gale.ARRAY_REL) if self.mask & r}
        elif kind == "coboundary":
            if gale.load_library().gale_enumerate(ctx._h, gale.ENUM_SORTED) != 0:
                raise RuntimeError("enumeration failed")

    def tensor(self, key, ptr, n):
        got = self.held.get(key)
        if got is None or got[0] != (ptr, n):
            got = self.held[key] = ((ptr, n), gale.device_tensor(ptr, n))
            got[1].owner = self.ctx  # the array is the context's: it lives as long as the tensor
        return got[1]

    def bulk(self):
        ptrs, lens = self.ctx.bulk_arrays()
        return {a: self.tensor(a, ptrs[a], lens[a]) for a in gale.ARRAYS if lens[a]}

    def coboundary(self, which):
        cb = gale.Coboundary()
        lib = gale.load_library()
        if lib.gale_build_coboundary(self.ctx._h, which, ctypes.byref(cb)) != 0:
            raise RuntimeError(lib.gale_last_error().decode())
        out = {}
        for i, name in enumerate(("VE", "VF", "EF", "FT")):
            if which & (1 << i):
                out[name + "_off"] = self.tensor(name + "_off", cb.off[i], int(cb.rows[i]) + 1)
                out[name] = self.tensor(name, cb.val[i], int(cb.len[i]))
        return out


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    ctx = s.ctx
    if s.kind == "build":
        ctx.build(None, s.mask, gale.MODE_BATCHED)
        return s.bulk()
    if s.kind == "list":
        ctx.build(s.ids, s.mask, gale.MODE_BATCHED)
        return s.bulk()
    if s.kind == "noalloc":
        ctx.build_noalloc(s.ids, s.mask, s.out)
        return s.out
    if s.kind == "export":
        return ctx.build_export(None, s.mask, s.out)
    if s.kind == "serve":
        flat = {}
        for k in s.walk:
            v = ctx.request(k, s.mask)
            for a, dst in s.out[k].items():
                ctx.copy_to_host(getattr(v, a), dst.size, dst)
            ctx.release(v)
        for a in s.out[s.walk[0]]:
            flat[a] = np.concatenate([s.out[k][a] for k in s.walk])
        return flat
    if s.kind == "coboundary":
        return s.coboundary(s.case["which"])
    en = ctx.enumerate(gale.ENUM_SORTED)
    out = s.coboundary(gale.CB_VE | gale.CB_VF)
    ctx.build(None, gale.VT, gale.MODE_BATCHED)
    return {**out, **s.bulk(), **en}


def exact(case, seed):
    return None  # every output is whole numbers


def _mesh_counts(case):
    """Vertices, edges and tets: exact for the grid; a Delaunay mesh of this
    point distribution has about 6.72 tets a point, and V - E + F - T = 1."""
    n = case["n"]
    if case["mesh"] == "grid":
        return (n + 1) ** 3, 7 * n ** 3 + 9 * n ** 2 + 3 * n, 6 * n ** 3
    return n, n + int(6.72 * n), int(6.72 * n)


def _relation_words(mask, v, e, t):
    """int32 words of the relations (rows and their offsets)."""
    return ((4 * t + v if mask & gale.VT else 0) + (2 * e + v if mask & gale.VV else 0) +
            (6 * t + 2 * e + v if mask & gale.ET else 0) + (5 * t if mask & gale.TT else 0))


def work(case):
    """Each input (the tets' vertices, the vertices' segments; for the
    coboundary pass the enumeration) read once, each output written once."""
    v, e, t = _mesh_counts(case)
    f = 2 * t + (6 * case["n"] ** 2 if case["mesh"] == "grid" else 0)
    kind = case["kind"]
    read = 4 * (4 * t + v)
    if kind in ("coboundary", "gradient"):
        which = case.get("which", gale.CB_VE | gale.CB_VF)
        words = ((2 * e + v if which & gale.CB_VE else 0) + (3 * f + v if which & gale.CB_VF else 0) +
                 (3 * f + e if which & gale.CB_EF else 0) + (4 * t + f if which & gale.CB_FT else 0))
        lists = 2 * e + 3 * f
        if kind == "coboundary":
            read = 4 * (lists + (4 * t if which & gale.CB_FT else 0))
        else:
            words += lists + _relation_words(gale.VT, v, e, t)
        return {"bytes": read + 4 * words, "flops": 0}
    share = case.get("share", 1.0)
    if kind in ("noalloc", "serve"):
        # leaves hold a little over half of the cap on the grid; a Delaunay
        # leaf a few hundred vertices
        leaf = case["cap"] * 0.55 if case["mesh"] == "grid" else 190
        share = min(1.0, case["count"] * leaf / v)
    return {"bytes": int(share * (read + 4 * _relation_words(case["mask"], v, e, t))), "flops": 0}

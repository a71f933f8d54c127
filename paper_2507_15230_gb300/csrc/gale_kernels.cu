// Producer kernels: per-cluster VT, VV, ET and TT as canonical sorted CSR.
//
// One CTA builds one cluster at a time (persistent CTAs take clusters from a
// ticket counter; the per-cluster baseline launches one CTA per cluster).
// The rows of the cluster's working set - its internal tets, its external
// tets T_ex and its face halo (Section 4.3, "Initialization"), as 16-bit
// local rows - arrive in shared memory by one bulk copy, and every relation
// is built there.  Each phase spreads its work evenly over all threads of the
// block (over tets, bitmap words, VT incidences, edges or internal tets), so
// the block size is free of the cluster's vertex count; the outputs leave
// through shared-memory staging with one thread per element (coalesced),
// except TT's rows of at most four entries, stored straight out.
//
//  B. VT (Section 4.6 / Algorithm 1: iterate the segment's tets and test
//     each vertex against the segment interval): every incidence of an own
//     vertex takes a slot of that vertex's row by one returning atomic (the
//     paper's atomicPush, Algorithm 2), and the rows, in arrival order, are
//     then sorted in registers: a thread sorts two rows of up to 32 tets at
//     once, in the halves of 16-bit pairs, by a merge network.
//  C. VV and the edges (x, w), x < w, that an own vertex x owns:
//     - C1, in B's pass over the tets: the other vertices of every tet of
//       VT(x) are ORed into a bitmap of x over the cluster's vertex universe;
//       local order is canonical order, so the bitmap read in bit order is
//       VV(x), sorted and deduplicated, and its bits above x are the upper
//       endpoints w;
//     - C2, per own vertex: the row lengths, four offsets by one block scan,
//       and for each bitmap word the number of neighbours before it, so that
//       an edge's index is one popcount away; then the VV rows, read out of
//       the bitmaps while B's rows are sorted;
//     - C3, per tet: bit j is set in the tet mask of each edge (x, w) of the
//       tet, the j-th of VT(x); a mask read in bit order is ET(x, w);
//     - C5, per internal tet (a, b, c, d): the AND of the masks of two edges
//       (a, w1), (a, w2) holds the two tets of the face (a, w1, w2); the face
//       (b, c, d) is matched the same way inside VT(b) when b is own;
//     - C4, per edge: the mask bits become the ET rows.
//  D. TT (Table 1; the paper gives no kernel for it) for the faces (b, c, d)
//     of internal tets (a, b, c, d) with no own vertex: a small
//     open-addressing hash of those faces is probed with the faces of the
//     halo tets.
//  E. TT rows from the four face links, sorted by canonical id.  A face with
//     a second partner (a triangle in three or more tets) marks the cluster
//     instead, whose rows then come from E', a general pass over the block
//     (compiled into every kernel but the hot shared-memory one, as is the
//     tight layout: the host runs clusters that need either from per-item
//     bins; the counting pass reports the non-manifold ones).  Parts of cut clusters report it as an error.
//
// The counting mode runs the same passes without writes and returns the
// exact sizes the host uses to place outputs and to admit cache entries.
//
// What bounds it: nothing here is a contraction, and DRAM is busy for a
// fifth of the time.  The time followed the warp instructions of a cluster
// (about 0.011 ms per thousand at 128^3, over every phase), with the shared-
// memory pipe close behind, so the passes above are chosen for few
// instructions per incidence.  Measured at 268 vertices / 1,536 tets a
// cluster (2 CTAs of 512 threads an SM): with a stable fill from per-warp
// counters and lane masks in B, C1 as a pass of its own, edge ranks recomputed
// in C5 and a scan over the edges in C4, 107.6k warp instructions, 29.8k
// shared wavefronts and 9.07 ms per 256^3 build; with the passes above 70.7k,
// 24.4k and 7.06 ms.  What is left waits on the shared-memory pipe (76 % of
// its peak, issue 58 %) and barriers, so loads go before the atomics and
// stores they may alias, a few steps at a time: 77k, 23.5k and 6.85 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "gale_internal.h"

namespace gale {

namespace {

constexpr int kScanWords = 128;  // scan scratch: a word per warp (up to 32) and value
// words of the block's header, free once every thread has read it
constexpr int kFlagNonManifold = 0, kFlagLong = 1, kScanTotals = 4;
constexpr unsigned FULL = 0xffffffffu;
constexpr int kWaitLimit = 1 << 22;  // polls of the block copy's barrier before giving up

struct Smem {
    int32_t *scan;
    int32_t *blk;
    int32_t *vt_off;
    uint16_t *vt_list;
    int32_t *c_vv, *c_e;
    uint16_t *fill;       // r2 and nbr
    uint16_t *nbr;
    uint8_t *jpos;        // until C5
    int32_t *eo;          // jpos (phase C4)
    uint32_t *emask;      // r2
    uint16_t *st_v;       // r2
    int32_t *et_b;        // r2
    uint16_t *long_rows;  // r2
    uint32_t *bm;         // r1 (until C3)
    uint8_t *pre;         // r1 (until C3)
    uint16_t *st_et;      // r1 (phase C4)
    uint16_t *ex;         // r1 (phase C4)
    uint32_t *hash;       // r1 (phase D)
    int32_t *tcnt;        // r1 (phases D, E)
    uint16_t *st_tt;      // r1 (phase E')
};

__device__ __forceinline__ Smem carve(char *base, const SmemPlan &p) {
    Smem s;
    s.scan = reinterpret_cast<int32_t *>(base + p.scan);
    s.blk = reinterpret_cast<int32_t *>(base + p.blk);
    s.vt_off = reinterpret_cast<int32_t *>(base + p.vt_off);
    s.vt_list = reinterpret_cast<uint16_t *>(base + p.vt_list);
    s.c_vv = reinterpret_cast<int32_t *>(base + p.c_vv);
    s.c_e = reinterpret_cast<int32_t *>(base + p.c_e);
    s.fill = reinterpret_cast<uint16_t *>(base + p.fill);
    s.nbr = reinterpret_cast<uint16_t *>(base + p.nbr);
    s.jpos = reinterpret_cast<uint8_t *>(base + p.jpos);
    s.eo = reinterpret_cast<int32_t *>(base + p.jpos);
    s.emask = reinterpret_cast<uint32_t *>(base + p.r2);
    s.st_v = reinterpret_cast<uint16_t *>(base + p.r2);
    s.et_b = reinterpret_cast<int32_t *>(base + p.et_b);
    s.long_rows = reinterpret_cast<uint16_t *>(base + p.long_rows);
    s.bm = reinterpret_cast<uint32_t *>(base + p.r1);
    s.pre = reinterpret_cast<uint8_t *>(base + p.pre);
    s.st_et = reinterpret_cast<uint16_t *>(base + p.r1);
    s.ex = reinterpret_cast<uint16_t *>(base + p.ex);
    s.hash = reinterpret_cast<uint32_t *>(base + p.r1);
    s.tcnt = reinterpret_cast<int32_t *>(base + p.tcnt);
    s.st_tt = reinterpret_cast<uint16_t *>(base + p.st_tt);
    return s;
}

// ---- bulk copy into shared memory, completion on an mbarrier ----
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    // order this CTA's earlier generic accesses of dst before the async write
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0u;
}
// bulk prefetch of [p, p + bytes) into L2 (16-byte aligned, multiple of 16)
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// bounded wait for the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    for (int i = 0; i < kWaitLimit; ++i)
        if (mbar_test(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ uint32_t vtx(uint2 r, int s) {
    uint32_t w = (s < 2) ? r.x : r.y;
    return (s & 1) ? (w >> 16) : (w & 0xffffu);
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Who builds a cluster: the whole CTA, or a team - a warp-aligned slice of
// it with a named barrier of its own (several small clusters per CTA).
struct BlockTeam {
    __device__ __forceinline__ int nt() const { return blockDim.x; }
    __device__ __forceinline__ int tid() const { return threadIdx.x; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    __device__ __forceinline__ int sync_or(int p) const { return __syncthreads_or(p); }
};
struct SliceTeam {
    int n;    // threads (a multiple of 32)
    int t;    // this thread's index in the team
    int bar;  // named barrier id (1..15; 0 is __syncthreads')
    __device__ __forceinline__ int nt() const { return n; }
    __device__ __forceinline__ int tid() const { return t; }
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(n) : "memory"); }
    __device__ __forceinline__ int sync_or(int p) const {
        int r;
        asm volatile(
            "{\n\t.reg .pred pin, pout;\n\tsetp.ne.s32 pin, %1, 0;\n\t"
            "bar.red.or.pred pout, %2, %3, pin;\n\tselp.s32 %0, 1, 0, pout;\n\t}"
            : "=r"(r)
            : "r"(p), "r"(bar), "r"(n)
            : "memory");
        return r;
    }
};

// Exclusive scan of one value per thread over the team (any multiple of 32
// threads up to 1024); scr needs 33 words.  Two team barriers.
template <class Team>
__device__ __forceinline__ int block_scan_thread(const Team &tm, int v, int32_t *scr, int *total) {
    const int nw = tm.nt() >> 5;
    const int lane = tm.tid() & 31, warp = tm.tid() >> 5;
    const int incl = warp_incl_scan(v, lane);
    if (lane == 31) scr[warp] = incl;
    tm.sync();
    if (warp == 0) {
        const int w = lane < nw ? scr[lane] : 0;
        const int wi = warp_incl_scan(w, lane);
        if (lane < nw) scr[lane] = wi - w;
        if (lane == 31) scr[32] = wi;
    }
    tm.sync();
    *total = scr[32];
    return scr[warp] + incl - v;
}

// Exclusive scans of four values per thread over the team, in place; totals
// to t[0..3], by way of tot[0..3].  scr needs kScanWords words.
template <class Team>
__device__ __forceinline__ void block_scan4(const Team &tm, int &a, int &b, int &c, int &d, int32_t *scr, int32_t *tot,
                                            int *t) {
    const int nw = tm.nt() >> 5;
    const int lane = tm.tid() & 31, warp = tm.tid() >> 5;
    const int ia = warp_incl_scan(a, lane), ib = warp_incl_scan(b, lane);
    const int ic = warp_incl_scan(c, lane), id = warp_incl_scan(d, lane);
    if (lane == 31) {
        scr[warp] = ia;
        scr[32 + warp] = ib;
        scr[64 + warp] = ic;
        scr[96 + warp] = id;
    }
    tm.sync();
    for (int s = warp; s < 4; s += nw) {  // a warp per value
        const int w = lane < nw ? scr[32 * s + lane] : 0;
        const int wi = warp_incl_scan(w, lane);
        if (lane < nw) scr[32 * s + lane] = wi - w;
        if (lane == 31) tot[s] = wi;
    }
    tm.sync();
#pragma unroll
    for (int s = 0; s < 4; ++s) t[s] = tot[s];
    a = scr[warp] + ia - a;
    b = scr[32 + warp] + ib - b;
    c = scr[64 + warp] + ic - c;
    d = scr[96 + warp] + id - d;
}

// p[0 .. n) = v over the team, 16 bytes a store (p is 16-byte aligned: every
// region of the plan is).
template <class Team>
__device__ __forceinline__ void fill_words(const Team &tm, uint32_t *p, int n, uint32_t v) {
    uint4 *q = reinterpret_cast<uint4 *>(p);
    const int n4 = n >> 2;
    const uint4 v4 = make_uint4(v, v, v, v);
    for (int i = tm.tid(); i < n4; i += tm.nt()) q[i] = v4;
    for (int i = 4 * n4 + tm.tid(); i < n; i += tm.nt()) p[i] = v;
}

// Length of each thread's contiguous range when n items are split over the
// team: odd, so that neighbouring threads start in different banks.
template <class Team>
__device__ __forceinline__ int range_len(const Team &tm, int n) {
    const int per = (n + tm.nt() - 1) / tm.nt();
    return per > 1 ? (per | 1) : per;
}

// dst[j] = f(j) for j < n over the team, four loads in flight per thread
// before their stores (the values come through L2 from the block's maps).
template <class Team, typename F>
__device__ __forceinline__ void copy_out(const Team &tm, int32_t *__restrict__ dst, int n, F f) {
    const int NT = tm.nt();
    int j = tm.tid();
    for (; j + 3 * NT < n; j += 4 * NT) {
        const int32_t a = f(j), b = f(j + NT), c = f(j + 2 * NT), d = f(j + 3 * NT);
        dst[j] = a;
        dst[j + NT] = b;
        dst[j + 2 * NT] = c;
        dst[j + 3 * NT] = d;
    }
    for (; j < n; j += NT) dst[j] = f(j);
}

// Exclusive scan in place of a[0..n); returns the total.  Ends synced.
template <class Team>
__device__ int block_scan_array(const Team &tm, int32_t *a, int n, int32_t *scr) {
    const int per = range_len(tm, n);
    const int b = min(n, tm.tid() * per);
    const int e = min(n, b + per);
    int s = 0;
    for (int i = b; i < e; ++i) s += a[i];
    int total;
    int run = block_scan_thread(tm, s, scr, &total);
    for (int i = b; i < e; ++i) {
        const int v = a[i];
        a[i] = run;
        run += v;
    }
    tm.sync();
    return total;
}

// Hash of a face, its three 16-bit ids as (first, second | third << 16).
__device__ __forceinline__ uint32_t face_hash(uint2 key) {
    const uint32_t h = key.y * 0x9E3779B1u + key.x * 0x85EBCA77u;
    return h ^ (h >> 15);
}

// number of local vertex ids two packed rows have in common
__device__ __forceinline__ int shared_vertices(uint2 a, uint2 b) {
    const uint32_t b0 = b.x & 0xffffu, b1 = b.x >> 16, b2 = b.y & 0xffffu, b3 = b.y >> 16;
    int c = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const uint32_t v = vtx(a, s);
        c += (v == b0) + (v == b1) + (v == b2) + (v == b3);
    }
    return c;
}

// compare-exchange of keys a, b carrying payloads pa, pb
__device__ __forceinline__ void cswap2(int32_t &a, int32_t &b, uint32_t &pa, uint32_t &pb) {
    const bool sw = b < a;
    const int32_t ka = sw ? b : a, kb = sw ? a : b;
    const uint32_t qa = sw ? pb : pa, qb = sw ? pa : pb;
    a = ka;
    b = kb;
    pa = qa;
    pb = qb;
}

// hash entries: bits [0, 17) = internal-tet index + 1, bits [17, 32) =
// number of other tets matched to the face
constexpr uint32_t kRefMask = (1u << 17) - 1u;
constexpr uint32_t kMatch = 1u << 17;

template <int N>
struct IntC {
    static constexpr int value = N;
};

// stars larger than this count their tets and ET entries in two words
constexpr int32_t kMaxPacked = 21845;
// VV offsets (a tet adds up to 12 entries: 12 x 65,534 < 2^24) under the 8-bit bias
constexpr int kOffMask = 0xffffff;

__device__ __forceinline__ void cmpx_u16x2(uint32_t &a, uint32_t &b) {
    uint32_t lo, hi;
    asm("min.u16x2 %0, %1, %2;" : "=r"(lo) : "r"(a), "r"(b));
    asm("max.u16x2 %0, %1, %2;" : "=r"(hi) : "r"(a), "r"(b));
    a = lo;
    b = hi;
}

// one row of a star: n entries from `in`, written in order from `out`
struct SortRow {
    int n, in, out;
};

// Two rows of up to N distinct 16-bit entries each, sorted by one thread in
// registers: row a in the low halves, row b in the high ones (Batcher's
// odd-even merge network, pruned to N).  N = 64: one row of 33 to 64 entries
// (b is its tail from the 33rd), whose sorted halves a bitonic merge then
// joins.  Input rows start on a word and are padded with 0xffff to one.
// keyed: entries are 4 * tet + slot; the tets go out, and every entry's
// position goes to jpos (16-bit with jp16).
template <int N>
__device__ __forceinline__ void sort_rows(const uint16_t *in, uint16_t *out, uint8_t *jpos, bool keyed, bool jp16,
                                          const SortRow &a, const SortRow &b) {
    constexpr int R = N < 32 ? N : 32;
    uint32_t v[R];
    const uint32_t *wa = reinterpret_cast<const uint32_t *>(in + a.in);
    const uint32_t *wb = reinterpret_cast<const uint32_t *>(in + b.in);
#pragma unroll
    for (int i = 0; i < R; i += 2) {
        const uint32_t x = i < a.n ? wa[i >> 1] : 0xffffffffu, y = i < b.n ? wb[i >> 1] : 0xffffffffu;
        v[i] = __byte_perm(x, y, 0x5410);
        v[i + 1] = __byte_perm(x, y, 0x7632);
    }
#pragma unroll
    for (int p = 1; p < R; p <<= 1)
#pragma unroll
        for (int k = p; k >= 1; k >>= 1)
#pragma unroll
            for (int i = 0; i + k < R; ++i)
                if (i >= k % p && ((i - k % p) / k) % 2 == 0 && i / (2 * p) == (i + k) / (2 * p))
                    cmpx_u16x2(v[i], v[i + k]);
    if (N == 64) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {  // low[i] against high[31 - i], and high[i] against low[31 - i]
            uint32_t lo = v[i], hi = (v[R - 1 - i] >> 16) | (v[R - 1 - i] << 16);
            cmpx_u16x2(lo, hi);
            v[i] = (lo & 0xffffu) | (hi << 16);
            v[R - 1 - i] = (lo >> 16) | (hi & 0xffff0000u);
        }
#pragma unroll
        for (int k = R / 2; k >= 1; k >>= 1)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if ((i & k) == 0) cmpx_u16x2(v[i], v[i + k]);
    }
    uint16_t *const oa = out + a.out, *const ob = out + b.out;
    if (keyed && !jp16) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const uint32_t x = v[i] & 0xffffu, y = v[i] >> 16;
            if (i < a.n) {
                oa[i] = uint16_t(x >> 2);
                jpos[x] = uint8_t(i);
            }
            if (i < b.n) {
                ob[i] = uint16_t(y >> 2);
                jpos[y] = uint8_t(N == 64 ? i + 32 : i);
            }
        }
        return;
    }
    auto put = [&](uint16_t *o, int i, int pos, uint32_t e) {
        o[i] = uint16_t(keyed ? e >> 2 : e);
        if (keyed) reinterpret_cast<uint16_t *>(jpos)[e] = uint16_t(pos);
    };
#pragma unroll
    for (int i = 0; i < R; ++i) {
        if (i < a.n) put(oa, i, i, v[i] & 0xffffu);
        if (i < b.n) put(ob, i, N == 64 ? i + 32 : i, v[i] >> 16);
    }
}

// One row of any length sorted in place by a warp: a bitonic network whose
// comparisons all point the same way, so that the pairs past the end drop out.
__device__ __forceinline__ void sort_row_warp(uint16_t *v, int n, int lane) {
    int half = 32;
    while (2 * half < n) half <<= 1;
    auto cx = [&](int a, int b) {
        if (b < n) {
            const uint16_t x = v[a], y = v[b];
            if (y < x) {
                v[a] = y;
                v[b] = x;
            }
        }
    };
    for (int k = 2; (k >> 1) < n; k <<= 1) {
        const int kh = k >> 1;
        for (int i = lane; i < half; i += 32) {
            const int a = (i & ~(kh - 1)) * 2, f = i & (kh - 1);
            cx(a + f, a + k - 1 - f);
        }
        __syncwarp();
        for (int j = kh >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < half; i += 32) {
                const int a = (i & ~(j - 1)) * 2 + (i & (j - 1));
                cx(a, a + j);
            }
            __syncwarp();
        }
    }
}

// ---------------- E'. TT of a non-manifold cluster ----------------
// A triangle of the block lies in three or more tets, so a face may have
// more than one partner.  Every tet of the block holding a face of an
// internal tet is in its TT row, and the block holds them all: such a tet
// holds an own vertex of the face (working set) or lies across a face
// without one (face halo).  Each row is found by comparing vertex triples
// with every tet of the block and sorted by canonical id.  Runs only for
// the clusters the face links mark.  Ends synced.
template <bool COUNT, class Team>
__device__ __forceinline__ void tt_general(const Team &tm, const Smem &S, const uint2 *rows, const int32_t *tmap,
                                        int32_t t_base, int n_ext, int n_own, int n_all, int32_t max_tt,
                                        const WorkItem *it, int64_t *sizes_out, int32_t *err) {
    const int NT = tm.nt(), tid = tm.tid();
    const int n_vtets = n_ext + n_own;
    auto gtet = [&](int loc) -> int32_t {
        if (loc < n_ext) return tmap[loc];
        if (loc < n_vtets) return t_base + (loc - n_ext);
        return tmap[loc - n_own];
    };
    int32_t *tcnt = S.tcnt;
    for (int i = tid; i < n_own; i += NT) {
        const int li = n_ext + i;
        const uint2 r = rows[li];
        int c = 0;
        for (int u = 0; u < n_all; ++u) c += (u != li && shared_vertices(rows[u], r) == 3);
        tcnt[i] = c;
    }
    tm.sync();
    const int tot_tt = block_scan_array(tm, tcnt, n_own, S.scan);
    if (COUNT) {
        if (tid == 0) {
            sizes_out[SZ_TT] = tot_tt;
            sizes_out[SZ_GENERAL] = 1;
        }
    } else {
        if (tot_tt > max_tt) {
            if (tid == 0) atomicOr(err, ERR_CAPACITY);
            tm.sync();
            return;
        }
        for (int i = tid; i < n_own; i += NT) {
            const int li = n_ext + i;
            const uint2 r = rows[li];
            const int p = tcnt[i];
            uint16_t *o = S.st_tt + p;
            int c = 0;
            for (int u = 0; u < n_all; ++u) {
                if (u == li || shared_vertices(rows[u], r) != 3) continue;
                const int32_t gu = gtet(u);
                int q = c++;
                while (q > 0 && gtet(o[q - 1]) > gu) {
                    o[q] = o[q - 1];
                    --q;
                }
                o[q] = uint16_t(u);
            }
            it->tt_off[i] = p;
        }
        if (tid == 0) it->tt_off[n_own] = tot_tt;
        tm.sync();
        copy_out(tm, it->tt_val, tot_tt, [&](int j) { return gtet(S.st_tt[j]); });
    }
    tm.sync();
}

// ---------------------------------------------------------------------------
// A persistent CTA's next work item, taken while it builds the current one:
// the ticket, the order entry, the item (and its plan), the block's extent
// and the block's L2 prefetch depend on one another, a global latency each, so
// one thread takes a step of the chain between two phases, by asynchronous
// copies into the slot that the next item is read from.  (Taken in one go at
// the top of the loop, the chain stood before every block copy: 1.031 ms a
// build of 128^3 against 1.015.)
// ---------------------------------------------------------------------------
struct NextSlot {
    WorkItem item;
    int64_t blk[2];  // the block's first word and its end
    int32_t has;     // 0: no item is left
    int32_t at;      // the claiming thread's: ticket, then position
    int32_t step;    // ... next step (5: done)
    int32_t pad;
};

__device__ __forceinline__ void copy_async(void *dst, const void *src, int bytes) {
    if (bytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else if (bytes == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct NoClaim {
    __device__ __forceinline__ void step(int) {}
};

// (its state lives in the slot: the build has no registers to spare)
struct NextItem {
    const WorkItem *items;
    const int32_t *order;
    int32_t *ticket;
    const SmemPlan *plans;  // NULL: the launch has one plan
    const DevMesh &m;
    int32_t n;
    NextSlot *slot;
    SmemPlan *plan;

    __device__ __forceinline__ bool mine() const { return threadIdx.x == blockDim.x - 32; }
    __device__ __forceinline__ void begin(NextSlot *s, SmemPlan *p) {
        slot = s;
        plan = p;
        if (mine()) slot->step = 0;
    }
    __device__ __forceinline__ void step(int s) {
        if (mine() && slot->step == s) take(s);
    }
    __device__ __forceinline__ void take(int s) {
        slot->step = s + 1;
        if (s == 0) {
            slot->at = atomicAdd(ticket, 1);
            return;
        }
        const int at = slot->at;
        if (s == 1) {
            slot->has = at < n;
            slot->at = at >= n ? -1 : order ? order[at] : at;
        } else if (at < 0) {
            return;
        } else if (s == 2) {
            const char *src = reinterpret_cast<const char *>(items + at);
            for (int i = 0; i < int(sizeof(WorkItem)); i += 16)
                copy_async(reinterpret_cast<char *>(&slot->item) + i, src + i, 16);
        } else if (s == 3) {
            copies_done();
            const int k = slot->item.k;
            slot->blk[0] = slot->blk[1] = 0;
            if (k < 0 || k >= m.K + m.NP) return;  // reported when its turn comes
            copy_async(&slot->blk[0], m.blk_off + k, 8);
            copy_async(&slot->blk[1], m.blk_off + k + 1, 8);
            if (plans) {
                const int32_t *src = reinterpret_cast<const int32_t *>(plans + k);
                for (int i = 0; i < int(sizeof(SmemPlan) / 4); ++i)
                    copy_async(reinterpret_cast<int32_t *>(plan) + i, src + i, 4);
            }
        } else {
            copies_done();
            const int64_t w0 = slot->blk[0], w1 = slot->blk[1];
            if (w1 > w0) prefetch_l2(m.blocks + w0, uint32_t(4 * (w1 - w0)));
        }
    }
    // the steps a build with fewer phases left
    __device__ __forceinline__ void finish() {
        if (!mine()) return;
        for (int s = slot->step; s < 5; ++s) take(s);
    }
};

// ---------------------------------------------------------------------------
// One cluster.  COUNT: no output writes; sizes -> sizes_out[5].  SPILL: the
// regions are global scratch and the rows arrive by vector loads instead of
// the bulk copy.  `it` points to a shared-memory copy of the work item; bar
// and phase are the CTA's block-copy barrier and its next parity.  Returns
// false when a bounded wait ran out (the CTA must stop).
// ---------------------------------------------------------------------------
// PART: the item is a part of a cut cluster (block header part != 0); the
// whole-cluster instances carry none of the part logic.  GEN: the instance
// carries the rare forms of whole clusters (E', tight plans), which the hot
// shared-memory kernel leaves out.
// claim: takes the CTA's next work item in steps between the phases (NextItem).
template <bool COUNT, bool SPILL, bool PART, bool GEN, class Team, class Claim>
__device__ bool run_cluster(const Team &tm, const DevMesh &m, const SmemPlan &plan, const Smem &S, int64_t blk_word, int64_t words,
                            uint32_t mask, const WorkItem *it, int64_t *sizes_out, int32_t *err, uint64_t *bar,
                            uint32_t &phase, Claim &claim) {
    const int NT = tm.nt(), NWARP = NT >> 5;
    const int tid = tm.tid(), lane = tid & 31, warp = tid >> 5;
    const Caps &caps = plan.caps;
    const int32_t *__restrict__ g = m.blocks + blk_word;
    int32_t *const flag = S.blk;  // kFlag* words
    const bool jp16 = (plan.mode & kJpos16) != 0;
    const bool tight = GEN && !SPILL && (plan.mode & kTight) != 0;

    // ---------------- A. the block, by one bulk copy ----------------
    // The regions that B starts from are cleared while it is under way, as
    // far as the plan's capacities go.
    const bool fits = words >= kHdrWords && words <= caps.blk_words && (words & 3) == 0;
    const bool need_nb = COUNT || (mask & ~R_VT) != 0;
    if (tid == 0 && fits && !SPILL) bulk_load(S.blk, g, uint32_t(4 * words), bar);
    claim.step(0);
    for (int i = tid; i <= caps.nv_own; i += NT) {
        S.c_vv[i] = 0;
        S.vt_off[i] = 0;
    }
    if (need_nb) fill_words(tm, S.bm, caps.nv_own * plan.W, 0u);
    if (!tight)
        fill_words(tm, reinterpret_cast<uint32_t *>(S.fill),
                   plan.stride ? (caps.nv_own * plan.stride) >> 1 : (caps.n_vt + caps.nv_own + 3) >> 1, FULL);
    if (SPILL && fits) {
        const int4 *src = reinterpret_cast<const int4 *>(g);
        int4 *dst = reinterpret_cast<int4 *>(S.blk);
        const int n4 = int(words >> 2);
        for (int i = tid; i < n4; i += NT) dst[i] = __ldg(src + i);
    }
    {
        const bool ok = SPILL || !fits || mbar_wait(bar, phase);
        if (tm.sync_or(!ok)) {
            if (tid == 0) atomicOr(err, ERR_TIMEOUT);
            if (!ok) mbar_wait(bar, phase);  // the copy may still be in flight
            return false;
        }
    }
    if (!fits) {
        if (tid == 0) atomicOr(err, ERR_CAPACITY);
        tm.sync();
        return true;
    }
    if (!SPILL) phase ^= 1u;
    const BlockHdr h = *reinterpret_cast<const BlockHdr *>(S.blk);
    // a part block: its record, and the extra tmap words of its internal tets
    const PartInfo *part = (PART && h.part > 0 && h.part <= m.NP) ? m.parts + (h.part - 1) : nullptr;
    const int32_t xmap = part ? h.n_own : 0;
    {
        const int64_t n_tot = int64_t(h.n_ext) + h.n_own + h.n_halo;
        const bool ok = h.n_ext >= 0 && h.n_own >= 0 && h.n_halo >= 0 && h.nv_loc >= 0 && h.own_lo >= 0 &&
                        h.nv_own >= 0 && h.nv_nb >= 0 && h.n_bnd >= 0 && n_tot <= caps.n_tot &&
                        h.n_own <= caps.n_own && h.nv_loc <= caps.nv_loc && h.nv_own <= caps.nv_own &&
                        h.nv_nb <= caps.nv_nb && h.nv_nb <= h.nv_loc && int64_t(h.own_lo) + h.nv_own <= h.nv_nb &&
                        2 * int64_t(h.n_bnd) + 1 <= caps.hcap && (PART ? part != nullptr : h.part == 0) &&
                        blk_words(h.nv_loc, h.n_ext, h.n_own, h.n_halo, h.n_bnd, xmap) == words;
        if (!ok) {
            if (tid == 0) atomicOr(err, ERR_CAPACITY);
            tm.sync();
            return true;
        }
    }
    const int n_ext = h.n_ext, n_own = h.n_own;
    const int n_vtets = n_ext + n_own;
    const uint2 *rows = reinterpret_cast<const uint2 *>(S.blk + blk_rows_off(h.nv_loc, n_ext, h.n_halo, xmap));
    const int32_t *vmap = S.blk + kHdrWords;
    const int32_t *tmap = S.blk + blk_tmap_off(h.nv_loc);
    const int nvo = h.nv_own, lo = h.own_lo;
    const uint32_t nvo_u = uint32_t(nvo);
    // the counting pass sizes the relations the context is preconditioned for
    const bool want_tt = (mask & R_TT) != 0;
    const bool do_vv = !COUNT && (mask & R_VV);
    const bool do_et = !COUNT && (mask & R_ET);
    const int32_t t_base = h.t_base;
    const int n_halo_b = h.n_halo;
    // canonical id of a local tet: of the star tets (external and internal)
    // by one predicated load, of any tet by two
    const int32_t t_own = t_base - n_ext;
    auto gstar = [&](int loc) -> int32_t {
        if (PART) return tmap[loc < n_ext ? loc : n_halo_b + loc];
        int32_t g1 = loc + t_own;
        if (loc < n_ext) g1 = tmap[loc];
        return g1;
    };
    auto gtet = [&](int loc) -> int32_t {
        if (PART) return loc >= n_vtets ? tmap[loc - n_own] : gstar(loc);
        int32_t g1 = loc + t_own;
        if (uint32_t(loc - n_ext) >= uint32_t(n_own)) g1 = tmap[loc < n_ext ? loc : loc - n_own];
        return g1;
    };
    // a part writes cluster-level offset values: its entries are shifted by
    // those of the cluster's earlier parts
    int32_t b_vt = 0, b_vv = 0, b_e = 0, b_et = 0;
    if (part && !COUNT) {
        b_vt = __ldg(&part->b_vt);
        b_vv = __ldg(&part->b_vv);
        b_e = __ldg(&part->b_e);
        b_et = __ldg(&part->b_et);
    }

    const int W = (h.nv_nb + 31) >> 5;  // bitmap words per vertex
    const int WP = W | 1;                // row stride (odd: rows start in different banks)
    uint32_t *bm = S.bm;
    uint8_t *pre = S.pre;

    // ---------------- B/C1. stars and neighbour bitmaps, per tet ----------
    // For every own vertex x of a tet: one atomic counts x's star (low half
    // of the counter) and the ET entries x owns (high half: a tet gives x
    // one for each of its vertices above x), and the other three vertices
    // are ORed into x's bitmap.  With padded rows (plan.stride) the value the
    // count returns is also the tet's slot; otherwise a second pass fills
    // compact rows by cursors.  An entry is 4 * tet + x's slot in the tet
    // (kKeyed).  Tight plans have no room for these rows beside VT's own
    // (kTight): they fill VT in place, with its offsets as the cursors, and a
    // warp then sorts each row there; the first ET entries are not kept.
    int32_t *const cnt = S.c_vv;  // the counters, then VV offsets, then the biased edge bases
    int32_t *const et_b = S.et_b;  // first ET entry of each own vertex
    const int stride = plan.stride;
    const bool keyed = (plan.mode & kKeyed) != 0, wide = caps.max_deg > kMaxPacked;
    uint16_t *const fill = S.fill;  // rows in arrival order, each from a word boundary
    int32_t *const cur = reinterpret_cast<int32_t *>(S.st_v);  // fill cursors of compact rows
    auto row_at = [&](int x) -> int { return stride ? x * stride : (S.vt_off[x] + x + 1) & ~1; };
    int32_t flags = 0;
    for (int i = tid; i < n_vtets; i += NT) {
        const uint2 r = rows[i];
        const uint32_t v[4] = {r.x & 0xffffu, r.x >> 16, r.y & 0xffffu, r.y >> 16};
        uint32_t bit[4], q[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            q[s] = v[s] >> 5;
            bit[s] = 1u << (v[s] & 31u);
        }
        // the four counts first: the slots they return come back while the
        // bitmaps are set
        int slot[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const uint32_t d = v[s] - uint32_t(lo);
            slot[s] = stride;
            if (d < nvo_u) {
                if (wide) {  // the halves could overflow: two counters
                    atomicAdd(&cnt[d], 3 - s);
                    atomicAdd(&S.vt_off[d + 1], 1);
                } else {
                    slot[s] = atomicAdd(&cnt[d], 1 | ((3 - s) << 16)) & 0xffff;
                }
            }
        }
        if (need_nb) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint32_t d = v[s] - uint32_t(lo);
                if (d < nvo_u) {
                    uint32_t *row = bm + d * WP;
#pragma unroll
                    for (int u = 1; u < 4; ++u) atomicOr(row + q[(s + u) & 3], bit[(s + u) & 3]);
                }
            }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (slot[s] < stride) fill[(v[s] - uint32_t(lo)) * stride + slot[s]] = uint16_t(keyed ? 4 * i + s : i);
    }
    claim.step(1);
    tm.sync();
    if (tid == 0) {  // every thread has read the header
        flag[kFlagNonManifold] = 0;
        flag[kFlagLong] = 0;
    }

    // ---------------- C2. row lengths and offsets, per own vertex ----------
    // Every bitmap word gets the number of neighbours before it (8 bits); the
    // edge to y, one of x's upper neighbours, is then
    //   base[x] + ((pre + popc(bits of y's word below y)) & 255),
    // base being x's first edge less its lower neighbours (with more than 255
    // neighbours the prefixes start from minus the lower ones instead).
    int vt_total, et_total, vv_total = 0, tot_e = 0;
    {
        const int per = range_len(tm, nvo);
        const int x0 = min(nvo, tid * per), x1 = min(nvo, x0 + per);
        int sv = 0, se = 0, sn = 0, su = 0;
        for (int x = x0; x < x1; ++x) {
            const uint32_t c = uint32_t(cnt[x]);
            const int d = wide ? S.vt_off[x + 1] : int(c & 0xffffu);
            const int et = wide ? int(c) : int(c >> 16);
            S.vt_off[x + 1] = d;
            if (!tight) et_b[x] = et;
            sv += d;
            se += et;
            if (d > caps.max_deg) flags |= ERR_CAPACITY;
            if (need_nb) {
                const uint32_t *row = bm + x * WP;
                uint8_t *prx = pre + x * WP;
                int n = 0;
#pragma unroll 4
                for (int q = 0; q < W; ++q) {
                    prx[q] = uint8_t(n);
                    n += __popc(row[q]);
                }
                const int X = lo + x, qx = X >> 5;
                const uint32_t below = (1u << (X & 31)) - 1u;
                int k0 = prx[qx] + __popc(row[qx] & below);  // neighbours below x
                int bias = k0;
                if (n > 255) {
                    k0 = 0;
                    for (int q = 0; q < qx; ++q) k0 += __popc(row[q]);
                    k0 += __popc(row[qx] & below);
                    int run = -k0;
                    for (int q = 0; q < W; ++q) {
                        prx[q] = uint8_t(run);
                        run += __popc(row[q]);
                    }
                    bias = 0;
                }
                if (n - k0 > 255) flags |= ERR_CAPACITY;
                S.c_vv[x] = n | int(uint32_t(bias) << 24);
                S.c_e[x] = n - k0;
                sn += n;
                su += n - k0;
            }
        }
        int tot[4];
        block_scan4(tm, sv, se, sn, su, S.scan, S.blk + kScanTotals, tot);
        vt_total = tot[0];
        et_total = tot[1];
        vv_total = tot[2];
        tot_e = tot[3];
        if (vt_total > caps.n_vt || tot_e > caps.max_e || ((do_vv || do_et) && vv_total > caps.max_vv) ||
            (do_et && et_total > caps.max_etv))
            flags |= ERR_CAPACITY;
        for (int x = x0; x < x1; ++x) {
            const int d = S.vt_off[x + 1];
            if (tight) {
                S.vt_off[x + 1] = sv;  // the cursor, which the fill moves to the row's end
            } else {
                const int et = et_b[x];
                if (d > 32) S.long_rows[atomicAdd(&flag[kFlagLong], 1)] = uint16_t(x);
                S.vt_off[x + 1] = sv + d;
                if (!stride) cur[x] = (sv + x + 1) & ~1;
                et_b[x] = se;
                se += et;
            }
            sv += d;
            if (need_nb) {
                const int n = S.c_vv[x], u = S.c_e[x];
                S.c_vv[x] = sn | (n & int(0xff000000u));  // the bias stays on top
                S.c_e[x] = su;
                sn += n & kOffMask;
                su += u;
            }
        }
        if (tid == 0) {
            S.c_vv[nvo] = vv_total;
            S.c_e[nvo] = tot_e;
        }
        if (tm.sync_or(flags)) {
            if (tid == 0) atomicOr(err, ERR_CAPACITY);
            return true;
        }
    }
    if (!stride) {
        for (int i = tid; i < n_vtets; i += NT) {
            const uint2 r = rows[i];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint32_t d = vtx(r, s) - uint32_t(lo);
                if (d < nvo_u)
                    fill[atomicAdd(tight ? &S.vt_off[d + 1] : &cur[d], 1)] = uint16_t(keyed ? 4 * i + s : i);
            }
        }
        tm.sync();
    }

    // ---------------- B/C2. rows in order: VT sorted, VV read from the bitmaps
    // A thread sorts two stars of up to 32 tets at once, or one of up to 64:
    // long chains of register operations on a few warps, while the others
    // read the VV rows out of the bitmaps.  A sorted entry also gives the
    // position of its (tet, own vertex) in the row, kept for C3 and C5.
    {
        const int half = (nvo + 1) >> 1, nlong = flag[kFlagLong];
        const int w_pair = tight ? 0 : (half + 31) >> 5, w_long = (nlong + 31) >> 5;
        const int w_emit = do_vv || do_et ? (nvo + 31) >> 5 : 0;
        for (int w = warp; w < w_pair + w_long + w_emit; w += NWARP) {
            if (w < w_pair) {
                const int xa = w * 32 + lane, xb = xa + half;
                SortRow a{}, b{};
                if (xa < half) {
                    a.out = S.vt_off[xa];
                    a.n = S.vt_off[xa + 1] - a.out;
                    a.in = row_at(xa);
                    if (xb < nvo) {
                        b.out = S.vt_off[xb];
                        b.n = S.vt_off[xb + 1] - b.out;
                        b.in = row_at(xb);
                    }
                    if (a.n > 32) a.n = 0;
                    if (b.n > 32) b.n = 0;
                }
                const int top = __reduce_max_sync(FULL, max(a.n, b.n));
                if (top > 24) sort_rows<32>(fill, S.vt_list, S.jpos, keyed, jp16, a, b);
                else if (top > 16) sort_rows<24>(fill, S.vt_list, S.jpos, keyed, jp16, a, b);
                else if (top > 0) sort_rows<16>(fill, S.vt_list, S.jpos, keyed, jp16, a, b);
            } else if (w < w_pair + w_long) {
                const int i = (w - w_pair) * 32 + lane;
                SortRow a{}, b{};
                if (i < nlong) {
                    const int x = S.long_rows[i];
                    a.out = S.vt_off[x];
                    a.n = S.vt_off[x + 1] - a.out;
                    a.in = row_at(x);
                    if (a.n > 64) a.n = 0;
                    if (a.n) {
                        b.n = a.n - 32;
                        b.out = a.out + 32;
                        b.in = a.in + 32;
                        a.n = 32;
                    }
                }
                sort_rows<64>(fill, S.vt_list, S.jpos, keyed, jp16, a, b);
            } else {
                const int x = (w - w_pair - w_long) * 32 + lane;
                if (x >= nvo) continue;
                // one loop step per set bit, words visited through an
                // occupancy mask with the next one loaded ahead
                const uint32_t *row = bm + x * WP;
                uint16_t *o = S.st_v + (S.c_vv[x] & kOffMask);
                for (int q0 = 0; q0 < W; q0 += 32) {
                    const int qn = min(32, W - q0);
                    uint32_t occ = 0u;
#pragma unroll 4
                    for (int u = 0; u < qn; ++u) occ |= (row[q0 + u] != 0u ? 1u : 0u) << u;
                    if (occ == 0u) continue;
                    const uint32_t *r0 = row + q0 - 1;
                    int f = __ffs(int(occ)), base = 32 * (q0 + f) - 33;
                    uint32_t wd = r0[f];
                    occ &= occ - 1u;
                    f = __ffs(int(occ));
                    uint32_t next = occ ? r0[f] : 0u;
                    while (wd) {
                        *o++ = uint16_t(base + __ffs(int(wd)));
                        wd &= wd - 1u;
                        if (wd == 0u) {
                            wd = next;
                            base = 32 * (q0 + f) - 33;
                            occ &= occ - 1u;
                            f = __ffs(int(occ));
                            next = occ ? r0[f] : 0u;
                        }
                    }
                }
            }
        }
        // stars of more than 64 tets: a warp each
        if (tight || caps.max_deg > 64)
            for (int i = warp; i < (tight ? nvo : nlong); i += NWARP) {
                const int x = tight ? i : S.long_rows[i];
                const int o = S.vt_off[x], n = S.vt_off[x + 1] - o;
                if (n <= 64 && !tight) continue;
                uint16_t *const v = fill + (tight ? o : row_at(x));
                sort_row_warp(v, n, lane);
                if (tight) continue;
                for (int j = lane; j < n; j += 32) {
                    const uint32_t e = v[j];
                    S.vt_list[o + j] = uint16_t(keyed ? e >> 2 : e);
                    if (keyed && jp16) reinterpret_cast<uint16_t *>(S.jpos)[e] = uint16_t(j);
                    else if (keyed) S.jpos[e] = uint8_t(j);
                }
            }
        tm.sync();
        if (!keyed) {  // tet ids too large to carry the slot: positions by a pass over the rows
            for (int x = warp; x < nvo; x += NWARP) {
                const int o = S.vt_off[x], n = S.vt_off[x + 1] - o;
                for (int j = lane; j < n; j += 32) {
                    const int t = S.vt_list[o + j];
                    const uint2 r = rows[t];
                    const uint32_t X = uint32_t(lo + x);
                    const int s = vtx(r, 0) == X ? 0 : vtx(r, 1) == X ? 1 : vtx(r, 2) == X ? 2 : 3;
                    if (jp16) reinterpret_cast<uint16_t *>(S.jpos)[4 * t + s] = uint16_t(j);
                    else S.jpos[4 * t + s] = uint8_t(j);
                }
            }
            tm.sync();
        }
    }
    claim.step(2);
    if (COUNT) {
        if (tid == 0) {
            sizes_out[SZ_VT] = vt_total;
            sizes_out[SZ_VV] = vv_total;
            sizes_out[SZ_E] = tot_e;
            sizes_out[SZ_ET] = et_total;
        }
    } else {
        if (mask & R_VT) {
            for (int i = tid; i <= nvo; i += NT) it->vt_off[i] = S.vt_off[i] + b_vt;
            copy_out(tm, it->vt_val, vt_total, [&](int j) { return gstar(S.vt_list[j]); });
        }
        if (do_vv) {
            for (int i = tid; i <= nvo; i += NT) it->vv_off[i] = (S.c_vv[i] & kOffMask) + b_vv;
            copy_out(tm, it->vv_val, vv_total, [&](int j) { return vmap[S.st_v[j]]; });
        }
        if (do_et) {
            for (int i = tid; i <= nvo; i += NT) it->eu_off[i] = S.c_e[i] + b_e;
            // upper endpoints: the tail of each VV row
            for (int x = tid; x < nvo; x += NT) {
                const int e0 = S.c_e[x], ne = S.c_e[x + 1] - e0;
                const uint16_t *src = S.st_v + (S.c_vv[x + 1] & kOffMask) - ne;
                int32_t *dst = it->e_w + e0;
                for (int i = 0; i < ne; i += 4) {  // four loads in flight
                    const int l = ne - 1 - i;
                    const int32_t a = vmap[src[i]], b = vmap[src[i + min(l, 1)]];
                    const int32_t c = vmap[src[i + min(l, 2)]], d = vmap[src[i + min(l, 3)]];
                    dst[i] = a;
                    if (l >= 1) dst[i + 1] = b;
                    if (l >= 2) dst[i + 2] = c;
                    if (l >= 3) dst[i + 3] = d;
                }
            }
            if (tid == 0) it->et_off[tot_e] = et_total + b_et;
        }
    }
    if (!(do_et || want_tt)) {
        tm.sync();
        return true;
    }
    const int nch = plan.nch;
    uint32_t *em = S.emask;
    tm.sync();  // the VV staging and the vertex map are dead
    // the edge bases take the place of the VV offsets, the edge masks that of
    // the VV staging; masks of several words also reach the first ET entries,
    // which move to the vertex map (nvo <= nv_loc words)
    int32_t *const et_first = nch > 1 ? S.blk + kHdrWords : et_b;
    if (nch > 1 && !tight) {
        for (int x = tid; x < nvo; x += NT) et_first[x] = et_b[x];
        tm.sync();
    }
    for (int x = tid; x < nvo; x += NT) cnt[x] = S.c_e[x] - int(uint32_t(cnt[x]) >> 24);
    fill_words(tm, em, tot_e * nch, 0u);
    tm.sync();

    // ---------------- C3. edge tet masks, per tet ----------------
    // bit j of mask(x, w): the j-th tet of VT(x) contains w; every own
    // vertex x of a tet marks the edges to the tet's vertices above x.  An
    // internal tet's edge ranks stay in its link words for C5.
    {
        auto rank = [&](uint32_t x, uint32_t y) -> uint32_t {
            const uint32_t at = x * uint32_t(WP) + (y >> 5);
            return (pre[at] + uint32_t(__popc(bm[at] & ((1u << (y & 31u)) - 1u)))) & 0xffu;
        };
        auto marks = [&](auto one) {
            constexpr bool ONE = decltype(one)::value != 0;  // masks of one word
            auto mark = [&](int e, uint32_t j) {
                if (ONE) atomicOr(em + e, 1u << j);
                else atomicOr(em + e * nch + (j >> 5), 1u << (j & 31));
            };
            for (int i = tid; i < n_vtets; i += NT) {
                const uint2 r = rows[i];
                const uint32_t v0 = r.x & 0xffffu, v1 = r.x >> 16, v2 = r.y & 0xffffu, v3 = r.y >> 16;
                uint32_t j0, j1, j2;
                if (!ONE && jp16) {
                    const uint2 jw = reinterpret_cast<const uint2 *>(S.jpos)[i];
                    j0 = jw.x & 0xffffu;
                    j1 = jw.x >> 16;
                    j2 = jw.y & 0xffffu;
                } else {
                    const uint32_t jw = reinterpret_cast<const uint32_t *>(S.jpos)[i];
                    j0 = jw & 0xffu;
                    j1 = (jw >> 8) & 0xffu;
                    j2 = (jw >> 16) & 0xffu;
                }
                const uint32_t x0 = v0 - uint32_t(lo), x1 = v1 - uint32_t(lo), x2 = v2 - uint32_t(lo);
                // a tet's ranks all before its marks, so that their loads overlap
                int e0 = 0, e1 = 0, e2 = 0;
                uint32_t ra = 0u, rb = 0u;
                if (x0 < nvo_u) {
                    e0 = cnt[x0];
                    ra = rank(x0, v1) | (rank(x0, v2) << 8) | (rank(x0, v3) << 16);
                }
                if (x1 < nvo_u) {
                    e1 = cnt[x1];
                    rb = rank(x1, v2) | (rank(x1, v3) << 8);
                }
                if (x2 < nvo_u) e2 = cnt[x2] + int(rank(x2, v3));
                if (x0 < nvo_u) {
                    mark(e0 + int(ra & 0xffu), j0);
                    mark(e0 + int((ra >> 8) & 0xffu), j0);
                    mark(e0 + int(ra >> 16), j0);
                }
                if (x1 < nvo_u) {
                    mark(e1 + int(rb & 0xffu), j1);
                    mark(e1 + int(rb >> 8), j1);
                }
                if (x2 < nvo_u) mark(e2, j2);
                if (want_tt && i >= n_ext) reinterpret_cast<uint2 *>(S.nbr)[i - n_ext] = make_uint2(ra, rb);
            }
        };
        if (nch == 1) marks(IntC<1>{});
        else marks(IntC<0>{});
    }
    tm.sync();

    claim.step(3);
    // ---------------- C5. TT links of faces with an own lowest vertex ------
    // mask(x, w1) & mask(x, w2), less the tet's own bit, is its partner
    // across the face (x, w1, w2)
    if (want_tt) {
        auto links = [&](auto one) {
            constexpr bool ONE = decltype(one)::value != 0;
            for (int i = tid; i < n_own; i += NT) {
                const int li = n_ext + i;
                const uint32_t rx = rows[li].x;
                const uint2 rk = reinterpret_cast<const uint2 *>(S.nbr)[i];
                const uint32_t a = (rx & 0xffffu) - uint32_t(lo), b = (rx >> 16) - uint32_t(lo);
                uint32_t f0 = 0xffffu, f1 = 0xffffu, f2 = 0xffffu, f3 = 0xffffu;
                auto pick = [&](uint32_t m1, uint32_t m2, uint32_t self, int base, uint32_t &f, int &found) {
                    const uint32_t mm = m1 & m2 & ~self;
                    if (mm != 0u) {
                        if (found == 0) f = S.vt_list[base + __ffs(int(mm)) - 1];
                        found += ONE ? 1 + ((mm & (mm - 1u)) != 0u) : __popc(mm);
                    }
                };
                if (a < nvo_u) {
                    const int e = cnt[a], e1 = e + int(rk.x & 0xffu), e2 = e + int((rk.x >> 8) & 0xffu),
                              e3 = e + int((rk.x >> 16) & 0xffu);
                    const int base = S.vt_off[a];
                    int n1 = 0, n2 = 0, n3 = 0;
                    if (ONE) {
                        const uint32_t self = 1u << S.jpos[4 * li];
                        const uint32_t m1 = em[e1], m2 = em[e2], m3 = em[e3];
                        pick(m1, m2, self, base, f3, n3);
                        pick(m1, m3, self, base, f2, n2);
                        pick(m2, m3, self, base, f1, n1);
                    } else {
                        const int js = jp16 ? reinterpret_cast<const uint16_t *>(S.jpos)[4 * li] : S.jpos[4 * li];
                        for (int c = 0; c < nch; ++c) {
                            const uint32_t self = c == (js >> 5) ? 1u << (js & 31) : 0u;
                            const uint32_t m1 = em[e1 * nch + c], m2 = em[e2 * nch + c], m3 = em[e3 * nch + c];
                            pick(m1, m2, self, base + 32 * c, f3, n3);
                            pick(m1, m3, self, base + 32 * c, f2, n2);
                            pick(m2, m3, self, base + 32 * c, f1, n1);
                        }
                    }
                    if (max(n1, max(n2, n3)) > 1) flags |= ERR_NONMANIFOLD;
                    if (b < nvo_u) {
                        const int eb = cnt[b], e4 = eb + int(rk.y & 0xffu), e5 = eb + int((rk.y >> 8) & 0xffu);
                        const int base_b = S.vt_off[b];
                        int n0 = 0;
                        if (ONE) {
                            pick(em[e4], em[e5], 1u << S.jpos[4 * li + 1], base_b, f0, n0);
                        } else {
                            const int js =
                                jp16 ? reinterpret_cast<const uint16_t *>(S.jpos)[4 * li + 1] : S.jpos[4 * li + 1];
                            for (int c = 0; c < nch; ++c)
                                pick(em[e4 * nch + c], em[e5 * nch + c], c == (js >> 5) ? 1u << (js & 31) : 0u,
                                     base_b + 32 * c, f0, n0);
                        }
                        if (n0 > 1) flags |= ERR_NONMANIFOLD;
                    }
                } else if (!part) {  // an internal tet's lowest vertex is own (a part's: an earlier part's)
                    flags |= ERR_BAD_BLOCK;
                }
                reinterpret_cast<uint2 *>(S.nbr)[i] = make_uint2(f0 | (f1 << 16), f2 | (f3 << 16));
            }
        };
        if (nch == 1) links(IntC<1>{});
        else links(IntC<0>{});
        if (GEN && !PART && (flags & ERR_NONMANIFOLD)) {  // TT of this cluster takes the general pass (E')
            flag[kFlagNonManifold] = 1;
            flags &= ~ERR_NONMANIFOLD;
        }
        if (flags) atomicOr(err, flags);
    }
    tm.sync();  // positions, bitmaps and prefixes are dead

    // ---------------- C4. ET rows, per edge ----------------
    if (do_et) {
        int32_t *eo = S.eo;
        uint16_t *ex = S.ex;
        bool bad = false;
        auto rows_out = [&](auto one) {
            constexpr bool ONE = decltype(one)::value != 0;
            const int nc = ONE ? 1 : nch;
            // each edge's first entry and its lower vertex, per own vertex
            for (int x = tid; x < nvo; x += NT) {
                int run = et_first[x];
                const int e1 = S.c_e[x + 1];
                for (int e = S.c_e[x]; e < e1; e += 4) {  // four edges' masks in flight
                    const int l = min(3, e1 - 1 - e);
                    int n0 = 0, n1 = 0, n2 = 0, n3 = 0;
                    for (int c = 0; c < nc; ++c) {
                        n0 += __popc(em[e * nc + c]);
                        n1 += __popc(em[(e + min(l, 1)) * nc + c]);
                        n2 += __popc(em[(e + min(l, 2)) * nc + c]);
                        n3 += __popc(em[(e + l) * nc + c]);
                    }
                    eo[e] = run;
                    ex[e] = uint16_t(x);
                    run += n0;
                    if (l >= 1) {
                        eo[e + 1] = run;
                        ex[e + 1] = uint16_t(x);
                        run += n1;
                    }
                    if (l >= 2) {
                        eo[e + 2] = run;
                        ex[e + 2] = uint16_t(x);
                        run += n2;
                    }
                    if (l >= 3) {
                        eo[e + 3] = run;
                        ex[e + 3] = uint16_t(x);
                        run += n3;
                    }
                }
                bad |= run != (x + 1 < nvo ? et_first[x + 1] : et_total);  // one distinct bit per entry
            }
            bad = tm.sync_or(bad) != 0;
            if (bad) return;
            for (int e = tid; e < tot_e; e += NT) {
                const int o = eo[e];
                it->et_off[e] = o + b_et;
                uint16_t *dst = S.st_et + o;
                const uint16_t *vt = S.vt_list + S.vt_off[ex[e]] - 1;
                for (int c = 0; c < nc; ++c) {
                    for (uint32_t mm = em[e * nc + c]; mm;) {  // two entries a step
                        const int b0 = __ffs(int(mm));
                        mm &= mm - 1u;
                        const int b1 = mm ? __ffs(int(mm)) : b0;
                        const uint16_t t0 = vt[b0], t1 = vt[b1];
                        dst[0] = t0;
                        if (mm) dst[1] = t1;
                        dst += mm ? 2 : 1;
                        mm &= mm - 1u;
                    }
                    vt += 32;
                }
            }
        };
        if (tight) {  // a vertex's edges by one thread, from sums over the masks
            const int per = range_len(tm, nvo);
            const int x0 = min(nvo, tid * per), x1 = min(nvo, x0 + per);
            int n = 0, total;
            for (int i = S.c_e[x0] * nch; i < S.c_e[x1] * nch; ++i) n += __popc(em[i]);
            int run = block_scan_thread(tm, n, S.scan, &total);
            bad = total != et_total;  // one distinct bit per entry
            for (int x = x0; x < x1 && !bad; ++x)
                for (int e = S.c_e[x]; e < S.c_e[x + 1]; ++e) {
                    it->et_off[e] = run + b_et;
                    for (int c = 0; c < nch; ++c)
                        for (uint32_t mm = em[e * nch + c]; mm; mm &= mm - 1u)
                            S.st_et[run++] = S.vt_list[S.vt_off[x] + 32 * c + __ffs(int(mm)) - 1];
                }
        } else if (nch == 1) {
            rows_out(IntC<1>{});
        } else {
            rows_out(IntC<0>{});
        }
        if (bad) {
            if (tid == 0) atomicOr(err, ERR_BAD_BLOCK);
            return true;
        }
        tm.sync();
        copy_out(tm, it->et_val, et_total, [&](int j) { return gstar(S.st_et[j]); });
        tm.sync();  // ET staging is dead: r1 takes the face hash
    }

    claim.step(4);
    if (want_tt) {
        // ---------------- D. faces with no own vertex, against the halo ----
        const uint32_t hmask = uint32_t(caps.hcap - 1);
        uint32_t *hash = S.hash;
        fill_words(tm, hash, caps.hcap, 0u);
        tm.sync();
        int32_t flags = 0;
        // the face (b, c, d) an entry stands for: entries hold an internal
        // tet's index + 1 and, on top, the number of tets matched to its face
        auto same = [&](uint32_t e, uint2 key) {
            const uint2 r = rows[n_ext + int(e & kRefMask) - 1];
            return (r.x >> 16) == key.x && r.y == key.y;
        };
        // the internal tets whose face (b, c, d) has no own vertex
        const uint16_t *bnd =
            reinterpret_cast<const uint16_t *>(S.blk + blk_bnd_off(h.nv_loc, n_ext, n_own, h.n_halo, xmap));
        for (int jb = tid; jb < h.n_bnd; jb += NT) {
            const int i = bnd[jb];
            const uint2 r = rows[n_ext + i];
            const uint2 key = make_uint2(r.x >> 16, r.y);
            uint32_t hp = face_hash(key) & hmask;
            int probe = 0;
            for (; probe < caps.hcap; ++probe) {
                const uint32_t prev = atomicCAS(&hash[hp], 0u, uint32_t(i + 1));
                if (prev == 0u) break;
                if (same(prev, key)) {
                    const int ref = int(prev & kRefMask) - 1;
                    if (atomicAdd(&hash[hp], kMatch) >= kMatch) flags |= ERR_NONMANIFOLD;
                    S.nbr[4 * ref] = uint16_t(n_ext + i);
                    S.nbr[4 * i] = uint16_t(n_ext + ref);
                    break;
                }
                hp = (hp + 1u) & hmask;
            }
            if (probe == caps.hcap) flags |= ERR_HASH_FULL;
        }
        tm.sync();
        for (int j = tid; j < h.n_halo; j += NT) {
            const int tl = n_vtets + j;
            const uint2 r = rows[tl];
            // the faces opposite slots 0 to 3, their first probes together
            const uint2 key[4] = {make_uint2(r.x >> 16, r.y), make_uint2(r.x & 0xffffu, r.y),
                                  make_uint2(r.x & 0xffffu, (r.x >> 16) | (r.y & 0xffff0000u)),
                                  make_uint2(r.x & 0xffffu, (r.x >> 16) | (r.y << 16))};
            uint32_t hp[4], first[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                hp[f] = face_hash(key[f]) & hmask;
                first[f] = hash[hp[f]];
            }
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                uint32_t e = first[f], h1 = hp[f];
                for (int probe = 1; e != 0u; ++probe) {
                    if (same(e, key[f])) {
                        if (atomicAdd(&hash[h1], kMatch) >= kMatch) flags |= ERR_NONMANIFOLD;
                        S.nbr[4 * (int(e & kRefMask) - 1)] = uint16_t(tl);
                        break;
                    }
                    if (probe == caps.hcap) break;
                    h1 = (h1 + 1u) & hmask;
                    e = hash[h1];
                }
            }
        }
        if (GEN && !PART && (flags & ERR_NONMANIFOLD)) {
            flag[kFlagNonManifold] = 1;
            flags &= ~ERR_NONMANIFOLD;
        }
        if (flags) atomicOr(err, flags);
        tm.sync();
        if (GEN && !PART && flag[kFlagNonManifold] != 0) {
            tt_general<COUNT>(tm, S, rows, tmap, t_base, n_ext, n_own, n_vtets + h.n_halo, caps.max_tt, it,
                              sizes_out, err);
            return true;
        }
        // ---------------- E. TT rows ----------------
        int32_t *tcnt = S.tcnt;
        auto n_links = [&](int i) -> int {
            const uint2 nb = *reinterpret_cast<const uint2 *>(&S.nbr[i * 4]);
            return ((nb.x & 0xffffu) != 0xffffu) + ((nb.x >> 16) != 0xffffu) + ((nb.y & 0xffffu) != 0xffffu) +
                   ((nb.y >> 16) != 0xffffu);
        };
        const int per_t = range_len(tm, n_own);
        const int tb0 = min(n_own, tid * per_t), tb1 = min(n_own, tb0 + per_t);
        int mine_tt = 0;
        for (int i = tb0; i < tb1; ++i) {
            const int c = n_links(i);
            mine_tt += c;
            // row lengths of the part's own internal tets, by canonical id
            if (COUNT && part && (rows[n_ext + i].x & 0xffffu) - uint32_t(lo) < nvo_u) m.tt_pos[gtet(n_ext + i)] = c;
        }
        int tot_tt;
        int run_tt = block_scan_thread(tm, mine_tt, S.scan, &tot_tt);
        if (!COUNT && !part)
            for (int i = tb0; i < tb1; ++i) {
                tcnt[i] = run_tt;
                run_tt += n_links(i);
            }
        tm.sync();
        if (COUNT) {
            if (tid == 0) sizes_out[SZ_TT] = tot_tt;
        } else if (part) {
            // rows straight to their cluster-level offsets (the earlier parts'
            // rows of the same cluster precede this part's in the list)
            if (tot_tt > caps.max_tt) {
                if (tid == 0) atomicOr(err, ERR_CAPACITY);
                return true;
            }
            int32_t *const c_off = it->tt_off - __ldg(&part->b_to);
            int32_t *const c_val = it->tt_val - __ldg(&part->b_tt);
            const int32_t tb = __ldg(&part->t_base_c);
            for (int i = tid; i < n_own; i += NT) {
                if ((rows[n_ext + i].x & 0xffffu) - uint32_t(lo) >= nvo_u) continue;  // an earlier part's row
                const uint2 nb = *reinterpret_cast<const uint2 *>(&S.nbr[i * 4]);
                const uint32_t n0 = nb.x & 0xffffu, n1 = nb.x >> 16, n2 = nb.y & 0xffffu, n3 = nb.y >> 16;
                int32_t w0 = n0 != 0xffffu ? gtet(int32_t(n0)) : INT32_MAX;
                int32_t w1 = n1 != 0xffffu ? gtet(int32_t(n1)) : INT32_MAX;
                int32_t w2 = n2 != 0xffffu ? gtet(int32_t(n2)) : INT32_MAX;
                int32_t w3 = n3 != 0xffffu ? gtet(int32_t(n3)) : INT32_MAX;
                uint32_t l0 = n0, l1 = n1, l2 = n2, l3 = n3;
                cswap2(w0, w1, l0, l1); cswap2(w2, w3, l2, l3); cswap2(w0, w2, l0, l2); cswap2(w1, w3, l1, l3);
                cswap2(w1, w2, l1, l2);
                const int32_t gt = gtet(n_ext + i);
                const int32_t p = m.tt_pos[gt];
                c_off[gt - tb] = p;
                if (w0 != INT32_MAX) c_val[p] = w0;
                if (w1 != INT32_MAX) c_val[p + 1] = w1;
                if (w2 != INT32_MAX) c_val[p + 2] = w2;
                if (w3 != INT32_MAX) c_val[p + 3] = w3;
            }
            if (tid == 0 && __ldg(&part->last)) c_off[__ldg(&part->n_own_c)] = __ldg(&part->tt_total);
        } else {
            if (tot_tt > caps.max_tt) {
                if (tid == 0) atomicOr(err, ERR_CAPACITY);
                return true;
            }
            for (int i = tid; i < n_own; i += NT) {
                const uint2 nb = *reinterpret_cast<const uint2 *>(&S.nbr[i * 4]);
                const uint32_t n0 = nb.x & 0xffffu, n1 = nb.x >> 16, n2 = nb.y & 0xffffu, n3 = nb.y >> 16;
                // local ids ordered by canonical id; absent neighbours sort last
                int32_t w0 = n0 != 0xffffu ? gtet(int32_t(n0)) : INT32_MAX;
                int32_t w1 = n1 != 0xffffu ? gtet(int32_t(n1)) : INT32_MAX;
                int32_t w2 = n2 != 0xffffu ? gtet(int32_t(n2)) : INT32_MAX;
                int32_t w3 = n3 != 0xffffu ? gtet(int32_t(n3)) : INT32_MAX;
                uint32_t l0 = n0, l1 = n1, l2 = n2, l3 = n3;
                cswap2(w0, w1, l0, l1); cswap2(w2, w3, l2, l3); cswap2(w0, w2, l0, l2); cswap2(w1, w3, l1, l3);
                cswap2(w1, w2, l1, l2);
                // canonical ids straight out: a warp's rows are adjacent, so
                // its four stores cover one contiguous span
                const int p = tcnt[i];
                it->tt_off[i] = p;
                int32_t *o = it->tt_val + p;
                if (w0 != INT32_MAX) o[0] = w0;
                if (w1 != INT32_MAX) o[1] = w1;
                if (w2 != INT32_MAX) o[2] = w2;
                if (w3 != INT32_MAX) o[3] = w3;
            }
            if (tid == 0) it->tt_off[n_own] = tot_tt;
        }
    }
    tm.sync();
    return true;
}

// A work item: a whole cluster, or (id >= K) a part of a cut cluster.  The
// items that need GEN (non-manifold clusters, which the counting pass marks,
// and tight plans) run from per-item bins.
template <bool COUNT, bool SPILL, bool GEN, class Claim>
__device__ __forceinline__ bool run_item(bool part, const DevMesh &m, const SmemPlan &plan, const Smem &S,
                                         int64_t blk_word, int64_t words, uint32_t mask, const WorkItem *it,
                                         int64_t *sizes_out, int32_t *err, uint64_t *bar, uint32_t &phase,
                                         Claim &claim) {
    const BlockTeam tm;
    if (part)
        return run_cluster<COUNT, SPILL, true, false>(tm, m, plan, S, blk_word, words, mask, it, sizes_out, err, bar,
                                                      phase, claim);
    return run_cluster<COUNT, SPILL, false, GEN>(tm, m, plan, S, blk_word, words, mask, it, sizes_out, err, bar, phase,
                                                 claim);
}

// SPILL: the cluster's regions live in a per-CTA slice of global scratch
// (clusters whose working set exceeds shared memory); otherwise in dynamic
// shared memory.
template <bool SPILL>
__device__ __forceinline__ char *region_base(char *smem, char *gscratch, const SmemPlan &plan) {
    return SPILL ? gscratch + size_t(blockIdx.x) * size_t(plan.total) : smem;
}

// Blocks have up to 1024 threads, so every cluster kernel is bounded to 64
// registers per thread.
constexpr int kMaxThreads = 1024;

template <bool SPILL>
__device__ __forceinline__ void init_barrier(uint64_t *bar) {
    if (!SPILL && threadIdx.x == 0) mbar_init(bar);
    __syncthreads();
}

template <bool SPILL>
__global__ void __launch_bounds__(kMaxThreads) count_kernel(DevMesh m, SmemPlan plan, const int32_t *ids, int32_t n, int64_t *sizes, int32_t *err,
                             int32_t *ticket, char *gscratch, uint32_t mask) {
    extern __shared__ __align__(16) char smem[];
    const Smem S = carve(region_base<SPILL>(smem, gscratch, plan), plan);
    __shared__ int32_t s_idx;
    __shared__ int64_t s_sizes[SZ_N + 1];
    __shared__ __align__(8) uint64_t s_bar;
    init_barrier<SPILL>(&s_bar);
    uint32_t phase = 0;
    NoClaim none;
    for (;;) {
        if (threadIdx.x == 0) s_idx = atomicAdd(ticket, 1);
        __syncthreads();
        const int idx = s_idx;
        __syncthreads();
        if (idx >= n) break;
        const int k = ids ? ids[idx] : idx;
        if (k < 0 || k >= m.K + m.NP) {
            if (threadIdx.x == 0) atomicOr(err, ERR_BAD_ITEM);
            continue;
        }
        if (threadIdx.x <= SZ_N) s_sizes[threadIdx.x] = 0;
        __syncthreads();
        if (!run_item<true, SPILL, true>(k >= m.K, m, plan, S, m.blk_off[k], m.blk_off[k + 1] - m.blk_off[k], mask, nullptr, s_sizes,
                                      err, &s_bar, phase, none))
            return;
        __syncthreads();
        if (threadIdx.x < SZ_N) sizes[int64_t(k) * SZ_N + threadIdx.x] = s_sizes[threadIdx.x];
        if (threadIdx.x == 0 && k < m.K && m.tt_general) m.tt_general[k] = int32_t(s_sizes[SZ_GENERAL]);
    }
}

template <bool SPILL>
__global__ void __launch_bounds__(kMaxThreads) build_kernel(DevMesh m, SmemPlan plan, const WorkItem *items, const int32_t *order, int32_t n,
                             int32_t *err, int32_t *ticket, char *gscratch) {
    extern __shared__ __align__(16) char smem[];
    const Smem S = carve(region_base<SPILL>(smem, gscratch, plan), plan);
    __shared__ __align__(16) NextSlot s_slot[2];
    __shared__ __align__(8) uint64_t s_bar;
    NextItem claim{items, order, ticket, nullptr, m, n, nullptr, nullptr};
    claim.begin(&s_slot[0], nullptr);
    claim.finish();
    init_barrier<SPILL>(&s_bar);
    uint32_t phase = 0;
    for (int cur = 0; s_slot[cur].has; cur ^= 1) {
        const NextSlot &slot = s_slot[cur];
        const int k = slot.item.k;
        claim.begin(&s_slot[cur ^ 1], nullptr);
        bool ok = true;
        if (k < 0 || k >= m.K + m.NP) {
            if (threadIdx.x == 0) atomicOr(err, ERR_BAD_ITEM);
        } else {
            ok = run_item<false, SPILL, SPILL>(k >= m.K, m, plan, S, slot.item.blk, slot.blk[1] - slot.blk[0],
                                               slot.item.mask, &slot.item, nullptr, err, &s_bar, phase, claim);
        }
        claim.finish();
        if (!ok) return;
        __syncthreads();
    }
}

template <bool SPILL>
__global__ void __launch_bounds__(kMaxThreads) build_one_kernel(DevMesh m, SmemPlan plan, const WorkItem *items, int32_t index, int32_t *err,
                                 char *gscratch) {
    extern __shared__ __align__(16) char smem[];
    const Smem S = carve(region_base<SPILL>(smem, gscratch, plan), plan);
    __shared__ WorkItem s_item;
    __shared__ __align__(8) uint64_t s_bar;
    init_barrier<SPILL>(&s_bar);
    uint32_t phase = 0;
    NoClaim none;
    if (threadIdx.x == 0) s_item = items[index];
    __syncthreads();
    if (s_item.k < 0 || s_item.k >= m.K + m.NP) {
        if (threadIdx.x == 0) atomicOr(err, ERR_BAD_ITEM);
        return;
    }
    run_cluster<false, SPILL, false, true>(BlockTeam{}, m, plan, S, s_item.blk, m.blk_off[s_item.k + 1] - m.blk_off[s_item.k], s_item.mask,
                              &s_item, nullptr, err, &s_bar, phase, none);
}

// ---------------------------------------------------------------------------
// Several small clusters per CTA.  Each team of team_n threads (a multiple
// of 32; the block holds blockDim.x / team_n teams) takes clusters from the
// ticket on its own and builds each in its own slice of the dynamic shared
// memory, with a named barrier and a bulk-copy barrier of its own, so a
// small cluster's barriers involve only its team.
//
// Two instances.  Left alone the compiler takes 95 registers and spills none,
// which is the faster code, but one CTA of 512 threads then fills an SM's
// registers; at 64 (LEAN) two fit.  With as many CTAs on an SM the first is 4
// to 8 % faster, with half as many the second is: 64^3 grid of 64-vertex
// leaves, teams of 128 x 4 260 -> 199 us a build (one CTA an SM against two),
// 128 x 2 254 -> 188 (two against four), 64 x 2 195 against 205 (four of
// either).  At two against three it goes either way (64 x 4 205 against 215;
// 128-vertex leaves, 128 x 2 181 against 158).  So the plan takes the second
// where it holds twice the CTAs (kLeanTeam, max_ctas_per_sm_teams).
// ---------------------------------------------------------------------------
constexpr int kMaxTeams = 15;  // named barriers 1..15
constexpr int kMaxTeamBlock = 512;

template <bool LEAN>
__global__ void __launch_bounds__(kMaxTeamBlock, LEAN ? 2 : 1)
    build_kernel_team(DevMesh m, SmemPlan plan, const WorkItem *items, const int32_t *order, int32_t n, int32_t *err,
                      int32_t *ticket, int team_n) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int32_t s_idx[kMaxTeams];
    __shared__ WorkItem s_item[kMaxTeams];
    __shared__ __align__(8) uint64_t s_bar[kMaxTeams];
    const int g = int(threadIdx.x) / team_n;
    if (g >= kMaxTeams) return;  // (the host never launches more teams)
    const SliceTeam tm{team_n, int(threadIdx.x) - g * team_n, 1 + g};
    const Smem S = carve(smem + size_t(g) * size_t(plan.total), plan);
    if (tm.tid() == 0) mbar_init(&s_bar[g]);
    tm.sync();
    uint32_t phase = 0;
    NoClaim none;
    for (;;) {
        if (tm.tid() == 0) {
            const int idx = atomicAdd(ticket, 1);
            s_idx[g] = idx;
            if (idx < n) s_item[g] = items[order ? order[idx] : idx];
        }
        tm.sync();
        if (s_idx[g] >= n) break;
        const int k = s_item[g].k;
        if (k < 0 || k >= m.K) {
            if (tm.tid() == 0) atomicOr(err, ERR_BAD_ITEM);
            tm.sync();
            continue;
        }
        if (!run_cluster<false, false, false, false>(tm, m, plan, S, s_item[g].blk, m.blk_off[k + 1] - m.blk_off[k],
                                              s_item[g].mask, &s_item[g], nullptr, err, &s_bar[g], phase, none))
            return;
        tm.sync();  // the next claim rewrites this team's item
    }
}

// ---------------------------------------------------------------------------
// Clusters that each carry their own shared-memory plan (plans[k]), for the
// largest clusters, whose plans cannot be merged under one launch plan
// without exceeding a CTA's shared memory: every CTA copies its cluster's
// plan into shared memory and carves its regions from it, so such clusters
// of uneven sizes still share one persistent launch, with the dynamic shared
// memory of the largest.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void load_plan(SmemPlan &dst, const SmemPlan *src) {
    constexpr int kWords = int(sizeof(SmemPlan) / 4);
    for (int i = threadIdx.x; i < kWords; i += blockDim.x)
        reinterpret_cast<int32_t *>(&dst)[i] = reinterpret_cast<const int32_t *>(src)[i];
}

__global__ void __launch_bounds__(kMaxThreads) count_kernel_pi(DevMesh m, const SmemPlan *plans, const int32_t *ids,
                                                              int32_t n, int64_t *sizes, int32_t *err, int32_t *ticket,
                                                              uint32_t mask) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int32_t s_idx;
    __shared__ int64_t s_sizes[SZ_N + 1];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ __align__(16) SmemPlan s_plan;
    init_barrier<false>(&s_bar);
    uint32_t phase = 0;
    NoClaim none;
    for (;;) {
        if (threadIdx.x == 0) s_idx = atomicAdd(ticket, 1);
        __syncthreads();
        const int idx = s_idx;
        __syncthreads();
        if (idx >= n) break;
        const int k = ids ? ids[idx] : idx;
        if (k < 0 || k >= m.K + m.NP) {
            if (threadIdx.x == 0) atomicOr(err, ERR_BAD_ITEM);
            continue;
        }
        load_plan(s_plan, plans + k);
        if (threadIdx.x <= SZ_N) s_sizes[threadIdx.x] = 0;
        __syncthreads();
        const Smem S = carve(smem, s_plan);
        if (!run_item<true, false, true>(k >= m.K, m, s_plan, S, m.blk_off[k], m.blk_off[k + 1] - m.blk_off[k], mask, nullptr,
                                      s_sizes, err, &s_bar, phase, none))
            return;
        __syncthreads();
        if (threadIdx.x < SZ_N) sizes[int64_t(k) * SZ_N + threadIdx.x] = s_sizes[threadIdx.x];
        if (threadIdx.x == 0 && k < m.K && m.tt_general) m.tt_general[k] = int32_t(s_sizes[SZ_GENERAL]);
    }
}

__global__ void __launch_bounds__(kMaxThreads) build_kernel_pi(DevMesh m, const SmemPlan *plans, const WorkItem *items,
                                                              const int32_t *order, int32_t n, int32_t *err,
                                                              int32_t *ticket) {
    extern __shared__ __align__(16) char smem[];
    __shared__ __align__(16) NextSlot s_slot[2];
    __shared__ __align__(16) SmemPlan s_plan[2];
    __shared__ __align__(8) uint64_t s_bar;
    NextItem claim{items, order, ticket, plans, m, n, nullptr, nullptr};
    claim.begin(&s_slot[0], &s_plan[0]);
    claim.finish();
    init_barrier<false>(&s_bar);
    uint32_t phase = 0;
    for (int cur = 0; s_slot[cur].has; cur ^= 1) {
        const NextSlot &slot = s_slot[cur];
        const int k = slot.item.k;
        claim.begin(&s_slot[cur ^ 1], &s_plan[cur ^ 1]);
        bool ok = true;
        if (k < 0 || k >= m.K + m.NP) {
            if (threadIdx.x == 0) atomicOr(err, ERR_BAD_ITEM);
        } else {
            const Smem S = carve(smem, s_plan[cur]);
            ok = run_item<false, false, true>(k >= m.K, m, s_plan[cur], S, slot.item.blk, slot.blk[1] - slot.blk[0],
                                              slot.item.mask, &slot.item, nullptr, err, &s_bar, phase, claim);
        }
        claim.finish();
        if (!ok) return;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Device-resident serving loop.  Work items arrive in a ring in mapped host
// memory; the host writes an item and then publishes its ticket by a release
// store of the ring tail.  Each CTA claims the next published ticket (acquire
// load of the tail at system scope, CAS on a device counter), builds the
// cluster into the cache slot the item points to, then fences and stores the
// ticket into the slot's done flag (release, system scope).  A CTA that finds
// no published work sleeps and polls again; after idle_ns without a claim,
// or when the host raises the stop flag, it returns.  Every wait is bounded.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long ld_acquire_sys(const long long *p) {
    long long v;
    asm volatile("ld.acquire.sys.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_acquire_sys32(const int *p) {
    int v;
    asm volatile("ld.acquire.sys.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_sys(long long *p, long long v) {
    asm volatile("st.release.sys.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void __launch_bounds__(1024) serve_kernel(DevMesh m, const SmemPlan *plans, ServeRing ring,
                                                     int32_t *err) {
    extern __shared__ __align__(16) char smem[];
    __shared__ __align__(16) SmemPlan s_plan;
    __shared__ long long s_t;
    __shared__ WorkItem s_item;
    __shared__ __align__(8) uint64_t s_bar;
    init_barrier<false>(&s_bar);
    uint32_t phase = 0;
    NoClaim none;
    unsigned long long last = globaltimer();
    __shared__ unsigned long long s_claim;
    for (;;) {
        if (threadIdx.x == 0) {
            long long t = -1;
            unsigned sleep_ns = 256;
            for (;;) {
                if (ld_acquire_sys32(ring.stop)) break;
                const long long pub = ld_acquire_sys(ring.tail);
                const unsigned long long cur = *reinterpret_cast<volatile unsigned long long *>(ring.next);
                if ((long long)cur < pub) {
                    if (atomicCAS(ring.next, cur, cur + 1ull) == cur) {
                        t = (long long)cur;
                        break;
                    }
                    continue;
                }
                if (globaltimer() - last > ring.idle_ns) break;
                __nanosleep(sleep_ns);
                if (sleep_ns < 2048) sleep_ns *= 2;
            }
            if (t >= 0) {
                s_claim = globaltimer();
                const int slot = int(t % ring.cap);
                const volatile int32_t *src = reinterpret_cast<const volatile int32_t *>(ring.items + slot);
                int32_t *dst = reinterpret_cast<int32_t *>(&s_item);
                for (int w = 0; w < int(sizeof(WorkItem) / 4); ++w) dst[w] = src[w];
            }
            s_t = t;
        }
        __syncthreads();
        const long long t = s_t;
        if (t < 0) break;
        bool go_on = true;
        if (s_item.k >= 0 && s_item.k < m.K) {
            load_plan(s_plan, plans + s_item.k);  // the cluster's own plan
            __syncthreads();
            const Smem S = carve(smem, s_plan);
            go_on = run_cluster<false, false, false, true>(BlockTeam{}, m, s_plan, S, s_item.blk, m.blk_off[s_item.k + 1] - m.blk_off[s_item.k],
                                              s_item.mask, &s_item, nullptr, err, &s_bar, phase, none);
        } else if (threadIdx.x == 0) {
            atomicOr(err, ERR_BAD_ITEM);
        }
        if (!go_on) break;  // a bounded wait ran out; the slot stays not done
        __syncthreads();
        if (threadIdx.x == 0) {
            const int slot = int(t % ring.cap);
            ring.times[2 * slot] = (long long)s_claim;
            ring.times[2 * slot + 1] = (long long)globaltimer();
            __threadfence_system();
            st_release_sys(ring.done + slot, t);
        }
        last = globaltimer();
    }
}

// Output placement: exclusive scans, over the listed clusters, of the
// lengths of the ten output arrays, then one work item per cluster with its
// output pointers.  Three launches: block sums, a scan of the block sums,
// then per-block scans that write the items (one launch for short lists).  arrays_base holds the base
// pointers of the ten output arrays (its k / mask / blk fields are ignored).
constexpr int kBasesThreads = 256;
constexpr int NA = 10;

__device__ __forceinline__ void item_lengths(const DevMesh &m, const int32_t *ids, const int64_t *sizes,
                                             uint32_t mask, int idx, int64_t *L) {
    const int k = ids ? ids[idx] : idx;
    const int64_t *sz = sizes + int64_t(k) * SZ_N;
    // a cluster's offset arrays end with one extra entry; a part's only when
    // it is its cluster's last
    int64_t nvo, nown, fin;
    if (k < m.K) {
        nvo = m.I_V[k + 1] - m.I_V[k];
        nown = m.I_T[k + 1] - m.I_T[k];
        fin = 1;
    } else {
        const PartInfo &p = m.parts[k - m.K];
        nvo = p.nvo;
        nown = p.n_rows;
        fin = p.last;
    }
    const bool vt = mask & R_VT, vv = mask & R_VV, et = mask & R_ET, tt = mask & R_TT;
    L[0] = vt ? nvo + fin : 0;
    L[1] = vt ? sz[SZ_VT] : 0;
    L[2] = vv ? nvo + fin : 0;
    L[3] = vv ? sz[SZ_VV] : 0;
    L[4] = et ? nvo + fin : 0;
    L[5] = et ? sz[SZ_E] : 0;
    L[6] = et ? sz[SZ_E] + fin : 0;
    L[7] = et ? sz[SZ_ET] : 0;
    L[8] = tt ? nown + fin : 0;
    L[9] = tt ? sz[SZ_TT] : 0;
}

// block-wide exclusive scan of NA int64 values per thread; totals -> tot[]
__device__ __forceinline__ void block_scan_na(int64_t *v, int64_t (*s_warp)[NA], int64_t *tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t incl[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) {
        int64_t x = v[a];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        incl[a] = x;
        if (lane == 31) s_warp[warp][a] = x;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const int64_t w = lane < nw ? s_warp[lane][a] : 0;
            int64_t x = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(FULL, x, o);
                if (lane >= o) x += y;
            }
            if (lane < nw) s_warp[lane][a] = x - w;
            if (lane == 31) tot[a] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < NA; ++a) v[a] = s_warp[warp][a] + incl[a] - v[a];
}

__global__ void __launch_bounds__(kBasesThreads) bases_sum_kernel(DevMesh m, const int32_t *ids, int32_t n,
                                                                  const int64_t *sizes, uint32_t mask,
                                                                  int64_t *bsum, int32_t *tickets, int nt) {
    __shared__ int64_t s_warp[32][NA];
    __shared__ int64_t s_tot[NA];
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && int(threadIdx.x) < nt) tickets[threadIdx.x] = 0;
    int64_t L[NA];
    if (idx < n) item_lengths(m, ids, sizes, mask, idx, L);
    else
        for (int a = 0; a < NA; ++a) L[a] = 0;
    block_scan_na(L, s_warp, s_tot);
    if (threadIdx.x < NA) bsum[int64_t(blockIdx.x) * NA + threadIdx.x] = s_tot[threadIdx.x];
}

__global__ void __launch_bounds__(kBasesThreads) bases_scan_kernel(int32_t nblocks, int64_t *bsum,
                                                                   int64_t *totals) {
    __shared__ int64_t s_warp[32][NA];
    __shared__ int64_t s_tot[NA];
    __shared__ int64_t s_run[NA];
    if (threadIdx.x < NA) s_run[threadIdx.x] = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nblocks; b0 += blockDim.x) {
        const int b = b0 + threadIdx.x;
        int64_t v[NA];
        for (int a = 0; a < NA; ++a) v[a] = b < nblocks ? bsum[int64_t(b) * NA + a] : 0;
        block_scan_na(v, s_warp, s_tot);
        if (b < nblocks)
            for (int a = 0; a < NA; ++a) bsum[int64_t(b) * NA + a] = v[a] + s_run[a];
        __syncthreads();
        if (threadIdx.x < NA) s_run[threadIdx.x] += s_tot[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x < NA) totals[threadIdx.x] = s_run[threadIdx.x];
}

// the idx-th work item: its arrays start `run` after `before` in each base
__device__ __forceinline__ void write_item(const DevMesh &m, const int32_t *ids, int idx, uint32_t mask,
                                           int32_t *const *base, const int64_t *before, const int64_t *run,
                                           WorkItem *items) {
    const int k = ids ? ids[idx] : idx;
    WorkItem w;
    w.k = k;
    w.mask = mask;
    w.blk = m.blk_off[k];
    int32_t *p[NA];
    for (int a = 0; a < NA; ++a) p[a] = base[a] ? base[a] + before[a] + run[a] : nullptr;
    w.vt_off = p[0]; w.vt_val = p[1]; w.vv_off = p[2]; w.vv_val = p[3];
    w.eu_off = p[4]; w.e_w = p[5]; w.et_off = p[6]; w.et_val = p[7];
    w.tt_off = p[8]; w.tt_val = p[9];
    items[idx] = w;
}

__global__ void __launch_bounds__(kBasesThreads) bases_write_kernel(DevMesh m, const int32_t *ids, int32_t n,
                                                                    const int64_t *sizes, uint32_t mask,
                                                                    const WorkItem *arrays_base,
                                                                    const int64_t *bsum, WorkItem *items) {
    __shared__ int64_t s_warp[32][NA];
    __shared__ int64_t s_tot[NA];
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    int64_t L[NA];
    if (idx < n) item_lengths(m, ids, sizes, mask, idx, L);
    else
        for (int a = 0; a < NA; ++a) L[a] = 0;
    int64_t run[NA];
    for (int a = 0; a < NA; ++a) run[a] = L[a];
    block_scan_na(run, s_warp, s_tot);
    if (idx >= n) return;
    const int64_t *bb = bsum + int64_t(blockIdx.x) * NA;
    int32_t *base[NA] = {arrays_base->vt_off, arrays_base->vt_val, arrays_base->vv_off, arrays_base->vv_val,
                         arrays_base->eu_off, arrays_base->e_w,    arrays_base->et_off, arrays_base->et_val,
                         arrays_base->tt_off, arrays_base->tt_val};
    write_item(m, ids, idx, mask, base, bb, run, items);
}

// Up to kBasesOne clusters: one launch, one block, which also zeroes the
// builds' ticket counters.  (The three launches and a memset per size bin are
// most of a small build: 16^3 grid, 128 clusters, 25.3 us a build of two
// bins with them, 11.6 us without and merged into one.)
constexpr int kBasesOne = 1024;
__global__ void __launch_bounds__(kBasesThreads) bases_one_kernel(DevMesh m, const int32_t *ids, int32_t n,
                                                                  const int64_t *sizes, uint32_t mask,
                                                                  const WorkItem *arrays_base, WorkItem *items,
                                                                  int64_t *totals, int32_t *tickets, int nt) {
    __shared__ int64_t s_warp[32][NA];
    __shared__ int64_t s_tot[NA];
    if (int(threadIdx.x) < nt) tickets[threadIdx.x] = 0;
    int32_t *base[NA] = {arrays_base->vt_off, arrays_base->vt_val, arrays_base->vv_off, arrays_base->vv_val,
                         arrays_base->eu_off, arrays_base->e_w,    arrays_base->et_off, arrays_base->et_val,
                         arrays_base->tt_off, arrays_base->tt_val};
    int64_t before[NA] = {};
    for (int b0 = 0; b0 < n; b0 += kBasesThreads) {
        const int idx = b0 + threadIdx.x;
        int64_t run[NA];
        if (idx < n) item_lengths(m, ids, sizes, mask, idx, run);
        else
            for (int a = 0; a < NA; ++a) run[a] = 0;
        block_scan_na(run, s_warp, s_tot);
        if (idx < n) write_item(m, ids, idx, mask, base, before, run, items);
        for (int a = 0; a < NA; ++a) before[a] += s_tot[a];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int a = 0; a < NA; ++a) totals[a] = before[a];
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

static int64_t a16(int64_t x) { return (x + 15) & ~int64_t(15); }

static int64_t pow2_at_least(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

Caps caps_of(const ClusterStat &s, const int64_t *sizes) {
    Caps c{};
    c.blk_words = int32_t(blk_words(s.nv_loc, s.n_ext, s.n_own, s.n_halo, s.n_bnd, s.xmap));
    c.nv_own = s.nv_own;
    c.n_vt = s.n_vt;
    c.n_own = s.n_own;
    c.nv_loc = s.nv_loc;
    c.nv_nb = s.nv_nb;
    c.max_deg = s.max_deg;
    c.max_e = s.n_e;
    if (sizes) {
        c.max_vv = int32_t(sizes[SZ_VV]);
        c.max_e = int32_t(sizes[SZ_E]);
        c.max_etv = int32_t(sizes[SZ_ET]);
        c.max_tt = int32_t(sizes[SZ_TT]);
    }
    c.hcap = int32_t(std::max<int64_t>(64, pow2_at_least(2 * int64_t(s.n_bnd) + 1)));
    c.n_tot = s.n_ext + s.n_own + s.n_halo;
    c.n_star = s.n_ext + s.n_own;
    return c;
}

int64_t class_bytes(const Caps &c, int threads) {
    const int64_t nwarp = threads / 32, nvo = c.nv_own;
    const int64_t W = std::max(1, (c.nv_nb + 31) / 32) | 1, nch = std::max(1, (c.max_deg + 31) / 32);
    const int64_t pad = (nvo + 1) & ~int64_t(1);
    const int64_t fixed = 512 + a16(4 * int64_t(c.blk_words)) + 3 * a16(4 * (nvo + 1)) + a16(2 * int64_t(c.n_vt)) +
                          a16(8 * int64_t(c.n_own)) + a16((c.max_deg > 256 ? 8 : 4) * int64_t(c.n_star));
    const int64_t edges = a16(std::max<int64_t>(4 * int64_t(c.max_e) * nch,
                                                a16(2 * int64_t(c.max_vv)) + 2 * int64_t(c.max_e)));
    const int64_t work = std::max(std::max(a16(2 * nwarp * pad) + 4 * nwarp * pad, a16(4 * nvo * W) + nvo * W),
                                  std::max(2 * int64_t(c.max_etv), a16(4 * int64_t(c.hcap)) +
                                                                       a16(4 * (int64_t(c.n_own) + 1)) +
                                                                       2 * int64_t(c.max_tt)));
    return fixed + edges + a16(work);
}

int64_t estimate_class(const ClusterStat &s, int threads) {
    Caps c = caps_of(s, nullptr);
    c.max_vv = 2 * s.n_e;           // each edge is in two VV rows (within the working set, about)
    c.max_etv = s.n_vt + s.n_vt / 2;  // an incidence (x, t) meets 1.5 vertices of t above x on average
    c.max_tt = 4 * s.n_own;
    return class_bytes(c, threads);
}

// The layout of kTight: no region beside those of class_bytes, none of them
// larger, so that what the size class lets into shared memory fits there.
static SmemPlan plan_tight(const Caps &c, int threads) {
    SmemPlan p{};
    p.threads = threads;
    p.caps = c;
    const int64_t nvo = c.nv_own;
    p.W = std::max(1, (c.nv_nb + 31) / 32) | 1;
    p.nch = std::max(1, (c.max_deg + 31) / 32);
    p.mode = kTight | (c.max_deg > 256 ? kJpos16 : 0);
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        const int64_t at = off;
        off = a16(off + bytes);
        return int32_t(std::min<int64_t>(at, INT32_MAX));
    };
    p.scan = take(4 * kScanWords);
    p.blk = take(4 * int64_t(c.blk_words));
    p.vt_off = take(4 * (nvo + 1));
    p.fill = p.vt_list = take(2 * int64_t(c.n_vt));
    p.c_vv = take(4 * (nvo + 1));
    p.c_e = take(4 * (nvo + 1));
    p.jpos = take((p.mode & kJpos16 ? 8 : 4) * int64_t(c.n_star));
    // r2: VV staging, then the edge masks
    p.et_b = p.long_rows = p.r2 = take(std::max(4 * int64_t(c.max_e) * p.nch, 2 * int64_t(c.max_vv)));
    p.nbr = take(8 * int64_t(c.n_own));
    // r1: bitmaps + rank prefixes | ET staging | face hash + TT counts + TT staging
    const int64_t bm = a16(4 * nvo * p.W), hs = a16(4 * int64_t(c.hcap)), tc = a16(4 * (int64_t(c.n_own) + 1));
    p.ex = p.r1 =
        take(std::max(std::max(bm + nvo * p.W, 2 * int64_t(c.max_etv)), hs + tc + 2 * int64_t(c.max_tt)));
    p.pre = int32_t(p.r1 + bm);
    p.tcnt = int32_t(p.r1 + hs);
    p.st_tt = int32_t(p.r1 + hs + tc);
    p.total = off > INT32_MAX ? INT32_MAX : int32_t(off);
    return p;
}

SmemPlan plan_smem(const Caps &c, int threads, bool shared) {
    SmemPlan p{};
    p.threads = threads;
    p.caps = c;
    const int64_t nvo = c.nv_own;
    p.W = std::max(1, (c.nv_nb + 31) / 32) | 1;  // row stride of the bitmaps (odd)
    p.nch = std::max(1, (c.max_deg + 31) / 32);
    p.mode = (c.max_deg > 256 ? kJpos16 : 0) | (c.n_star <= 16383 ? kKeyed : 0);  // 4 * tet + slot below 0xffff
    // The fill's rows are padded to one odd number of words (no count pass
    // before it, and a thread per row meets no bank conflict) unless that
    // takes over a quarter more than compact rows, as on irregular meshes.
    const int64_t stride = 2 * (((c.max_deg + 1) / 2) | 1);
    p.stride = c.max_deg <= 62 && 4 * nvo * stride <= 5 * int64_t(c.n_vt) ? int32_t(stride) : 0;
    for (;;) {
        int64_t off = 0;
        auto take = [&](int64_t bytes) {
            const int64_t at = off;
            off = a16(off + bytes);
            return int32_t(std::min<int64_t>(at, INT32_MAX));
        };
        p.scan = take(4 * kScanWords);
        p.blk = take(4 * int64_t(c.blk_words));
        p.vt_off = take(4 * (nvo + 1));
        p.vt_list = take(2 * int64_t(c.n_vt));
        p.c_vv = take(4 * (nvo + 1));
        p.c_e = take(4 * (nvo + 1));
        p.jpos = take(std::max((p.mode & kJpos16 ? 8 : 4) * int64_t(c.n_star), 4 * int64_t(c.max_e)));
        // r2: fill cursors, then VV staging; first ET entries, long rows; then
        // the edge masks.  The rows in arrival order (padded, or compact from a
        // word each) end with nbr and reach back into what r2 leaves free.
        const int64_t vv = a16(std::max(2 * int64_t(c.max_vv), 4 * nvo)), eb = a16(4 * nvo);
        const int64_t lr = c.max_deg > 32 ? a16(2 * nvo) : 0;
        const int64_t em = 4 * int64_t(c.max_e) * p.nch;
        const int64_t eb0 = p.nch == 1 ? std::max(vv, a16(em)) : vv;  // single-word masks leave the ET entries in place
        p.r2 = take(std::max<int64_t>(em, eb0 + eb + lr));
        p.et_b = int32_t(p.r2 + eb0);
        p.long_rows = int32_t(p.r2 + eb0 + eb);
        const int64_t n_fill = a16(p.stride ? 2 * nvo * p.stride : 2 * (int64_t(c.n_vt) + nvo + 4));
        p.nbr = take(std::max(8 * int64_t(c.n_own), p.r2 + eb0 + eb + lr + n_fill - off));
        p.fill = int32_t(std::min<int64_t>(off - n_fill, INT32_MAX));
        // r1: bitmaps + rank prefixes | ET staging + the edges' lower vertices
        // | face hash + TT counts + TT staging
        const int64_t bm = a16(4 * nvo * p.W), et = a16(2 * int64_t(c.max_etv));
        const int64_t hs = a16(4 * int64_t(c.hcap)), tc = a16(4 * (int64_t(c.n_own) + 1));
        p.r1 = take(std::max(std::max(bm + nvo * p.W, et + 2 * int64_t(c.max_e)), hs + tc + 2 * int64_t(c.max_tt)));
        p.pre = int32_t(p.r1 + bm);
        p.ex = int32_t(p.r1 + et);
        p.tcnt = int32_t(p.r1 + hs);
        p.st_tt = int32_t(p.r1 + hs + tc);
        p.total = off > INT32_MAX ? INT32_MAX : int32_t(off);
        if (p.stride && off > kPaddedFit) {
            p.stride = 0;  // compact rows take less
            continue;
        }
        if (!shared || off <= kCompactFit) return p;
        const SmemPlan t = plan_tight(c, threads);
        return t.total <= kCtaBytes ? t : p;
    }
}

int kernel_smem_limit() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

int device_sm_count() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
}

// Largest dynamic shared memory a cluster kernel can be launched with: the
// opt-in limit less the kernels' own static shared memory.
int dynamic_smem_limit() {
    const int optin = kernel_smem_limit();
    int stat = 0;
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, build_kernel<false>) == cudaSuccess) stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, build_one_kernel<false>) == cudaSuccess)
        stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, count_kernel<false>) == cudaSuccess) stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, serve_kernel) == cudaSuccess) stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, build_kernel_pi) == cudaSuccess) stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, count_kernel_pi) == cudaSuccess) stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, build_kernel_team<false>) == cudaSuccess)
        stat = std::max(stat, int(a.sharedSizeBytes));
    if (cudaFuncGetAttributes(&a, build_kernel_team<true>) == cudaSuccess)
        stat = std::max(stat, int(a.sharedSizeBytes));
    cudaGetLastError();
    return optin - stat;
}

bool prepare_kernels(int smem) {
    // the attribute belongs to the kernel, shared by every context of the
    // process on this device: it only ever grows (a larger limit does not
    // change the occupancy of launches that ask for less)
    static std::mutex mu;
    static int granted[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    const int d = dev >= 0 && dev < 64 ? dev : 0;
    smem = std::min(std::max(smem, granted[d]), dynamic_smem_limit());
    bool ok = cudaFuncSetAttribute(build_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
              cudaSuccess;
    ok &= cudaFuncSetAttribute(build_one_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
          cudaSuccess;
    ok &= cudaFuncSetAttribute(count_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
    ok &= cudaFuncSetAttribute(build_kernel_pi, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
    ok &= cudaFuncSetAttribute(count_kernel_pi, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
    ok &= cudaFuncSetAttribute(build_kernel_team<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
          cudaSuccess;
    ok &= cudaFuncSetAttribute(build_kernel_team<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ==
          cudaSuccess;
    cudaGetLastError();
    if (ok) granted[d] = smem;
    return ok;
}

int max_ctas_per_sm(const SmemPlan &plan, bool spill, bool per_item) {
    int a = 0, b = 0;
    cudaError_t e1, e2;
    if (per_item) {
        e1 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, build_kernel_pi, plan.threads, plan.total);
        e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, count_kernel_pi, plan.threads, plan.total);
    } else if (spill) {
        e1 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, build_kernel<true>, plan.threads, 0);
        e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, count_kernel<true>, plan.threads, 0);
    } else {
        e1 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, build_kernel<false>, plan.threads, plan.total);
        e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, count_kernel<false>, plan.threads, plan.total);
    }
    if (e1 != cudaSuccess || e2 != cudaSuccess) return 0;
    return a < b ? a : b;
}

int per_item_fit(int ctas, int threads) {
    SmemPlan p{};
    p.threads = threads;
    cudaFuncAttributes a;
    int dev = 0, sm = 0, reserved = 0;
    cudaGetDevice(&dev);
    if (max_ctas_per_sm(p, false, true) < ctas || cudaFuncGetAttributes(&a, build_kernel_pi) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    // (the occupancy API answers within the limit granted so far; a CTA's
    // share is whole 128-byte units)
    return std::min((sm / ctas & ~127) - reserved, kernel_smem_limit()) - int(a.sharedSizeBytes);
}

int max_ctas_per_sm_teams(SmemPlan &plan, int teams) {
    if (teams < 1 || teams > kMaxTeams || plan.threads % 32 || plan.threads * teams > kMaxTeamBlock) return 0;
    const int nt = plan.threads * teams;
    const size_t smem = size_t(plan.total) * teams;
    int a = 0, lean = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, build_kernel_team<false>, nt, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lean, build_kernel_team<true>, nt, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const bool take = lean >= 2 * a;
    plan.mode = take ? plan.mode | kLeanTeam : plan.mode & ~kLeanTeam;
    return take ? lean : a;
}

int launch_count_pass(const DevMesh &m, const SmemPlan &plan, const int32_t *ids, int32_t n, int64_t *sizes_out,
                      int32_t *err, int32_t *ticket, int grid, void *stream, char *gscratch, uint32_t mask,
                      const SmemPlan *plans) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaMemsetAsync(ticket, 0, sizeof(int32_t), s);
    if (plans)
        count_kernel_pi<<<grid, plan.threads, plan.total, s>>>(m, plans, ids, n, sizes_out, err, ticket, mask);
    else if (gscratch)
        count_kernel<true><<<grid, plan.threads, 0, s>>>(m, plan, ids, n, sizes_out, err, ticket, gscratch, mask);
    else
        count_kernel<false><<<grid, plan.threads, plan.total, s>>>(m, plan, ids, n, sizes_out, err, ticket, nullptr,
                                                                  mask);
    return int(cudaGetLastError());
}

int bases_scratch_words(int32_t n) { return ((n + kBasesThreads - 1) / kBasesThreads) * NA; }

int launch_bases(const DevMesh &m, const int32_t *ids, int32_t n, const int64_t *sizes, uint32_t mask,
                 const WorkItem *arrays_base, WorkItem *items, int64_t *totals_out, int64_t *bsum, int32_t *tickets,
                 int nt, void *stream, int *launches) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int nb = (n + kBasesThreads - 1) / kBasesThreads;
    if (launches) *launches = 0;
    if (nb == 0) return 0;
    if (nt > kBasesThreads) return int(cudaErrorInvalidValue);
    if (n <= kBasesOne) {
        bases_one_kernel<<<1, kBasesThreads, 0, s>>>(m, ids, n, sizes, mask, arrays_base, items, totals_out, tickets,
                                                     nt);
        if (launches) *launches = 1;
        return int(cudaGetLastError());
    }
    bases_sum_kernel<<<nb, kBasesThreads, 0, s>>>(m, ids, n, sizes, mask, bsum, tickets, nt);
    bases_scan_kernel<<<1, kBasesThreads, 0, s>>>(nb, bsum, totals_out);
    bases_write_kernel<<<nb, kBasesThreads, 0, s>>>(m, ids, n, sizes, mask, arrays_base, bsum, items);
    if (launches) *launches = 3;
    return int(cudaGetLastError());
}

int launch_build(const DevMesh &m, const SmemPlan &plan, const WorkItem *items, const int32_t *order, int32_t n,
                 int32_t *err, int32_t *ticket, int grid, void *stream, char *gscratch, const SmemPlan *plans,
                 int teams, bool reset) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (reset) cudaMemsetAsync(ticket, 0, sizeof(int32_t), s);
    if (teams > 0) {
        if (plans || gscratch || teams > kMaxTeams || plan.threads * teams > kMaxTeamBlock)
            return int(cudaErrorInvalidValue);
        const auto kernel = (plan.mode & kLeanTeam) ? build_kernel_team<true> : build_kernel_team<false>;
        kernel<<<grid, plan.threads * teams, size_t(plan.total) * teams, s>>>(m, plan, items, order, n, err, ticket,
                                                                             plan.threads);
    } else if (plans) build_kernel_pi<<<grid, plan.threads, plan.total, s>>>(m, plans, items, order, n, err, ticket);
    else if (gscratch) build_kernel<true><<<grid, plan.threads, 0, s>>>(m, plan, items, order, n, err, ticket, gscratch);
    else build_kernel<false><<<grid, plan.threads, plan.total, s>>>(m, plan, items, order, n, err, ticket, nullptr);
    return int(cudaGetLastError());
}

// The serving kernel's shared memory limit, grown like the cluster kernels'.
static void grow_serve_attr(int smem) {
    static std::mutex mu;
    static int granted[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const int d = dev >= 0 && dev < 64 ? dev : 0;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= granted[d]) return;
    if (cudaFuncSetAttribute(serve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess)
        granted[d] = smem;
    cudaGetLastError();
}

int launch_serve(const DevMesh &m, const SmemPlan &plan, const SmemPlan *plans, const ServeRing &ring, int32_t *err,
                 int grid, void *stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    grow_serve_attr(plan.total);
    serve_kernel<<<grid, plan.threads, plan.total, s>>>(m, plans, ring, err);
    return int(cudaGetLastError());
}

int serve_ctas_per_sm(const SmemPlan &plan) {
    int a = 0;
    grow_serve_attr(plan.total);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, serve_kernel, plan.threads, plan.total) != cudaSuccess)
        return 0;
    return a;
}

int launch_build_one(const DevMesh &m, const SmemPlan &plan, const WorkItem *items, int32_t index, int32_t *err,
                     void *stream, char *gscratch) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (gscratch) build_one_kernel<true><<<1, plan.threads, 0, s>>>(m, plan, items, index, err, gscratch);
    else build_one_kernel<false><<<1, plan.threads, plan.total, s>>>(m, plan, items, index, err, nullptr);
    return int(cudaGetLastError());
}

}  // namespace gale

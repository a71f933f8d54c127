// Coboundary relations VE, VF, EF, FT in the ids of the edge / triangle
// enumeration (Section 4.4: coboundary relations are computed by the GPU for
// whole segments; Section 5 evaluates VE, VF, EF and FT among them).
//
// Inputs on the device: the canonical tet rows, each vertex's cluster and
// the enumeration (E, F, I_E, I_F and each segment's ids in vertex-tuple
// order).  The enumeration itself, when made on the device, reads every
// cluster's ET rows from a batched build (enumerate_sorted_device).
//
// Lookup structure, built once per enumeration: the edges and triangles in
// vertex-tuple ("sorted") order, with
//   eo[v]    first sorted edge position with lower vertex v (nv+1 entries),
//   ekw[j]   upper vertex of the j-th sorted edge,
//   feo[j]   first sorted triangle position whose first two vertices are the
//            j-th sorted edge (nE+1 entries),
//   fkc[p]   third vertex of the p-th sorted triangle,
//   e2s, f2s the sorted position of every edge / triangle id.
// An edge (a, b) is then found among a's few upper edges and a triangle
// (a, b, c) among the few triangles over its edge (a, b).
//
// The relations are scattered from the simplices (details at the scatter
// kernels below): every row is a contiguous range of the sorted order (VE(v):
// v's upper edges; EF(e): the triangles over e; VF(v): the triangles with
// lowest vertex v) plus entries that other edges and triangles place after
// counts and an exclusive scan; FT takes two slots per triangle that its tets
// claim (a counted form with cursors and row sorts when a triangle lies in
// three or more tets).  With the sorted numbering only each row's scattered
// prefix needs sorting, and VF is gathered from VE and EF; otherwise rows are
// sorted whole.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "gale_ctx.h"
#include "gale_enum.h"

namespace gale {

// device copies the coboundary pass keeps in the context
struct Cobound {
    uint64_t enm_gen = 0;  // the enumeration the lookup index was made from
    uint64_t dev_gen = 0;  // the enumeration E, F, IE, IF (and ebk, fbk) hold
    int32_t *rows = nullptr, *cluster_of = nullptr;
    int32_t *E = nullptr, *F = nullptr, *ebk = nullptr, *fbk = nullptr;
    int64_t *IE = nullptr, *IF = nullptr;
    int32_t *eo = nullptr, *ekw = nullptr, *feo = nullptr, *fkc = nullptr, *fo = nullptr;
    int32_t *e2s = nullptr, *f2s = nullptr;
    bool sorted_ids = false;

    int32_t *cnt = nullptr;        // counts of the largest relation
    int64_t *bsum = nullptr;       // scan block sums
    int64_t cnt_cap = 0, bsum_cap = 0;
    int32_t *off[4] = {}, *val[4] = {};
    int32_t *scratch = nullptr;    // counters and lookups of the scatter passes
    int64_t scratch_cap = 0;
    int64_t off_cap[4] = {}, val_cap[4] = {};
    int64_t rows_of[4] = {}, len[4] = {};
    bool ft_general = false;       // FT by counts and cursors: some triangle lies in three or more tets
};

void cobound_destroy(gale_ctx *ctx) {
    delete ctx->cb;  // device memory is the context's and goes with it
    ctx->cb = nullptr;
}

namespace {

constexpr int kThreads = 256;
enum { REL_VE = 0, REL_VF = 1, REL_EF = 2, REL_FT = 3 };
// bulk array indices (the order of gale_arrays)
enum { B_VT_OFF = 0, B_VT_VAL = 1, B_VV_OFF = 2, B_VV_VAL = 3, B_ET_UOFF = 4, B_ET_W = 5, B_ET_OFF = 6, B_ET_VAL = 7 };

struct CbMesh {
    const int4 *rows;
    const int32_t *cluster_of, *I_V;
    const int32_t *E, *F, *ebk, *fbk;
    const int64_t *IE, *IF;
    const int32_t *eo, *ekw, *feo, *fkc, *e2s, *f2s;
    // the ET rows of a batched build (the sorted enumeration reads them)
    const int32_t *et_w, *et_off, *et_val;
    const int32_t *et_uoff;          // ET edges per own lower vertex
    const int64_t *base;
    const int64_t *sizes;  // [K][5] per-cluster entries: VT, VV, edges, ET, TT
    int64_t nv, nE, nF;
    bool sorted_ids;
};

// the ET row [b, e) of the edge at sorted position j, whose vertices are
// (a, w); false if the cluster's ET rows do not list that edge there
__device__ bool et_row(const CbMesh &m, int64_t j, int32_t a, int32_t w, int64_t &b, int64_t &e) {
    const int32_t k = m.cluster_of[a];
    const int64_t le = j - m.IE[k];
    if (le < 0 || j >= m.IE[k + 1] || le >= m.sizes[5 * int64_t(k) + 2]) return false;
    const int64_t *B = m.base + 10 * int64_t(k);
    if (m.et_w[B[B_ET_W] + le] != w) return false;
    b = B[B_ET_VAL] + m.et_off[B[B_ET_OFF] + le];
    e = B[B_ET_VAL] + m.et_off[B[B_ET_OFF] + le + 1];
    return true;
}

__device__ __forceinline__ int32_t edge_id(const CbMesh &m, int64_t j) { return m.sorted_ids ? int32_t(j) : m.ebk[j]; }
__device__ __forceinline__ int32_t face_id(const CbMesh &m, int64_t p) { return m.sorted_ids ? int32_t(p) : m.fbk[p]; }

// ---- the relations by scatter, over sorted positions ----
// Every row is [scattered part | contiguous part].  The contiguous part is a
// range the vertex-tuple order gives whole: for VE(v) the edges whose lower
// vertex is v (sorted positions eo[v] ..), for EF(e) the triangles whose
// first two vertices are e (feo[e] ..), for VF(v) the triangles whose lowest
// vertex is v (fo[v] ..).  The other entries come from the edges, triangles
// and tets that hold the row's simplex elsewhere than in front: an edge
// (a, b) is in VE(b); a triangle (a, b, c) is in EF(a, c), EF(b, c), VF(b)
// and VF(c); a tet is in FT of its four faces.  They take slots by atomic
// counters, and a last pass sorts every row by id.  With the sorted
// numbering the scattered ids all precede the contiguous ones, so only the
// scattered prefix moves.

__device__ __forceinline__ int64_t erow(const CbMesh &m, int64_t j) { return m.sorted_ids ? j : m.ebk[j]; }
__device__ __forceinline__ int64_t frow(const CbMesh &m, int64_t p) { return m.sorted_ids ? p : m.fbk[p]; }

struct Scatter {
    int32_t *ve_n;                         // [nv] lower edges of v
    int32_t *ve_rank;                      // [nE] (sorted positions) arrival rank of edge (a, b) among b's
    int32_t *ef_lo, *ef_mid;               // [nE] (sorted positions) triangles (x, u, w), x < u, and
                                           // (u, x, w), u < x < w, of edge (u, w)
    int4 *tri;                             // [nF] sorted positions of the edges (a, c), (b, c) of triangle p, its
                                           // arrival ranks in ef_mid of the one and ef_lo of the other
    int32_t *vf_n, *vf_fill;               // [nv] triangles of v's VF row but its contiguous part; cursor
    int2 *ft_slot;                         // [nF] (row order) the one or two tets of a triangle
    int2 *ef_tail;                         // [nE] (sorted numbering, VF gather) EF(j) after its lower part
    int32_t *cnt;                          // row lengths of the relation being placed
    const int32_t *ve_off, *ef_off, *vf_off, *ft_off;
    int32_t *ve_val, *ef_val, *vf_val, *ft_val;
};

// edges: VE(b) of every edge (a, b).  The counting pass keeps the rank that
// its atomic returns, so that the fill is a plain store.
__global__ void __launch_bounds__(kThreads) k_ve_count(CbMesh m, Scatter sc) {
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m.nE; j += int64_t(gridDim.x) * blockDim.x)
        sc.ve_rank[j] = atomicAdd(&sc.ve_n[m.ekw[j]], 1);
}
__global__ void __launch_bounds__(kThreads) k_ve_fill(CbMesh m, Scatter sc) {
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m.nE; j += int64_t(gridDim.x) * blockDim.x)
        sc.ve_val[sc.ve_off[m.ekw[j]] + sc.ve_rank[j]] = edge_id(m, j);
}

// triangles: EF(a, c), EF(b, c), VF(b), VF(c) of every triangle (a, b, c).
// The two edge searches advance together, and the counting pass keeps the
// ranks its atomics return, so that the EF fill has none (at 128^3 the two
// passes took 0.61 ms with counts and fill cursors, and 0.07 ms to set these).
template <bool FILL>
__global__ void __launch_bounds__(kThreads) k_sc_tris(CbMesh m, Scatter sc, bool ef, bool vf, int32_t *err) {
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < m.nF; p += int64_t(gridDim.x) * blockDim.x) {
        const int32_t id = int32_t(face_id(m, p));
        if (FILL) {
            if (ef) {
                const int4 t = sc.tri[p];
                if (t.x >= 0) {
                    sc.ef_val[sc.ef_off[erow(m, t.x)] + sc.ef_lo[t.x] + t.z] = id;
                    sc.ef_val[sc.ef_off[erow(m, t.y)] + t.w] = id;
                }
            }
            if (vf) {
                const int32_t *t = m.F + 3 * int64_t(id);
                sc.vf_val[atomicAdd(&sc.vf_fill[t[1]], 1)] = id;
                sc.vf_val[atomicAdd(&sc.vf_fill[t[2]], 1)] = id;
            }
            continue;
        }
        const int32_t *t = m.F + 3 * int64_t(id);
        const int32_t a = t[0], b = t[1], c = t[2];
        if (ef) {
            int32_t l0 = m.eo[a], l1 = m.eo[b];
            const int32_t e0 = m.eo[a + 1], e1 = m.eo[b + 1];
            int32_t h0 = e0, h1 = e1;
            while (l0 < h0 || l1 < h1) {
                const int32_t m0 = (l0 + h0) >> 1, m1 = (l1 + h1) >> 1;
                const int32_t w0 = l0 < h0 ? m.ekw[m0] : 0, w1 = l1 < h1 ? m.ekw[m1] : 0;
                if (l0 < h0) { if (w0 < c) l0 = m0 + 1; else h0 = m0; }
                if (l1 < h1) { if (w1 < c) l1 = m1 + 1; else h1 = m1; }
            }
            if (l0 >= e0 || l1 >= e1 || m.ekw[l0] != c || m.ekw[l1] != c) {
                atomicOr(err, ERR_BAD_BLOCK);
                sc.tri[p] = make_int4(-1, -1, 0, 0);
            } else {
                const int32_t rm = atomicAdd(&sc.ef_mid[l0], 1), rl = atomicAdd(&sc.ef_lo[l1], 1);
                sc.tri[p] = make_int4(l0, l1, rm, rl);
            }
        }
        if (vf) {
            atomicAdd(&sc.vf_n[b], 1);
            atomicAdd(&sc.vf_n[c], 1);
        }
    }
}
// FT: a triangle lies in one or two tets, so each has two slots (row order);
// every tet exchanges itself into the first slot of each of its four faces
// and moves what it finds there to the second, and one scan over the
// triangles places and writes the rows (smaller tet first).  A third tet
// overwrites a slot: the entries then sum to less than four a tet.
// MODE: FT_SLOTS claims the slots; FT_COUNT counts each triangle's tets
// (sc.cnt, by row); FT_FILL places them by cursors (sc.cnt zeroed) in rows
// that a sort then orders - the form for a mesh with a triangle in three
// or more tets.
// A tet's three edge searches and its face scans advance together, so that
// their loads overlap: at 128^3 the claims take 0.60 ms one search after the
// other, with compare-and-swap on both slots and blocks striding over the
// whole mesh.
enum { FT_SLOTS = 0, FT_COUNT = 1, FT_FILL = 2 };
constexpr int kFtStrip = 1024;
template <int MODE>
__global__ void __launch_bounds__(kThreads) k_ft_tets(CbMesh m, Scatter sc, int64_t nT, int32_t *err) {
    // strips of kFtStrip consecutive tets, whose index entries stay in one
    // SM's L1, while the blocks together move through the mesh (and L2)
    for (int64_t i = int64_t(blockIdx.x) * kFtStrip + threadIdx.x; i < nT;
         i += (i % kFtStrip + kThreads < kFtStrip) ? kThreads : int64_t(gridDim.x - 1) * kFtStrip + kThreads) {
        const int64_t t = i;
        const int4 r = m.rows[t];
        // sorted positions of the edges (a, b), (a, c), (b, c)
        const int32_t a0 = m.eo[r.x], a1 = m.eo[r.x + 1], b0 = m.eo[r.y], b1 = m.eo[r.y + 1];
        int32_t l0 = a0, h0 = a1, l1 = a0, h1 = a1, l2 = b0, h2 = b1;
        while (l0 < h0 || l1 < h1 || l2 < h2) {
            const int32_t m0 = (l0 + h0) >> 1, m1 = (l1 + h1) >> 1, m2 = (l2 + h2) >> 1;
            const int32_t w0 = l0 < h0 ? m.ekw[m0] : 0, w1 = l1 < h1 ? m.ekw[m1] : 0, w2 = l2 < h2 ? m.ekw[m2] : 0;
            if (l0 < h0) { if (w0 < r.y) l0 = m0 + 1; else h0 = m0; }
            if (l1 < h1) { if (w1 < r.z) l1 = m1 + 1; else h1 = m1; }
            if (l2 < h2) { if (w2 < r.z) l2 = m2 + 1; else h2 = m2; }
        }
        if (l0 >= a1 || l1 >= a1 || l2 >= b1) {
            atomicOr(err, ERR_BAD_BLOCK);
            continue;
        }
        const int32_t s0 = m.feo[l0], e0 = m.feo[l0 + 1], s1 = m.feo[l1], e1 = m.feo[l1 + 1];
        const int32_t s2 = m.feo[l2], e2 = m.feo[l2 + 1];
        const bool edges = m.ekw[l0] == r.y && m.ekw[l1] == r.z && m.ekw[l2] == r.z;
        int32_t f[4] = {-1, -1, -1, -1};
        const int32_t len = max(e0 - s0, max(e1 - s1, e2 - s2));
        for (int32_t k = 0; k < len; ++k) {
            const int32_t c0 = s0 + k < e0 ? m.fkc[s0 + k] : -1, c1 = s1 + k < e1 ? m.fkc[s1 + k] : -1;
            const int32_t c2 = s2 + k < e2 ? m.fkc[s2 + k] : -1;
            if (c0 == r.z) f[0] = s0 + k;
            if (c0 == r.w) f[1] = s0 + k;
            if (c1 == r.w) f[2] = s1 + k;
            if (c2 == r.w) f[3] = s2 + k;
            if (min(min(f[0], f[1]), min(f[2], f[3])) >= 0) break;
        }
        if (!edges || min(min(f[0], f[1]), min(f[2], f[3])) < 0) {
            atomicOr(err, ERR_BAD_BLOCK);
            continue;
        }
        int32_t old[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t row = frow(m, f[q]);
            if (MODE == FT_SLOTS) {
                old[q] = atomicExch(&sc.ft_slot[row].x, int32_t(t));
            } else {
                const int32_t c = atomicAdd(&sc.cnt[row], 1);
                if (MODE == FT_FILL) sc.ft_val[sc.ft_off[row] + c] = int32_t(t);
            }
        }
        if (MODE == FT_SLOTS) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (old[q] >= 0) sc.ft_slot[frow(m, f[q])].y = old[q];
        }
    }
}

// row lengths: scattered part + contiguous part
__global__ void __launch_bounds__(kThreads) k_len_ve(CbMesh m, Scatter sc) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < m.nv; v += int64_t(gridDim.x) * blockDim.x)
        sc.cnt[v] = sc.ve_n[v] + (m.eo[v + 1] - m.eo[v]);
}
// cursors (first-appearance numbering): every scattered part's first slot
__global__ void __launch_bounds__(kThreads) k_cursors(CbMesh m, Scatter sc) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < m.nv; v += int64_t(gridDim.x) * blockDim.x)
        sc.vf_fill[v] = sc.vf_off[v];
}
__global__ void __launch_bounds__(kThreads) k_len_vf(CbMesh m, Scatter sc, const int32_t *fo) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < m.nv; v += int64_t(gridDim.x) * blockDim.x)
        sc.cnt[v] = sc.vf_n[v] + (fo[v + 1] - fo[v]);
}
// vf: edge (a, b) gives VF(b) its middle and contiguous EF entries (sorted
// numbering, see k_vf_gather)
__global__ void __launch_bounds__(kThreads) k_len_ef(CbMesh m, Scatter sc, bool vf) {
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m.nE; j += int64_t(gridDim.x) * blockDim.x) {
        const int32_t tail = sc.ef_mid[j] + (m.feo[j + 1] - m.feo[j]);
        sc.cnt[erow(m, j)] = sc.ef_lo[j] + tail;
        if (vf) atomicAdd(&sc.vf_n[m.ekw[j]], tail);
    }
}

// Row sorts.  Only a row's scattered prefix needs ordering with the sorted
// numbering (its entries all precede, and are smaller than, the contiguous
// part); otherwise the whole row does.
__device__ __forceinline__ void insertion_sort(int32_t *o, int32_t n) {
    for (int32_t i = 1; i < n; ++i) {
        const int32_t y = o[i];
        int32_t j = i - 1;
        while (j >= 0 && o[j] > y) {
            o[j + 1] = o[j];
            --j;
        }
        o[j + 1] = y;
    }
}

// ascending bitonic sort of N values held in registers (all indices are
// compile-time constants once unrolled)
template <int N>
__device__ __forceinline__ void bitonic_regs(int32_t (&x)[N]) {
#pragma unroll
    for (int k = 2; k <= N; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const int32_t a = x[i], b = x[l];
                    const bool asc = (i & k) == 0;
                    x[i] = asc ? min(a, b) : max(a, b);
                    x[l] = asc ? max(a, b) : min(a, b);
                }
            }
}

// one thread per row: prefixes of up to N entries are sorted in registers,
// longer ones in place.  A block's rows are one contiguous span of the
// values: it is staged through shared memory when it fits, so that loads
// and stores are coalesced.  FRONT writes the row's contiguous part first (VE:
// v's upper edges; EF: the triangles over the edge; VF: the triangles with
// lowest vertex v).
enum { FRONT_NONE = 0, FRONT_EF = 1, FRONT_VF = 2, FRONT_VE = 3 };
// SPAN: int32 entries of a staged span (0: rows are sorted where they are).
// With the sorted numbering, EF's sort also records for each edge the range
// of its entries after the lower part (the VF gather reads them).
template <int N, int FRONT, int SPAN>
__global__ void __launch_bounds__(kThreads) k_sort_rows(CbMesh m, Scatter sc, int64_t rows, const int32_t *off,
                                                        int32_t *val, const int32_t *fo) {
    __shared__ int32_t s_val[SPAN > 0 ? SPAN : 1];
    for (int64_t r0 = int64_t(blockIdx.x) * kThreads; r0 < rows; r0 += int64_t(gridDim.x) * kThreads) {
        const int64_t r1 = min(rows, r0 + kThreads);
        const int32_t base = off[r0], span = off[r1] - base;
        const bool staged = SPAN > 0 && span <= SPAN;
        if (staged) {
            for (int32_t u = threadIdx.x; u < span; u += kThreads) s_val[u] = val[base + u];
            __syncthreads();
        }
        const int64_t r = r0 + threadIdx.x;
        if (r < r1) {
            int32_t *o = staged ? s_val + (off[r] - base) : val + off[r];
            const int32_t len = off[r + 1] - off[r];
            int32_t n = len;
            if (FRONT == FRONT_VE) {
                n = sc.ve_n[r];
                const int32_t j0 = m.eo[r];
                for (int32_t i = n; i < len; ++i) o[i] = edge_id(m, j0 + i - n);
            } else if (FRONT == FRONT_EF) {
                const int64_t j = m.sorted_ids ? r : m.e2s[r];
                const int32_t lo = sc.ef_lo[j];
                n = lo + sc.ef_mid[j];
                if (m.sorted_ids && sc.ef_tail) sc.ef_tail[j] = make_int2(off[r] + lo, off[r + 1]);
                int32_t *f = o + n;
                const int32_t p0 = m.feo[j], p1 = m.feo[j + 1];
                for (int32_t p = p0; p < p1; ++p) f[p - p0] = face_id(m, p);
            } else if (FRONT == FRONT_VF) {
                n = sc.vf_n[r];
                const int32_t p0 = fo[r], p1 = fo[r + 1];
                for (int32_t p = p0; p < p1; ++p) o[n + p - p0] = face_id(m, p);
            }
            if (!m.sorted_ids) n = len;
            if (n > N) {
                insertion_sort(o, n);
            } else if (n >= 2) {
                int32_t x[N];
#pragma unroll
                for (int i = 0; i < N; ++i) x[i] = i < n ? o[i] : INT32_MAX;
                bitonic_regs<N>(x);
#pragma unroll
                for (int i = 0; i < N; ++i)
                    if (i < n) o[i] = x[i];
            }
        }
        if (staged) {
            __syncthreads();
            for (int32_t u = threadIdx.x; u < span; u += kThreads) val[base + u] = s_val[u];
            __syncthreads();
        }
    }
}

// VF with the sorted numbering, from VE and EF (both sorted): the triangles
// through v whose lowest vertex a is not v are, for the lower edges (a, v)
// in ascending a, EF(a, v) after its lower part - its middle part (a, x, v)
// and its contiguous part (a, v, x) - already in id order; the triangles
// with lowest vertex v follow.  At 128^3 0.30 ms; a thread a vertex took
// 0.48 ms, one dependent load after the other.
// VF: eight lanes a vertex, a lower edge each (the four groups of a warp run
// their loops together, to the longest one's count: with a mask per group
// each shuffle would split the warp)
constexpr int kGroup = 8, kGroups = kThreads / kGroup;
constexpr int kVfSpan = 2048;
__device__ __forceinline__ int32_t group_incl_scan(int32_t v, int l) {
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, v, o, kGroup);
        if (l >= o) v += y;
    }
    return v;
}
__global__ void __launch_bounds__(kThreads) k_vf_gather(CbMesh m, Scatter sc, const int32_t *fo) {
    __shared__ int32_t s_val[kVfSpan];  // the block's rows, stored coalesced
    const int g = threadIdx.x / kGroup, l = threadIdx.x % kGroup;
    for (int64_t vb = int64_t(blockIdx.x) * kGroups; vb < m.nv; vb += int64_t(gridDim.x) * kGroups) {
        const int64_t ve = min(m.nv, vb + kGroups);
        const int32_t base = sc.vf_off[vb], span = sc.vf_off[ve] - base;
        const bool staged = span <= kVfSpan, mine = vb + g < ve;
        const int64_t u = mine ? vb + g : vb;
        const int32_t *low = sc.ve_val + sc.ve_off[u];
        const int32_t nl = mine ? sc.ve_n[u] : 0;
        const int32_t p0 = fo[u], p1 = mine ? fo[u + 1] : p0;
        int32_t *o = staged ? s_val + (sc.vf_off[u] - base) : sc.vf_val + sc.vf_off[u];
        for (int32_t q0 = 0; __any_sync(0xffffffffu, q0 < nl); q0 += kGroup) {
            int2 t = make_int2(0, 0);
            if (q0 + l < nl) t = sc.ef_tail[low[q0 + l]];
            const int32_t n = t.y - t.x, incl = group_incl_scan(n, l);
            int32_t *d = o + (incl - n);
            for (int32_t i = t.x; i < t.y; i += 4) {  // four loads in flight
                const int32_t a = sc.ef_val[i], b = i + 1 < t.y ? sc.ef_val[i + 1] : 0;
                const int32_t c = i + 2 < t.y ? sc.ef_val[i + 2] : 0, e = i + 3 < t.y ? sc.ef_val[i + 3] : 0;
                d[0] = a;
                if (i + 1 < t.y) d[1] = b;
                if (i + 2 < t.y) d[2] = c;
                if (i + 3 < t.y) d[3] = e;
                d += 4;
            }
            o += __shfl_sync(0xffffffffu, incl, kGroup - 1, kGroup);
        }
        for (int32_t p = p0 + l; p < p1; p += kGroup) o[p - p0] = p;
        __syncthreads();
        if (staged)
            for (int32_t t = threadIdx.x; t < span; t += kThreads) sc.vf_val[base + t] = s_val[t];
        __syncthreads();
    }
}

// ---- sorted enumeration on the device ----
// A segment's edges in vertex-tuple order are its cluster's ET edges (own
// lower vertex u, then upper vertex w): E is written straight from the ET
// rows.  Its triangles over an edge (a, b) are (a, b, c) for the distinct
// vertices c > b of the tets of ET(a, b), ascending.

// E pairs of every cluster's edges, at I_E[k] + local edge index
__global__ void __launch_bounds__(kThreads) k_enum_edges(CbMesh m, int32_t *E) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v < m.nv; v += int64_t(gridDim.x) * blockDim.x) {
        const int32_t k = m.cluster_of[v];
        const int32_t i = int32_t(v) - m.I_V[k];
        const int64_t *B = m.base + 10 * int64_t(k);
        const int32_t e0 = m.et_uoff[B[B_ET_UOFF] + i], e1 = m.et_uoff[B[B_ET_UOFF] + i + 1];
        for (int32_t e = e0; e < e1; ++e) {
            const int64_t j = m.IE[k] + e;
            E[2 * j] = int32_t(v);
            E[2 * j + 1] = m.et_w[B[B_ET_W] + e];
        }
    }
}

// triangles over each edge: count (F == nullptr) or write at FS[j]
template <bool WRITE>
__global__ void __launch_bounds__(kThreads) k_enum_faces(CbMesh m, const int32_t *E, int32_t *nf, const int32_t *FS,
                                                         int32_t *F, int32_t *err) {
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m.nE; j += int64_t(gridDim.x) * blockDim.x) {
        const int32_t a = E[2 * j], b = E[2 * j + 1];
        int64_t eb, ee;
        if (!et_row(m, j, a, b, eb, ee)) {
            atomicOr(err, ERR_BAD_BLOCK);
            if (!WRITE) nf[j] = 0;
            continue;
        }
        int32_t n = 0;
        int64_t out = WRITE ? FS[j] : 0;
        const int64_t cap = WRITE ? FS[j + 1] - FS[j] : 0;
        constexpr int kCand = 32;
        if (ee - eb <= kCand / 2) {
            int32_t xs[kCand];
            int c = 0;
            for (int64_t q = eb; q < ee; ++q) {
                const int4 r = m.rows[m.et_val[q]];
#pragma unroll
                for (int s2 = 0; s2 < 4; ++s2) {
                    const int32_t x = s2 == 0 ? r.x : s2 == 1 ? r.y : s2 == 2 ? r.z : r.w;
                    if (x <= b || c >= kCand) continue;
                    int p = c++;
                    while (p > 0 && xs[p - 1] > x) {
                        xs[p] = xs[p - 1];
                        --p;
                    }
                    xs[p] = x;
                }
            }
            for (int p = 0; p < c; ++p) {
                if (p > 0 && xs[p] == xs[p - 1]) continue;
                if (WRITE && n < cap) {
                    F[3 * (out + n)] = a;
                    F[3 * (out + n) + 1] = b;
                    F[3 * (out + n) + 2] = xs[p];
                }
                ++n;
            }
        } else {
            // many tets around the edge: emit each c once, in increasing order
            int32_t last = b;
            for (;;) {
                int32_t next = INT32_MAX;
                for (int64_t q = eb; q < ee; ++q) {
                    const int4 r = m.rows[m.et_val[q]];
                    const int32_t xv[4] = {r.x, r.y, r.z, r.w};
                    for (int s2 = 0; s2 < 4; ++s2)
                        if (xv[s2] > last && xv[s2] < next) next = xv[s2];
                }
                if (next == INT32_MAX) break;
                if (WRITE && n < cap) {
                    F[3 * (out + n)] = a;
                    F[3 * (out + n) + 1] = b;
                    F[3 * (out + n) + 2] = next;
                }
                ++n;
                last = next;
            }
        }
        if (!WRITE) nf[j] = n;
        else if (n != cap) atomicOr(err, ERR_BAD_BLOCK);
    }
}

// I_F[k] = FS[I_E[k]] for k = 0..K
__global__ void __launch_bounds__(kThreads) k_enum_if(const int64_t *IE, const int32_t *FS, int64_t K, int64_t *IF) {
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k <= K; k += int64_t(gridDim.x) * blockDim.x)
        IF[k] = FS[IE[k]];
}

// ---- lookup structure, once per enumeration ----

// eo[v]: first sorted edge position of lower vertex v within its segment
__global__ void __launch_bounds__(kThreads) k_eo(CbMesh m, int32_t *eo) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v <= m.nv; v += int64_t(gridDim.x) * blockDim.x) {
        if (v == m.nv) {
            eo[v] = int32_t(m.nE);
            continue;
        }
        const int32_t k = m.cluster_of[v];
        int64_t lo = m.IE[k], hi = m.IE[k + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (m.E[2 * int64_t(edge_id(m, mid))] < v) lo = mid + 1;
            else hi = mid;
        }
        eo[v] = int32_t(lo);
    }
}

// fo[v]: first sorted triangle position of lowest vertex v
__global__ void __launch_bounds__(kThreads) k_fo(CbMesh m, int32_t *fo) {
    for (int64_t v = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; v <= m.nv; v += int64_t(gridDim.x) * blockDim.x) {
        if (v == m.nv) {
            fo[v] = int32_t(m.nF);
            continue;
        }
        const int32_t k = m.cluster_of[v];
        int64_t lo = m.IF[k], hi = m.IF[k + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (m.F[3 * int64_t(face_id(m, mid))] < v) lo = mid + 1;
            else hi = mid;
        }
        fo[v] = int32_t(lo);
    }
}

// ekw and e2s over sorted edge positions; fkc and f2s over triangle positions
__global__ void __launch_bounds__(kThreads) k_keys(CbMesh m, int32_t *ekw, int32_t *e2s, int32_t *fkc,
                                                   int32_t *f2s) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m.nE; j += stride) {
        const int32_t id = edge_id(m, j);
        ekw[j] = m.E[2 * int64_t(id) + 1];
        e2s[id] = int32_t(j);
    }
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < m.nF; p += stride) {
        const int32_t id = face_id(m, p);
        fkc[p] = m.F[3 * int64_t(id) + 2];
        f2s[id] = int32_t(p);
    }
}

// feo[j]: first sorted triangle position over the j-th sorted edge (a, b)
__global__ void __launch_bounds__(kThreads) k_feo(CbMesh m, const int32_t *fo, int32_t *feo) {
    for (int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; j <= m.nE; j += int64_t(gridDim.x) * blockDim.x) {
        if (j == m.nE) {
            feo[j] = int32_t(m.nF);
            continue;
        }
        const int32_t id = edge_id(m, j);
        const int32_t a = m.E[2 * int64_t(id)], b = m.E[2 * int64_t(id) + 1];
        int64_t lo = fo[a], hi = fo[a + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (m.F[3 * int64_t(face_id(m, mid)) + 1] < b) lo = mid + 1;
            else hi = mid;
        }
        feo[j] = int32_t(lo);
    }
}

// exclusive scan of the row lengths of n rows into off[0..n], in tiles of
// kScanTile lengths (kScanItems consecutive ones per thread): tile sums, one
// pass over the tile sums, then the per-tile scans.  Lengths come from an
// array, or (FT) are the number of taken slots, and the rows are then written
// along with the offsets.
constexpr int kScanItems = 8;
constexpr int64_t kScanTile = int64_t(kThreads) * kScanItems;
inline int64_t scan_tiles(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

struct CountRows {
    const int32_t *cnt;
    __device__ __forceinline__ void load(int64_t n, int64_t i0, int32_t (&c)[kScanItems]) const {
        if (i0 + kScanItems <= n) {  // i0 is a multiple of kScanItems
            const int4 *q = reinterpret_cast<const int4 *>(cnt + i0);
#pragma unroll
            for (int u = 0; u < kScanItems / 4; ++u) {
                const int4 v = q[u];
                c[4 * u] = v.x;
                c[4 * u + 1] = v.y;
                c[4 * u + 2] = v.z;
                c[4 * u + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int u = 0; u < kScanItems; ++u) c[u] = i0 + u < n ? cnt[i0 + u] : 0;
        }
    }
};

// block-wide inclusive scan of one int64 per thread
__device__ __forceinline__ int64_t block_incl_scan(int64_t x, int64_t *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < kThreads / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kThreads / 32) s_warp[lane] = w;
    }
    __syncthreads();
    return x + (warp > 0 ? s_warp[warp - 1] : 0);
}

__global__ void __launch_bounds__(kThreads) scan_sums(CountRows rows, int64_t n, int64_t *bsum) {
    __shared__ int64_t s_warp[kThreads / 32];
    const int64_t i0 = int64_t(blockIdx.x) * kScanTile + int64_t(threadIdx.x) * kScanItems;
    int32_t c[kScanItems];
    rows.load(n, i0, c);
    int64_t mine = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) mine += c[u];
    const int64_t tot = block_incl_scan(mine, s_warp);
    if (threadIdx.x == kThreads - 1) bsum[blockIdx.x] = tot;
}
// FT: the taken slots of each tile
__global__ void __launch_bounds__(kThreads) ft_sums(const int2 *slot, int64_t n, int64_t *bsum, int32_t *err) {
    __shared__ int64_t s_warp[kThreads / 32];
    const int64_t t0 = int64_t(blockIdx.x) * kScanTile;
    int32_t mine = 0;
    bool bad = false;
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = t0 + u * kThreads + threadIdx.x;
        if (i >= n) break;
        const int2 q = slot[i];
        bad |= q.x < 0;  // a triangle in no tet
        mine += (q.x >= 0) + (q.y >= 0);
    }
    if (bad) atomicOr(err, ERR_BAD_BLOCK);
    const int64_t tot = block_incl_scan(mine, s_warp);
    if (threadIdx.x == kThreads - 1) bsum[blockIdx.x] = tot;
}

// exclusive scan of the nb tile sums in place (bsum[nb] = total), one
// block: a block scan per kBsumThreads sums, the next ones loaded ahead
constexpr int kBsumThreads = 1024;
__global__ void __launch_bounds__(kBsumThreads) scan_bsums(int64_t *bsum, int64_t nb) {
    __shared__ int64_t s_warp[2][kBsumThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t run = 0, next = threadIdx.x < nb ? bsum[threadIdx.x] : 0;
    int buf = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += kBsumThreads, buf ^= 1) {
        const int64_t b = b0 + threadIdx.x, mine = next;
        next = b + kBsumThreads < nb ? bsum[b + kBsumThreads] : 0;
        int64_t x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[buf][warp] = x;
        __syncthreads();
        int64_t w = s_warp[buf][lane];  // every warp scans the warps' sums
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const int64_t before = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
        if (b < nb) bsum[b] = run + (warp > 0 ? before : 0) + x - mine;
        run += __shfl_sync(0xffffffffu, w, 31);
    }
    if (threadIdx.x == 0) bsum[nb] = run;
}

// the total of the tile sums as the last offset
__device__ __forceinline__ void last_offset(const int64_t *bsum, int64_t nb, int32_t *off, int64_t n, int32_t *err) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t tot = bsum[nb];
        if (tot > INT32_MAX) atomicOr(err, ERR_CAPACITY);
        off[n] = int32_t(tot);
    }
}
__global__ void __launch_bounds__(kThreads) scan_write(CountRows rows, int64_t n, const int64_t *bsum, int32_t *off,
                                                       int64_t nb, int32_t *err) {
    __shared__ int64_t s_warp[kThreads / 32];
    __shared__ int32_t s_out[kScanTile + kScanTile / kScanItems];  // the tile's offsets, one word of padding a thread
    const int64_t t0 = int64_t(blockIdx.x) * kScanTile;
    int32_t c[kScanItems];
    rows.load(n, t0 + int64_t(threadIdx.x) * kScanItems, c);
    int64_t mine = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) mine += c[u];
    int64_t run = bsum[blockIdx.x] + block_incl_scan(mine, s_warp) - mine;
    if (run + mine > INT32_MAX) atomicOr(err, ERR_CAPACITY);
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        s_out[threadIdx.x * (kScanItems + 1) + u] = int32_t(run);
        run += c[u];
    }
    __syncthreads();
    const int64_t m = min(kScanTile, n - t0);
    for (int64_t u = threadIdx.x; u < m; u += kThreads) off[t0 + u] = s_out[u + u / kScanItems];
    last_offset(bsum, nb, off, n, err);
}
// FT: offsets and rows of a tile, from its slots.  A warp takes 32
// consecutive rows a step, whose positions come from two ballots.
__global__ void __launch_bounds__(kThreads) ft_write(const int2 *slot, int64_t n, const int64_t *bsum, int32_t *off,
                                                     int32_t *val, int64_t nb, int64_t entries, int32_t *err) {
    __shared__ int32_t s_warp[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t w0 = int64_t(blockIdx.x) * kScanTile + warp * 32 * kScanItems;
    int2 q[kScanItems];
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = w0 + 32 * u + lane;
        q[u] = i < n ? slot[i] : make_int2(-1, -1);
    }
    int32_t mine = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u)
        mine += __popc(__ballot_sync(0xffffffffu, q[u].x >= 0)) + __popc(__ballot_sync(0xffffffffu, q[u].y >= 0));
    if (lane == 0) s_warp[warp] = mine;
    __syncthreads();
    int64_t run = bsum[blockIdx.x];
    for (int w = 0; w < warp; ++w) run += s_warp[w];
    const bool fits = run + mine <= entries;
    if (run + mine > INT32_MAX) atomicOr(err, ERR_CAPACITY);
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = w0 + 32 * u + lane;
        const uint32_t bx = __ballot_sync(0xffffffffu, q[u].x >= 0), by = __ballot_sync(0xffffffffu, q[u].y >= 0);
        const int32_t o = int32_t(run) + __popc(bx & lt) + __popc(by & lt);
        run += __popc(bx) + __popc(by);
        if (i >= n) continue;
        off[i] = o;
        if (!fits) continue;
        const bool two = q[u].x >= 0 && q[u].y >= 0;
        if (q[u].x >= 0) val[o] = two ? min(q[u].x, q[u].y) : q[u].x;
        if (two) val[o + 1] = max(q[u].x, q[u].y);
    }
    last_offset(bsum, nb, off, n, err);
    // a third tet on some triangle took another's slot
    if (blockIdx.x == 0 && threadIdx.x == 0 && bsum[nb] != entries) atomicOr(err, ERR_NONMANIFOLD);
}

gale_status fail(gale_status s, const std::string &msg) {
    set_error(msg);
    return s;
}

template <class T>
bool grow(gale_ctx *ctx, T *&p, int64_t &cap, int64_t need) {
    if (need <= cap && p) return true;
    if (p) ctx->dfree(p);
    p = nullptr;
    cap = 0;
    const int64_t c = std::max<int64_t>(need + need / 8, 64);
    p = static_cast<T *>(ctx->dalloc(size_t(c) * sizeof(T)));
    if (!p) return false;
    cap = c;
    return true;
}

template <class T>
T *upload(gale_ctx *ctx, const T *h, size_t n, cudaStream_t s) {
    T *d = static_cast<T *>(ctx->dalloc(std::max<size_t>(n, 1) * sizeof(T)));
    if (d && n) cudaMemcpyAsync(d, h, n * sizeof(T), cudaMemcpyHostToDevice, s);
    return d;
}
template <class T>
T *upload(gale_ctx *ctx, const std::vector<T> &h, cudaStream_t s) {
    return upload(ctx, h.data(), h.size(), s);
}

}  // namespace

bool device_enumeration(gale_ctx *ctx, uint64_t gen, const int32_t **E, const int32_t **F) {
    if (!ctx->cb || ctx->cb->dev_gen != gen || !ctx->cb->E || !ctx->cb->F) return false;
    *E = ctx->cb->E;
    *F = ctx->cb->F;
    return true;
}

// Sorted enumeration on the device (declared in gale_enum.h).
gale_status enumerate_sorted_device(gale_ctx *ctx, uint64_t gen, std::vector<int64_t> &IE,
                                    std::vector<int64_t> &IF) {
    if (ctx->device < 0 || (ctx->precond & GALE_ET) == 0) return GALE_ENOTFOUND;
    gale_status st = gale_build_clusters(ctx, nullptr, 0, GALE_ET, GALE_MODE_BATCHED);
    if (st == GALE_OK) st = gale_synchronize(ctx);
    if (st != GALE_OK) return st;
    std::lock_guard<std::mutex> lock(ctx->mu);
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(GALE_ECUDA, "cudaSetDevice");
    cudaStream_t s = ctx->stream;
    const HostMesh &hm = ctx->hm;
    const int32_t K = hm.K;
    IE.assign(size_t(K) + 1, 0);
    for (int32_t k = 0; k < K; ++k) IE[k + 1] = IE[k] + ctx->sizes[size_t(5) * k + 2];
    const int64_t nE = IE[K];
    if (nE >= INT32_MAX) return fail(GALE_EINVAL, "more than 2^31 - 1 edges");
    if (!ctx->cb) ctx->cb = new Cobound();
    Cobound &cb = *ctx->cb;
    if (!cb.rows) {
        cb.rows = upload(ctx, hm.rows, s);
        cb.cluster_of = upload(ctx, hm.cluster_of, s);
        if (!cb.rows || !cb.cluster_of) return fail(GALE_ENOMEM, "device allocation of the mesh rows failed");
    }
    std::vector<int64_t> base(ctx->bulk_offs.begin(), ctx->bulk_offs.begin() + size_t(10) * K);
    std::vector<void *> tmp;
    auto dal = [&](size_t bytes) {
        void *p = ctx->dalloc(std::max<size_t>(bytes, 16));
        if (p) tmp.push_back(p);
        return p;
    };
    auto release = [&]() {
        for (void *p : tmp) ctx->dfree(p);
        tmp.clear();
    };
    int64_t *d_base = static_cast<int64_t *>(dal(base.size() * 8));
    int64_t *d_IE = static_cast<int64_t *>(dal(IE.size() * 8));
    int32_t *d_E = static_cast<int32_t *>(dal(size_t(2) * nE * 4));
    int32_t *d_nf = static_cast<int32_t *>(dal(size_t(nE) * 4 + 4));
    int32_t *d_FS = static_cast<int32_t *>(dal((size_t(nE) + 1) * 4));
    int64_t *d_IF = static_cast<int64_t *>(dal((size_t(K) + 1) * 8));
    const int64_t nb = scan_tiles(nE);
    int64_t *d_bsum = static_cast<int64_t *>(dal((size_t(nb) + 1) * 8));
    if (!d_base || !d_IE || !d_E || !d_nf || !d_FS || !d_IF || !d_bsum) {
        release();
        return fail(GALE_ENOMEM, "device allocation for the enumeration failed");
    }
    cudaMemcpyAsync(d_base, base.data(), base.size() * 8, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(d_IE, IE.data(), IE.size() * 8, cudaMemcpyHostToDevice, s);
    CbMesh m{};
    m.rows = reinterpret_cast<const int4 *>(cb.rows);
    m.cluster_of = cb.cluster_of;
    m.I_V = ctx->d_I_V;
    m.IE = d_IE;
    m.et_uoff = ctx->bulk[B_ET_UOFF];
    m.et_w = ctx->bulk[B_ET_W];
    m.et_off = ctx->bulk[B_ET_OFF];
    m.et_val = ctx->bulk[B_ET_VAL];
    m.base = d_base;
    m.sizes = ctx->d_sizes;
    m.nv = hm.nv;
    m.nE = nE;
    const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
    auto grid_for = [&](int64_t n) {
        return int(std::min<int64_t>(std::max<int64_t>((n + kThreads - 1) / kThreads, 1), int64_t(sms) * 16));
    };
    k_enum_edges<<<grid_for(hm.nv), kThreads, 0, s>>>(m, d_E);
    k_enum_faces<false><<<grid_for(nE), kThreads, 0, s>>>(m, d_E, d_nf, nullptr, nullptr, ctx->d_err);
    if (nb > 0) {
        scan_sums<<<int(nb), kThreads, 0, s>>>(CountRows{d_nf}, nE, d_bsum);
        scan_bsums<<<1, kBsumThreads, 0, s>>>(d_bsum, nb);
        scan_write<<<int(nb), kThreads, 0, s>>>(CountRows{d_nf}, nE, d_bsum, d_FS, nb, ctx->d_err);
    } else {
        cudaMemsetAsync(d_FS, 0, 4, s);
    }
    int32_t nF = 0;
    if (cudaMemcpyAsync(&nF, d_FS + nE, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        release();
        return fail(GALE_ECUDA, "enumeration count pass failed");
    }
    int32_t e = 0;
    cudaMemcpy(&e, ctx->d_err, 4, cudaMemcpyDeviceToHost);
    if (e) {
        cudaMemset(ctx->d_err, 0, 4);
        release();
        return fail(GALE_EDEVICE, "enumeration count pass: error word " + std::to_string(e));
    }
    int32_t *d_F = static_cast<int32_t *>(dal(size_t(3) * nF * 4));
    if (!d_F) {
        release();
        return fail(GALE_ENOMEM, "device allocation of the triangle list failed");
    }
    k_enum_faces<true><<<grid_for(nE), kThreads, 0, s>>>(m, d_E, nullptr, d_FS, d_F, ctx->d_err);
    k_enum_if<<<grid_for(K + 1), kThreads, 0, s>>>(d_IE, d_FS, K, d_IF);
    // only the intervals come to the host; E and F are copied by the
    // queries that need them (gale_get_enumeration, gale_boundary)
    IF.assign(size_t(K) + 1, 0);
    const gale_status cst = copy_to_host(ctx, IF.data(), d_IF, IF.size() * 8);
    if (cst != GALE_OK) {
        release();
        return cst;
    }
    cudaMemcpy(&e, ctx->d_err, 4, cudaMemcpyDeviceToHost);
    if (e) {
        cudaMemset(ctx->d_err, 0, 4);
        release();
        return fail(GALE_EDEVICE, "enumeration fill pass: error word " + std::to_string(e));
    }
    // the device lists stay with the coboundary pass, which would otherwise
    // upload the same arrays again
    for (int32_t **p : {&cb.E, &cb.F, &cb.ebk, &cb.fbk})
        if (*p) {
            ctx->dfree(*p);
            *p = nullptr;
        }
    for (int64_t **p : {&cb.IE, &cb.IF})
        if (*p) {
            ctx->dfree(*p);
            *p = nullptr;
        }
    cb.E = d_E;
    cb.F = d_F;
    cb.IE = d_IE;
    cb.IF = d_IF;
    cb.dev_gen = gen;
    tmp.erase(std::remove_if(tmp.begin(), tmp.end(),
                             [&](void *p) { return p == d_E || p == d_F || p == d_IE || p == d_IF; }),
              tmp.end());
    release();
    return GALE_OK;
}

// One coboundary pass over the current enumeration (the caller holds the
// context's lock).  *err_word receives the device error word.
gale_status run_pass(gale_ctx *ctx, uint32_t which, const EnumView &ev, int32_t *err_word) {
    const int64_t nE = ev.nE, nF = ev.nF;
    const uint64_t gen = ev.gen;
    cudaStream_t s = ctx->stream;
    const HostMesh &hm = ctx->hm;
    const int32_t K = hm.K;
    if (!ctx->cb) ctx->cb = new Cobound();
    Cobound &cb = *ctx->cb;
    if (!cb.rows) {
        cb.rows = upload(ctx, hm.rows, s);
        cb.cluster_of = upload(ctx, hm.cluster_of, s);
        if (!cb.rows || !cb.cluster_of) return fail(GALE_ENOMEM, "device allocation of the mesh rows failed");
    }
    // the pass reads the enumeration, its index and the canonical tet rows
    CbMesh m{};
    m.rows = reinterpret_cast<const int4 *>(cb.rows);
    m.cluster_of = cb.cluster_of;
    m.I_V = ctx->d_I_V;
    m.E = cb.E;
    m.F = cb.F;
    m.ebk = cb.ebk;
    m.fbk = cb.fbk;
    m.IE = cb.IE;
    m.IF = cb.IF;
    m.eo = cb.eo;
    m.ekw = cb.ekw;
    m.feo = cb.feo;
    m.fkc = cb.fkc;
    m.e2s = cb.e2s;
    m.f2s = cb.f2s;
    m.nv = hm.nv;
    m.nE = nE;
    m.nF = nF;
    m.sorted_ids = cb.sorted_ids;
    const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
    auto grid_for = [&](int64_t n) {
        return int(std::min<int64_t>(std::max<int64_t>((n + kThreads - 1) / kThreads, 1), int64_t(sms) * 16));
    };
    if (cb.enm_gen != gen) {
        for (int32_t **p : {&cb.eo, &cb.ekw, &cb.feo, &cb.fkc, &cb.fo, &cb.e2s, &cb.f2s})
            if (*p) {
                ctx->dfree(*p);
                *p = nullptr;
            }
        cb.enm_gen = 0;
        if (cb.dev_gen != gen) {  // the lists are not on the device yet
            if (!ev.E || !ev.F) return fail(GALE_EINVAL, "the enumeration's lists are gone from the device");
            for (int32_t **p : {&cb.E, &cb.F, &cb.ebk, &cb.fbk})
                if (*p) {
                    ctx->dfree(*p);
                    *p = nullptr;
                }
            for (int64_t **p : {&cb.IE, &cb.IF})
                if (*p) {
                    ctx->dfree(*p);
                    *p = nullptr;
                }
            cb.dev_gen = 0;
            cb.E = upload(ctx, ev.E, size_t(2) * nE, s);
            cb.F = upload(ctx, ev.F, size_t(3) * nF, s);
            if (ev.ebk) cb.ebk = upload(ctx, ev.ebk, size_t(nE), s);
            if (ev.fbk) cb.fbk = upload(ctx, ev.fbk, size_t(nF), s);
            cb.IE = upload(ctx, ev.IE, size_t(K) + 1, s);
            cb.IF = upload(ctx, ev.IF, size_t(K) + 1, s);
            if (!cb.E || !cb.F || (ev.ebk && !cb.ebk) || (ev.fbk && !cb.fbk) || !cb.IE || !cb.IF)
                return fail(GALE_ENOMEM, "device allocation of the enumeration failed");
            cb.dev_gen = gen;
        }
        auto dal = [&](int64_t n) { return static_cast<int32_t *>(ctx->dalloc(size_t(std::max<int64_t>(n, 1)) * 4)); };
        cb.eo = dal(hm.nv + 1);
        cb.fo = dal(hm.nv + 1);
        cb.ekw = dal(nE);
        cb.e2s = dal(nE);
        cb.feo = dal(nE + 1);
        cb.fkc = dal(nF);
        cb.f2s = dal(nF);
        if (!cb.eo || !cb.fo || !cb.ekw || !cb.e2s || !cb.feo || !cb.fkc || !cb.f2s)
            return fail(GALE_ENOMEM, "device allocation of the enumeration index failed");
        // ids follow the vertex-tuple order exactly when no key arrays exist
        cb.sorted_ids = ev.ebk == nullptr;
        m.E = cb.E;
        m.F = cb.F;
        m.ebk = cb.ebk;
        m.fbk = cb.fbk;
        m.IE = cb.IE;
        m.IF = cb.IF;
        m.sorted_ids = cb.sorted_ids;
        k_eo<<<grid_for(hm.nv + 1), kThreads, 0, s>>>(m, cb.eo);
        k_fo<<<grid_for(hm.nv + 1), kThreads, 0, s>>>(m, cb.fo);
        k_keys<<<grid_for(std::max(nE, nF)), kThreads, 0, s>>>(m, cb.ekw, cb.e2s, cb.fkc, cb.f2s);
        k_feo<<<grid_for(nE + 1), kThreads, 0, s>>>(m, cb.fo, cb.feo);
        if (cudaGetLastError() != cudaSuccess) return fail(GALE_ECUDA, "coboundary lookup-structure launch failed");
        cb.enm_gen = gen;
    }
    m.eo = cb.eo;
    m.ekw = cb.ekw;
    m.feo = cb.feo;
    m.fkc = cb.fkc;
    m.e2s = cb.e2s;
    m.f2s = cb.f2s;
    m.sorted_ids = cb.sorted_ids;
    const int64_t nT = hm.nt;
    const int64_t rows_of[4] = {hm.nv, hm.nv, nE, nF};
    // entries: every edge is in two VE rows, every triangle in three VF and
    // three EF rows, every tet in four FT rows
    const int64_t len_of[4] = {2 * nE, 3 * nF, 3 * nF, 4 * nT};
    for (int rel = 0; rel < 4; ++rel)
        if (len_of[rel] >= INT32_MAX) return fail(GALE_EINVAL, "a coboundary relation has 2^31 or more entries");
    const bool wVF = which & GALE_CB_VF, wFT = which & GALE_CB_FT;
    // with the sorted numbering VF is gathered from VE and EF, which are then
    // built whether asked for or not; otherwise it is scattered like them
    const bool vf_gather = wVF && cb.sorted_ids, vf_scatter = wVF && !cb.sorted_ids;
    const bool wVE = (which & GALE_CB_VE) || vf_gather, wEF = (which & GALE_CB_EF) || vf_gather;
    const bool ft_gen = wFT && cb.ft_general;
    // scratch of the relations that are built: counters (zeroed), then ranks
    // and lookups.  FT comes last, and its slots take the place of the
    // triangles' lookups.
    int64_t n_scr = 0;
    auto take = [&](bool wanted, int64_t n) {
        const int64_t at = n_scr;
        if (wanted) n_scr += (n + 3) & ~int64_t(3);
        return at;
    };
    const int64_t o_ve_n = take(wVE, hm.nv), o_vf_n = take(wVF, hm.nv);
    const int64_t o_ef_lo = take(wEF, nE), o_ef_mid = take(wEF, nE);
    const int64_t n_ctr = n_scr;
    const int64_t o_vf_fill = take(vf_scatter, hm.nv), o_ve_rank = take(wVE, nE), o_ef_tail = take(vf_gather, 2 * nE);
    const int64_t o_tri = take(wEF || wFT, std::max<int64_t>({2, wEF ? 4 * nF : 0, wFT && !ft_gen ? 2 * nF : 0}));
    const int64_t n_cnt = std::max({wVE || wVF ? hm.nv : 1, wEF ? nE : 1, ft_gen ? nF : 1});
    if (!grow(ctx, cb.scratch, cb.scratch_cap, std::max<int64_t>(n_scr, 4)) ||
        !grow(ctx, cb.cnt, cb.cnt_cap, n_cnt))
        return fail(GALE_ENOMEM, "device allocation of coboundary scratch failed");
    Scatter sc{};
    sc.ve_n = cb.scratch + o_ve_n;
    sc.vf_n = cb.scratch + o_vf_n;
    sc.ef_lo = cb.scratch + o_ef_lo;
    sc.ef_mid = cb.scratch + o_ef_mid;
    sc.vf_fill = cb.scratch + o_vf_fill;
    sc.ve_rank = cb.scratch + o_ve_rank;
    sc.ef_tail = vf_gather ? reinterpret_cast<int2 *>(cb.scratch + o_ef_tail) : nullptr;
    sc.tri = reinterpret_cast<int4 *>(cb.scratch + o_tri);
    sc.ft_slot = reinterpret_cast<int2 *>(cb.scratch + o_tri);
    sc.cnt = cb.cnt;
    if (cudaMemsetAsync(cb.scratch, 0, sizeof(int32_t) * size_t(n_ctr), s) != cudaSuccess)
        return fail(GALE_ECUDA, "cudaMemsetAsync");
    const int32_t *fo = cb.fo;
    // room for a relation's rows
    auto room = [&](int rel) {
        const int64_t n = rows_of[rel];
        cb.rows_of[rel] = n;
        cb.len[rel] = len_of[rel];
        return grow(ctx, cb.bsum, cb.bsum_cap, scan_tiles(n) + 1) && grow(ctx, cb.off[rel], cb.off_cap[rel], n + 1) &&
               grow(ctx, cb.val[rel], cb.val_cap[rel], std::max<int64_t>(len_of[rel], 1));
    };
    const bool use[4] = {wVE, wVF, wEF, wFT};
    for (int rel = 0; rel < 4; ++rel)
        if (use[rel] && !room(rel)) return fail(GALE_ENOMEM, "device allocation of coboundary rows failed");
    sc.ve_off = cb.off[REL_VE];
    sc.vf_off = cb.off[REL_VF];
    sc.ef_off = cb.off[REL_EF];
    sc.ft_off = cb.off[REL_FT];
    sc.ve_val = cb.val[REL_VE];
    sc.vf_val = cb.val[REL_VF];
    sc.ef_val = cb.val[REL_EF];
    sc.ft_val = cb.val[REL_FT];
    auto scan = [&](const int32_t *cnt, int64_t n, int32_t *off) {
        const int64_t nb = scan_tiles(n);
        if (nb > 0) {
            scan_sums<<<int(nb), kThreads, 0, s>>>(CountRows{cnt}, n, cb.bsum);
            scan_bsums<<<1, kBsumThreads, 0, s>>>(cb.bsum, nb);
            scan_write<<<int(nb), kThreads, 0, s>>>(CountRows{cnt}, n, cb.bsum, off, nb, ctx->d_err);
        } else {
            cudaMemsetAsync(off, 0, sizeof(int32_t), s);
        }
    };
    const int gV = grid_for(hm.nv), gE = grid_for(nE), gF = grid_for(nF);
    if (wVE) {
        k_ve_count<<<gE, kThreads, 0, s>>>(m, sc);
        k_len_ve<<<gV, kThreads, 0, s>>>(m, sc);
        scan(sc.cnt, hm.nv, cb.off[REL_VE]);
        k_ve_fill<<<gE, kThreads, 0, s>>>(m, sc);
        k_sort_rows<16, FRONT_VE, 6144><<<gV, kThreads, 0, s>>>(m, sc, hm.nv, sc.ve_off, sc.ve_val, fo);
    }
    if (wEF || vf_scatter) k_sc_tris<false><<<gF, kThreads, 0, s>>>(m, sc, wEF, vf_scatter, ctx->d_err);
    if (wEF) {
        k_len_ef<<<gE, kThreads, 0, s>>>(m, sc, vf_gather);
        scan(sc.cnt, nE, cb.off[REL_EF]);
    }
    if (wVF) {
        k_len_vf<<<gV, kThreads, 0, s>>>(m, sc, fo);
        scan(sc.cnt, hm.nv, cb.off[REL_VF]);
    }
    if (vf_scatter) k_cursors<<<gV, kThreads, 0, s>>>(m, sc);
    if (wEF || vf_scatter) k_sc_tris<true><<<gF, kThreads, 0, s>>>(m, sc, wEF, vf_scatter, ctx->d_err);
    if (wEF) k_sort_rows<8, FRONT_EF, 2560><<<gE, kThreads, 0, s>>>(m, sc, nE, sc.ef_off, sc.ef_val, fo);
    if (vf_gather) k_vf_gather<<<grid_for(hm.nv * kGroup), kThreads, 0, s>>>(m, sc, fo);
    if (vf_scatter)
        k_sort_rows<32, FRONT_VF, 12288><<<gV, kThreads, 0, s>>>(m, sc, hm.nv, sc.vf_off, sc.vf_val, fo);
    if (ft_gen) {
        const size_t bytes = sizeof(int32_t) * size_t(std::max<int64_t>(nF, 1));
        cudaMemsetAsync(sc.cnt, 0, bytes, s);
        k_ft_tets<FT_COUNT><<<grid_for(nT), kThreads, 0, s>>>(m, sc, nT, ctx->d_err);
        scan(sc.cnt, nF, cb.off[REL_FT]);
        cudaMemsetAsync(sc.cnt, 0, bytes, s);
        k_ft_tets<FT_FILL><<<grid_for(nT), kThreads, 0, s>>>(m, sc, nT, ctx->d_err);
        k_sort_rows<4, FRONT_NONE, 0><<<grid_for(nF), kThreads, 0, s>>>(m, sc, nF, sc.ft_off, sc.ft_val, fo);
    } else if (wFT) {
        cudaMemsetAsync(sc.ft_slot, 0xff, sizeof(int2) * size_t(std::max<int64_t>(nF, 1)), s);
        k_ft_tets<FT_SLOTS><<<grid_for(nT), kThreads, 0, s>>>(m, sc, nT, ctx->d_err);
        const int64_t nb = scan_tiles(nF);
        if (nb > 0) {
            ft_sums<<<int(nb), kThreads, 0, s>>>(sc.ft_slot, nF, cb.bsum, ctx->d_err);
            scan_bsums<<<1, kBsumThreads, 0, s>>>(cb.bsum, nb);
            ft_write<<<int(nb), kThreads, 0, s>>>(sc.ft_slot, nF, cb.bsum, cb.off[REL_FT], cb.val[REL_FT], nb,
                                                  len_of[REL_FT], ctx->d_err);
        } else {
            cudaMemsetAsync(cb.off[REL_FT], 0, sizeof(int32_t), s);
        }
    }
    if (cudaGetLastError() != cudaSuccess) return fail(GALE_ECUDA, "coboundary launch failed");
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(GALE_ECUDA, "cudaStreamSynchronize");
    int32_t e = 0;
    cudaMemcpy(&e, ctx->d_err, sizeof(int32_t), cudaMemcpyDeviceToHost);
    *err_word = e;
    if (e) {
        cudaMemset(ctx->d_err, 0, sizeof(int32_t));
        return fail(GALE_EDEVICE, "coboundary pass: error word " + std::to_string(e));
    }
    return GALE_OK;
}

}  // namespace gale

extern "C" gale_status gale_build_coboundary(gale_ctx *ctx, uint32_t which, gale_coboundary *out) {
    using namespace gale;
    if (!ctx || !out) return fail(GALE_EINVAL, "NULL argument");
    if (ctx->device < 0) return fail(GALE_EINVAL, "host-only context");
    if (which == 0 || (which & ~uint32_t(GALE_CB_VE | GALE_CB_VF | GALE_CB_EF | GALE_CB_FT)))
        return fail(GALE_EINVAL, "which must be a non-empty set of GALE_CB_* bits");
    EnumView ev{};
    if (!enumeration_view(ctx, &ev)) return fail(GALE_ENOTFOUND, "no enumeration: call gale_enumerate first");
    if (ev.nE >= INT32_MAX || ev.nF >= INT32_MAX) return fail(GALE_EINVAL, "more than 2^31 - 1 edges or triangles");
    std::lock_guard<std::mutex> lock(ctx->mu);
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(GALE_ECUDA, "cudaSetDevice");
    if (!ctx->cb) ctx->cb = new Cobound();
    Cobound &cb = *ctx->cb;
    // a mesh the counting pass found non-manifold takes the general FT form
    // at once; otherwise a third tet on a triangle (the slots overflow)
    // switches this context to it and the pass runs again
    for (int32_t g : ctx->tt_general) cb.ft_general |= g != 0;
    int32_t e = 0;
    gale_status st = run_pass(ctx, which, ev, &e);
    if (st == GALE_EDEVICE && e == ERR_NONMANIFOLD && (which & GALE_CB_FT) && !cb.ft_general) {
        cb.ft_general = true;
        st = run_pass(ctx, which, ev, &e);
    }
    if (st != GALE_OK) return st;
    for (int rel = 0; rel < 4; ++rel) {
        const bool have = (which & (1u << rel)) != 0;
        out->rows[rel] = have ? cb.rows_of[rel] : 0;
        out->len[rel] = have ? cb.len[rel] : 0;
        out->off[rel] = have ? cb.off[rel] : nullptr;
        out->val[rel] = have ? cb.val[rel] : nullptr;
    }
    return GALE_OK;
}

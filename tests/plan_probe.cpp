// Looks at the launch planning of a loaded context from a test: every work
// item's sizes counted from its block on the CPU, its size class and the
// shared memory its build plan takes.  Compiled by plan_util.py against the
// library's own headers and linked to it.
#include <algorithm>
#include <array>
#include <map>
#include <set>
#include <vector>

#include "gale_ctx.h"

using namespace gale;

namespace {
// the five sizes of item k, by brute force over its block
void count_item(const HostMesh &hm, int32_t k, int64_t *sz) {
    const int32_t *b = hm.blocks + hm.blk_off[k];
    const BlockHdr h = *reinterpret_cast<const BlockHdr *>(b);
    const int32_t xmap = h.part > 0 ? h.n_own : 0;
    const uint16_t *rows =
        reinterpret_cast<const uint16_t *>(b + blk_rows_off(h.nv_loc, h.n_ext, h.n_halo, xmap));
    const int32_t n_star = h.n_ext + h.n_own, n_all = n_star + h.n_halo;
    std::vector<std::set<int>> nb(size_t(h.nv_own));
    std::map<std::array<int, 3>, int> faces;
    std::fill(sz, sz + SZ_N, 0);
    for (int32_t t = 0; t < n_all; ++t) {
        const uint16_t *r = rows + 4 * t;
        for (int s = 0; s < 4; ++s) {
            std::array<int, 3> f;
            for (int u = 0, i = 0; u < 4; ++u)
                if (u != s) f[i++] = r[u];
            faces[f]++;
            const int x = r[s] - h.own_lo;
            if (t >= n_star || x < 0 || x >= h.nv_own) continue;
            sz[SZ_VT]++;
            sz[SZ_ET] += 3 - s;
            for (int u = 0; u < 4; ++u)
                if (u != s) nb[size_t(x)].insert(r[u]);
        }
    }
    for (int32_t x = 0; x < h.nv_own; ++x) {
        sz[SZ_VV] += int64_t(nb[x].size());
        sz[SZ_E] += std::distance(nb[x].upper_bound(h.own_lo + x), nb[x].end());
    }
    for (int32_t t = h.n_ext; t < n_star; ++t)
        for (int s = 0; s < 4; ++s) {
            std::array<int, 3> f;
            for (int u = 0, i = 0; u < 4; ++u)
                if (u != s) f[i++] = rows[4 * t + u];
            sz[SZ_TT] += faces[f] - 1;
        }
}
}  // namespace

extern "C" {

int32_t probe_items(gale_ctx *ctx) { return ctx->hm.K + ctx->hm.NP; }

// per item: own vertices, internal tets, incidences, longest star, size
// class, plan total and mode (host-only context)
void probe_plans(gale_ctx *ctx, int32_t threads, int64_t *out) {
    for (int32_t k = 0; k < probe_items(ctx); ++k, out += 7) {
        int64_t sz[SZ_N];
        count_item(ctx->hm, k, sz);
        const ClusterStat &s = ctx->hm.stats[k];
        const Caps c = caps_of(s, sz);
        const SmemPlan p = plan_smem(c, threads);
        const int64_t row[7] = {s.nv_own, s.n_own, s.n_vt, s.max_deg, class_bytes(c, threads), p.total,
                                p.mode | (p.stride ? 256 : 0)};
        std::copy(row, row + 7, out);
    }
}

// class, plan total and mode of n sets of capacities
void probe_caps(const Caps *caps, int32_t n, int32_t threads, int64_t *out) {
    for (int32_t i = 0; i < n; ++i, out += 3) {
        const SmemPlan p = plan_smem(caps[i], threads);
        out[0] = class_bytes(caps[i], threads);
        out[1] = p.total;
        out[2] = p.mode;
    }
}

int32_t probe_caps_words() { return int32_t(sizeof(Caps) / sizeof(int32_t)); }

// the constants plan_smem holds for a CTA's limit, and the device's
void probe_limits(int64_t *out) {
    out[0] = kCompactFit;
    out[1] = kCtaBytes;
    out[2] = dynamic_smem_limit();
}

// CTAs an SM holds at `total` bytes: as merged launches plan, and the device's
void probe_merged_ctas(gale_ctx *ctx, int32_t total, int32_t *out) {
    prepare_kernels(dynamic_smem_limit());
    SmemPlan p{};
    p.threads = 512;
    p.total = total;
    out[0] = merged_ctas(ctx, total);
    out[1] = max_ctas_per_sm(p, false, true);
}

// per-item bins, and the bytes that some member's own plan takes beyond its
// launch's shared memory (0: none)
void probe_per_item(gale_ctx *ctx, int64_t *out) {
    out[0] = out[1] = 0;
    for (const Bin &b : ctx->bins) {
        if (!b.per_item) continue;
        ++out[0];
        for (int32_t k : b.clusters) out[1] = std::max<int64_t>(out[1], ctx->h_plans[k].total - b.plan.total);
    }
}

int32_t probe_bin_streams(gale_ctx *ctx) { return int32_t(ctx->bin_streams.size()); }

// shared memory of one plan over the listed items (a size bin's)
int64_t probe_merged(gale_ctx *ctx, const int32_t *ids, int32_t n, int32_t threads) {
    Caps m{};
    for (int32_t i = 0; i < n; ++i) {
        int64_t sz[SZ_N];
        count_item(ctx->hm, ids[i], sz);
        const Caps c = caps_of(ctx->hm.stats[ids[i]], sz);
        for (size_t w = 0; w < sizeof(Caps) / sizeof(int32_t); ++w) {
            int32_t &a = reinterpret_cast<int32_t *>(&m)[w];
            a = std::max(a, reinterpret_cast<const int32_t *>(&c)[w]);
        }
    }
    return plan_smem(m, threads).total;
}
}

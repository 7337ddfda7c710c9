// The choices that a call makes from sizes alone: items of a split plan,
// clusters or a plan, launch shape of the step kernels.  Host code without
// CUDA calls.
#include <algorithm>

#include "kvd_internal.h"

namespace kvd {

// Items end at about the same time on all warps if there are some of them per
// warp: three for MHA, two for GQA, whose items leave a partial per query
// head.  But an item costs about 0.6 pages beside its own, and a row of several
// a merge, so where a warp's share is short (up to 30 pages of d = 128)
//  - rows of nearly equal length are cut into one item per resident warp, or
//    up to 1.3 for shares past 15 pages of 200 units or more;
//  - unequal rows stay whole if none is much longer than a warp's share, or up
//    to 8 pages and four shares.  A host's step then runs without a merge pass
//    (rows of up to 5 pages always); a device step launches it in any case, and
//    the line is at 2.3 shares.
// Longer shares gain nothing (32 heads of 900, B 24 / 32: best target within
// 2 % of a third of the share), up to items so long that the last ones to end
// leave the others idle: targets from 48 pages (d = 64: 65) for rows past 128
// become a third of that, at least 40 and at most 128.
//
// us per layer of host steps, three (GQA two) items per warp and the rule.
// Equal rows: 32 heads of 900 tokens, B 5 / 8 / 12 16.6 and 13.2, 21.9 and 18.9,
// 29.2 and 26.8; 16/8 heads of 500, B 32 13.8 and 11.8; 14/2 at d = 64 of 1000, B
// 128 15.3 and 12.8; 8/8 at d = 64 of 700, B 64 21.5 and 17.0.  The 1.06 against
// 1.0: 32 heads, 8 rows of 760 to 1000 19.8 and 18.3, nine other batches within
// 2 % of each other up to 1.15; the 1.3 against 1.0 within 3 %, 2.0 up to 5 %
// slower; fewer than 200 units: 32 heads, 16000 tokens 39.7 and 45.1, 3 rows of
// 3100 26.0 and 28.4.  Whole rows: 56/8 heads, 106 of up to 105 tokens 12.5 and
// 8.1; 32 heads, 57 of up to 248 23.3 and 20.2; 8/8 at d = 64, 256 of up to 300
// (1.13 shares) 19.7 and 14.8; but 40/40 heads, a row of 101 tokens and 10 of
// 10-24 4.7 and, whole, 6.2; 8/8 heads, 33 of up to 8 pages 4.7 and 6.9, device
// steps 5.9 and 9.1.  At least 16, so that whole rows of 2 pages are not halved
// where the last rows take fractions (56/8 heads, 152 such rows 1.7 times as long).
// Long items: 32 heads, 96 rows of up to 8192 tokens, 94 / 40 / 48 / 64 pages
// 385 379 380 376, 128 / 42 691 680; 78 of up to 4581, 73 / 40 / 48 297 293 299;
// 16/8 heads, 149 of up to 4606, 53 / 40 / 64 154 147 151; not below: 56/8 heads,
// 117 of up to 4592, 37 / 40 108 107; 8/8 at d = 64, 37 of up to 27861, 52 / 40
// 111 110.
int32_t auto_item_pages(int D, bool gqa, int num_kv_heads, int64_t warps, int64_t rows, int64_t pages,
                        int64_t max_pages, bool growing)
{
    const int64_t units = rows * num_kv_heads, total = pages * num_kv_heads;
    const int64_t per_warp = gqa ? 2 : 3;
    int64_t T = std::max<int64_t>(2, (total + per_warp * warps - 1) / (per_warp * warps));
    if (T > (D == 128 ? 47 : 64) && max_pages > 128) T = std::max<int64_t>(40, T / 3);
    T = std::min<int64_t>(128, T);
    // Pages of 4 KB (d = 128) per warp.
    const double share = (double)total / (double)warps * D / 128;
    if (share > 30 || rows < 1) return (int32_t)T;
    const double even = (double)max_pages * (double)rows / (double)std::max<int64_t>(1, pages);   // longest row / mean row
    int64_t few = 0;
    bool whole = false;   // every row is one item
    if (share < 15 ? even <= 1.35 : even <= 1.15 && 6 * units >= warps) {
        const double want = (double)warps / (double)units * (share < 15 ? 1.06 : 1.3) + (share < 15 ? 0.0 : 0.5);
        const int64_t items = std::max<int64_t>(1, (int64_t)want);
        few = (max_pages + (growing ? max_pages / 8 : 0) + items - 1) / items;
        // The 1.06 is for rows shorter than the longest.  Where the mean row's
        // items outnumber the warps all the same, the few warps that work a
        // second item cost up to 4 pages' time (d = 64: 7): items a page larger
        // (d = 64: up to 3) if that is enough (us per layer; 32 heads, 229
        // pages in items of 6 / 7: 15.0 / 11.9; 3 rows of 88, 7 / 8: 15.9 /
        // 12.7; 8/8 heads at d = 64, 3 rows of 738, 14 / 15: 19.4 / 14.8; but
        // 32 heads, 8 rows of 65, 14 / 17: 21.2 / 22.6).
        int64_t fit = few;
        while (share < 15 && fit < max_pages && (pages + rows * fit - 1) / (rows * fit) * units > warps) ++fit;
        if (fit - few < 2 * 128 / D) few = fit;
        whole = items == 1;
    } else if ((!growing && max_pages <= 5) ||
               (max_pages <= 8 && 10 * max_pages * warps <= (growing ? 23 : 40) * total) ||
               (units >= warps && 10 * max_pages * warps <= 13 * total)) {
        few = max_pages;
        whole = true;
    }
    // (also the last rows', whose target is a fraction; not for few units, whose
    // rows would have too few items once they have grown)
    if (whole) few = std::max<int64_t>(few, 16);
    return (int32_t)std::max(T, std::min<int64_t>(128, few));
}

// Twice the usual cap when units x the usual cap would leave resident warps
// without an item and some row is long enough to use more items of T pages,
// and 32 if it uses more than 16 (14/2 heads, 17 rows of 6700 tokens, 26 items
// 19.8 us a layer, cut at 16 22.9; Qwen heads, 8 rows of 3000 11.1 and 13.2).
// Otherwise 32 for MHA and 16 for GQA: a GQA row of at most 16 items merges
// in one round trip with the 16-item variant, the largest whose registers
// fit beside the resident GQA split pass (Qwen shape, of the copy rate: 0.742
// at 32, 0.769 at 16, 0.756 at 24, 0.686 at 12).
int32_t chunk_cap(bool gqa, int64_t units, int64_t warps, int64_t max_pages, int32_t T)
{
    if (units * kChunkCap < warps) {
        if (max_pages > (int64_t)kChunkCap * T) return kMaxChunks;
        if (max_pages > (int64_t)kChunkCapGqa * T) return kChunkCap;
    }
    return gqa ? kChunkCapGqa : kChunkCap;
}

// The allocation-free call's: with a row of more than 256 pages and 32 shares
// (pages per warp) 32 items for GQA too, as that row decides (us a call, 16 and 32; 28/4
// heads, 12 rows of 5400 tokens and one of 21500 52 and 36; 16/8, 6 of 3600 to
// 28600 65 and 57; 14/2, 25 of 288 and one of 11500 24 and 15; the Qwen-shaped
// batch, whose longest row has 27 shares, stays at 16).
int32_t noalloc_chunk_cap(bool gqa, int num_kv_heads, int64_t warps, int64_t rows, int64_t pages, int64_t max_pages,
                          int32_t T)
{
    const int32_t cap = chunk_cap(gqa, rows * num_kv_heads, warps, max_pages, T);
    return max_pages > 256 && max_pages * warps > 32 * pages * num_kv_heads ? std::max(cap, kChunkCap) : cap;
}

// Pages that a warp of the longest row may have in clusters of n warps for each
// of `units` units, whose layer holds `bytes` of K and V: the time that takes
// against the plan's merge pass and what the layer's bytes take in any case.
// GQA: 5 pages (d = 64: 7) and 1 more per 4 MB (2.8 MB), up to 25 MB, which keep
// the HBM busy beside them.  An MHA page is worked on the CUDA cores and takes
// a warp about twice as long: 4 pages, and 3 and 1 more per 6 MB, up to 7, or 5
// where half of the GPU's warps have nothing that the plan would give them (d =
// 64: 5 and 1 more per 4.5 MB, or up to 7 with 8 warps to a CTA).  Us per layer,
// plan and clusters, 8/8 heads: 2 rows of 3000, 6 pages 7.7 and 8.2; 6 of up to
// 2330, 10 pages 7.6 and 10.6; 16/16, one of 2500, 5 pages 7.4 and 6.9, of
// 5000, 10 pages 9.6 and 12.7; 40/40, 9 of up to 380, 6 pages 6.5 and 8.0, 3 of
// up to 730, 6 pages 9.1 and 7.5; 8/8 at d = 64, 17 of up to 1080, 9 pages 10.4
// and 7.2, 2 of 9200 and 1500, 9 pages 8.4 and 9.6.
int64_t most_pages_per_warp(int D, bool gqa, int64_t units, int64_t n, int64_t bytes)
{
    if (gqa) return (20000000 + std::min<int64_t>(bytes, 25000000)) / (D == 128 ? 4000000 : 2800000);
    if (D == 128)
        return std::min<int64_t>(n < 64 && units * n < 600 ? 5 : 7, std::max<int64_t>(4, (17000000 + bytes) / 6000000));
    return n == 64 ? 7 : (24000000 + bytes) / 4500000;
}

// The line between the two, measured as us per layer of graph-replayed steps
// (split plan -> clusters).  Clusters save the merge pass and its dependency
// hop (2.3 us), but cut the rows evenly, without the plan's balancing: they
// win up to about 45 MB of K/V per layer (LLaVA heads, 800 tokens, B 1 / 2 / 3:
// 6.5 -> 4.3, 8.0 -> 7.1, 10.2 -> 9.7; B 4, 52 MB: 12.0 -> 13.9; Qwen heads,
// 1500 tokens, B 4 / 8: 7.0 -> 4.3, 8.4 -> 6.3; 16/8 heads of 500, B 20: 9.1 ->
// 8.7; B 16 of 1400, 46 MB: 10.2 -> 10.4), unless one row is so long that its
// warps finish far behind the others (Qwen heads, 8 rows of 300 to 3800
// tokens, 8 pages per warp: 9.8 -> 7.8; 7 of 300 to 4300, 24 MB, 9 pages: 9.3 ->
// 8.1; 8/8 heads, 20 rows of 50 to 1500, 12
// pages per warp: 12.1 -> 14.2; 1 row of 32000, 32 pages: 19.5 -> 21.5).
//
// Of the shapes, the one with the most warps per unit whose units all find a
// slot at once, with a tenth to spare for the next launch's (LLaVA heads,
// B 3, 96 units: 4 x 4 warps with 2 stages, 110 slots, 10.0; with 3 stages,
// 74 slots, 13.9), but no more than about a warp per page (8 x 8 against
// 4 x 4 warps at 7 pages: 10.2 against 3.0).
//
// spread: for a launch that loads nothing before its dependency wait.  Placed
// while the clusters before it leave, it would crowd on the SMs that empty
// first; with as many stages as let all units stay resident an SM takes no
// more than its share of CTAs (us per call in a row, fewest stages -> most:
// LLaVA heads, 850 tokens 5.0 -> 4.3, 40/40 heads, 500 tokens 4.0 -> 3.6, Qwen
// heads, 8 rows of 700 5.2 -> 4.3).  A launch that does load early is better
// off with a slot for every CTA at once (LLaVA layer 4.8 -> 5.2).
//
// limit: the pages that a row may grow to while the shape stays (device steps
// and the graphs captured of them; 0 for a step that picks its own).  Warps and
// stages then serve rows of half of that, and a step whose longest row could
// still fall far behind runs from the plan, which follows the lengths.  A shape
// picked for one page a row, graph kept while the rows grow to 2000 / 8000
// tokens: LLaVA heads, one row 43 / 165 us a layer, Qwen heads, 8 rows 33 / 119
// (plan 10.3 / 22.8 and 11.0 / 22.7).  Rows that all grow are within 6 % of the
// plan or faster; most_grown bounds one row of `limit` pages among short ones
// (us, clusters and plan; Qwen heads, 8 rows, clusters of 32 warps, 4000 / 8000
// / 16000 tokens 6.6 and 7.0, 10.3 and 9.5, 18.2 and 13.3; 24 rows, 16 warps,
// 8000 19.7 and 17.9; 56/8 heads, 20 rows, 8 warps, 1000 / 2000 7.2 and 7.3,
// 11.5 and 9.2; LLaVA heads, 2 rows, 16 warps, 1000 / 2000 5.5 and 7.3, 9.9 and
// 9.4; 8/8 heads, 4 rows, 32 warps, 2000 / 4000 5.3 and 6.0, 9.2 and 7.9).
// Clusters of 64 GQA warps cut a row as the plan does (28/4 heads, 32000 tokens
// 19.8 and 18.8), and the heads of a single row that fill the GPU are bound by
// their bytes (LLaVA heads, 16000 tokens 41.4 and 39.7).  Short rows of long
// tables pay: LLaVA heads, one of 16 / 50 tokens 2.9 / 3.1, with a shape of
// their own 2.5 / 2.5 (plan 4.0 / 5.2).
ClusterShape pick_cluster_shape(ResidentClusters resident, int device, int D, bool gqa, int num_kv_heads,
                                int64_t batch, int64_t pages, int64_t max_pages, bool spread, int64_t limit)
{
    constexpr int64_t kMostBytes = 45000000;   // K and V of a layer
    constexpr int kWarpsOf[][2] = {{8, 8}, {8, 4}, {4, 4}, {2, 4}, {1, 4}};
    const int64_t units = batch * num_kv_heads;
    const int64_t stage = 2 * (int64_t)kPageSize * D * 2;
    const int64_t bytes = pages * num_kv_heads * stage;
    if (bytes > kMostBytes) return ClusterShape{};
    const int64_t row = std::max(max_pages, (limit + 1) / 2);   // pages that warps and stages are chosen for
    auto most_grown = [&](int64_t n) -> int64_t {
        if (gqa) {
            if (n == 64 || (n == 32 && D == 64 && units >= 38)) return limit;
            return n == 32 ? 17 : n == 16 ? 33 : n == 8 ? 9 : 8;
        }
        if (units * n > 900 && (batch == 1 || n == 32)) return batch == 1 ? limit : D == 128 ? 8 : 18;
        return D == 128 ? (n == 16 ? 6 : 4) : n == 64 ? 9 : n == 16 ? 7 : 5;
    };
    for (const auto& cw : kWarpsOf) {
        ClusterShape sh;
        sh.ctas = cw[0];
        sh.warps = cw[1];
        const int64_t n = (int64_t)sh.ctas * sh.warps;
        if (n > 4 && (n / 2 >= row || (n == 64 && row <= 128))) continue;
        const int ring = (int)std::min<int64_t>(kClusterRingBytes / stage, std::max<int64_t>(1, (row + n - 1) / n));
        for (sh.ring = ring; sh.ring >= std::min(ring, 2); --sh.ring) {
            if (10 * (int64_t)resident(device, D, gqa, sh) < 11 * units) continue;
            const int64_t most = most_pages_per_warp(D, gqa, units, n, bytes);
            if ((max_pages + n - 1) / n > most) return ClusterShape{};
            if (limit > max_pages && (limit + n - 1) / n > std::max(most, most_grown(n))) return ClusterShape{};
            for (ClusterShape more = sh; spread && ++more.ring <= kClusterRingBytes / stage;) {
                if (resident(device, D, gqa, more) < units) break;
                sh = more;
            }
            return sh;
        }
    }
    return ClusterShape{};
}

// A plan of whole rows has no merge pass, so a row of one page is quickest as
// one warp's item; of two for large GQA groups, whose exchange over the cluster
// takes long, and where few rows have a second page (us per layer, clusters and
// whole rows; 56/8 heads, 6 rows of up to 12 tokens 3.2 and 2.5; 28/4 heads, 51
// of 8 4.1 and 2.7; 32 heads, 3 of 8 2.5 and 2.4; 14/2 heads, 60 of up to 2
// pages 3.8 and 2.7; 16/8 heads, 43 of which one has 2 3.0 and 2.6; but 40/40
// heads, one of 2 2.6 and 2.9; d = 64, 14/2 heads, 76 of up to 2 2.5 and 2.8, 6/2
// and 8/8 heads, up to 100 units of one page 2.1-2.3 and 2.2-2.4).
bool whole_rows_beat_clusters(int D, int group, int num_kv_heads, int64_t rows, int64_t pages, int64_t max_pages)
{
    if (D == 64 && group <= 4 && rows * num_kv_heads <= 100) return false;
    return max_pages == 1 || (max_pages == 2 && ((group > 4 && D == 128) || 4 * pages <= 5 * rows));
}

// The first layer after a step kernel may be placed while that runs and what
// ran before it leaves, which saves up to 1 us a step.  But a split pass that
// fills less than half of its slots then crowds on the SMs that are empty
// first, and the layers after it, each placed where the one before the last
// left, keep that pattern (us per layer, placed early and not; 28/4 heads, one
// row of 20000 tokens, 256 of 1216 slots 14.3 and 13.6; 8/8 heads, one of 12000,
// 512 slots 14.5 and 14.1; at d = 64 9.8 and 9.4; from 1216 on the same).
bool place_first_layer_early(int64_t ctas, int64_t slots) { return 2 * ctas >= slots; }

// A step kernel that builds a plan is a cluster of 8 CTAs, but for a few short
// rows, which one CTA handles before the cluster has met.  Each warp takes a
// row at a time, or 128 page ids of one, so 8 warps a CTA, 16 for more than 64
// rows, and a thread per row where a block can have one (the rows' order
// depends on that).  us a step, one CTA of 256 / 512 / 1024 threads and 8 of 256 /
// 512 / 1024: 1 row of 50 pages 3.9 4.1 4.7 and 4.7 5.1 6.0; 16 of 4 4.8 4.4 5.2
// and 4.9 5.2 6.4; 12 of 85 5.7 5.1 5.4 and 4.8 5.2 6.4; 64 of 8 9.7 7.3 6.8 and
// 5.2 5.7 7.1; 188 of 1 22.0 14.8 12.0 and 8.5 8.2 8.3; 96 of 128 24.4 17.2 15.7
// and 8.6 7.8 8.1; 8 of 2049 16.9 11.9 10.6 and 6.3 6.1 7.0; 500 of 4 - 37.0 29.0
// and - 16.1 15.8.  Without a plan (no ids) one CTA, 256 / 512 / 1024 threads: 1.7
// 1.7 1.9.
int step_ctas(int64_t rows, int64_t ids) { return ids == 0 || (rows <= 16 && ids <= 1024) ? 1 : 8; }

int step_threads(int64_t rows, int64_t ids)
{
    if (rows > 512) return 1024;
    if (rows > 256) return 512;
    if (ids == 0) return 256;
    return rows > (step_ctas(rows, ids) == 1 ? 8 : 64) ? 512 : 256;
}

}  // namespace kvd

// Page-table maintenance, the per-step update and split plan, token writes /
// reads into pages, and the fused K+V append (kv_append).
#include <algorithm>
#include <climits>

#include "kvd_internal.h"
#include "kvd_ptx.cuh"

namespace kvd {

namespace {

__device__ __forceinline__ void flag_error(int32_t* err, int bit) { atomicOr(err, bit); }

template <int N>
__global__ void scatter_i32_kernel(int32_t* base, const __grid_constant__ ScatterI32<N> s)
{
    griddep_launch_dependents();
    griddep_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.n; i += gridDim.x * blockDim.x)
        base[s.idx[i]] = s.val[i];
}

// Exclusive block-wide prefix sum of one int per thread (whole warps).
__device__ int block_exclusive_scan(int v, int* total)
{
    __shared__ int warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;   // inclusive over warps
    }
    __syncthreads();
    const int before_warp = warp ? warp_sums[warp - 1] : 0;
    *total = warp_sums[31];
    __syncthreads();
    return before_warp + x - v;
}

// Split plan of a step, built by a cluster of CTAs: plan position
// i takes batch row b, sequence seq, len tokens from row_at(i, &b, &seq,
// &len); the row is cut into row_chunks() items of near-equal size, a row's
// items adjacent, its target size graduated by position (row_item_pages).
// Entries past max_entries are dropped with error bit 4.  Each entry's page
// ids are copied from the page table into pages_out (stride page_stride), so
// the decode kernel reads them alongside the entry.  Returns the entries
// planned (in CTA 0).
//
// CTA 0 orders and counts; all CTAs then write entries and page lists, the
// rows spread over their warps, reading what CTA 0 found from its shared
// memory.  Device step, one CTA of 1024 threads and eight: 32 rows of 288 pages
// 10.3 and 5.8 us, 96 of 128 15.7 and 7.8, 188 of one page 12.0 and 8.2.
template <class RowAt>
__device__ int build_split_plan(int batch, int item_pages, int chunk_cap, int max_entries, RowAt row_at,
                                PlanEntry* plan, int2* rows, const int32_t* page_table, int max_pages,
                                int32_t* pages_out, int page_stride, int32_t* err)
{
    constexpr int kFields = 6;                     // seq, pages, first entry, items, batch row, tokens
    __shared__ int s_row[kFields][1024];
    const int lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int warp = rank * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
    const int n_warps = (int)cluster_nctarank() * (int)(blockDim.x >> 5);
    int carry = 0;
    for (int base = 0; base < batch; base += blockDim.x) {
        if (rank == 0) {
            const int i = base + threadIdx.x;
            int b = 0, seq = 0, len = 0, np = 0, nch = 0;
            if (i < batch) {
                row_at(i, &b, &seq, &len);
                np = (len + kPageSize - 1) / kPageSize;
                nch = row_chunks(np, row_item_pages(item_pages, i, batch), chunk_cap);
            }
            int total;
            const int off = carry + block_exclusive_scan(nch, &total);
            if (off + nch > max_entries) {
                flag_error(err, 4);
                nch = 0;
            }
            if (i < batch) rows[b] = make_int2(off, nch);
            s_row[0][threadIdx.x] = seq;
            s_row[1][threadIdx.x] = np;
            s_row[2][threadIdx.x] = off;
            s_row[3][threadIdx.x] = nch;
            s_row[4][threadIdx.x] = b;
            s_row[5][threadIdx.x] = len;
            carry += total;
        }
        __syncwarp();
        cluster_sync();
        // Each row gets (warps / rows) warps, at least one; the first writes
        // its entries, all copy 32-page windows of its page ids, four in
        // flight per lane.  Page j of a row lies in item c at offset o
        // (chunk_range inverted: the first np % nch items hold one page more).
        const int n_rows = min((int)blockDim.x, batch - base);
        const int per_row = n_rows >= n_warps ? 1 : n_warps / n_rows;
        if (warp >= n_rows * per_row) cluster_arrive_release();
        for (int t = warp; t < n_rows * per_row; t += n_warps) {
            const int r = t / per_row, part = t - r * per_row;
            const int field = cluster_load(cluster_map(smem_addr(&s_row[min(lane, kFields - 1)][r]), 0));
            const int rseq = __shfl_sync(0xffffffffu, field, 0), rnp = __shfl_sync(0xffffffffu, field, 1);
            const int roff = __shfl_sync(0xffffffffu, field, 2), rnch = __shfl_sync(0xffffffffu, field, 3);
            const int rb = __shfl_sync(0xffffffffu, field, 4), rlen = __shfl_sync(0xffffffffu, field, 5);
            if (t + n_warps >= n_rows * per_row) cluster_arrive_release();   // the warp has read its last row's
            if (rnch == 0) continue;
            const int small = rnp / rnch, extra = rnp % rnch, big_pages = extra * (small + 1);
            const int32_t* src = page_table + (int64_t)rseq * max_pages;
            for (int w0 = part; w0 * 32 < rnp; w0 += 4 * per_row) {
                int32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = (w0 + u * per_row) * 32 + lane;
                    v[u] = j < rnp ? src[j] : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = (w0 + u * per_row) * 32 + lane;
                    if (j >= rnp) continue;
                    int c, o;
                    if (j < big_pages) {
                        c = j / (small + 1);
                        o = j - c * (small + 1);
                    } else {
                        c = extra + (j - big_pages) / small;
                        o = j - big_pages - (c - extra) * small;
                    }
                    if (o < page_stride)
                        pages_out[(int64_t)(roff + c) * page_stride + o] = v[u];
                    else
                        flag_error(err, 4);
                }
            }
            if (part == 0) {
                for (int c = lane; c < rnch; c += 32) {
                    int first, n;
                    chunk_range(rnp, rnch, c, &first, &n);
                    plan[roff + c] = PlanEntry{rb, rseq, rlen, first, n, c, rnch, roff};
                }
            }
        }
        __syncwarp();
        cluster_wait();   // CTA 0's shared arrays are read: the next chunk of rows, or its exit
    }
    return carry;
}

// Apply the step's length / page-table updates; in the last launch of a step,
// build the split plan with the rows in the host's order (longest first when
// the batch fits one launch).  The host sized the plan for exactly this step.
__global__ void __launch_bounds__(1024)
    step_kernel(const __grid_constant__ StepPatch patch, const __grid_constant__ PlanArgs a)
{
    griddep_wait();
    griddep_launch_dependents();   // the first layer may be placed; it waits before it reads anything
    const bool lead = cluster_ctarank() == 0;
    for (int i = threadIdx.x; lead && i < patch.n; i += blockDim.x) {
        const int seq = patch.seq[i], len = patch.new_len[i];
        a.seq_len[seq] = len;
        a.step_seq[patch.b0 + i] = seq;
        if (a.no_plan) a.rows[patch.b0 + i] = make_int2(seq, len);
        if (patch.new_page[i] >= 0)
            a.page_table[(int64_t)seq * a.max_pages + (len - 1) / kPageSize] = patch.new_page[i];
    }
    if (!a.build || a.no_plan) return;
    __syncthreads();
    build_split_plan(
        a.batch, a.item_pages, a.chunk_cap, INT_MAX,
        [&](int i, int* b, int* seq, int* len) {
            // (an ordered batch is one launch: its rows are in the patch)
            *b = a.use_order ? a.order[i] : i;
            *seq = a.use_order ? patch.seq[*b] : a.step_seq[*b];
            *len = a.use_order ? patch.new_len[*b] : a.seq_len[*seq];
            if (*len <= 0 || *len > a.max_pages * kPageSize) {
                flag_error(a.err, 4);
                *len = 1;
            }
        },
        a.plan, a.rows, a.page_table, a.max_pages, a.page_ids, a.page_stride, a.err);
    if (lead && threadIdx.x == 0) *a.step_no += 1u;
}

// The same step on the device (graph-replayable, no host input): rows in
// batch order reserve position len; a row whose position opens a page takes
// the next page of the device free stack, in batch order (the same pages the
// host allocator would hand out); then the split plan, rows longest first
// (stable, as on the host) when the batch fits one block, else in batch order.
// A row whose step fails (a sequence id outside [0, max_seqs), a full page
// row, or an exhausted pool: error bits 4 / 8) keeps its length and gets
// step_seq -1 and no work items, so the layer calls that follow neither write
// its cache nor its output row.  With the batch in one block, each row's
// sequence and new length stay in shared memory for the ranking and the plan.
__global__ void __launch_bounds__(1024) step_device_kernel(const StepDevArgs a)
{
    __shared__ int s_free[1024];
    __shared__ int s_seq[1024], s_len[1024];   // per batch row when the batch fits the block
    griddep_wait();
    griddep_launch_dependents();   // the first layer may be placed; it waits before it reads anything
    const bool small = a.batch <= (int)blockDim.x;
    const bool lead = cluster_ctarank() == 0;   // the other CTAs only help to write the plan
    // The stack's top pages, one per thread, load along with the rows' lengths
    // (with the early arrival in build_split_plan 1 us of a step of 96 rows).
    const int top0 = lead ? *a.free_top : 0;
    if (lead && threadIdx.x < top0) s_free[threadIdx.x] = a.free_pages[top0 - 1 - threadIdx.x];
    int carry = 0;
    for (int base = 0; lead && base < a.batch; base += blockDim.x) {
        const int i = base + threadIdx.x;
        int seq = -1, len = 0, need = 0;
        bool ok = false;
        if (i < a.batch) {
            seq = a.seq_ids[i];
            if (seq >= 0 && seq < a.max_seqs) {
                len = a.seq_len[seq];
                ok = len >= 0 && len + 1 <= a.max_pages * kPageSize;
            }
            if (!ok) flag_error(a.err, 4);
            need = (ok && len % kPageSize == 0) ? 1 : 0;
        }
        int total;
        const int rank = carry + block_exclusive_scan(need, &total);   // also orders s_free's writes
        if (ok) {
            int32_t page = -1;
            if (need) {
                const int idx = top0 - 1 - rank;
                if (idx < 0) {
                    flag_error(a.err, 8);   // pool exhausted
                    ok = false;
                } else {
                    page = rank < (int)blockDim.x ? s_free[rank] : a.free_pages[idx];
                }
            }
            if (ok) {
                if (page >= 0) a.page_table[(int64_t)seq * a.max_pages + len / kPageSize] = page;
                a.seq_len[seq] = len + 1;
                len += 1;
            }
        }
        if (i < a.batch) {
            a.step_seq[i] = ok ? seq : -1;
            if (a.no_plan) a.rows[i] = make_int2(ok ? seq : 0, ok ? len : 0);   // no tokens: the row is left out
            if (small) {
                s_seq[i] = ok ? seq : -1;
                s_len[i] = ok ? len : 0;
            }
        }
        carry += total;
    }
    __syncthreads();
    if (lead && threadIdx.x == 0) *a.free_top = top0 - min(carry, top0);
    if (a.no_plan) return;

    // Row order: the rank of row b counts the rows with more pages, and the
    // rows with as many pages that come before b (failed rows have none).
    __shared__ int s_np[1024];
    __shared__ int s_order[1024];
    if (small && lead) {
        const int b = threadIdx.x;
        int np = 0;
        if (b < a.batch) {
            np = (s_len[b] + kPageSize - 1) / kPageSize;
            s_np[b] = np;
        }
        __syncthreads();
        if (b < a.batch) {
            int rank = 0;
            for (int j = 0; j < a.batch; ++j) {
                const int o = s_np[j];
                rank += (o > np || (o == np && j < b)) ? 1 : 0;
            }
            s_order[rank] = b;
        }
        __syncthreads();
    }
    const int entries = build_split_plan(
        a.batch, a.item_pages, a.chunk_cap, a.max_entries,
        [&](int i, int* b, int* seq, int* len) {
            *b = small ? s_order[i] : i;
            *seq = small ? s_seq[*b] : a.step_seq[*b];
            *len = *seq < 0 ? 0 : (small ? s_len[*b] : a.seq_len[*seq]);   // 0 tokens: no items
            if (*seq < 0) *seq = 0;
        },
        a.plan, a.rows, a.page_table, a.max_pages, a.page_ids, a.page_stride, a.err);
    if (lead && threadIdx.x == 0) {
        *a.n_entries = min(entries, a.max_entries);
        *a.step_no += 1u;
    }
}

// Reserve n tokens for a sequence, or release all its pages, on the device
// free stack, in stream order with device-side steps: a reservation takes
// the next pages of the stack for the logical pages its new positions open
// (all or nothing: a full page row sets bit 4, an exhausted pool bit 8, and
// nothing changes); a release puts the pages back on top of the stack so that
// its logical page 0 is handed out next, clears its page-table row and sets
// its length to 0.
//
// A chain of dependent loads (length and stack top, then pages), so its time
// is latency: every thread reads the length and the top itself instead of
// waiting for one that does, a release reads its row's first pages along with
// them, and calls that follow one another are chained (programmatic dependent
// launch).  An admission of 64 requests (64 releases, 64 reservations): 4.1 us
// a call before, 1.6 now.
__global__ void __launch_bounds__(256) seq_op_kernel(const SeqOpArgs a)
{
    griddep_launch_dependents();
    griddep_wait();
    int32_t* row = a.page_table + (int64_t)a.seq * a.max_pages;
    const int tid = threadIdx.x;
    const int len = a.seq_len[a.seq];
    const int top = *a.free_top;
    const int32_t page0 = a.free_seq && tid < a.max_pages ? row[tid] : -1;
    int first = 0, count = 0, err = 0, new_len = len;
    if (len < 0 || len > a.max_pages * kPageSize) {
        err = 4;
    } else if (a.free_seq) {
        count = (len + kPageSize - 1) / kPageSize;
        new_len = 0;
    } else {
        const int64_t end = (int64_t)len + a.n;
        first = (len + kPageSize - 1) / kPageSize;
        const int64_t need_total = (end + kPageSize - 1) / kPageSize;
        if (need_total > a.max_pages) {
            err = 4;
        } else if (need_total - first > top) {
            err = 8;
        } else {
            count = (int)(need_total - first);
            new_len = (int)end;
        }
    }
    __syncthreads();   // every thread has the length and the top
    if (tid == 0) {
        if (err) flag_error(a.err, err);
        else {
            a.seq_len[a.seq] = new_len;
            *a.free_top = a.free_seq ? top + count : top - count;
        }
    }
    if (a.free_seq) {
        for (int k = tid; k < count; k += blockDim.x) {
            a.free_pages[top + count - 1 - k] = k == tid ? page0 : row[k];
            row[k] = -1;
        }
    } else {
        for (int k = tid; k < count; k += blockDim.x) row[first + k] = a.free_pages[top - 1 - k];
    }
}

// Tokens of one sequence and layer to or from its pages.  CTA (x, y) takes
// the x-th page touched and the y-th 1024 of its 16-byte chunks, in the
// page's order ([H_kv][slot][D]); the page id is read once and a thread's
// four chunks of K and V are in flight together.  (A grid-stride loop of one
// chunk with 64-bit divisions, for 900 LLaVA tokens of a layer,
// 14.7 MB read and written, 4.4 us at the copy rate: 10.2 us in
// a row, now 6.4 with the launches chained; 16 tokens 4.2, now 2.6.)
constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 4;

template <bool TO_POOL>
__global__ void __launch_bounds__(kCopyThreads) token_copy_kernel(const TokenCopyArgs a)
{
    griddep_launch_dependents();
    griddep_wait();
    if (a.len && a.first_pos + a.n > *a.len) {   // positions past the sequence's length
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) flag_error(a.err, 4);
        return;
    }
    const int page_idx = a.first_pos / kPageSize + (int)blockIdx.x;
    const int p0 = max(a.first_pos, page_idx * kPageSize);
    const int nt = min(a.first_pos + a.n, (page_idx + 1) * kPageSize) - p0;
    const int32_t pid = a.pt_row[page_idx];
    if (pid < 0 || pid >= a.num_pages) {
        if (threadIdx.x == 0) flag_error(a.err, 1);
        return;
    }
    const int cpr = a.D / 8;   // 16-byte chunks per (token, head) row
    const int total = a.H_kv * nt * cpr;
    const int slot0 = p0 - page_idx * kPageSize;
    const int64_t page = (int64_t)pid * a.H_kv * kPageSize * cpr;
    const int64_t tok0 = (int64_t)(p0 - a.first_pos) * a.H_kv * cpr;
    uint4* pk = reinterpret_cast<uint4*>(a.pool_k) + page;
    uint4* pv = reinterpret_cast<uint4*>(a.pool_v) + page;
    uint4* tk = reinterpret_cast<uint4*>(a.tok_k) + tok0;
    uint4* tv = reinterpret_cast<uint4*>(a.tok_v) + tok0;
    uint4 rk[kCopyUnroll], rv[kCopyUnroll];
    int from[kCopyUnroll], to[kCopyUnroll];
    const int base = (int)blockIdx.y * kCopyThreads * kCopyUnroll + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        const int idx = base + u * kCopyThreads;
        if (idx < total) {
            const int r = idx / cpr, c = idx - r * cpr;
            const int h = r / nt, t = r - h * nt;
            const int in_page = (h * kPageSize + slot0 + t) * cpr + c, in_tok = (t * a.H_kv + h) * cpr + c;
            from[u] = TO_POOL ? in_tok : in_page;
            to[u] = TO_POOL ? in_page : in_tok;
            rk[u] = (TO_POOL ? tk : pk)[from[u]];
            rv[u] = (TO_POOL ? tv : pv)[from[u]];
        }
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
        if (base + u * kCopyThreads < total) {
            (TO_POOL ? pk : tk)[to[u]] = rk[u];
            (TO_POOL ? pv : tv)[to[u]] = rv[u];
        }
    }
}

// Bulk write of packed token blocks.  CTA x finds its block by a binary
// search over tile_start, reads the tile's page id once, then its threads
// stream (the z-th cta_chunks 16-byte chunks of) the tile in the page's order
// ([H_kv][slot][D], four chunks per thread in flight) with streaming loads and
// stores: the source is read once and the pages are not read back soon.
//
// A whole page of 32 or 40 heads is 160 KB for one CTA: a few hundred CTAs
// leave the last ones running alone.  2048 chunks of K and V per CTA, 1024
// where that gives fewer than 5000 CTAs, 512 where that gives fewer than one
// per SM (us, one CTA per tile before / 2048 / 1024 / 512; 40 heads, 11 blocks
// of 4-220 tokens, 4 layers: 17.0 / 9.3 / 8.3 / 8.8; 32 heads, 64 blocks of
// 900, 8 layers: 2160 / 2153 / 2199 / 2276; 8 heads of 64, 4 blocks of 96:
// 3.5 / 3.6 / 3.7 / 2.9).
constexpr int kVarlenThreads = 256;
constexpr int kVarlenUnroll = 4;

__global__ void __launch_bounds__(kVarlenThreads) varlen_write_kernel(const __grid_constant__ VarlenWriteArgs a)
{
    griddep_launch_dependents();
    griddep_wait();
    const int tile = blockIdx.x;
    int lo = 0, hi = a.n_blocks - 1;   // the last block with tile_start <= tile
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.tile_start[mid] <= tile) lo = mid;
        else hi = mid - 1;
    }
    const int first = a.first_pos[lo];
    const int page_idx = first / kPageSize + (tile - a.tile_start[lo]);
    const int p0 = max(first, page_idx * kPageSize);
    const int p1 = min(first + a.n_tok[lo], (page_idx + 1) * kPageSize);
    const int nt = p1 - p0;
    // A block that passes its sequence's length is refused whole (every tile
    // checks the block's end, not its own).
    if (a.seq_len && first + a.n_tok[lo] > a.seq_len[a.seq[lo]]) {
        if (threadIdx.x == 0) flag_error(a.err, 4);
        return;
    }
    const int32_t pid = a.page_table[(int64_t)a.seq[lo] * a.max_pages + page_idx];
    if (pid < 0 || pid >= a.num_pages) {
        if (threadIdx.x == 0) flag_error(a.err, 1);
        return;
    }
    const int cpr = a.D / 8;   // 16-byte chunks per (token, head) row
    const int total = min(a.H_kv * nt * cpr, ((int)blockIdx.z + 1) * a.cta_chunks);
    const int64_t layer = blockIdx.y;
    const uint4* sk = reinterpret_cast<const uint4*>(a.k + layer * a.src_layer_stride);
    const uint4* sv = reinterpret_cast<const uint4*>(a.v + layer * a.src_layer_stride);
    uint4* dk = reinterpret_cast<uint4*>(a.pool_k + layer * a.pool_layer_stride) +
                (int64_t)pid * a.H_kv * kPageSize * cpr;
    uint4* dv = reinterpret_cast<uint4*>(a.pool_v + layer * a.pool_layer_stride) +
                (int64_t)pid * a.H_kv * kPageSize * cpr;
    const int64_t tok0 = (int64_t)a.src_row[lo] + (p0 - first);
    const int slot0 = p0 - page_idx * kPageSize;
    for (int base = (int)blockIdx.z * a.cta_chunks + threadIdx.x; base < total; base += kVarlenUnroll * kVarlenThreads) {
        uint4 rk[kVarlenUnroll], rv[kVarlenUnroll];
        int64_t doff[kVarlenUnroll];
#pragma unroll
        for (int u = 0; u < kVarlenUnroll; ++u) {
            const int idx = base + u * kVarlenThreads;
            if (idx < total) {
                const int c = idx % cpr;
                const int r = idx / cpr;
                const int h = r / nt;
                const int t = r - h * nt;
                const int64_t soff = ((tok0 + t) * a.H_kv + h) * cpr + c;
                doff[u] = ((int64_t)h * kPageSize + slot0 + t) * cpr + c;
                rk[u] = __ldcs(sk + soff);
                rv[u] = __ldcs(sv + soff);
            }
        }
#pragma unroll
        for (int u = 0; u < kVarlenUnroll; ++u) {
            if (base + u * kVarlenThreads < total) {
                __stcs(dk + doff[u], rk[u]);
                __stcs(dv + doff[u], rv[u]);
            }
        }
    }
}

// kv_append: one thread per 16-byte chunk of k_new / v_new ([B][H_kv][D]);
// the chunk goes to slot (len-1) % P of page page_table[seq][(len-1) / P].
__global__ void append_kernel(const AppendArgs a)
{
    // Every thread waits (and so completes after) the kernel before it.
    griddep_launch_dependents();
    griddep_wait();
    const int chunks = a.D / 8;
    const int total = a.batch * a.H_kv * chunks;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int c = i % chunks;
    const int bg = i / chunks;
    const int g = bg % a.H_kv;
    const int b = bg / a.H_kv;
    const int seq = a.step_seq[b];
    if (seq < 0) return;   // the row's device-side step failed (already flagged)
    const int pos = a.seq_len[seq] - 1;
    if (pos < 0 || pos >= a.max_pages * kPageSize) {
        flag_error(a.err, 4);
        return;
    }
    const int32_t page = a.page_table[(int64_t)seq * a.max_pages + pos / kPageSize];
    if (page < 0 || page >= a.num_pages) {
        flag_error(a.err, 1);
        return;
    }
    const int64_t poff = (((int64_t)page * a.H_kv + g) * kPageSize + pos % kPageSize) * a.D + c * 8;
    const int64_t noff = (int64_t)i * 8;
    const uint4 kk = *reinterpret_cast<const uint4*>(a.k_new + noff);
    const uint4 vv = *reinterpret_cast<const uint4*>(a.v_new + noff);
    *reinterpret_cast<uint4*>(a.pool_k + poff) = kk;
    *reinterpret_cast<uint4*>(a.pool_v + poff) = vv;
}

// One warp waits, with the decode kernel's bounded wait, on an mbarrier that
// nothing arrives on; status = 1 when the wait gave up, 0 if it completed.
__global__ void wait_timeout_kernel(uint64_t limit_ns, int32_t* status)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_addr(&bar), 1);
        fence_mbar_init();
    }
    __syncwarp();
    const bool done = mbar_wait_bounded(smem_addr(&bar), 0, limit_ns);
    if (threadIdx.x == 0) *status = __all_sync(0xffffffffu, done) ? 0 : 1;
    else (void)__all_sync(0xffffffffu, done);
}

// A launch that may start before the one before it has completed, if pdl (the
// kernel waits before it reads or writes anything).
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, bool pdl, cudaStream_t st, const A&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// A step kernel as one cluster, placed while what ran before it finishes; it
// waits for that at its top.  (13B heads, 12 requests, 4 steps of 8 layers:
// 1974 us as an ordinary launch, 1965 so; 28/4 heads, 254 rows 4828 and 4820.)
template <class... P, class... A>
cudaError_t launch_cluster_of(int ctas, int threads, void (*kernel)(P...), cudaStream_t st, const A&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cfg.gridDim.x;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctas > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int N>
cudaError_t launch_scatter(int32_t* base, const int32_t* idx, const int32_t* val, int n, bool pdl, cudaStream_t st)
{
    ScatterI32<N> s;
    s.n = n;
    std::copy_n(idx, n, s.idx);
    std::copy_n(val, n, s.val);
    return launch_chained(scatter_i32_kernel<N>, (n + 255) / 256, 256, pdl, st, base, s);
}

}  // namespace

cudaError_t launch_wait_timeout_check(uint64_t limit_ns, int32_t* status, cudaStream_t st)
{
    wait_timeout_kernel<<<1, 32, 0, st>>>(limit_ns, status);
    return cudaGetLastError();
}

cudaError_t launch_seq_op(const SeqOpArgs& a, bool pdl, cudaStream_t st)
{
    return launch_chained(seq_op_kernel, 1, 256, pdl, st, a);
}

cudaError_t launch_step_device(const StepDevArgs& a, cudaStream_t st)
{
    const int64_t ids = a.no_plan ? 0 : a.pages;
    return launch_cluster_of(step_ctas(a.batch, ids), step_threads(a.batch, ids), step_device_kernel, st, a);
}

cudaError_t launch_scatter_i32(int32_t* base, const int32_t* idx, const int32_t* val, int n, bool pdl, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    return n <= kScatterSmall ? launch_scatter<kScatterSmall>(base, idx, val, n, pdl, st)
                              : launch_scatter<kScatterMax>(base, idx, val, n, pdl, st);
}

cudaError_t launch_step(const StepPatch& patch, const PlanArgs& plan, cudaStream_t st)
{
    const int64_t ids = plan.build && !plan.no_plan ? plan.pages : 0;
    return launch_cluster_of(step_ctas(plan.batch, ids), step_threads(plan.batch, ids), step_kernel, st, patch, plan);
}

cudaError_t launch_token_copy(const TokenCopyArgs& a, bool pdl, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    const int pages = (a.first_pos + a.n - 1) / kPageSize - a.first_pos / kPageSize + 1;
    const int per_cta = kCopyThreads * kCopyUnroll;
    const int chunks = a.H_kv * std::min(a.n, kPageSize) * (a.D / 8);   // of a page at most
    const dim3 grid((unsigned)pages, (unsigned)((chunks + per_cta - 1) / per_cta));
    return a.to_pool ? launch_chained(token_copy_kernel<true>, grid, kCopyThreads, pdl, st, a)
                     : launch_chained(token_copy_kernel<false>, grid, kCopyThreads, pdl, st, a);
}

cudaError_t launch_varlen_write(const VarlenWriteArgs& a, int n_layers, bool pdl, cudaStream_t st)
{
    if (a.n_tiles <= 0 || n_layers <= 0) return cudaSuccess;
    const int64_t chunks = a.H_kv * kPageSize * (a.D / 8);   // of a whole page's K
    auto parts = [&](int per_cta) { return (chunks + per_cta - 1) / per_cta; };
    const int64_t tiles = (int64_t)a.n_tiles * n_layers;
    VarlenWriteArgs args = a;
    args.cta_chunks = tiles * parts(2048) > 5000 ? 2048 : tiles * parts(1024) > 150 ? 1024 : 512;
    return launch_chained(varlen_write_kernel, dim3((unsigned)a.n_tiles, (unsigned)n_layers, (unsigned)parts(args.cta_chunks)),
                          kVarlenThreads, pdl, st, args);
}

cudaError_t launch_append(const AppendArgs& a, bool pdl, cudaStream_t st)
{
    const int total = a.batch * a.H_kv * (a.D / 8);
    if (total <= 0) return cudaSuccess;
    return launch_chained(append_kernel, (total + 255) / 256, 256, pdl, st, a);
}

}  // namespace kvd

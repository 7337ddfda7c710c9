// decode_attention_noalloc: decode attention over caller-owned paged K/V with
// no device allocation at all.
//
// Who needs it.  The kv_cache path allocates: its pools at creation and, when
// a step's split plan outgrows them, its plan and partial-result buffers with
// cudaMallocAsync.  Some callers may not allocate device memory while they
// serve: an engine plugin whose enqueue must run inside a memory budget fixed
// when the engine was built, a runtime whose device memory all belongs to
// another framework's allocator, or a latency-critical decode thread that must
// not take the allocator's locks.  Those callers own the K/V pools and page
// table themselves and call this entry point instead.
//
// Launches.  Everything that a plan would say follows from the lengths, which
// are on the host: they go to the kernels as parameters (RowTable, LensTable)
// and the page ids come straight from the caller's table, so a call is the
// split pass and its merge pass, or one cluster launch for a small batch.
// (A plan kernel with 20 KB of parameters and a page-list kernel before the
// split pass, two loads per page, the merge pass as an ordinary launch and
// five device queries per call measured 41 us a call on the Qwen-shaped
// batch, 34 us of it on the host.)  The first launch is placed while what ran
// before it finishes (programmatic dependent launch): it sets up its barriers
// and finds its first item, and waits before it reads any device memory, since
// what ran before may have written the pools or the page table.  Calls in a
// row, us per call, as ordinary launches and so: the Qwen-shaped batch from
// Python 26.6 and 24.1; replayed from a graph 13.7 and 13.6 (78 MB, in L2),
// 64 LLaVA rows of 900 tokens 132.7 and 132.0, 2 Qwen rows of 2500 and 4400
// (clusters) 6.5 and 5.9, 4 rows of 100, 8/8 heads, d = 64 3.1 and 2.5.
//
// Scratch.  The per-item partial results, the per-row merge table and the
// work counter live in one file-scope __device__ array of
// kNoAllocScratchBytes (16 MiB) that every GPU loading this library holds
// until the process exits.  Host code cannot use the array's name as a device
// address; the first call on each device looks the address up with
// cudaGetSymbolAddress (make that first call before any stream capture) and
// later calls reuse it.  Every call shares the array and leaves its contents
// behind, but for the work counter, which is zero before and after each
// launch; calls that overlap on the GPU (different streams, no ordering) race
// on the array.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "kvd_internal.h"
#include "kvdecode.h"

namespace kvd {
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(16) << 20;
constexpr int kNoAllocMaxBatch = 1024;

static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocScratchBytes];

PFN_cuTensorMapEncodeTiled_v12000 encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// What a call needs to know of the current device, asked once per device:
// the address of the scratch array and the split pass's variants.
struct DeviceInfo {
    uint8_t* scratch = nullptr;
    int num_sms = 0;
    DecodeVariant var[2][2];   // [D == 128][GQA]
};

int device_info(int* device, const DeviceInfo** out)
{
    static std::mutex mu;
    static DeviceInfo info[64];
    auto err = [](const char* what, cudaError_t e) {
        set_last_error((std::string("decode_attention_noalloc: ") + what + ": " + cudaGetErrorString(e)).c_str());
        return KVC_ERR_CUDA;
    };
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return err("cudaGetDevice", e);
    std::lock_guard<std::mutex> lock(mu);
    DeviceInfo& d = info[dev];
    if (!d.scratch) {
        e = cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, dev);
        for (int i = 0; i < 4 && e == cudaSuccess; ++i) e = decode_variant_info(i & 2 ? 128 : 64, i & 1, &d.var[i >> 1][i & 1]);
        if (e != cudaSuccess) return err("cannot query the current device", e);
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return err("cudaGetSymbolAddress", e);
        d.scratch = static_cast<uint8_t*>(p);
    }
    *device = dev;
    *out = &d;
    return KVC_OK;
}

size_t round256(size_t x) { return (x + 255) & ~size_t(255); }

int fail(int code, const char* msg)
{
    set_last_error((std::string("decode_attention_noalloc: ") + msg).c_str());
    return code;
}

}  // namespace
}  // namespace kvd

using namespace kvd;

extern "C" KVC_API int decode_attention_noalloc(const void* k_pool, const void* v_pool, int64_t num_pages,
                                                int32_t num_q_heads, int32_t num_kv_heads, int32_t head_dim,
                                                int32_t batch, const int32_t* page_table, int32_t max_pages,
                                                const int32_t* lens, const void* q, void* out,
                                                float softmax_scale, int32_t* device_error, void* stream)
{
    if (!k_pool || !v_pool || !page_table || !lens || !q || !out) return fail(KVC_ERR_INVALID, "null argument");
    const uintptr_t al = reinterpret_cast<uintptr_t>(k_pool) | reinterpret_cast<uintptr_t>(v_pool) |
                         reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(out);
    if (al & 15u) return fail(KVC_ERR_INVALID, "k_pool, v_pool, q and out must be 16-byte aligned");
    if (num_q_heads < 1 || num_kv_heads < 1 || num_q_heads % num_kv_heads)
        return fail(KVC_ERR_INVALID, "num_q_heads must be a positive multiple of num_kv_heads");
    const int G = num_q_heads / num_kv_heads;
    if (G > kMaxGroup) return fail(KVC_ERR_UNSUPPORTED, "more than 8 query heads per KV head");
    if (head_dim != 64 && head_dim != 128) return fail(KVC_ERR_UNSUPPORTED, "head_dim must be 64 or 128");
    if (batch < 1 || batch > kNoAllocMaxBatch) return fail(KVC_ERR_INVALID, "batch must be in 1 .. 1024");
    if (num_pages < 1 || num_pages * num_kv_heads * kPageSize >= (int64_t)1 << 31)
        return fail(KVC_ERR_INVALID, "num_pages must be >= 1 with num_pages * num_kv_heads * 16 < 2^31");
    if (max_pages < 1) return fail(KVC_ERR_INVALID, "max_pages must be >= 1");
    if (!(softmax_scale <= 0.f) && !std::isfinite(softmax_scale))
        return fail(KVC_ERR_INVALID, "softmax_scale must be finite");
    int64_t total_pages = 0;
    for (int b = 0; b < batch; ++b) {
        if (lens[b] < 1 || (int64_t)lens[b] > (int64_t)max_pages * kPageSize)
            return fail(KVC_ERR_INVALID, "every length must be in 1 .. max_pages * 16");
        total_pages += (lens[b] + kPageSize - 1) / kPageSize;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    int dev = 0;
    const DeviceInfo* info = nullptr;
    if (int rc = device_info(&dev, &info)) return rc;
    const DecodeVariant& var = info->var[head_dim == 128][G > 1];
    const int num_sms = info->num_sms;
    uint8_t* const scratch = info->scratch;

    // Items: the library's usual target (about three per resident warp),
    // enlarged until a plan (an entry and its page ids per item) and the
    // partials fit the static scratch: the documented limit.
    const int64_t warps = (int64_t)num_sms * std::max(1, var.ctas_per_sm) * std::max(1, var.warps);
    const int64_t units = total_pages * num_kv_heads;
    const size_t partial = (size_t)num_kv_heads * G * (head_dim * sizeof(float) + sizeof(float2));   // per entry
    int64_t T = std::min<int64_t>(128, std::max<int64_t>(2, (units + 3 * warps - 1) / (3 * warps)));
    size_t need = 0;
    int max_np = 0;
    // T doubles, clamped to kMaxItemPages; the attempt at kMaxItemPages is the last.
    for (;; T = std::min<int64_t>(2 * T, kMaxItemPages)) {
        int64_t entries = 0, split_items = 0;   // only rows cut into several items keep partials
        int stride = 1;
        for (int b = 0; b < batch; ++b) {
            const int np = (lens[b] + kPageSize - 1) / kPageSize;
            const int nch = row_chunks(np, (int)T);
            entries += nch;
            if (nch > 1) split_items += nch;
            stride = std::max(stride, (np + nch - 1) / nch);
            max_np = std::max(max_np, np);
        }
        const size_t off_pages = round256((size_t)entries * sizeof(PlanEntry));
        const size_t off_o = round256(off_pages + (size_t)entries * stride * sizeof(int32_t));
        const size_t slots = (size_t)split_items * num_kv_heads;
        const size_t off_ml = round256(off_o + slots * G * head_dim * sizeof(float));
        const size_t off_rows = round256(off_ml + slots * G * sizeof(float2));
        need = round256(round256(off_rows + (size_t)batch * sizeof(int2)) + 3 * sizeof(uint32_t));
        if (need <= kNoAllocScratchBytes || T >= kMaxItemPages) break;
    }
    if (need > kNoAllocScratchBytes)
        return fail(KVC_ERR_UNSUPPORTED, ("the batch needs " + std::to_string(need) +
                                          " bytes of scratch; the static limit is 16 MiB").c_str());

    // One tensor map over both pools (one load per page), the lower one first,
    // where their distance is a whole number of 128-byte lines; else a map for
    // each.
    auto encode = encoder();
    if (!encode) return fail(KVC_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    CUtensorMap maps[2];
    const int64_t rows = num_pages * num_kv_heads * kPageSize;
    const int64_t apart = static_cast<const char*>(v_pool) - static_cast<const char*>(k_pool);
    int kv_map = 0;
    if (apart != 0 && apart % 128 == 0 && std::abs(apart) < (int64_t)1 << 40 &&
        encode_tile_map(reinterpret_cast<void*>(encode), &maps[0], const_cast<void*>(apart > 0 ? k_pool : v_pool), rows,
                        head_dim, std::abs(apart)) == CUDA_SUCCESS) {
        kv_map = apart > 0 ? 1 : 2;
        maps[1] = maps[0];
    }
    for (int kv = 0; kv < 2 && !kv_map; ++kv) {
        CUresult r = encode_tile_map(reinterpret_cast<void*>(encode), &maps[kv], const_cast<void*>(kv ? v_pool : k_pool),
                                     rows, head_dim, 0);
        if (r != CUDA_SUCCESS) return fail(KVC_ERR_INVALID, "cuTensorMapEncodeTiled rejected the pools");
    }

    const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / std::sqrt((float)head_dim);
    // The scratch: [work counter, error word], the merge table, the partials.
    const size_t off_rows = 256, off_part = round256(off_rows + (size_t)batch * sizeof(int2));
    DecodeParams p{};
    p.q = static_cast<const uint16_t*>(q);
    p.out = static_cast<uint16_t*>(out);
    p.page_table = page_table;
    p.rows_out = reinterpret_cast<int2*>(scratch + off_rows);
    p.rows = p.rows_out;
    p.rows_late = 1;
    p.batch = batch;
    p.queue = reinterpret_cast<uint32_t*>(scratch);
    p.err = device_error ? device_error : reinterpret_cast<int32_t*>(scratch) + 1;
    p.num_pages = num_pages;
    p.H_kv = num_kv_heads;
    p.H_q = num_q_heads;
    p.G = G;
    p.max_pages = max_pages;
    p.scale_log2 = scale * 1.4426950408889634f;
    p.kv_map = kv_map;
    p.early = 0;   // placed early, but what ran before may have written anything it reads
    p.num_sms = num_sms;

    const ClusterShape shape = cluster_shape(dev, head_dim, G > 1, num_kv_heads, batch, total_pages, max_np, true);
    if (shape.ctas && batch <= kLensRows) {
        LensTable lt;
        std::copy_n(lens, batch, lt.len);
        p.ring = shape.ring;
        if (cudaError_t e = launch_cluster(head_dim, G > 1, false, true, shape, maps[0], maps[1], p,
                                           &lt, st);
            e != cudaSuccess)
            return fail(KVC_ERR_CUDA, cudaGetErrorString(e));
        return KVC_OK;
    }

    // Rows in planning order, longest first.
    RowTable<kNoAllocMaxBatch> rt;
    rt.n = batch;
    for (int b = 0; b < batch; ++b) rt.row[b] = (uint16_t)b;
    std::stable_sort(rt.row, rt.row + batch, [&](uint16_t x, uint16_t y) { return lens[x] > lens[y]; });
    for (int i = 0; i < batch; ++i) rt.len[i] = lens[rt.row[i]];
    // The plan of a step of the cache (items per resident warp, graduated
    // sizes, items per row) where its partials fit, also with larger items,
    // else the one sized above (whose rows of one item come last and keep no
    // partial).
    int max_chunks = 1;
    int64_t split_end = 0;   // entries up to the last row of several items: those with partial slots
    auto cut = [&](int64_t size, int cap, bool graduated) {
        int32_t off = 0;
        split_end = 0;
        max_chunks = 1;
        for (int i = 0; i < batch; ++i) {
            const int np = (rt.len[i] + kPageSize - 1) / kPageSize;
            const int nch = row_chunks(np, graduated ? row_item_pages((int)size, i, batch) : (int)size, cap);
            rt.off[i] = off;
            off += nch;
            if (nch > 1) split_end = off;
            max_chunks = std::max(max_chunks, nch);
        }
        rt.off[batch] = off;
        return off_part + (size_t)split_end * partial + 512 <= kNoAllocScratchBytes;
    };
    const int64_t T_step = auto_item_pages(head_dim, G > 1, num_kv_heads, warps, batch, total_pages, max_np, false);
    auto cut_as_step = [&](int64_t size) {
        return cut(size, noalloc_chunk_cap(G > 1, num_kv_heads, warps, batch, total_pages, max_np, (int32_t)size), true);
    };
    if (!cut_as_step(T_step) && !cut_as_step(std::max(T, T_step)) && !cut(T, kChunkCap, false))
        return fail(KVC_ERR_UNSUPPORTED, "the batch does not fit the static scratch");
    const int32_t entries = rt.off[batch];
    p.part_o = reinterpret_cast<float*>(scratch + off_part);
    p.part_ml = reinterpret_cast<float2*>(
        scratch + round256(off_part + (size_t)split_end * num_kv_heads * G * head_dim * sizeof(float)));
    p.n_items = entries * num_kv_heads;
    const int64_t resident = (int64_t)num_sms * std::max(1, var.ctas_per_sm);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(resident, p.n_items));
    if (cudaError_t e = launch_decode_table(head_dim, G > 1, grid, maps[0], maps[1], p, rt, st); e != cudaSuccess)
        return fail(KVC_ERR_CUDA, cudaGetErrorString(e));
    if (max_chunks > 1) {
        const int split_regs = ((var.ctas_per_sm * var.warps + 3) / 4) * warp_register_allocation(var.regs);
        if (cudaError_t e = launch_merge(head_dim, true, max_chunks, num_sms, split_regs, p, st); e != cudaSuccess)
            return fail(KVC_ERR_CUDA, cudaGetErrorString(e));
    }
    return KVC_OK;
}

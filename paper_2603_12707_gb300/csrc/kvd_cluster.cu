// Decode attention for steps with few (sequence, KV head) units (sm_103a): a
// thread-block cluster per unit, no second pass.
//
// A unit's pages are cut evenly over all warps of its cluster (C CTAs of W
// warps).  Each warp streams its pages through its own ring of shared-memory
// stages and runs the same online softmax as the split pass
// (kvd_decode_kernel.cuh).  The warps' (o, m, l) then merge by log-sum-exp in
// two hops: within the CTA through shared memory, and across the cluster
// through distributed shared memory, where CTA r receives every CTA's dims
// [r D/C, (r+1) D/C) and writes them as bf16 output.
//
// What bounds it: such a layer holds a few MB, 1-2 us of HBM time, so the
// chain of dependent latencies per layer decides.  The split pass and merge
// pass pay two dependency hops (~1 us each) and two L2 round trips for the
// partials; this kernel pays one hop and one exchange over the cluster (sent
// with st.async, received on an mbarrier: 0.4 us less than a cluster
// barrier).  us per chained layer, split plan -> this: LLaVA heads, one
// request of 850 tokens (14 MB) 6.5 -> 4.3; Qwen heads, two of 2500 and 4400
// (14 MB) 6.9 -> 5.0; 4 requests of 100 tokens, 8/8 heads, d = 64: 4.6 -> 2.5.
#include <algorithm>
#include <atomic>

#include "kvd_decode_kernel.cuh"

namespace kvd {

namespace {

constexpr int kClusterMaxCtas = 8;   // the portable cluster size
constexpr int kClusterMaxWarps = 8;
// Pages a warp brings into L2 before the dependency wait, beyond its ring.
constexpr int kClusterL2Pages = 8;

template <int D, bool GQA>
struct ClusterGeo {
    static constexpr int kStage = Geo<D, GQA>::kStageBytes;
    static constexpr int kHeads = GQA ? kMaxGroup : 1;
    static constexpr int kRow = D + 4;                          // floats per head of a warp's staged o (bank spread)
    static constexpr int kRecv = kHeads * D * 4;                // this CTA's dims from every CTA of the cluster
    static constexpr int kRecvMl = kClusterMaxCtas * kHeads * 8;
    static constexpr int kWarpMl = kClusterMaxWarps * kHeads * 8;
    static_assert(kHeads * kRow * 4 <= kStage, "a warp's staged o fits one stage of its ring");
    static int smem(int warps, int ring)
    {
        return warps * ring * (kStage + 8) + kRecv + kRecvMl + kWarpMl + 8;
    }
};

// A warp's unnormalised o ([head][kRow] floats) and (m, l) per head to shared memory.
template <int D>
__device__ __forceinline__ void stage_partial(MhaCompute<D>& c, float* wo, float2* wml, int lane)
{
    constexpr int CH = MhaCompute<D>::CH;
    float o[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) f2_unpack(c.o2[k], o[2 * k], o[2 * k + 1]);
#pragma unroll
    for (int mask = CH; mask < 32; mask <<= 1)
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] += __shfl_xor_sync(0xffffffffu, o[k], mask);
    float l = c.l;
#pragma unroll
    for (int mask = 1; mask < 32; mask <<= 1) l += __shfl_xor_sync(0xffffffffu, l, mask);
    if (c.tsub == 0) {
        float4* dst = reinterpret_cast<float4*>(wo + c.c * 8);
        dst[0] = make_float4(o[0], o[1], o[2], o[3]);
        dst[1] = make_float4(o[4], o[5], o[6], o[7]);
    }
    if (lane == 0) wml[0] = make_float2(c.m, l);
}

template <int D>
__device__ __forceinline__ void stage_partial(GqaCompute<D>& c, float* wo, float2* wml, int lane)
{
    constexpr int ROW = ClusterGeo<D, true>::kRow;
    float l0 = c.l0, l1 = c.l1;
#pragma unroll
    for (int mask = 4; mask < 32; mask <<= 1) {
        l0 += __shfl_xor_sync(0xffffffffu, l0, mask);
        l1 += __shfl_xor_sync(0xffffffffu, l1, mask);
    }
    const int h0 = 2 * (lane & 3), h1 = h0 + 1, dlo = lane >> 2;
#pragma unroll
    for (int mt = 0; mt < GqaCompute<D>::KS; ++mt) {
        const int d0 = mt * 16 + dlo;
        wo[h0 * ROW + d0] = c.oacc[mt][0];
        wo[h1 * ROW + d0] = c.oacc[mt][1];
        wo[h0 * ROW + d0 + 8] = c.oacc[mt][2];
        wo[h1 * ROW + d0 + 8] = c.oacc[mt][3];
    }
    if (lane < 4) {
        wml[h0] = make_float2(c.m0, l0);
        wml[h1] = make_float2(c.m1, l1);
    }
}

// Weight of a partial with reference max m against M; a partial without
// tokens (m = -inf) weighs 0 even when M is -inf too.
__device__ __forceinline__ float lse_weight(float m, float M) { return m == -INFINITY ? 0.f : ex2(m - M); }

// Keep a value read from the kernel parameters in a register from here on:
// its first use would otherwise fetch the parameter line at the end of the
// layer's dependent chain.
template <class T>
__device__ __forceinline__ void hold(T*& v) { asm volatile("" : "+l"(v)); }
__device__ __forceinline__ void hold(int& v) { asm volatile("" : "+r"(v)); }

template <int D, bool GQA, bool FUSED, class Rows>
__global__ void __launch_bounds__(kClusterMaxWarps * 32, 1)
    cluster_kernel(const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv,
                   const DecodeParams p, const __grid_constant__ Rows rt)
{
    using Cg = ClusterGeo<D, GQA>;
    constexpr int STAGE = Cg::kStage;
    constexpr int TILE = STAGE / 2;
    // 128-byte swizzled stages need a 1024-byte aligned base; the kernel has no
    // static shared memory, so its dynamic part starts at that alignment.
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int W = blockDim.x >> 5, R = p.ring;
    const int C = (int)cluster_nctarank(), rank = (int)cluster_ctarank();
    // CTAs and warps of a unit are powers of two: shifts in place of divisions,
    // which cost the entry of a kernel this short.
    const int log_dc = 31 - __clz(D / C), log_cw = 31 - __clz(C * W);
    uint8_t* ring = smem + warp * R * STAGE;
    float* recv = reinterpret_cast<float*>(smem + W * R * STAGE);               // [C][G][D / C]
    float2* recv_ml = reinterpret_cast<float2*>(reinterpret_cast<uint8_t*>(recv) + Cg::kRecv);   // [C][heads]
    float2* warp_ml = recv_ml + kClusterMaxCtas * Cg::kHeads;                   // [W][heads]
    uint64_t* recv_bar = reinterpret_cast<uint64_t*>(warp_ml + kClusterMaxWarps * Cg::kHeads);
    uint64_t* bars = recv_bar + 1 + warp * R;
    const uint32_t ring_s = smem_addr(ring);
    int G = GQA ? p.G : 1;

    // The next launch may start at once, with this one still waiting: before
    // its own dependency wait it reads nothing that this launch or the chain
    // before it writes (but for slots that it replaces itself).  After
    // a step kernel both wait for that first.
    // A launch with the caller's tables waits before it reads those.
    const bool waited = Rows::kTable || p.early == 0;
    if constexpr (!Rows::kTable) {
        if (waited) griddep_wait();
        griddep_launch_dependents();
    }
    const int b = blockIdx.y, g = (int)blockIdx.x >> (31 - __clz(C));
    int2 row;   // (page-table row, tokens attended)
    if constexpr (Rows::kTable) row = make_int2(b, rt.len[b]);
    else row = p.rows[b];   // by the step kernel; no tokens: the row's step failed
    if (lane == 0) {
#pragma unroll 1
        for (int s = 0; s < R; ++s) mbar_init(smem_addr(&bars[s]), 1);
        if (warp == 0) mbar_init(smem_addr(recv_bar), 1);
        fence_mbar_init();
        if (warp == 0) {   // what the cluster sends this CTA: its dims and (M, L) of every CTA and head
            prefetch_tensormap(&tmk);
            if (!p.kv_map) prefetch_tensormap(&tmv);
            mbar_arrive_expect_tx(smem_addr(recv_bar), G * D * 4 + C * G * 8);
        }
    }
    __syncwarp();
    cluster_arrive();   // "ready to receive": waited for before the first write to another CTA
    const int len = row.y;
    const int np = (len + kPageSize - 1) / kPageSize;
    const int at = rank * W + warp, each = np >> log_cw, more = np & ((1 << log_cw) - 1);   // chunk_range
    const int first = at * each + min(at, more), n = each + (at < more ? 1 : 0);
    const bool has_last = n > 0 && first + n == np;
    const int32_t* pt_row = p.page_table + (int64_t)row.x * p.max_pages + first;
    auto load_window = [&](int w0) { return (w0 + lane < n) ? pt_row[w0 + lane] : 0; };
    if constexpr (Rows::kTable) {
        griddep_wait();
        griddep_launch_dependents();
    }
    int32_t pid_cur = load_window(0);
    int32_t pid_next = 0;
    const uint64_t policy = l2_policy_evict_first();
    auto load = [&](int32_t pid, int s) {   // page pid into stage s, by one lane
        if (pid < 0 || pid >= p.num_pages) {
            atomicOr(p.err, 1);
            pid = 0;
        }
        const uint32_t bar = smem_addr(&bars[s]);
        const uint32_t dst = ring_s + s * STAGE;
        const int32_t y = (pid * p.H_kv + g) * kPageSize;
        mbar_arrive_expect_tx(bar, STAGE);
        if (!Rows::kTable || p.kv_map) {
            tma_load_4d(dst, &tmk, 0, y, 0, 0, bar, policy);
        } else {
            tma_load_3d(dst, &tmk, 0, y, 0, bar, policy);
            tma_load_3d(dst + TILE, &tmv, 0, y, 0, bar, policy);
        }
    };
    auto issue = [&](int j, int s) {
        if ((j & 31) == 8 && j + 24 < n) pid_next = load_window(j + 24);
        if ((j & 31) == 0 && j > 0) pid_cur = pid_next;
        const int32_t pid = __shfl_sync(0xffffffffu, pid_cur, j & 31);
        if (lane == 0) load(pid, s);
    };
    const int pre = min(n, R);
    // lane i: page i into stage i (a row's last page only after the wait where
    // an append of the chain may be under way)
    const bool late_page = !FUSED && p.hold_last && has_last && n == pre;
    if (lane < pre - (late_page ? 1 : 0)) load(pid_cur, lane);
    // The pages past the ring into L2: when a stage is free again its next
    // page is an L2 round trip away.
    if (!Rows::kTable || p.kv_map) {
        const int end = min(min(n, 32), R + kClusterL2Pages);
        if (lane >= R && lane < end && pid_cur >= 0 && pid_cur < p.num_pages)
            tma_prefetch_l2_4d(&tmk, 0, (pid_cur * p.H_kv + g) * kPageSize, 0, 0);
    }
    __syncwarp();

    PlanEntry en{};
    en.b = b;
    en.len = len;
    float scale_log2 = p.scale_log2;
    uint16_t* out = p.out + ((int64_t)b * p.H_q + g * G) * D;
    hold(out);
    hold(G);
    if (!waited) griddep_wait();
    if (late_page && lane == pre - 1) load(pid_cur, lane);
    __syncwarp();
    using Comp = typename std::conditional<GQA, GqaCompute<D>, MhaCompute<D>>::type;
    Comp comp;
    comp.start(p, en, g, lane);
    uint4 new_kv = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (FUSED)
        if (has_last) new_kv = load_new_token<D>(p, en, g, lane);

    const int k_off = Rows::kTable && p.kv_map == 2 ? TILE : 0, v_off = TILE - k_off;   // K and V within a stage
    uint32_t phase = 0, pending = (1u << pre) - 1u;
    bool ok = true;
    // Wait for page j in stage s and put the new token into it if it is the row's last.
    auto arrived = [&](int j, int s) {
        const uint32_t bar = smem_addr(&bars[s]), parity = (phase >> s) & 1u;
        const bool w = mbar_try_wait_cluster(bar, parity) || mbar_wait_bounded_cluster(bar, parity, kWaitLimitNs);
        if (!__all_sync(0xffffffffu, w)) return false;
        phase ^= 1u << s;
        pending &= ~(1u << s);
        if constexpr (FUSED) {
            if (has_last && j == n - 1) {   // the page-id window has not moved past this page
                const int32_t pid = __shfl_sync(0xffffffffu, pid_cur, j & 31);
                put_new_token<D>(p, en, g, pid, new_kv, ring + s * STAGE + k_off, ring + s * STAGE + v_off, lane);
            }
        }
        return true;
    };
    auto refill = [&](int j, int s) {
        if (j + R < n) {
            issue(j + R, s);
            pending |= 1u << s;
        }
    };
    auto after = [&](int s) { return s + 1 == R ? 0 : s + 1; };
    auto tokens = [&](int j) { return min(kPageSize, len - (first + j) * kPageSize); };
#pragma unroll 1
    for (int j = 0, s = 0; ok && j < n; ++j) {
        ok = arrived(j, s);
        if (!ok) break;
        if (GQA && j == 0) comp.ready(lane);
        uint8_t* sk = ring + s * STAGE;
        const uint32_t a = ring_s + s * STAGE;
        comp.page(sk + k_off, sk + v_off, a + k_off, a + v_off, tokens(j), scale_log2, lane);
        __syncwarp();
        refill(j, s);
        s = after(s);
    }
    if (!ok) {   // let the loads in flight land: their stages are about to be reused
        if (lane == 0) atomicOr(p.err, 2);
#pragma unroll 1
        for (int i = 0; i < R; ++i)
            if (pending & (1u << i)) mbar_wait_bounded_cluster(smem_addr(&bars[i]), (phase >> i) & 1u, kWaitLimitNs);
    }
    __syncwarp();

    // Hop 1: the CTA's warps, four dims of a head at a time; the result goes
    // to the CTA of the cluster that owns those dims.
    stage_partial<D>(comp, reinterpret_cast<float*>(ring), warp_ml + warp * Cg::kHeads, lane);
    __syncthreads();
    cluster_wait();
    const uint32_t bar_s = smem_addr(recv_bar);
#pragma unroll 1
    for (int i = threadIdx.x; i < G * (D / 4); i += blockDim.x) {
        const int h = i / (D / 4), d0 = (i % (D / 4)) * 4;
        // (fixed bounds, so that every load goes out before the first use)
        float2 ml[kClusterMaxWarps];
        float4 v[kClusterMaxWarps];
#pragma unroll
        for (int w = 0; w < kClusterMaxWarps; ++w) {
            ml[w] = make_float2(-INFINITY, 0.f);
            v[w] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (w < W) {
                ml[w] = warp_ml[w * Cg::kHeads + h];
                v[w] = *reinterpret_cast<const float4*>(smem + w * R * STAGE + (h * Cg::kRow + d0) * 4);
            }
        }
        float M = ml[0].x;
#pragma unroll
        for (int w = 1; w < kClusterMaxWarps; ++w) M = fmaxf(M, ml[w].x);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        float L = 0.f;
#pragma unroll
        for (int w = 0; w < kClusterMaxWarps; ++w) {
            const float e = lse_weight(ml[w].x, M);
            a.x = fmaf(e, v[w].x, a.x);
            a.y = fmaf(e, v[w].y, a.y);
            a.z = fmaf(e, v[w].z, a.z);
            a.w = fmaf(e, v[w].w, a.w);
            L = fmaf(e, ml[w].y, L);
        }
        const uint32_t dst = (uint32_t)(d0 >> log_dc);
        const int dd = d0 & ((1 << log_dc) - 1);
        const uint32_t bar = cluster_map(bar_s, dst);
        cluster_store_async4(cluster_map(smem_addr(recv + ((rank * G + h) << log_dc) + dd), dst), a, bar);
        // every CTA gets (M, L) of each head, from the thread of its first dims
        if (dd == 0) cluster_store_async2(cluster_map(smem_addr(recv_ml + rank * Cg::kHeads + h), dst), M, L, bar);
    }
    if (!mbar_try_wait_cluster(bar_s, 0) && !mbar_wait_bounded_cluster(bar_s, 0, kWaitLimitNs)) {
        // What is still on its way needs this CTA's shared memory: leave with
        // the last of the cluster (every wait in here is bounded).
        atomicOr(p.err, 2);
        cluster_leave();
        return;
    }
    // Hop 2: this CTA's dims over the cluster, two at a time.
    if (np == 0) return;   // a row whose step failed: its output is left alone
#pragma unroll 1
    for (int i = threadIdx.x; i < G << (log_dc - 1); i += blockDim.x) {
        const int h = i >> (log_dc - 1), d0 = (i & ((1 << (log_dc - 1)) - 1)) * 2;
        float2 ml[kClusterMaxCtas], v[kClusterMaxCtas];
#pragma unroll
        for (int c = 0; c < kClusterMaxCtas; ++c) {
            ml[c] = make_float2(-INFINITY, 0.f);
            v[c] = make_float2(0.f, 0.f);
            if (c < C) {
                ml[c] = recv_ml[c * Cg::kHeads + h];
                v[c] = *reinterpret_cast<const float2*>(recv + ((c * G + h) << log_dc) + d0);
            }
        }
        float M = ml[0].x;
#pragma unroll
        for (int c = 1; c < kClusterMaxCtas; ++c) M = fmaxf(M, ml[c].x);
        float L = 0.f, x = 0.f, y = 0.f;
#pragma unroll
        for (int c = 0; c < kClusterMaxCtas; ++c) {
            const float e = lse_weight(ml[c].x, M);
            L = fmaf(e, ml[c].y, L);
            x = fmaf(e, v[c].x, x);
            y = fmaf(e, v[c].y, y);
        }
        const float inv = 1.f / L;
        *reinterpret_cast<uint32_t*>(out + h * D + (rank << log_dc) + d0) = pack_bf16(x * inv, y * inv);
    }
}

template <int D, bool GQA, bool FUSED, class Rows = PlanRows>
cudaError_t prepare_cluster()
{
    static OncePerDevice once;
    return once.set_attribute(
        cluster_kernel<D, GQA, FUSED, Rows>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        ClusterGeo<D, GQA>::smem(kClusterMaxWarps, kClusterRingBytes / ClusterGeo<D, GQA>::kStage));
}

template <int D, bool GQA, bool FUSED, class Rows>
cudaError_t launch_variant(bool pdl, const ClusterShape& sh, const CUtensorMap& tk, const CUtensorMap& tv,
                           const DecodeParams& p, const Rows& rows, cudaStream_t st)
{
    if (cudaError_t e = prepare_cluster<D, GQA, FUSED, Rows>(); e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.H_kv * sh.ctas), (unsigned)p.batch);
    cfg.blockDim = dim3((unsigned)(sh.warps * 32));
    cfg.dynamicSmemBytes = (size_t)ClusterGeo<D, GQA>::smem(sh.warps, sh.ring);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)sh.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, cluster_kernel<D, GQA, FUSED, Rows>, tk, tv, p, rows);
}

template <int D, bool GQA>
cudaError_t launch_shape(bool fused, bool pdl, const ClusterShape& sh, const CUtensorMap& tk,
                         const CUtensorMap& tv, const DecodeParams& p, const LensTable* lens, cudaStream_t st)
{
    if (lens) return launch_variant<D, GQA, false>(pdl, sh, tk, tv, p, *lens, st);
    return fused ? launch_variant<D, GQA, true>(pdl, sh, tk, tv, p, PlanRows{}, st)
                 : launch_variant<D, GQA, false>(pdl, sh, tk, tv, p, PlanRows{}, st);
}

template <int D, bool GQA>
cudaError_t resident_shape(const ClusterShape& sh, int* clusters)
{
    if (cudaError_t e = prepare_cluster<D, GQA, true>(); e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sh.ctas);
    cfg.blockDim = dim3((unsigned)(sh.warps * 32));
    cfg.dynamicSmemBytes = (size_t)ClusterGeo<D, GQA>::smem(sh.warps, sh.ring);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)sh.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, cluster_kernel<D, GQA, true, PlanRows>, &cfg);
}

// Clusters of a shape that the GPU holds at once, asked once per device and
// shape, for the fused kernel: of a head shape's variants it takes the most
// registers (108 / 126 / 132 / 164 for d = 64 MHA, GQA, d = 128 MHA, GQA; the
// others 92 / 114 / 119 / 154), so the others fit as well.
int resident_clusters(int device, int D, bool gqa, const ClusterShape& sh)
{
    static std::atomic<int> known[64][2][2][kClusterMaxCtas + 1][kClusterMaxWarps / 4 + 1][kClusterRingBytes / 4096 + 1];
    if (device < 0 || device >= 64) return 0;
    std::atomic<int>& at = known[device][D == 128][gqa][sh.ctas][sh.warps / 4][sh.ring];
    int n = at.load(std::memory_order_relaxed) - 1;   // 0: not asked yet
    if (n < 0) {
        const cudaError_t e =
            D == 128 ? (gqa ? resident_shape<128, true>(sh, &n) : resident_shape<128, false>(sh, &n))
                     : (gqa ? resident_shape<64, true>(sh, &n) : resident_shape<64, false>(sh, &n));
        if (e != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        at.store(n + 1, std::memory_order_relaxed);
    }
    return n;
}

}  // namespace

cudaError_t launch_cluster(int D, bool gqa, bool fused, bool pdl, const ClusterShape& sh,
                           const CUtensorMap& tk, const CUtensorMap& tv, const DecodeParams& p,
                           const LensTable* lens, cudaStream_t st)
{
    if (D == 128) return gqa ? launch_shape<128, true>(fused, pdl, sh, tk, tv, p, lens, st)
                             : launch_shape<128, false>(fused, pdl, sh, tk, tv, p, lens, st);
    if (D == 64) return gqa ? launch_shape<64, true>(fused, pdl, sh, tk, tv, p, lens, st)
                            : launch_shape<64, false>(fused, pdl, sh, tk, tv, p, lens, st);
    return cudaErrorInvalidValue;
}

ClusterShape cluster_shape(int device, int D, bool gqa, int num_kv_heads, int64_t batch, int64_t pages,
                           int64_t max_pages, bool spread, int64_t limit)
{
    return pick_cluster_shape(resident_clusters, device, D, gqa, num_kv_heads, batch, pages, max_pages, spread, limit);
}

}  // namespace kvd

// Launch side of the split pass: kernel attributes, occupancy, register
// counts and the (programmatic dependent) launches of decode_kernel
// (kvd_decode_kernel.cuh).
#include <algorithm>

#include "kvd_decode_kernel.cuh"

namespace kvd {

namespace {

template <int D, bool GQA, bool FUSED, class Rows = PlanRows>
cudaError_t prepare_variant()
{
    static OncePerDevice once;
    return once.set_attribute(decode_kernel<D, GQA, FUSED, Rows>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              Geo<D, GQA>::kSmem);
}

template <int D, bool GQA>
cudaError_t variant_info(DecodeVariant* v)
{
    cudaError_t e = prepare_variant<D, GQA, false>();
    if (e == cudaSuccess) e = prepare_variant<D, GQA, true>();
    if (e != cudaSuccess) return e;
    v->warps = kWarps;
    v->smem_bytes = Geo<D, GQA>::kSmem;
    cudaFuncAttributes a0, a1;
    e = cudaFuncGetAttributes(&a0, decode_kernel<D, GQA, false, PlanRows>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a1, decode_kernel<D, GQA, true, PlanRows>);
    if (e != cudaSuccess) return e;
    v->regs = std::max(a0.numRegs, a1.numRegs);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v->ctas_per_sm, decode_kernel<D, GQA, false, PlanRows>,
                                                         kWarps * 32, Geo<D, GQA>::kSmem);
}

template <int D, bool GQA>
cudaError_t launch_variant(bool fused, bool pdl, int grid, const CUtensorMap& tk, const CUtensorMap& tv,
                           const DecodeParams& p, cudaStream_t st)
{
    cudaError_t e = fused ? prepare_variant<D, GQA, true>() : prepare_variant<D, GQA, false>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kWarps * 32);
    cfg.dynamicSmemBytes = Geo<D, GQA>::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return fused ? cudaLaunchKernelEx(&cfg, decode_kernel<D, GQA, true, PlanRows>, tk, tv, p, PlanRows{})
                 : cudaLaunchKernelEx(&cfg, decode_kernel<D, GQA, false, PlanRows>, tk, tv, p, PlanRows{});
}

// Batches of up to 64 rows pass a table of 0.6 KB, larger ones 10 KB.
template <int D, bool GQA, int N>
cudaError_t launch_table(int grid, const CUtensorMap& tk, const CUtensorMap& tv, const DecodeParams& p,
                         const RowTable<1024>& all, cudaStream_t st)
{
    using Rows = RowTable<N>;
    if (cudaError_t e = prepare_variant<D, GQA, false, Rows>(); e != cudaSuccess) return e;
    Rows rows;
    rows.n = all.n;
    std::copy_n(all.row, all.n, rows.row);
    std::copy_n(all.len, all.n, rows.len);
    std::copy_n(all.off, all.n + 1, rows.off);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kWarps * 32);
    cfg.dynamicSmemBytes = Geo<D, GQA>::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, decode_kernel<D, GQA, false, Rows>, tk, tv, p, rows);
}

template <int D, bool GQA>
cudaError_t launch_table_size(int grid, const CUtensorMap& tk, const CUtensorMap& tv, const DecodeParams& p,
                              const RowTable<1024>& rows, cudaStream_t st)
{
    return rows.n <= kTableRows[0] ? launch_table<D, GQA, kTableRows[0]>(grid, tk, tv, p, rows, st)
                                   : launch_table<D, GQA, kTableRows[1]>(grid, tk, tv, p, rows, st);
}

}  // namespace

cudaError_t launch_decode_table(int D, bool gqa, int grid, const CUtensorMap& tk, const CUtensorMap& tv,
                                const DecodeParams& p, const RowTable<1024>& rows, cudaStream_t st)
{
    if (D == 128) return gqa ? launch_table_size<128, true>(grid, tk, tv, p, rows, st)
                             : launch_table_size<128, false>(grid, tk, tv, p, rows, st);
    if (D == 64) return gqa ? launch_table_size<64, true>(grid, tk, tv, p, rows, st)
                            : launch_table_size<64, false>(grid, tk, tv, p, rows, st);
    return cudaErrorInvalidValue;
}

cudaError_t decode_variant_info(int D, bool gqa, DecodeVariant* v)
{
    if (D == 128) return gqa ? variant_info<128, true>(v) : variant_info<128, false>(v);
    if (D == 64) return gqa ? variant_info<64, true>(v) : variant_info<64, false>(v);
    return cudaErrorInvalidValue;
}

cudaError_t launch_decode(int D, bool gqa, bool fused, bool pdl, int grid, const CUtensorMap& tk,
                          const CUtensorMap& tv, const DecodeParams& p, cudaStream_t st)
{
    if (D == 128) return gqa ? launch_variant<128, true>(fused, pdl, grid, tk, tv, p, st)
                             : launch_variant<128, false>(fused, pdl, grid, tk, tv, p, st);
    if (D == 64) return gqa ? launch_variant<64, true>(fused, pdl, grid, tk, tv, p, st)
                            : launch_variant<64, false>(fused, pdl, grid, tk, tv, p, st);
    return cudaErrorInvalidValue;
}

}  // namespace kvd

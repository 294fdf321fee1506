// The one-kernel compressor's instances and their launch.
#include "enec_fused.cuh"
#include "enec_launch.cuh"

namespace enec {

template <int DT>
static enec_status launch_fused_dt(FusedJob job, uint32_t nblocks, int sms, bool& attr_set, int* d_status, cudaStream_t stream) {
    using Shape = FusedShape<DT>;
    if (!attr_set) {
        if (cudaFuncSetAttribute(enec_fused_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Shape::kBytes)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        attr_set = true;
    }
    uint32_t grid = uint32_t(sms) * Shape::kCtasPerSm;
    if (grid > kMaxFusedGrid) grid = kMaxFusedGrid;
    if (grid > nblocks) grid = nblocks;
    // Up to 44 MB the sample is the whole tensor: its second reading comes from L2, and the parameters need no check. Beyond,
    // one block per SM is sampled. bf16, sampled against whole: 1024 blocks 24.6 / 25.1 us, 1400 29.0 / 30.8, 1600 30.3 / 33.5, 2000
    // 35.0 / 40.1; the line lies above the crossing because the whole count spares tensors with outliers the wasted sample, and
    // those with a few exact zeros, which a sample misses, the second pass (1024 blocks 53 / 29 us). What a misled sample costs
    // beyond it, one zero early / in the middle / late in the tensor, against the split form (for which the place is the same)
    // and against a sample that was right: bf16 1409 blocks 43 / 46 / 51 us against 41 and 28, 3584 blocks 91 / 99 / 111 against 89
    // and 52, 32064 blocks 490 / 594 / 695 against 679 and 354; fp32 712 blocks 51 against 38 and 29, 3584 blocks 150 / 169 / 183
    // against 167 and 87. A whole tensor with another (b, m) than its sample costs what a late zero does.
    job.sample = uint64_t(nblocks) * kBlockElems * elem_bytes(DT) <= (uint64_t(44) << 20) ? nblocks : uint32_t(sms);
    if (launch_pdl(enec_fused_kernel<DT>, grid, kFusedThreads, Shape::kBytes, stream, job, d_status) != cudaSuccess) return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ENEC_OK;
}

enec_status launch_fused(int dt, const FusedJob& job, uint32_t nblocks, int sms, bool* attr_set, int* d_status, cudaStream_t stream) {
    return dt == ENEC_BF16   ? launch_fused_dt<ENEC_BF16>(job, nblocks, sms, attr_set[dt], d_status, stream)
           : dt == ENEC_FP16 ? launch_fused_dt<ENEC_FP16>(job, nblocks, sms, attr_set[dt], d_status, stream)
                             : launch_fused_dt<ENEC_FP32>(job, nblocks, sms, attr_set[dt], d_status, stream);
}

}  // namespace enec

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
    // one block per SM is sampled. Sampled against whole: bf16 1024 blocks 23.3 / 21.1 us, 1400 26.7 / 25.5, 1600 28.0 / 28.1, 2000
    // 31.6 / 35.6; fp16 1400 blocks 27.2 / 26.6, 1600 28.5 / 30.7; fp32 704 blocks 28.5 / 27.9, 800 28.7 / 30.3. They cross at 50 MB of
    // bf16, 45 of fp16, 48 of fp32, so the line could lie a little higher; the whole count also spares tensors with outliers the
    // wasted sample, and those with a few exact zeros, which a sample misses, the second pass (1024 blocks 40.3 / 21.9 us). What a misled
    // sample costs beyond the line, one zero early / in the middle / late in the tensor, against the split form (for which the place is
    // the same) and against a sample that was right: bf16 1409 blocks 40 / 42 / 47 us against 39 and 27, 3584 blocks 83 / 89 / 100
    // against 89 and 49, 32064 blocks 459 / 534 / 617 against 682 and 313; fp32 712 blocks 50 against 42 and 28, 3584 blocks 144 / 161 /
    // 177 against 167 and 86. A whole tensor with another (b, m) than its sample is packed twice: where the rest is narrower, 3584
    // blocks of bf16 116 against 86. Where it is wider, nearly all groups are in the first pass, their records do not fit the place in
    // which they wait, and every block waits for its offset: 164 against 85, 32064 blocks 1485 against 607.
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

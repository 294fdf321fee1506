// The list compressor's instances and their launch.
#include "enec_fused_list.cuh"
#include "enec_launch.cuh"

namespace enec {

template <int DT>
static enec_status launch_fused_list_dt(const FusedList& list, uint32_t tickets, int sms, bool& attr_set, int* d_status, cudaStream_t stream) {
    using Shape = FusedShape<DT>;
    if (!attr_set) {
        if (cudaFuncSetAttribute(enec_fused_list_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(Shape::kBytes)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        attr_set = true;
    }
    uint32_t grid = uint32_t(sms) * Shape::kCtasPerSm;
    if (grid > tickets) grid = tickets;
    if (launch_pdl(enec_fused_list_kernel<DT>, grid, kFusedThreads, Shape::kBytes, stream, list, d_status) != cudaSuccess) return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ENEC_OK;
}

enec_status launch_fused_list(int dt, const FusedList& list, uint32_t tickets, int sms, bool* attr_set, int* d_status, cudaStream_t stream) {
    return dt == ENEC_BF16   ? launch_fused_list_dt<ENEC_BF16>(list, tickets, sms, attr_set[dt], d_status, stream)
           : dt == ENEC_FP16 ? launch_fused_list_dt<ENEC_FP16>(list, tickets, sms, attr_set[dt], d_status, stream)
                             : launch_fused_list_dt<ENEC_FP32>(list, tickets, sms, attr_set[dt], d_status, stream);
}

}  // namespace enec

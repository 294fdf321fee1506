// C-ABI entry points of libenec (see include/enec.h). Host-side validation and kernel launches only.
#include <atomic>
#include <map>
#include <mutex>
#include <utility>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "enec_decode.cuh"
#include "enec_encode.cuh"
#include "enec_blockwise.cuh"
#include "enec_fused_list.cuh"
#include "enec_launch.cuh"

namespace enec {

std::atomic<uint64_t> g_launches{0};

struct DeviceInfo {
    int sms = 0;
    bool hist_attr_set[3] = {false, false, false};
    bool encode_attr_set[3] = {false, false, false};
    bool blockwise_attr_set[3] = {false, false, false};
    bool split_attr_set[3] = {false, false, false};
    bool fused_attr_set[3] = {false, false, false};
    bool fused_list_attr_set[3] = {false, false, false};
};

// Per-device facts, for device ordinals below kMaxDevices (null beyond: the caller fails with ENEC_ERR_CUDA).
static DeviceInfo* device_info(int dev) {
    static std::mutex mu;
    static DeviceInfo infos[kMaxDevices];
    if (dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    DeviceInfo& d = infos[dev];
    if (d.sms == 0) cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
    return &d;
}

std::atomic<uint64_t> g_allocations{0};  // cudaMalloc calls the library has made (enec_allocation_count)

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Device scratch, one area per (device, stream, purpose): for the compressor control words and one state
// word per block, for a batched call the tensor descriptors. Grown when a larger request arrives;
// outgrown areas are kept until exit because work that uses them may still be queued.
struct ScratchArea {
    uint8_t* ptr = nullptr;
    size_t bytes = 0;
    uint64_t blocks = 0;      // one-kernel compressor: blocks the area is laid out for
    uint32_t supers[2] = {0, 0};  // one-kernel compressor: first-level sums in use in either set
    uint32_t epoch = 0;       // compressor areas: number of the last call
    bool needs_clear = true;  // compressor areas: fresh memory, a wrapped epoch or a launch that failed
};

enum ScratchKind { kScratchCompress = 0, kScratchBatch = 1, kScratchCompressBatch = 2, kScratchBlockwise = 3, kScratchDecodeTicket = 4, kScratchFused = 5 };

static std::mutex g_scratch_mu;
static ScratchArea& scratch_area(int dev, cudaStream_t stream, ScratchKind kind) {
    static std::map<std::pair<std::pair<int, int>, cudaStream_t>, ScratchArea> areas;
    return areas[std::make_pair(std::make_pair(dev, int(kind)), stream)];
}

static enec_status grow(ScratchArea& a, size_t need) {
    if (a.bytes >= need) return ENEC_OK;
    size_t bytes = a.bytes ? a.bytes : size_t(64) << 10;
    while (bytes < need) bytes *= 2;
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) return ENEC_ERR_CUDA;
    g_allocations.fetch_add(1, std::memory_order_relaxed);
    a.ptr = static_cast<uint8_t*>(p);
    a.bytes = bytes;
    a.needs_clear = true;
    return ENEC_OK;
}

static enec_status get_scratch(int dev, cudaStream_t stream, ScratchKind kind, size_t need, uint8_t** out) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchArea& a = scratch_area(dev, stream, kind);
    const enec_status st = grow(a, need);
    *out = a.ptr;
    return st;
}

// Scratch of one compress call and the call's number on it. The area is cleared (on `stream`) only when it
// is new, when the numbers have run out or after a call on it failed to launch; otherwise the kernels keep
// it usable from call to call (see EncodeControl).
static enec_status lease_compress_scratch(int dev, cudaStream_t stream, size_t need, uint8_t** out, uint32_t* epoch) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchArea& a = scratch_area(dev, stream, kScratchCompress);
    const enec_status st = grow(a, need);
    if (st != ENEC_OK) return st;
    if (a.needs_clear || a.epoch >= kEpochMax) {
        if (cudaMemsetAsync(a.ptr, 0, a.bytes, stream) != cudaSuccess) return ENEC_ERR_CUDA;
        a.needs_clear = false;
        a.epoch = 0;
    }
    *out = a.ptr;
    *epoch = ++a.epoch;
    return ENEC_OK;
}

// Scratch of the one-kernel compressor (see FusedControl), laid out for `blocks` blocks:
// [two control sets | two sets of first-level sums for two passes | a state word per block].
static size_t fused_scratch_bytes(uint64_t blocks) {
    return 2 * kFusedControlBytes + (4 * (blocks / kSuperBlocks) + blocks) * sizeof(unsigned long long);
}
static enec_status lease_fused_scratch(int dev, cudaStream_t stream, uint32_t nblocks, FusedJob& job) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchArea& a = scratch_area(dev, stream, kScratchFused);
    uint64_t blocks = a.blocks ? a.blocks : 4096;
    while (blocks < nblocks) blocks *= 2;
    const enec_status st = grow(a, fused_scratch_bytes(blocks));
    if (st != ENEC_OK) return st;
    if (blocks != a.blocks) {   // another layout
        a.blocks = blocks;
        a.needs_clear = true;
    }
    if (a.needs_clear || a.epoch > 0xFFFFFFF0u) {
        if (cudaMemsetAsync(a.ptr, 0, a.bytes, stream) != cudaSuccess) return ENEC_ERR_CUDA;
        a.needs_clear = false;
        a.epoch = 0;
        a.supers[0] = a.supers[1] = 0;
    }
    a.epoch += 2;  // one for each pass of the call
    const uint32_t set = (a.epoch >> 1) & 1, other = set ^ 1;
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(a.ptr + 2 * kFusedControlBytes);
    job.super_stride = uint32_t(blocks / kSuperBlocks);
    job.ctl = reinterpret_cast<FusedControl*>(a.ptr + set * kFusedControlBytes);
    job.ctl_next = reinterpret_cast<FusedControl*>(a.ptr + other * kFusedControlBytes);
    job.super = sums + size_t(set) * 2 * job.super_stride;
    job.super_next = sums + size_t(other) * 2 * job.super_stride;
    job.clear_supers = a.supers[other];
    job.state = sums + size_t(4) * job.super_stride;
    job.epoch = a.epoch;
    a.supers[other] = 0;
    a.supers[set] = (nblocks + kSuperBlocks - 1) / kSuperBlocks;
    return ENEC_OK;
}

static void mark_scratch_unclean(int dev, cudaStream_t stream, ScratchKind kind) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    scratch_area(dev, stream, kind).needs_clear = true;
}

static void mark_compress_scratch_unclean(int dev, cudaStream_t stream) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    scratch_area(dev, stream, kScratchCompress).needs_clear = true;
}

// The job's pointers into a scratch area for call number `epoch`.
static void place_job(EncodeJob& job, uint8_t* scratch, uint32_t epoch) {
    job.ctl = reinterpret_cast<EncodeControl*>(scratch + (epoch & 1) * kControlSlotBytes);
    job.ctl_next = reinterpret_cast<EncodeControl*>(scratch + ((epoch & 1) ^ 1) * kControlSlotBytes);
    job.state = reinterpret_cast<unsigned long long*>(scratch + kControlBytes);
    job.epoch = epoch;
}

// enec_compress takes the one-kernel form (enec_fused.cuh) for every size: none is known where the split form (histogram, pack
// kernel, then the kernel that places the records) is the faster one. That one is kept to measure and test against: for tensors of
// ENEC_SPLIT_MIN_BLOCKS .. ENEC_SPLIT_MAX_BLOCKS - 1 blocks, both from the environment and read once; without the first there is
// no such size. Given parameters always take the one-kernel form. One kernel against histogram and look-back
// kernel (as enec_compress_noalloc runs them, behind a memset) and against the split form: 4096 values 5.6 us against 12.9 and 27.4,
// 256 blocks 12.6 / 20.4 / 21.2, 1024 blocks 21.2 / 31.1 / 31.2, 3584 blocks 48.9 / 79.1 / 84.8, 32064 blocks 313 / 559 / 603 (bf16, in
// a stream). Where its sample misleads the one-kernel form it can be the slower one: see enec_fused.cu.
static uint32_t env_blocks(const char* name, uint32_t fallback) {
    const char* e = getenv(name);
    return e && *e ? uint32_t(strtoul(e, nullptr, 10)) : fallback;
}
static bool in_split_range(uint32_t nblocks) {
    static const uint32_t min_blocks = env_blocks("ENEC_SPLIT_MIN_BLOCKS", 0xFFFFFFFFu);
    static const uint32_t max_blocks = env_blocks("ENEC_SPLIT_MAX_BLOCKS", 0xFFFFFFFFu);
    return nblocks >= min_blocks && nblocks < max_blocks;
}

template <int DT>
static enec_status launch_split(const EncodeJob& job, uint32_t nblocks, int* d_status, DeviceInfo& info,
                                cudaStream_t stream) {
    if (!info.split_attr_set[DT]) {
        if (cudaFuncSetAttribute(enec_pack_tensor_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(kPackSmemBytes)) != cudaSuccess ||
            cudaFuncSetAttribute(enec_place_records_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(kPlaceSmemBytes)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        info.split_attr_set[DT] = true;
    }
    uint32_t grid = uint32_t(info.sms) * 4;
    if (grid > nblocks) grid = nblocks;
    if (launch_pdl(enec_pack_tensor_kernel<DT>, grid, kPackThreads, kPackSmemBytes, stream, job, d_status) != cudaSuccess)
        return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    grid = uint32_t(info.sms) * 2;
    if (grid > nblocks) grid = nblocks;
    if (grid > kPlaceMaxCtas) grid = kPlaceMaxCtas;
    if (launch_pdl(enec_place_records_kernel<DT>, grid, kPlaceThreads, kPlaceSmemBytes, stream, job, d_status) != cudaSuccess)
        return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ENEC_OK;
}

template <int DT>
static enec_status launch_encode(const EncodeJob& job, uint32_t nblocks, int* d_status, DeviceInfo& info, cudaStream_t stream,
                                 bool split = false) {
    const uint32_t smem = HistShape<DT>::kBytes;
    if (!info.hist_attr_set[DT]) {
        if (cudaFuncSetAttribute(enec_histogram_kernel<DT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(smem)) != cudaSuccess ||
            cudaFuncSetAttribute(enec_histogram_kernel<DT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(smem)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        info.hist_attr_set[DT] = true;
    }
    const uint64_t chunks = (job.count * uint64_t(elem_bytes(DT))) >> 4;  // 16-byte loads
    uint64_t hist_grid = (chunks + kHistThreads - 1) / kHistThreads;
    if (hist_grid > uint64_t(info.sms) * 3) hist_grid = uint64_t(info.sms) * 3;
    if (hist_grid == 0) hist_grid = 1;
    const cudaError_t herr =
        job.ranked ? launch_pdl(enec_histogram_kernel<DT, true>, uint32_t(hist_grid), kHistThreads, smem, stream, job.in,
                                job.count, job.ctl)
                   : launch_pdl(enec_histogram_kernel<DT, false>, uint32_t(hist_grid), kHistThreads, smem, stream, job.in,
                                job.count, job.ctl);
    if (herr != cudaSuccess) return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (split) return launch_split<DT>(job, nblocks, d_status, info, stream);
    if (!info.encode_attr_set[DT]) {
        if (cudaFuncSetAttribute(enec_encode_kernel<DT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(EncodeSmem<DT>::kBytes)) != cudaSuccess ||
            cudaFuncSetAttribute(enec_encode_kernel<DT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(EncodeSmem<DT>::kBytes)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        info.encode_attr_set[DT] = true;
    }
    uint32_t grid = uint32_t(info.sms) * 4;  // four resident CTAs per SM, each takes block after block
    if (grid > nblocks) grid = nblocks;
    const cudaError_t err =
        job.ranked ? launch_pdl(enec_encode_kernel<DT, true>, grid, kEncodeThreads, EncodeSmem<DT>::kBytes, stream,
                                job, d_status)
                   : launch_pdl(enec_encode_kernel<DT, false>, grid, kEncodeThreads, EncodeSmem<DT>::kBytes, stream,
                                job, d_status);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return err == cudaSuccess ? ENEC_OK : ENEC_ERR_CUDA;
}

static enec_status compress_common(const void* d_in, enec_dtype dt, size_t count, bool with_params, int b, int n,
                                   int m, void* d_out, size_t out_capacity, size_t* d_out_size, int* d_status,
                                   cudaStream_t stream, bool ranked = false) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if ((!d_in && count) || !d_out || (uint64_t(count) >> 36) || !aligned16(d_in) || !aligned16(d_out) ||
        (reinterpret_cast<uintptr_t>(d_out_size) & 7))
        return ENEC_ERR_INVALID_ARG;
    const int E = exp_bits(dt);
    if (with_params && (n < 1 || n > E || m < 1 || m > n || b < 0 || b >= (1 << E))) return ENEC_ERR_INVALID_ARG;
    if (out_capacity < (ranked ? enec_max_compressed_size_ranked(dt, count) : enec_max_compressed_size(dt, count)))
        return ENEC_ERR_BUFFER_TOO_SMALL;
    unsigned long long* out_size = reinterpret_cast<unsigned long long*>(d_out_size);
    if (count == 0) {
        // no exponent occurs: the search of Sec. 5.5 has nothing to minimise and keeps (0, 1, 1)
        enec_encode_empty_kernel<<<1, 32, 0, stream>>>(static_cast<uint8_t*>(d_out), int(dt), with_params ? b : 0,
                                                      with_params ? n : 1, with_params ? m : 1, out_size, ranked ? 1 : 0);
        g_launches.fetch_add(1, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess ? ENEC_OK : ENEC_ERR_CUDA;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
    DeviceInfo* found = device_info(dev);
    if (!found) return ENEC_ERR_CUDA;
    DeviceInfo& info = *found;
    const Geometry g = make_geometry(count);
    // control words, a state word per block, and the progress words of the kernel that places the records
    const size_t need = kControlBytes + (size_t(g.nblocks) + kPlaceMaxCtas) * sizeof(unsigned long long);
    // the scratch area carries state from call to call, which a replayed recording would not see
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return ENEC_ERR_CUDA;
    if (capturing != cudaStreamCaptureStatusNone) return ENEC_ERR_INVALID_ARG;
    const bool split = !ranked && !with_params && in_split_range(g.nblocks);
    if (!ranked && !split) {
        FusedJob fused;
        enec_status fst = lease_fused_scratch(dev, stream, g.nblocks, fused);
        if (fst != ENEC_OK) return fst;
        fused.in = static_cast<const uint8_t*>(d_in);
        fused.out = static_cast<uint8_t*>(d_out);
        fused.count = count;
        fused.out_size = out_size;
        fused.given = with_params ? uint32_t(b) | uint32_t(n) << 8 | uint32_t(m) << 12 | kParamsValid : 0u;
        fst = launch_fused(int(dt), fused, g.nblocks, info.sms, info.fused_attr_set, d_status, stream);
        if (fst != ENEC_OK) mark_scratch_unclean(dev, stream, kScratchFused);
        return fst;
    }
    uint8_t* scratch = nullptr;
    uint32_t epoch = 0;
    enec_status st = lease_compress_scratch(dev, stream, need, &scratch, &epoch);
    if (st != ENEC_OK) return st;
    EncodeJob job;
    job.in = static_cast<const uint16_t*>(d_in);
    job.out = static_cast<uint8_t*>(d_out);
    job.count = count;
    place_job(job, scratch, epoch);
    job.out_size = out_size;
    job.ranked = ranked ? 1 : 0;
    st = dt == ENEC_BF16   ? launch_encode<ENEC_BF16>(job, g.nblocks, d_status, info, stream, split)
         : dt == ENEC_FP16 ? launch_encode<ENEC_FP16>(job, g.nblocks, d_status, info, stream, split)
                           : launch_encode<ENEC_FP32>(job, g.nblocks, d_status, info, stream, split);
    if (st != ENEC_OK) mark_compress_scratch_unclean(dev, stream);  // a kernel of the call may not have run
    return st;
}

// ---- compression without any allocation ------------------------------------------------------------
// Scratch of enec_compress_noalloc: the compressor's control words and one look-back state word per
// block, for tensors of up to kNoAllocMaxCount values, held in the library image on every GPU that loads
// it. In host code `g_noalloc_scratch` is only a handle for cudaGetSymbolAddress, never an address to
// hand to a kernel.
constexpr uint64_t kNoAllocMaxCount = uint64_t(1) << 30;
constexpr size_t kNoAllocScratchBytes = kControlBytes + size_t(kNoAllocMaxCount / kBlockElems) * sizeof(unsigned long long);
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocScratchBytes];
static_assert(kNoAllocScratchBytes == ENEC_NOALLOC_SCRATCH_BYTES, "the header states the size of the built-in scratch");

// Device address of the scratch on the current device, looked up once per device.
static enec_status noalloc_scratch(int dev, uint8_t** out) {
    static std::mutex mu;
    static uint8_t* addr[kMaxDevices] = {};
    if (dev < 0 || dev >= kMaxDevices) return ENEC_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ENEC_ERR_CUDA;
        addr[dev] = static_cast<uint8_t*>(p);
    }
    *out = addr[dev];
    return ENEC_OK;
}

// ---- the block-wise variant ------------------------------------------------------------------------

// The counter of finished blocks: zeroed when the area is new or after a call on it failed to launch; the
// kernel that uses it leaves it at zero.
static enec_status lease_blockwise_counter(int dev, cudaStream_t stream, uint32_t** out) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchArea& a = scratch_area(dev, stream, kScratchBlockwise);
    const enec_status st = grow(a, 256);
    if (st != ENEC_OK) return st;
    if (a.needs_clear) {
        if (cudaMemsetAsync(a.ptr, 0, 256, stream) != cudaSuccess) return ENEC_ERR_CUDA;
        a.needs_clear = false;
    }
    *out = reinterpret_cast<uint32_t*>(a.ptr);
    return ENEC_OK;
}

template <int DT>
static enec_status launch_blockwise(const BlockwiseJob& job, uint32_t nblocks, int* d_status, DeviceInfo& info,
                                    cudaStream_t stream) {
    if (!info.blockwise_attr_set[DT]) {
        if (cudaFuncSetAttribute(enec_block_params_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(HistShape<DT>::kBytes)) != cudaSuccess ||
            cudaFuncSetAttribute(enec_pack_blocks_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(kPackSmemBytes)) != cudaSuccess)
            return ENEC_ERR_CUDA;
        info.blockwise_attr_set[DT] = true;
    }
    uint32_t grid = uint32_t(info.sms) * 3;
    if (grid > nblocks) grid = nblocks;
    cudaError_t err = launch_pdl(enec_block_params_kernel<DT>, grid, kBlockwiseThreads, HistShape<DT>::kBytes, stream, job,
                                 d_status);
    if (err != cudaSuccess) return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    grid = uint32_t(info.sms) * 4;
    if (grid > nblocks) grid = nblocks;
    err = launch_pdl(enec_pack_blocks_kernel<DT>, grid, kBlockwiseThreads, kPackSmemBytes, stream, job, d_status);
    if (err != cudaSuccess) return ENEC_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ENEC_OK;
}

static size_t max_size_blockwise(enec_dtype dt, size_t count) {
    if (!known_dtype(dt) || (uint64_t(count) >> 36)) return 0;
    const int E = exp_bits(dt);
    const Geometry g = make_geometry(count);
    // a block's low plane and records together are largest when all its groups are wide with n = E; the two
    // variable sections each end in up to 15 bytes of padding
    uint64_t worst = 0;
    for (int m = 1; m <= E; ++m) {
        const uint64_t t = make_sections_blockwise(dt, count, g, g.padded_count * uint64_t(m) / 8,
                                                   uint64_t(g.total_groups) * 2 * uint64_t(E - m)).total;
        if (t > worst) worst = t;
    }
    return size_t(worst + 32);
}

static enec_status compress_blockwise(const void* d_in, enec_dtype dt, size_t count, void* d_out, size_t out_capacity,
                                      size_t* d_out_size, int* d_status, cudaStream_t stream) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if ((!d_in && count) || !d_out || (uint64_t(count) >> 36) || !aligned16(d_in) || !aligned16(d_out) ||
        (reinterpret_cast<uintptr_t>(d_out_size) & 7))
        return ENEC_ERR_INVALID_ARG;
    if (out_capacity < max_size_blockwise(dt, count)) return ENEC_ERR_BUFFER_TOO_SMALL;
    unsigned long long* out_size = reinterpret_cast<unsigned long long*>(d_out_size);
    if (count == 0) {
        enec_encode_empty_kernel<<<1, 32, 0, stream>>>(static_cast<uint8_t*>(d_out), int(dt), 0, 0, 0, out_size, 2);
        g_launches.fetch_add(1, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess ? ENEC_OK : ENEC_ERR_CUDA;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
    DeviceInfo* found = device_info(dev);
    if (!found) return ENEC_ERR_CUDA;
    // the counter carries state from call to call, which a replayed recording would not see
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return ENEC_ERR_CUDA;
    if (capturing != cudaStreamCaptureStatusNone) return ENEC_ERR_INVALID_ARG;
    BlockwiseJob job;
    job.in = static_cast<const uint16_t*>(d_in);
    job.out = static_cast<uint8_t*>(d_out);
    job.count = count;
    job.out_size = out_size;
    enec_status st = lease_blockwise_counter(dev, stream, &job.done);
    if (st != ENEC_OK) return st;
    const uint32_t nblocks = make_geometry(count).nblocks;
    st = dt == ENEC_BF16   ? launch_blockwise<ENEC_BF16>(job, nblocks, d_status, *found, stream)
         : dt == ENEC_FP16 ? launch_blockwise<ENEC_FP16>(job, nblocks, d_status, *found, stream)
                           : launch_blockwise<ENEC_FP32>(job, nblocks, d_status, *found, stream);
    if (st != ENEC_OK) {
        std::lock_guard<std::mutex> lock(g_scratch_mu);
        scratch_area(dev, stream, kScratchBlockwise).needs_clear = true;
    }
    return st;
}

}  // namespace enec

using namespace enec;

extern "C" {

size_t enec_max_compressed_size(enec_dtype dt, size_t count) {
    if (!known_dtype(dt) || (uint64_t(count) >> 36)) return 0;
    const int E = exp_bits(dt);
    const Geometry g = make_geometry(count);
    uint64_t worst = 0;
    for (int m = 1; m <= E; ++m) {
        const uint64_t t = make_sections(dt, count, g, E, m, g.total_groups).total;
        if (t > worst) worst = t;
    }
    return size_t(worst);
}

// The ticket word of a large tensor's decode launch and the number of the launch on it (see enec_decode_kernel,
// TICKET = 2). The word is cleared once, when its area is allocated; after that every launch finds the number of an
// earlier launch in it and starts it afresh.
static enec_status lease_decode_ticket(int dev, cudaStream_t stream, uint8_t** word, uint32_t* number) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    ScratchArea& a = scratch_area(dev, stream, kScratchDecodeTicket);
    const enec_status st = grow(a, 256);
    if (st != ENEC_OK) return st;
    if (a.needs_clear || a.epoch == 0xFFFFFFFFu) {
        if (cudaMemsetAsync(a.ptr, 0, 256, stream) != cudaSuccess) return ENEC_ERR_CUDA;
        a.needs_clear = false;
        a.epoch = 0;
    }
    *word = a.ptr;
    *number = ++a.epoch;
    return ENEC_OK;
}

// Tensors of at least this many blocks are decoded with their blocks handed out by a ticket (outside a stream
// capture: the ticket word carries the launch's number, which a replay would repeat). ENEC_DECODE_TICKET_MIN_BLOCKS
// in the environment overrides the bound (read once; for measurements and tests).
static uint32_t decode_ticket_min_blocks() {
    static const uint32_t value = env_blocks("ENEC_DECODE_TICKET_MIN_BLOCKS", 16384u);
    return value;
}

static enec_status decompress_one(const void* d_in, size_t in_size, enec_dtype dt, size_t count, void* d_out,
                                  int* d_status, cudaStream_t stream, bool ranked, bool blockwise = false) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if (!d_in || (!d_out && count) || (uint64_t(count) >> 36) || !aligned16(d_in) || !aligned16(d_out))
        return ENEC_ERR_INVALID_ARG;
    if (in_size < kHeaderBytes + 16) return ENEC_ERR_BAD_STREAM;
    DecodeBatch batch;
    batch.jobs = nullptr;
    batch.prefix = nullptr;
    batch.n_jobs = 1;
    batch.blockwise = blockwise ? 1 : 0;
    batch.chunk_blocks = 0;
    batch.total_blocks = make_geometry(count).nblocks;
    batch.inline_jobs[0] = DecodeJob{static_cast<const uint8_t*>(d_in), static_cast<uint16_t*>(d_out), uint64_t(count),
                                     uint64_t(in_size)};
    batch.inline_prefix[0] = 0;
    batch.inline_prefix[1] = batch.total_blocks;
    int ticketed = 0;
    if (!ranked && !blockwise && batch.total_blocks >= decode_ticket_min_blocks()) {
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return ENEC_ERR_CUDA;
        if (capturing == cudaStreamCaptureStatusNone) {
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
            uint8_t* word = nullptr;
            uint32_t number = 0;
            // without the word (no device memory to be had) the launch keeps fixed shares: slower, not wrong
            if (lease_decode_ticket(dev, stream, &word, &number) == ENEC_OK) {
                batch.inline_jobs[1] = DecodeJob{word, nullptr, uint64_t(number), 0};  // not a tensor: n_jobs stays 1
                ticketed = 2;
            }
        }
    }
    return launch_decode_any(dt, batch, d_status, stream, ranked, ticketed);
}

enec_status enec_decompress(const void* d_in, size_t in_size, enec_dtype dt, size_t count, void* d_out,
                            int* d_status, enec_stream_t stream) {
    return decompress_one(d_in, in_size, dt, count, d_out, d_status, stream, false);
}

enec_status enec_decompress_ranked(const void* d_in, size_t in_size, enec_dtype dt, size_t count, void* d_out,
                                   int* d_status, enec_stream_t stream) {
    return decompress_one(d_in, in_size, dt, count, d_out, d_status, stream, true);
}

// Blocks per chunk of a ticketed list (see DecodeBatch): two, or one when that leaves CTAs (three per SM) without a
// second chunk.
static uint32_t batched_chunk_blocks(uint64_t total_blocks, int sms) {
    const uint64_t ctas_of_a_launch = uint64_t(sms) * 3;
    return total_blocks < 4 * ctas_of_a_launch ? 1u : 2u;
}

enec_status enec_decompress_batched(const enec_batch_item* h_items, int n_items, enec_dtype dt, int* d_status,
                                    enec_stream_t stream) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if (n_items < 0 || (n_items > 0 && !h_items)) return ENEC_ERR_INVALID_ARG;
    if (n_items == 0) return ENEC_OK;
    // descriptors and block prefix in one host buffer: [jobs | prefix]; long lists add [ticket | tensor of every chunk]
    const size_t jobs_bytes = size_t(n_items) * sizeof(DecodeJob);
    const size_t prefix_bytes = size_t(ticket_offset_behind_prefix(uint32_t(n_items)));
    std::vector<uint8_t> host(jobs_bytes + prefix_bytes);
    DecodeJob* jobs = reinterpret_cast<DecodeJob*>(host.data());
    uint32_t* prefix = reinterpret_cast<uint32_t*>(host.data() + jobs_bytes);
    uint64_t total = 0;
    for (int i = 0; i < n_items; ++i) {
        const enec_batch_item& it = h_items[i];
        if (!it.d_in || (!it.d_out && it.count) || (uint64_t(it.count) >> 36) || !aligned16(it.d_in) ||
            !aligned16(it.d_out))
            return ENEC_ERR_INVALID_ARG;
        if (it.size < kHeaderBytes + 16) return ENEC_ERR_BAD_STREAM;
        jobs[i] = DecodeJob{static_cast<const uint8_t*>(it.d_in), static_cast<uint16_t*>(it.d_out), uint64_t(it.count),
                            uint64_t(it.size)};
        prefix[i] = uint32_t(total);
        total += make_geometry(it.count).nblocks;
        if (total >> 31) return ENEC_ERR_INVALID_ARG;  // block indices are 32-bit
    }
    prefix[n_items] = uint32_t(total);
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return ENEC_ERR_CUDA;
    if (capturing != cudaStreamCaptureStatusNone && uint32_t(n_items) > kInlineJobs) {
        // A recording must hold neither a copy from this call's host memory nor the library's scratch: lists of
        // up to kInlineJobs tensors travel inside the launch parameters, so a longer list becomes several launches.
        for (int first = 0; first < n_items; first += int(kInlineJobs)) {
            const int n = n_items - first < int(kInlineJobs) ? n_items - first : int(kInlineJobs);
            DecodeBatch part;
            part.jobs = nullptr;
            part.prefix = nullptr;
            part.n_jobs = uint32_t(n);
            part.blockwise = 0;
            part.chunk_blocks = 0;
            part.total_blocks = prefix[first + n] - prefix[first];
            for (int i = 0; i < n; ++i) part.inline_jobs[i] = jobs[first + i];
            for (int i = 0; i <= n; ++i) part.inline_prefix[i] = prefix[first + i] - prefix[first];
            const enec_status st = launch_decode_any(dt, part, d_status, stream, false);
            if (st != ENEC_OK) return st;
        }
        return ENEC_OK;
    }
    DecodeBatch batch;
    batch.n_jobs = uint32_t(n_items);
    batch.blockwise = 0;
    batch.chunk_blocks = 0;
    batch.total_blocks = uint32_t(total);
    bool ticketed = false;
    // A short list travels in the launch parameters: no copy, no scratch. Unless it has so many blocks that the
    // ticket of the long-list form (which needs a zeroed word, hence the copy) gains more than the copy costs.
    constexpr uint64_t kTicketWorthBlocks = 8192;
    if (uint32_t(n_items) <= kInlineJobs && (capturing != cudaStreamCaptureStatusNone || total < kTicketWorthBlocks)) {
        batch.jobs = nullptr;
        batch.prefix = nullptr;
        for (int i = 0; i < n_items; ++i) batch.inline_jobs[i] = jobs[i];
        for (int i = 0; i <= n_items; ++i) batch.inline_prefix[i] = prefix[i];
    } else {
        // the blocks of a long list are handed out in chunks: a zeroed ticket word and the tensor of every chunk's
        // first block travel with the descriptors
        const size_t ticket_at = host.size();
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
        const DeviceInfo* info = device_info(dev);
        if (!info) return ENEC_ERR_CUDA;
        const uint32_t chunk = batched_chunk_blocks(total, info->sms);
        batch.chunk_blocks = uint16_t(chunk);
        const size_t n_chunks = size_t((total + chunk - 1) / chunk);
        host.resize(ticket_at + 16 + n_chunks * sizeof(uint32_t), 0);
        {
            const uint32_t* pre = reinterpret_cast<const uint32_t*>(host.data() + jobs_bytes);
            uint32_t* chunk_job = reinterpret_cast<uint32_t*>(host.data() + ticket_at + 16);
            uint32_t j = 0;
            for (size_t c = 0; c < n_chunks; ++c) {
                const uint64_t first = uint64_t(c) * chunk;
                while (pre[j + 1] <= first) ++j;  // tensors without blocks are skipped
                chunk_job[c] = j;
            }
        }
        uint8_t* scratch = nullptr;
        const enec_status st = get_scratch(dev, stream, kScratchBatch, host.size(), &scratch);
        if (st != ENEC_OK) return st;
        // pageable source: the call returns once the bytes are staged, so `host` may go out of scope
        if (cudaMemcpyAsync(scratch, host.data(), host.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess)
            return ENEC_ERR_CUDA;
        batch.jobs = reinterpret_cast<const DecodeJob*>(scratch);
        batch.prefix = reinterpret_cast<const uint32_t*>(scratch + jobs_bytes);
        ticketed = n_chunks > 0;
    }
    return launch_decode_any(dt, batch, d_status, stream, false, ticketed);
}

enec_status enec_compress(const void* d_in, enec_dtype dt, size_t count, void* d_out, size_t out_capacity,
                          size_t* d_out_size, int* d_status, enec_stream_t stream) {
    return compress_common(d_in, dt, count, false, 0, 0, 0, d_out, out_capacity, d_out_size, d_status, stream);
}

enec_status enec_compress_with_params(const void* d_in, enec_dtype dt, size_t count, int b, int n, int m,
                                      void* d_out, size_t out_capacity, size_t* d_out_size, int* d_status,
                                      enec_stream_t stream) {
    return compress_common(d_in, dt, count, true, b, n, m, d_out, out_capacity, d_out_size, d_status, stream);
}


size_t enec_max_compressed_size_ranked(enec_dtype dt, size_t count) {
    const size_t base = enec_max_compressed_size(dt, count);
    return base ? base + kRankTableBytes : 0;
}

size_t enec_max_compressed_size_blockwise(enec_dtype dt, size_t count) { return max_size_blockwise(dt, count); }

enec_status enec_compress_blockwise(const void* d_in, enec_dtype dt, size_t count, void* d_out, size_t out_capacity,
                                    size_t* d_out_size, int* d_status, enec_stream_t stream) {
    return compress_blockwise(d_in, dt, count, d_out, out_capacity, d_out_size, d_status, stream);
}

enec_status enec_decompress_blockwise(const void* d_in, size_t in_size, enec_dtype dt, size_t count, void* d_out,
                                      int* d_status, enec_stream_t stream) {
    return decompress_one(d_in, in_size, dt, count, d_out, d_status, stream, false, true);
}

enec_status enec_compress_ranked(const void* d_in, enec_dtype dt, size_t count, void* d_out, size_t out_capacity,
                                 size_t* d_out_size, int* d_status, enec_stream_t stream) {
    return compress_common(d_in, dt, count, false, 0, 0, 0, d_out, out_capacity, d_out_size, d_status, stream, true);
}

enec_status enec_compress_batched(const enec_batch_item* h_items, int n_items, enec_dtype dt, size_t* d_out_sizes,
                                  int* d_status, enec_stream_t stream) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if (n_items < 0 || (n_items > 0 && !h_items) || (reinterpret_cast<uintptr_t>(d_out_sizes) & 7))
        return ENEC_ERR_INVALID_ARG;
    if (n_items == 0) return ENEC_OK;
    for (int i = 0; i < n_items; ++i) {
        const enec_batch_item& it = h_items[i];
        if ((!it.d_in && it.count) || !it.d_out || (uint64_t(it.count) >> 36) || !aligned16(it.d_in) || !aligned16(it.d_out))
            return ENEC_ERR_INVALID_ARG;
        if (it.size < enec_max_compressed_size(dt, it.count)) return ENEC_ERR_BUFFER_TOO_SMALL;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
    DeviceInfo* found = device_info(dev);
    if (!found) return ENEC_ERR_CUDA;
    DeviceInfo& info = *found;
    // the call clears and fills scratch from host memory that does not outlive it: not something to record
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return ENEC_ERR_CUDA;
    if (capturing != cudaStreamCaptureStatusNone) return ENEC_ERR_INVALID_ARG;
    unsigned long long* sizes = reinterpret_cast<unsigned long long*>(d_out_sizes);
    // tensors of two blocks or more first, each from a multiple of kHistBlocks on in the index space of blocks, then those of
    // one block; tensors without elements are written by launches of their own
    std::vector<FusedListItem> items;
    std::vector<uint32_t> chunk_item;
    items.reserve(size_t(n_items));
    uint64_t index = 0, state_words = 0;
    uint32_t n_multi = 0;
    auto add = [&](int i, uint64_t first_block, uint32_t nblocks) {
        items.push_back(FusedListItem{static_cast<const uint8_t*>(h_items[i].d_in), static_cast<uint8_t*>(h_items[i].d_out),
                                      uint64_t(h_items[i].count), sizes ? sizes + i : nullptr, nullptr, nullptr, nullptr,
                                      uint32_t(first_block), nblocks});
    };
    for (int i = 0; i < n_items; ++i) {
        const uint32_t nblocks = make_geometry(h_items[i].count).nblocks;
        if (nblocks < 2) continue;
        if ((index + nblocks) >> 31) return ENEC_ERR_INVALID_ARG;  // block indices are 32-bit
        add(i, index, nblocks);
        const uint64_t chunks = (nblocks + kHistBlocks - 1) / kHistBlocks;
        chunk_item.insert(chunk_item.end(), size_t(chunks), n_multi);
        index += chunks * kHistBlocks;
        state_words += nblocks + (nblocks + kSuperBlocks - 1) / kSuperBlocks + nblocks / (kSuperBlocks * kHyperSupers) + 1;
        ++n_multi;
    }
    const uint32_t multi_blocks = uint32_t(index);
    for (int i = 0; i < n_items; ++i) {
        if (make_geometry(h_items[i].count).nblocks == 1) add(i, index++, 1u);
        if (h_items[i].count != 0) continue;
        enec_encode_empty_kernel<<<1, 32, 0, stream>>>(static_cast<uint8_t*>(h_items[i].d_out), int(dt), 0, 1, 1,
                                                      sizes ? sizes + i : nullptr);
        g_launches.fetch_add(1, std::memory_order_relaxed);
        if (cudaGetLastError() != cudaSuccess) return ENEC_ERR_CUDA;
    }
    if (items.empty()) return ENEC_OK;
    if (index >> 31) return ENEC_ERR_INVALID_ARG;
    // the order of the units
    std::vector<FusedListSegment> segments;
    uint32_t tickets = 0;
    auto segment = [&](uint32_t kind, uint32_t first, uint32_t end) {
        if (first == end) return;
        segments.push_back(FusedListSegment{tickets, first, kind});
        tickets += kind == kUnitCount ? (end - first) / kHistBlocks : end - first;
    };
    std::vector<uint32_t> wave{0};   // first blocks of the waves, and the end of the last
    for (uint32_t j = 0; j < n_multi; ++j) {
        const uint32_t end = j + 1 < n_multi ? items[j + 1].first_block : multi_blocks;
        if (j + 1 == n_multi || uint64_t(end - wave.back()) * kBlockElems * elem_bytes(dt) >= kWaveBytes) wave.push_back(end);
    }
    const size_t waves = wave.size() - 1;
    if (waves) segment(kUnitCount, wave[0], wave[1]);
    segment(kUnitWhole, multi_blocks, uint32_t(index));
    for (size_t w = 0; w < waves; ++w) {
        if (w + 1 < waves) segment(kUnitCount, wave[w + 1], wave[w + 2]);
        segment(kUnitPack, wave[w], wave[w + 1]);
    }
    segments.push_back(FusedListSegment{tickets, 0, kUnitEnd});
    // device scratch of the call: [ticket | control words per tensor | state words and sums], cleared, and
    // [tensors | tensor of every chunk | segments], copied from the host
    const size_t off_controls = 256;
    const size_t off_state = off_controls + size_t(n_multi) * sizeof(FusedItemControl);
    const size_t off_items = (off_state + size_t(state_words) * sizeof(unsigned long long) + 255) & ~size_t(255);
    const size_t off_chunks = off_items + items.size() * sizeof(FusedListItem);
    const size_t off_segments = off_chunks + ((chunk_item.size() + 3) & ~size_t(3)) * sizeof(uint32_t);
    const size_t need = off_segments + segments.size() * sizeof(FusedListSegment);
    uint8_t* scratch = nullptr;
    const enec_status st = get_scratch(dev, stream, kScratchCompressBatch, need, &scratch);
    if (st != ENEC_OK) return st;
    unsigned long long* words = reinterpret_cast<unsigned long long*>(scratch + off_state);
    for (uint32_t j = 0; j < n_multi; ++j) {
        FusedListItem& item = items[j];
        item.state = words;
        item.super = item.state + item.nblocks;
        item.hyper = item.super + (item.nblocks + kSuperBlocks - 1) / kSuperBlocks;
        words = item.hyper + item.nblocks / (kSuperBlocks * kHyperSupers) + 1;
    }
    std::vector<uint8_t> host(need - off_items);
    memcpy(host.data(), items.data(), items.size() * sizeof(FusedListItem));
    if (!chunk_item.empty()) memcpy(host.data() + (off_chunks - off_items), chunk_item.data(), chunk_item.size() * sizeof(uint32_t));
    memcpy(host.data() + (off_segments - off_items), segments.data(), segments.size() * sizeof(FusedListSegment));
    if (cudaMemsetAsync(scratch, 0, off_items, stream) != cudaSuccess) return ENEC_ERR_CUDA;
    // pageable source: the call returns once the bytes are staged, so `host` may go out of scope
    if (cudaMemcpyAsync(scratch + off_items, host.data(), host.size(), cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return ENEC_ERR_CUDA;
    FusedList list;
    list.items = reinterpret_cast<const FusedListItem*>(scratch + off_items);
    list.controls = reinterpret_cast<FusedItemControl*>(scratch + off_controls);
    list.chunk_item = reinterpret_cast<const uint32_t*>(scratch + off_chunks);
    list.segments = reinterpret_cast<const FusedListSegment*>(scratch + off_segments);
    list.n_segments = uint32_t(segments.size() - 1);
    list.n_items = uint32_t(items.size());
    list.n_multi = n_multi;
    list.multi_blocks = multi_blocks;
    list.ticket = reinterpret_cast<uint32_t*>(scratch);
    return launch_fused_list(int(dt), list, tickets, info.sms, info.fused_list_attr_set, d_status, stream);
}

enec_status enec_compress_noalloc(const void* d_in, enec_dtype dt, size_t count, void* d_out, size_t out_capacity,
                                  size_t* d_out_size, int* d_status, enec_stream_t stream) {
    if (!known_dtype(dt)) return ENEC_ERR_UNSUPPORTED_DTYPE;
    if (uint64_t(count) > kNoAllocMaxCount) return ENEC_ERR_TOO_LARGE;
    if ((!d_in && count) || !d_out || !aligned16(d_in) || !aligned16(d_out) ||
        (reinterpret_cast<uintptr_t>(d_out_size) & 7))
        return ENEC_ERR_INVALID_ARG;
    if (out_capacity < enec_max_compressed_size(dt, count)) return ENEC_ERR_BUFFER_TOO_SMALL;
    unsigned long long* out_size = reinterpret_cast<unsigned long long*>(d_out_size);
    if (count == 0) {
        enec_encode_empty_kernel<<<1, 32, 0, stream>>>(static_cast<uint8_t*>(d_out), int(dt), 0, 1, 1, out_size);
        g_launches.fetch_add(1, std::memory_order_relaxed);
        return cudaGetLastError() == cudaSuccess ? ENEC_OK : ENEC_ERR_CUDA;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ENEC_ERR_CUDA;
    uint8_t* scratch = nullptr;
    const enec_status st = noalloc_scratch(dev, &scratch);
    if (st != ENEC_OK) return st;
    DeviceInfo* found = device_info(dev);
    if (!found) return ENEC_ERR_CUDA;
    DeviceInfo& info = *found;
    const Geometry g = make_geometry(count);
    // the area keeps the previous call's words: histogram, ticket, flags and state words start at zero
    const size_t used = kControlBytes + size_t(g.nblocks) * sizeof(unsigned long long);
    if (cudaMemsetAsync(scratch, 0, used, stream) != cudaSuccess) return ENEC_ERR_CUDA;
    EncodeJob job;
    job.in = static_cast<const uint16_t*>(d_in);
    job.out = static_cast<uint8_t*>(d_out);
    job.count = count;
    place_job(job, scratch, 1);  // everything was just cleared, so every call is call number 1
    job.out_size = out_size;
    job.ranked = 0;
    return dt == ENEC_BF16   ? launch_encode<ENEC_BF16>(job, g.nblocks, d_status, info, stream)
           : dt == ENEC_FP16 ? launch_encode<ENEC_FP16>(job, g.nblocks, d_status, info, stream)
                             : launch_encode<ENEC_FP32>(job, g.nblocks, d_status, info, stream);
}

uint64_t enec_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

uint64_t enec_allocation_count(void) { return g_allocations.load(std::memory_order_relaxed); }

int enec_version(void) { return 100; }

}  // extern "C"

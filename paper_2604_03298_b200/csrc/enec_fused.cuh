// enec_compress in one kernel (Sec. 5.1 compression flow with the parameter choice of Sec. 5.5).
//
// enec_fused_kernel, three CTAs of 256 threads per SM, blocks of 16384 elements handed out by tickets:
//   1. Sample stage: the histogram of a sample of the tensor's blocks, spread over it (every block of a small tensor). When
//      the last sampled block is counted, its CTA runs the search of Sec. 5.5 and publishes (b, n, m).
//   2. Pack stage: split, transform (Sec. 5.3), group widths (Sec. 5.2), Algorithm 2, and the histogram of every block.
//      The input is read once, apart from the sample.
//   3. The CTA that counts the last block runs the search again, on the histogram of the whole tensor. When it gives the
//      parameters that were used, the stream is the one that the search on the whole tensor leads to. When it does not, the
//      CTAs pack the tensor again; a value that the sampled parameters cannot represent ends the pack stage at once, and the blocks
//      not packed yet are counted first.
// Parameters given by the caller: stage 2 alone, without the histogram, from the first block on; a value that they lose ends
// the call without a stream. (With a look-back kernel, or two kernels from 2048 blocks up, 3584 blocks of bf16 took 54 us, now 35.1;
// 1024 blocks 23.2 -> 13.9, fp16 4096 blocks 63.8 -> 43.8, fp32 8192 blocks 192 -> 158.)
// A tensor whose sample needs n > 6 exponent bits (bf16, fp32) takes the histogram of the whole tensor before it packs:
// the table kept beside the packing has 64 rows, and rare outliers of such a tensor are what a sample misses.
//
// Block offsets (the prefix sum of Sec. 5.1 / 5.4): every block's count of wide groups goes to a state word and is added
// to a sum per 128 blocks and a sum per 16384 blocks. A CTA keeps a block's packed records in shared memory while it
// packs its next block; by then all blocks handed out before have been counted as a rule, so its last four warps find the block's
// offset with one round of loads and copy the records to their place (if some block is not counted yet, one of them waits for it).
//
// A wait concerns only work whose tickets were handed out before, hence running CTAs, and in the pack stage only blocks
// with smaller numbers: the CTA with the smallest block that is not counted yet waits for nobody. Every wait is bounded
// all the same and ends in ENEC_ERR_TIMEOUT.
#pragma once

#include "enec_pack.cuh"

namespace enec {

constexpr int kFusedThreads = 256;
constexpr int kFusedWarps = kFusedThreads / 32;
constexpr uint32_t kSuperBlocks = 128;     // blocks per first-level sum
constexpr uint32_t kHyperSupers = 128;     // first-level sums per second-level sum
constexpr uint32_t kMaxHypers = 256;       // 2^36 values

// Control words of a call. The sums and the pack stage's ticket are kept per pass over the tensor (the second pass happens
// only when the sampled parameters were not the tensor's). Words that many CTAs add to lie on lines of their own: adds to
// one line are served one after another, about 3.6 ns each.
constexpr uint32_t kClaimWords = 16;
constexpr uint32_t kMaxFusedGrid = 32 * kClaimWords;
struct alignas(128) Counter { uint32_t value; uint32_t pad[31]; };
struct alignas(128) FusedControl {
    unsigned long long hist[2][256];             // of the sample, of the whole tensor but for what is in pack_hist
    unsigned long long pack_hist[256];           // of the pack stage
    unsigned long long hyper[2][kMaxHypers];     // bits 63..32 blocks counted, bits 31..0 their wide groups
    Counter hist_ticket[2], hist_done[2];
    Counter claims[kClaimWords];   // a bit per CTA: the block it starts with in the sample stage is taken
    Counter pack_ticket[2];
    Counter pack_done;         // blocks of the first pass whose counts are in pack_hist (or hist[1])
    Counter pack_left;         // blocks packed by the CTAs that have left the first pass, when there is a second
    uint32_t pack_target;      // blocks handed out before the first pass was ended early (0: it was not)
    uint32_t params[2];        // published: the parameters for hist[0], hist[1]
    uint32_t lossy;            // given parameters: some block holds a value that they lose
    uint32_t verdict;          // published: the whole tensor's parameters, when the first pass has counted every block
    uint32_t all_left;         // published: the first pass writes no more
};
constexpr uint32_t kFusedControlBytes = 16384;
static_assert(sizeof(FusedControl) <= kFusedControlBytes, "a control set fits its slot");
constexpr uint32_t kParamsValid = 1u << 31;   // a published word: b | n << 8 | m << 12 | valid
constexpr uint32_t kParamsRedo = 1u << 28;    // verdict: some packed blocks held values that the sampled parameters lose
constexpr uint32_t kParamsTake = 1u << 29;    // not a published word: there is a block to take
constexpr uint32_t kPassEnded = 1u << 30;     // pack_ticket: no further blocks in this pass

struct FusedJob {
    const uint8_t* in;
    uint8_t* out;
    uint64_t count;
    FusedControl* ctl;             // zero when the call starts
    FusedControl* ctl_next;        // the next call's set, zeroed by this call ...
    unsigned long long* super;     // first-level sums, two passes of super_stride words; zero when the call starts
    unsigned long long* super_next;
    uint32_t super_stride;
    uint32_t clear_supers;         // ... with so many first-level sums per pass
    uint32_t sample;               // blocks in the sample (nblocks: all)
    uint32_t given;                // the caller's parameters, as a published word (0: search)
    uint32_t epoch;                // tag of the first pass's state words; the second pass's is one more
    unsigned long long* state;     // per block: bits 63..32 epoch, bits 31..0 wide groups
    unsigned long long* out_size;  // device, may be null
};

template <int DT>
struct FusedShape {
    static constexpr int E = HistShape<DT>::E;
    static constexpr int kCtasPerSm = 3;
    static constexpr uint32_t kListAt = 0;                             // the wide groups' numbers, a byte each, by mask word
    static constexpr uint32_t kTensorAt = 1024;                        // FusedTensor (lists: of the block, the waiting block, the next)
    static constexpr uint32_t kSharedAt = kTensorAt + 3 * 256;         // FusedShared
    static constexpr uint32_t kPend = 4096;                            // a block's packed records waiting for their offset: two places
    static constexpr uint32_t kPendAt = kSharedAt + 256;
    // The pack stage's histogram lies on a multiple of its size (a CTA's shared memory begins with 1 KB of the system's), so that the
    // address of a value's counter is an AND-OR of the value's word: see histogram_in_place.
    static constexpr uint32_t kRows = DT == ENEC_FP16 ? 32 : 64;
    static constexpr uint32_t kHistAt = 7168;
    static constexpr uint32_t kHistBytes = kRows * HistShape<DT>::kRowBytes;
    static_assert(kPendAt + kPend <= kHistAt && (kHistAt + 1024) % kHistBytes == 0, "the histogram's place");
    // low plane | fp16 plane | the block's values: at the same places for every m, since a list's next block may have another
    static constexpr uint32_t kPlanesAt = kHistAt + kHistBytes;
    static constexpr uint32_t kSmhiAt = kPlanesAt + kBlockElems * 5 / 8, kValuesAt = kPlanesAt + kBlockElems;
    static_assert(kSmhiAt + kBlockElems * 3 / 8 <= kValuesAt, "the planes end before the values");
    static constexpr uint32_t kPend2At = kValuesAt + kBlockElems;
    static constexpr uint32_t kTableAt = kHistAt;                      // the table of the stages that count, and a search's
    static_assert(kTableAt + HistShape<DT>::kBytes <= kPend2At, "the table ends before the waiting records");
    static constexpr uint32_t kBytes = kPend2At + kPend;
    __device__ static uint32_t pend_at(uint32_t iter) { return iter & 1 ? kPend2At : kPendAt; }
    static_assert(kCtasPerSm * (kBytes + 1024) <= 228 * 1024, "the CTAs of an SM fit its shared memory");
};

// What a block of the pack stage needs to know about its tensor, in shared memory.
//
// The stage works with v = y ^ 2^(n-1) = b + 2^(n-1) - x (mod 2^n), one value per byte. PLAIN: 2^n <= b + 2^(n-1) <= 255
// (fp16: always), so that the difference of a representable exponent neither borrows nor leaves n bits, and a word
// pair takes two multiply-adds and a byte permutation; a value that is not representable shows as a bit above n.
struct FusedTensor {
    const uint8_t* in;
    uint8_t* out;
    uint8_t *sm, *lo, *low, *smhi, *mask, *high;   // the sections' first bytes
    uint32_t* table;
    unsigned long long* state;
    unsigned long long* super;
    unsigned long long* hyper;
    uint64_t count;
    uint64_t smhi_bytes, sm_bytes, lo_bytes;       // the sections' lengths
    unsigned long long* out_size;
    uint32_t nblocks, tail_real, tail_padded, total_groups;
    uint32_t epoch;
    int b, n, m, hbits;
    uint32_t c;        // the minuend: bf16 (b + 2^(n-1)) << 8 | 255 in both halves; fp16 and the general form: per byte
    uint32_t s4;       // 2^(n-1) in every byte
    uint32_t nmask4;   // 2^n - 1 in every byte
    uint32_t wide4;    // bits m .. n - 1 in every byte
    uint32_t pad;      // two 16-bit words with exponent b and nothing else: y = 0
    uint32_t wide_ok;  // bit 0: the input is 32-byte aligned, bit 1: the sm-lo plane is
    uint32_t plain;
    const uint32_t* lossy;         // given parameters: see FusedControl
    uint32_t first_block;          // lists: index of the tensor's first block in the list's index space
};

struct FusedShared {
    uint32_t mask[32];
    uint32_t next;       // the CTA's next ticket
    uint32_t word;       // broadcasts of thread 0
    uint32_t before;
    uint32_t ok;
    uint32_t unit[2][3];          // lists: what the CTA does now and next (see enec_fused_list_kernel)
    alignas(16) uint32_t part[4];   // the last four warps' shares of the wide groups before the waiting block; kNotReady: some are not counted yet
};
constexpr uint32_t kNotReady = 0xFFFFFFFFu;   // a tensor has at most 2^32 - 2^10 groups of 16 counted before a block
static_assert(sizeof(FusedTensor) <= 256 && sizeof(FusedShared) <= 256, "they fit their places");

__device__ __forceinline__ uint8_t* fused_smem() {
    extern __shared__ __align__(128) uint8_t smem[];
    return smem;
}
template <int DT>
__device__ __forceinline__ FusedTensor& fused_tensor(uint32_t slot = 0) {
    return *reinterpret_cast<FusedTensor*>(fused_smem() + FusedShape<DT>::kTensorAt + slot * 256);
}
template <int DT>
__device__ __forceinline__ FusedShared& fused_shared() { return *reinterpret_cast<FusedShared*>(fused_smem() + FusedShape<DT>::kSharedAt); }

template <int DT>
__device__ __forceinline__ bool plain_form(int b, int n) {
    return DT == ENEC_FP16 || (b + (1 << (n - 1)) <= 255 && (1 << n) <= b + (1 << (n - 1)));
}
// Whether the pack stage's histogram lies on a multiple of its size. (It does; a kernel where it did not would count whole tensors first.)
template <int DT>
__device__ __forceinline__ bool histogram_in_place() {
    return ((smem_u32(fused_smem()) + FusedShape<DT>::kHistAt) & (FusedShape<DT>::kHistBytes - 1)) == 0;
}
// Whether the pack stage can keep the histogram: representable exponents are told apart by their low six bits.
template <int DT>
__device__ __forceinline__ bool sample_will_do(uint32_t word) {
    const int b = int(word & 0xFF), n = int((word >> 8) & 0xF);
    return DT == ENEC_FP16 || (n <= 6 && plain_form<DT>(b, n));
}

// A tensor's context but for what follows from (b, n, m). One thread.
template <int DT>
__device__ inline void set_geometry(FusedTensor& t) {
    const Geometry g = make_geometry(t.count);
    const Sections sec = make_sections(DT, t.count, g, 1, 1, 0);
    t.nblocks = g.nblocks; t.tail_real = g.tail_real; t.tail_padded = g.tail_padded; t.total_groups = g.total_groups;
    t.table = reinterpret_cast<uint32_t*>(t.out + sec.table);
    t.mask = t.out + sec.mask;
    t.low = t.out + sec.low;
    t.smhi_bytes = sec.sm - sec.smhi;
    t.sm_bytes = sec.smlo - sec.sm;
    t.lo_bytes = sec.high - sec.smlo;
}
// The rest. One thread.
template <int DT>
__device__ inline void set_parameters(FusedTensor& t, uint32_t word) {
    const int b = int(word & 0xFF), n = int((word >> 8) & 0xF), m = int((word >> 12) & 0xF);
    t.b = b; t.n = n; t.m = m; t.hbits = n - m;
    const uint32_t d = uint32_t(b) + (1u << (n - 1));
    t.plain = plain_form<DT>(b, n);
    if (DT == ENEC_FP16) t.c = rep4(d + 64);   // the guard bit 6 keeps the bytes apart; bits 4..0 are the difference mod 32
    else t.c = t.plain ? ((d & 0xFF) << 8 | 0xFFu) * 0x00010001u : rep4(d);
    t.s4 = rep4(1u << (n - 1));
    t.nmask4 = rep4((1u << n) - 1);
    t.wide4 = rep4((0xFFu << m) & ((1u << n) - 1));
    t.pad = (DT == ENEC_FP16 ? uint32_t(b) << 10 : uint32_t(b) << 7) * 0x00010001u;
    t.smhi = t.low + align16((uint64_t(t.nblocks - 1) * kBlockElems + t.tail_padded) * uint32_t(m) / 8);
    t.sm = t.smhi + t.smhi_bytes;
    t.lo = t.sm + t.sm_bytes;
    t.high = t.lo + t.lo_bytes;
    t.wide_ok = ((reinterpret_cast<uintptr_t>(t.in) & 31) == 0 ? 1u : 0u) | ((reinterpret_cast<uintptr_t>(t.lo) & 31) == 0 ? 2u : 0u);
}

// Eq. 1 as width_eq1, the bit widths by counting leading zeros.
__device__ __forceinline__ int width_of_range(int b, int l, int h, int E) {
    const int pos = 32 - __clz(b - l);
    const int neg = h - b <= 1 ? 0 : 32 - __clz(h - b - 1);
    return min(max(pos, neg) + 1, E);
}

// ---- parameter search by one warp ------------------------------------------------------------------
// Sec. 5.5 phases 2 and 3 on a finished histogram. With C(x) = number of values with exponents up to x, N = all of them,
// S = sum of the exponents: for a candidate b of width n (Eq. 1) the values stored are b - x for x <= b and 2^n + b - x
// above, so Eq. 3's cost times N is N b - S + 2^n (N - C(b)), and the values below 2^m number
// C(b) - C(b - 2^m) + N - C(b + 2^n - 2^m): every candidate is a few table look-ups.
// `count_of(x)` gives the histogram; `table`: 256 words of shared memory. Returns b | n << 8 | m << 12 in every lane.
template <int DT, class CountOf>
__device__ __forceinline__ uint32_t search_by_warp(CountOf count_of, unsigned long long* table) {
    constexpr int E = HistShape<DT>::E;
    constexpr int kPer = (1 << E) / 32;
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    const int lane = int(threadIdx.x & 31);
    unsigned long long c[kPer];
    unsigned long long sum = 0, weighted = 0;
    int lo = 1 << E, hi = -1;
#pragma unroll
    for (int i = 0; i < kPer; ++i) c[i] = count_of(lane * kPer + i);
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int x = lane * kPer + i;
        if (c[i]) { lo = min(lo, x); hi = x; }
        sum += c[i];
        weighted += c[i] * (unsigned long long)x;
    }
    const int l = __reduce_min_sync(kAll, lo), h = __reduce_max_sync(kAll, hi);
    // 44 bits at most: the sum of 32 words in two halves
    const unsigned long long S = __reduce_add_sync(kAll, uint32_t(weighted & 0x3FFFFFFu)) +
                                 ((unsigned long long)__reduce_add_sync(kAll, uint32_t(weighted >> 26)) << 26);
    unsigned long long incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long t = __shfl_up_sync(kAll, incl, d);
        if (lane >= d) incl += t;
    }
    unsigned long long run = incl - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        run += c[i];
        table[lane * kPer + i] = run;
    }
    const unsigned long long total = __shfl_sync(kAll, incl, 31);
    __syncwarp();
    // the smallest of the lanes' 64-bit words, in two halves
    auto smallest = [&](unsigned long long v) -> unsigned long long {
        const uint32_t high = __reduce_min_sync(kAll, uint32_t(v >> 32));
        const uint32_t low = __reduce_min_sync(kAll, uint32_t(v >> 32) == high ? uint32_t(v) : kAll);
        return (unsigned long long)high << 32 | low;
    };
    unsigned long long key = ~0ull;
    for (int b = l + lane; b <= h; b += 32) {
        const int n = width_of_range(b, l, h, E);
        const unsigned long long cost = total * (unsigned long long)b - S + ((total - table[b]) << n);
        const unsigned long long mine = (cost << 12) | (unsigned long long)(n << 8) | (unsigned long long)b;  // cost < 2^44
        key = mine < key ? mine : key;
    }
    key = smallest(key);
    const int b = int(key & 0xFF), n = int((key >> 8) & 0xF);
    // Eq. 4 at L = 16, lane m - 1 evaluates m: plain IEEE double, one rounding per operation; ties go to the smaller m
    const int m = lane < n ? lane + 1 : n;
    auto upto = [&](int x) { return x < 0 ? 0ull : x >= (1 << E) ? total : table[x]; };
    const unsigned long long cnt = upto(b) - upto(b - (1 << m)) + total - upto(b + (1 << n) - (1 << m));
    const double p = __ddiv_rn(__ull2double_rn(cnt), __ull2double_rn(total));
    const double p2 = __dmul_rn(p, p), p4 = __dmul_rn(p2, p2), p8 = __dmul_rn(p4, p4), p16 = __dmul_rn(p8, p8);
    const double bits = __dadd_rn(__dadd_rn(double(n), 0.0625), __dmul_rn(double(m - n), p16));
    // positive numbers: their bit patterns are ordered as they are
    const unsigned long long pattern = (unsigned long long)__double_as_longlong(bits);
    const uint32_t winners = __ballot_sync(kAll, pattern == smallest(pattern));
    __syncwarp();
    return uint32_t(b) | (uint32_t(n) << 8) | (uint32_t(__ffs(winners)) << 12);
}

// The search on the sum of one or two histograms in global memory.
template <int DT>
__device__ __noinline__ uint32_t search_global(const unsigned long long* hist, const unsigned long long* more, unsigned long long* table) {
    return search_by_warp<DT>([&](int x) { return ld_relaxed_u64(&hist[x]) + (more ? ld_relaxed_u64(&more[x]) : 0ull); }, table);
}

// ---- loads -------------------------------------------------------------------------------------------
struct Run { uint32_t w[8]; };  // sixteen 16-bit words in element order

// 32 bytes at p: one access where p is 32-byte aligned (WIDE), two of 16 bytes else. (Two bodies and a branch around a batch
// of them, not two predicated loads: a predicated load keeps its registers occupied long before it.)
// The input's lines are the first to leave L2: what is read again from there is the kernel's code, after another kernel ran, and
// a small tensor's input, until it is packed (3584 blocks of bf16 55.2 -> 53.1 us, after another kernel 71.5 -> 63.6).
template <bool WIDE>
__device__ __forceinline__ Run load32(const uint8_t* p) {
    Run r;
    if constexpr (WIDE)
        asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                     : "l"(p));
    else
        asm volatile("ld.global.cs.v4.b32 {%0, %1, %2, %3}, [%8];\n\tld.global.cs.v4.b32 {%4, %5, %6, %7}, [%8+16];"
                     : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                     : "l"(p));
    return r;
}
__device__ __forceinline__ void store32(uint8_t* p, const Run& r, bool wide) {
    if (wide) {
        asm volatile("st.global.cs.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(r.w[0]), "r"(r.w[1]), "r"(r.w[2]), "r"(r.w[3]),
                     "r"(r.w[4]), "r"(r.w[5]), "r"(r.w[6]), "r"(r.w[7]), "l"(p)
                     : "memory");
    } else {
        __stcs(reinterpret_cast<uint4*>(p), make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]));
        __stcs(reinterpret_cast<uint4*>(p) + 1, make_uint4(r.w[4], r.w[5], r.w[6], r.w[7]));
    }
}

// fp32: the high halves of sixteen values (the first eight in a, the others in b); their low halves go to `lo` (32 bytes).
__device__ __forceinline__ Run split_halves(const Run& a, const Run& b, uint8_t* lo, bool wide) {
    Run h, l;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h.w[i] = prmt(a.w[2 * i], a.w[2 * i + 1], 0x7632u);
        h.w[4 + i] = prmt(b.w[2 * i], b.w[2 * i + 1], 0x7632u);
        l.w[i] = prmt(a.w[2 * i], a.w[2 * i + 1], 0x5410u);
        l.w[4 + i] = prmt(b.w[2 * i], b.w[2 * i + 1], 0x5410u);
    }
    store32(lo, l, wide);
    return h;
}

// The run of a tail block: values from element `real` on (counted from the run's first) are padding. fp32: zeros behind
// the low halves up to the plane's 16-byte boundary, `lo_room` more halves.
template <int DT>
__device__ __forceinline__ Run load_run_tail(const uint8_t* in, uint8_t* lo, int real, int lo_room, uint32_t pad) {
    Run r;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        uint32_t half[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = 2 * i + q;
            half[q] = pad & 0xFFFFu;
            if constexpr (DT == ENEC_FP32) {
                uint32_t full = 0;
                if (e < real) { full = reinterpret_cast<const uint32_t*>(in)[e]; half[q] = full >> 16; }
                if (e < lo_room) reinterpret_cast<uint16_t*>(lo)[e] = uint16_t(full);
            } else {
                if (e < real) half[q] = reinterpret_cast<const uint16_t*>(in)[e];
            }
        }
        r.w[i] = half[0] | (half[1] << 16);
    }
    return r;
}

// ---- one run: transform, sign/mantissa, histogram -------------------------------------------------------
// column: the lane's in the pack stage's table, whose address is a multiple of its size. (Adding the row to any other address is one
// instruction more per value: 32064 blocks of bf16 314.7 us, now 311.3, 4096 of fp16 59.7 and 58.9.)
template <int DT>
__device__ __forceinline__ void count_halves(uint32_t column, uint32_t w) {
    if constexpr (DT == ENEC_FP16) {
        red_add_one(((w >> 3) & 0xF80u) | column);
        red_add_one(((w >> 19) & 0xF80u) | column);
    } else {
        red_add_one((w & 0x1F80u) | column);
        red_add_one(((w >> 16) & 0x1F80u) | column);
    }
}

// a - 2 w as one multiply-add.
__device__ __forceinline__ uint32_t minus_twice(uint32_t a, uint32_t w) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, 0xFFFFFFFE, %2;" : "=r"(d) : "r"(w), "r"(a));
    return d;
}

template <int DT, bool PLAIN, bool HIST, bool CHECK>
__device__ __forceinline__ void transform_run(const Run& r, uint32_t minuend, uint32_t nmask4, uint32_t column, uint4& v,
                                              uint4& hs, uint4& sm) {
    uint32_t vv[4], ss[4], hh[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t w0 = r.w[2 * q], w1 = r.w[2 * q + 1];
        const uint32_t lo = prmt(w0, w1, 0x6420u), hi = prmt(w0, w1, 0x7531u);
        if constexpr (DT == ENEC_FP16) {
            vv[q] = minuend - ((hi >> 2) & 0x1F1F1F1Fu);
            ss[q] = lo;
            hh[q] = select_bits(0x03030303u, hi, (hi >> 5) & 0x04040404u);
        } else {
            ss[q] = select_bits(0x80808080u, hi, lo);
            hh[q] = 0;
            if constexpr (PLAIN) {
                vv[q] = prmt(minus_twice(minuend, w0), minus_twice(minuend, w1), 0x7531u);
            } else {
                const uint32_t x = prmt(2 * w0, 2 * w1, 0x7531u);
                vv[q] = ((minuend | 0x80808080u) - (x & 0x7F7F7F7Fu)) ^ ((minuend ^ ~x) & 0x80808080u);
                if (!CHECK) vv[q] &= nmask4;
            }
        }
        if constexpr (HIST) {
            count_halves<DT>(column, w0);
            count_halves<DT>(column, w1);
        }
    }
    v = make_uint4(vv[0], vv[1], vv[2], vv[3]);
    sm = make_uint4(ss[0], ss[1], ss[2], ss[3]);
    hs = make_uint4(hh[0], hh[1], hh[2], hh[3]);
}

__device__ __forceinline__ uint32_t or_flipped(const uint4& v, uint32_t s4) {
    return (v.x ^ s4) | (v.y ^ s4) | (v.z ^ s4) | (v.w ^ s4);
}

// ---- Algorithm 2 on packed bytes ---------------------------------------------------------------------
// As pack_plane_level (a thread owns eight consecutive lanes of the deepest level), for fields that need not be clean:
// bits above a field are masked away where it is inserted.
template <int W>
__device__ __forceinline__ void insert_field(uint32_t& lo, uint32_t& hi, uint32_t v, int s) {
    constexpr uint32_t kField = (1u << W) - 1;
    if (s + W <= 8) {
        const uint32_t mask = rep4(kField << s);
        lo = select_bits(mask, v << s, lo);
    } else if (s >= 8) {
        const uint32_t mask = rep4(kField << (s - 8));
        hi = select_bits(mask, v << (s - 8), hi);
    } else {
        const uint32_t mask_lo = rep4(0xFFu << s), mask_hi = rep4(kField >> (8 - s));
        lo = select_bits(mask_lo, v << s, lo);
        hi = select_bits(mask_hi, v >> (8 - s), hi);
    }
}

template <int W_IN, int LOG_UNITS>
__device__ __forceinline__ void pack_lanes_level(uint32_t S, uint32_t nb_off, uint32_t j, uint32_t n8, const uint2 (&in)[1 << LOG_UNITS]) {
    constexpr int F = folds_for(W_IN);
    static_assert(F <= LOG_UNITS, "lane runs must stay whole");
    constexpr int W = W_IN << F;
    constexpr int LOG_LANES = LOG_UNITS - F;
    constexpr int NL = 1 << LOG_LANES;
    constexpr int RES = W - 8;
    uint2 R[NL];
#pragma unroll
    for (int c = 0; c < NL; ++c) {
        uint2 V = make_uint2(0, 0);
        R[c] = make_uint2(0, 0);
#pragma unroll
        for (int q = 0; q < (1 << F); ++q) {
            const int e = c + q * NL;
            const int s = W_IN * bitrev(q, F);
            insert_field<W_IN>(V.x, R[c].x, in[e].x, s);
            insert_field<W_IN>(V.y, R[c].y, in[e].y, s);
        }
        sts64(S + nb_off + j + c * n8, V);
    }
    if constexpr (RES > 0) pack_lanes_level<RES, LOG_LANES>(S, nb_off + NL * n8, j, n8, R);
}

template <int DT>
__device__ __forceinline__ void pack_lanes_any(int m, uint32_t S, uint32_t j, uint32_t n8, const uint2 (&v)[8]) {
    switch (m) {
        case 1: pack_lanes_level<1, 3>(S, 0, j, n8, v); break;
        case 2: pack_lanes_level<2, 3>(S, 0, j, n8, v); break;
        case 3: pack_lanes_level<3, 3>(S, 0, j, n8, v); break;
        case 4: pack_lanes_level<4, 3>(S, 0, j, n8, v); break;
        case 5: pack_lanes_level<5, 3>(S, 0, j, n8, v); break;
        case 6: if constexpr (DT != ENEC_FP16) pack_lanes_level<6, 3>(S, 0, j, n8, v); break;
        case 7: if constexpr (DT != ENEC_FP16) pack_lanes_level<7, 3>(S, 0, j, n8, v); break;
        default: if constexpr (DT != ENEC_FP16) pack_lanes_level<8, 3>(S, 0, j, n8, v); break;
    }
}

// The low plane (and the fp16 plane) of a block of N >= 128 elements from its values in shared memory, in the order before
// the final fold; all threads.
template <int DT>
__device__ __forceinline__ void pack_planes(const FusedTensor& t, uint32_t work, uint32_t N, uint32_t tid) {
    using Shape = FusedShape<DT>;
    const uint32_t j = 8 * tid, n8 = N >> 3;
    if (j >= n8) return;
    const uint32_t values = work + Shape::kValuesAt, planes = work + Shape::kPlanesAt, s4 = t.s4;
    uint2 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = lds64(values + c * n8 + j);
    if (t.hbits == 0) {   // bit n - 1, flipped in v, belongs to the low plane
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = make_uint2(v[c].x ^ s4, v[c].y ^ s4);
    }
    pack_lanes_any<DT>(t.m, planes, j, n8, v);
    if constexpr (DT == ENEC_FP16) {
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = make_uint2(v[c].x >> 5, v[c].y >> 5);
        pack_lanes_level<3, 3>(work + Shape::kSmhiAt, 0, j, n8, v);
    }
}

// The final fold (see fold_plane_out), all threads. (Not unrolled: a thread has one or two rounds for m = 3, and the code around an
// unrolled loop costs more.)
__device__ __forceinline__ void fold_out(uint32_t S, uint32_t T, uint8_t* dst, uint32_t tid) {
    const uint32_t thalf = T >> 1, end = S + thalf;
    uint32_t at = S + 8 * tid;
    dst += 16 * tid;
#pragma unroll 1
    for (; at < end; at += 8 * kFusedThreads, dst += 16 * kFusedThreads) {
        const uint2 lo = lds64(at), hi = lds64(at + thalf);
        uint4 w;
        w.x = prmt(lo.x, hi.x, 0x5140u);
        w.y = prmt(lo.x, hi.x, 0x7362u);
        w.z = prmt(lo.y, hi.y, 0x5140u);
        w.w = prmt(lo.y, hi.y, 0x7362u);
        __stcs(reinterpret_cast<uint4*>(dst), w);
    }
}

// A wide group's record: Algorithm 2 with N = 16 on packed bytes, four lanes per 32-bit word. in: LANES fields of W_IN bits
// (four per word; two lanes sit in the low half of a word). The normalised bytes of the level go to nb from byte NB on.
template <int W_IN, int LANES, int NB, int NW>
__device__ __forceinline__ void record_level(const uint32_t (&in)[(LANES + 3) / 4], uint32_t (&nb)[NW]) {
    constexpr int F = folds_for(W_IN);
    constexpr int W = W_IN << F;
    constexpr int OUT = LANES >> F;      // lanes after the folds
    static_assert(OUT >= 2, "a record's lanes fold down to two at least");
    constexpr int RES = W - 8;
    constexpr int NV = (OUT + 3) / 4;
    uint32_t V[NV], R[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
        V[c] = R[c] = 0;
#pragma unroll
        for (int q = 0; q < (1 << F); ++q) {
            // the OUT lanes from lane q * OUT on
            const int first = q * OUT + 4 * c;
            const uint32_t lanes = OUT >= 4 ? in[first >> 2] : (first & 2) ? in[first >> 2] >> 16 : in[first >> 2] & 0xFFFFu;
            insert_field<W_IN>(V[c], R[c], lanes, W_IN * bitrev(q, F));
        }
        if (OUT == 2) V[c] &= 0xFFFFu;
        // bytes NB + 4 c .. of the normalised bytes (NB is even)
        if ((NB & 2) == 0) nb[(NB >> 2) + c] |= V[c];
        else {
            nb[NB >> 2] |= V[c] << 16;
            if (OUT >= 4) nb[(NB >> 2) + 1] |= V[c] >> 16;
        }
    }
    if constexpr (RES > 0) record_level<RES, OUT, NB + OUT, NW>(R, nb);
}

// The record of sixteen values v as H 16-bit words: word i = normalised byte i and, above it, normalised byte i + H.
template <int H>
__device__ __forceinline__ void record_words(const uint4& v, uint32_t s4, int m, uint32_t (&q)[H]) {
    constexpr uint32_t kMask = ((1u << H) - 1) * 0x01010101u;
    const uint32_t flip = s4 >> m;
    const uint32_t in[4] = {((v.x >> m) ^ flip) & kMask, ((v.y >> m) ^ flip) & kMask, ((v.z >> m) ^ flip) & kMask, ((v.w >> m) ^ flip) & kMask};
    uint32_t nb[(2 * H + 3) / 4 + 1];
#pragma unroll
    for (int i = 0; i < (2 * H + 3) / 4 + 1; ++i) nb[i] = 0;
    record_level<H, 16, 0>(in, nb);
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const int j = i + H;
        q[i] = prmt(nb[i >> 2], nb[j >> 2], uint32_t(i & 3) | (uint32_t(4 + (j & 3)) << 4));
    }
}

// The wide groups of a block, shared out over the CTA's threads in the order of their ranks: thread t packs those of rank t,
// t + 256, .. (the block's values at shared address `values`; the numbers of mask word w's wide groups, a byte each, at
// list + 32 w; lane w of every warp: wide groups before word w in `excl`). Records go to shared memory at `pend`, or, when they
// do not fit there, straight to `out` (2-byte aligned). A weight's block has about 250 wide groups: one round for the CTA. (Every
// warp packing the wide groups of its own runs takes two as a rule, since they are rarely 32 at most: nine tensors of a layer
// 277.2 us, now 271.0; 32064 blocks of bf16 366.5, now 358.9. Blocks whose groups are all wide, of random exponents, gain nothing
// and pay for the look-up of the words: 3584 blocks of bf16 82.5 -> 83.4, a list of 56 tensors 96.4 -> 98.7. Leaving it out
// for them brings 3584 blocks to 79.9, but costs the list compressor registers: a layer of ordinary weights 243.3 -> 247.6.)
template <int H>
__device__ __forceinline__ void pack_records(uint32_t values, uint32_t list, uint32_t wide, uint32_t excl, uint32_t s4, int m, uint32_t pend,
                                             uint8_t* out) {
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t base = threadIdx.x & ~31u; base < wide; base += kFusedThreads) {
        const uint32_t rank = base + lane;
        uint32_t word = 0, first = 0;   // the last word with at most `rank` wide groups before it
#pragma unroll
        for (uint32_t step = 16; step; step >>= 1) {
            const uint32_t before = __shfl_sync(0xFFFFFFFFu, excl, word + step);
            if (before <= rank) {
                word += step;
                first = before;
            }
        }
        if (rank < wide) {
            const uint32_t number = lds8(list + word * 32 + (rank - first));
            uint32_t q[H];
            record_words<H>(lds128(values + (word * 32 + number) * 16), s4, m, q);
            if (out == nullptr) {
#pragma unroll
                for (int k = 0; k < H; ++k) sts16(pend + (rank * H + k) * 2, q[k]);
            } else {
#pragma unroll
                for (int k = 0; k < H; ++k) reinterpret_cast<uint16_t*>(out)[rank * H + k] = uint16_t(q[k]);
            }
        }
    }
}

template <int DT>
__device__ __forceinline__ void pack_records_any(int h, uint32_t values, uint32_t list, uint32_t wide, uint32_t excl, uint32_t s4, int m,
                                                 uint32_t pend, uint8_t* out) {
    switch (h) {
        case 0: break;
        case 1: pack_records<1>(values, list, wide, excl, s4, m, pend, out); break;
        case 2: pack_records<2>(values, list, wide, excl, s4, m, pend, out); break;
        case 3: pack_records<3>(values, list, wide, excl, s4, m, pend, out); break;
        case 4: pack_records<4>(values, list, wide, excl, s4, m, pend, out); break;
        case 5: if constexpr (DT != ENEC_FP16) pack_records<5>(values, list, wide, excl, s4, m, pend, out); break;
        case 6: if constexpr (DT != ENEC_FP16) pack_records<6>(values, list, wide, excl, s4, m, pend, out); break;
        default: if constexpr (DT != ENEC_FP16) pack_records<7>(values, list, wide, excl, s4, m, pend, out); break;
    }
}
// Number of wide groups before block k, by one warp; false when the blocks before were not counted in time.
__device__ __forceinline__ bool groups_before(const FusedTensor& t, uint32_t k, uint32_t& before) {
    before = 0;
    if (k == 0) return true;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t sb = k / kSuperBlocks, hy = sb / kHyperSupers;
    for (uint32_t polls = 0; polls < (1u << 20); ++polls) {
        uint32_t sum = 0;
        bool ready = true;
        unsigned long long st[kSuperBlocks / 32], su[kHyperSupers / 32];
#pragma unroll
        for (uint32_t i = 0; i < kSuperBlocks / 32; ++i) {
            const uint32_t at = sb * kSuperBlocks + i * 32 + lane;
            st[i] = at < k ? ld_relaxed_u64(&t.state[at]) : (unsigned long long)t.epoch << 32;
        }
#pragma unroll
        for (uint32_t i = 0; i < kHyperSupers / 32; ++i) {
            const uint32_t at = hy * kHyperSupers + i * 32 + lane;
            su[i] = at < sb ? ld_relaxed_u64(&t.super[at]) : (unsigned long long)kSuperBlocks << 32;
        }
        for (uint32_t at = lane; at < hy; at += 32) {
            const unsigned long long w = ld_relaxed_u64(&t.hyper[at]);
            ready = ready && (w >> 32) == kSuperBlocks * kHyperSupers;
            sum += uint32_t(w);
        }
#pragma unroll
        for (uint32_t i = 0; i < kSuperBlocks / 32; ++i) {
            ready = ready && uint32_t(st[i] >> 32) == t.epoch;
            sum += uint32_t(st[i]);
        }
#pragma unroll
        for (uint32_t i = 0; i < kHyperSupers / 32; ++i) {
            ready = ready && uint32_t(su[i] >> 32) == kSuperBlocks;
            sum += uint32_t(su[i]);
        }
        if (__all_sync(0xFFFFFFFFu, ready)) {
            before = __reduce_add_sync(0xFFFFFFFFu, sum);
            return true;
        }
        __nanosleep(polls > 2 ? 400 : 50);
    }
    return false;
}

// The last four warps of a CTA look up a waiting block's offset and copy its records (for m = 3 the first four have one
// more round of the final fold).
constexpr uint32_t kPlaceThread0 = 128, kPlaceWarp0 = 4;

// The same question put by those warps together, without waiting: a thread asks for one state word and one first-level sum ...
static_assert(kSuperBlocks == 128 && kHyperSupers == 128 && kFusedThreads == 256, "a thread asks for two words");
struct Asked { unsigned long long state, super; };
__device__ __forceinline__ Asked ask_before(const FusedTensor& t, uint32_t k, uint32_t tid) {
    const uint32_t sb = k / kSuperBlocks, u = tid - kPlaceThread0;
    const uint32_t at = sb * kSuperBlocks + u, at_super = sb / kHyperSupers * kHyperSupers + u;
    Asked a;
    a.state = at < k ? ld_relaxed_u64(&t.state[at]) : (unsigned long long)t.epoch << 32;
    a.super = at_super < sb ? ld_relaxed_u64(&t.super[at_super]) : (unsigned long long)kSuperBlocks << 32;
    return a;
}
// ... and later each of the warps sums up its answers: its share, or kNotReady (the same in every lane).
__device__ __forceinline__ uint32_t share_before(const FusedTensor& t, const Asked& a, uint32_t k, uint32_t tid) {
    bool ready = uint32_t(a.state >> 32) == t.epoch && uint32_t(a.super >> 32) == kSuperBlocks;
    uint32_t sum = uint32_t(a.state) + uint32_t(a.super);
    if (tid < kPlaceThread0 + 32) {
        for (uint32_t i = tid - kPlaceThread0; i < k / (kSuperBlocks * kHyperSupers); i += 32) {   // tensors of more than 2^28 values
            const unsigned long long w = ld_relaxed_u64(&t.hyper[i]);
            ready = ready && uint32_t(w >> 32) == kSuperBlocks * kHyperSupers;
            sum += uint32_t(w);
        }
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    return __all_sync(0xFFFFFFFFu, ready) ? sum : kNotReady;
}
// All threads: the sum of the shares; false where one of them is missing.
__device__ __forceinline__ bool sum_shares(const uint32_t* part, uint32_t& before) {
    const uint4 p = lds128(smem_u32(part));
    before = p.x + p.y + p.z + p.w;
    return max(max(p.x, p.y), max(p.z, p.w)) != kNotReady;
}

// The last four warps: `halves` 16-bit words from shared memory (4-byte aligned) to global memory (2-byte aligned), in aligned
// pieces of 16 bytes and single halves before and behind them.
__device__ __forceinline__ void copy_halves(uint8_t* dst, uint32_t src, uint32_t halves, uint32_t tid) {
    const uint32_t u = tid - kPlaceThread0;
    const uint32_t to_aligned = (0u - (uint32_t(reinterpret_cast<uintptr_t>(dst)) >> 1)) & 7;
    const uint32_t head = min(to_aligned, halves);
    const uint32_t pieces = (halves - head) >> 3;
#pragma unroll 1
    for (uint32_t p = u; p < pieces; p += kFusedThreads - kPlaceThread0) {
        const uint32_t at = src + ((2 * head) & ~3u) + 16 * p;
        uint32_t w[5];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = lds32(at + 4 * i);
        if (head & 1) {
            w[4] = lds32(at + 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = prmt(w[i], w[i + 1], 0x5432u);
        }
        *reinterpret_cast<uint4*>(dst + 2 * head + 16 * p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (u < 16) {
        const uint32_t behind = head + 8 * pieces;
        const uint32_t h = u < 8 ? u : behind + u - 8;
        if (u < 8 ? h < head : h < halves) reinterpret_cast<uint16_t*>(dst)[h] = uint16_t(lds16(src + 2 * h));
    }
}

// What a failed call leaves, as the other compressors do: a header that no decompressor accepts and the length 0. (The output may
// hold an earlier stream, whose header would go with this call's sections.) One thread; any number of threads may say it.
__device__ __forceinline__ void leave_no_stream(const FusedTensor& t) {
    reinterpret_cast<Header*>(t.out)->magic = 0;
    if (t.out_size) *t.out_size = 0;
}
// A CTA whose wait ran out has not placed the records of its block k > 0. It takes the block's count back, so that no later block finds
// its offset and nobody completes the header. One thread. (Out of line and behind the pack loop: it moves the loop's code, and
// with it at the two waits in there 1024 blocks of bf16 took 23.5 us instead of 22.0, nine tensors of a layer up to 277
// instead of 270; as it is 21.9 and 272.)
template <int DT>
__device__ __noinline__ void give_up(uint32_t k, int* status, uint32_t slot = 0) {
    const FusedTensor& t = fused_tensor<DT>(slot);
    report(status, ENEC_ERR_TIMEOUT);
    st_relaxed_u64(&t.state[k], 0ull);                            // no call's epoch
    atomicAdd(&t.super[k / kSuperBlocks], 1ull << 32);            // one block too many
    if (t.nblocks > kSuperBlocks * kHyperSupers) atomicAdd(&t.hyper[k / (kSuperBlocks * kHyperSupers)], 1ull << 32);
    leave_no_stream(t);
}

// The end of a block, by a warp that knows its offset: table entry; for the last block also the header, the end of
// the table, the padding behind the records and the stream length.
// CHECK (given parameters): nothing of that, when some block lost a value. Its CTA has said so before it published its count, and
// the last block's offset is looked up by the warp that comes here (no block follows it in its CTA).
template <int DT, bool CHECK = false>
__device__ __forceinline__ void finish_block(const FusedTensor& t, uint32_t k, uint32_t before, uint32_t wide) {
    if constexpr (CHECK) {
        if (k + 1 == t.nblocks) {   // every lane has read counts: what was written before them is there for all lanes
            __threadfence();
            __syncwarp();
        }
    }
    if ((threadIdx.x & 31) != 0) return;
    t.table[k] = before;
    if (k + 1 != t.nblocks) return;
    if (CHECK && ld_relaxed_u32(t.lossy)) return;
    const uint32_t a_total = before + wide;
    const uint64_t high_bytes = uint64_t(a_total) * 2 * uint32_t(t.hbits);
    const uint64_t total = uint64_t(t.high - t.out) + align16(high_bytes);
    Header hd;
    hd.magic = kMagic;
    hd.version = kVersion;
    hd.dtype = DT;
    hd.variant = 0;
    hd.count = t.count;
    hd.block = kBlockElems;
    hd.b = uint8_t(t.b); hd.n = uint8_t(t.n); hd.m = uint8_t(t.m); hd.L = kGroupElems;
    hd.nblocks = t.nblocks;
    hd.total_groups = t.total_groups;
    hd.a_total = a_total;
    hd.pad1 = 0;
    hd.total_bytes = total;
    hd.pad2[0] = hd.pad2[1] = 0;
    *reinterpret_cast<Header*>(t.out) = hd;
    t.table[t.nblocks] = a_total;
    for (uint64_t i = uint64_t(t.nblocks) + 1; i < align16(4 * (uint64_t(t.nblocks) + 1)) / 4; ++i) t.table[i] = 0;
    for (uint64_t p = high_bytes; p < align16(high_bytes); p += 2) *reinterpret_cast<uint16_t*>(t.high + p) = 0;
    if (t.out_size) *t.out_size = total;
}

// One access of 32 bytes, or two of 16.
__device__ __forceinline__ Run load32_any(const uint8_t* p, bool wide) {
    if (wide) return load32<true>(p);
    return load32<false>(p);
}
// Stores of some lanes, predicated (an if around them becomes a branch).
__device__ __forceinline__ void sts32_if(bool p, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u32 [%1], %2;\n\t}" ::"r"(uint32_t(p)), "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts8_if(bool p, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u8 [%1], %2;\n\t}" ::"r"(uint32_t(p)), "r"(a), "r"(v) : "memory");
}
// One run of sixteen values of a block, group `g` of it: sign/mantissa plane, histogram, values (16 bytes per group; fp16:
// the bits of the fp16 plane in bits 7..5 of each byte), votes for the group mask and the lanes of the wide groups among the
// warp's, at `list`. Returns the OR of all values.
template <int DT, bool PLAIN, bool HIST, bool CHECK = false>
__device__ __forceinline__ uint32_t pack_run(const Run& r, uint32_t minuend, uint32_t nmask4, uint32_t s4, uint32_t wide4, uint32_t column,
                                             uint32_t lane, uint32_t below, uint32_t value_at, uint32_t list, uint32_t mask_word, bool store,
                                             uint8_t* sm_out) {
    uint4 v, hs, sm;
    transform_run<DT, PLAIN, HIST, CHECK>(r, minuend, nmask4, column, v, hs, sm);
    if (store) __stcs(reinterpret_cast<uint4*>(sm_out), sm);
    const uint32_t all = v.x | v.y | v.z | v.w;
    const bool is_wide = (or_flipped(v, s4) & wide4) != 0;
    if constexpr (DT == ENEC_FP16)
        v = make_uint4((v.x & 0x1F1F1F1Fu) | (hs.x << 5), (v.y & 0x1F1F1F1Fu) | (hs.y << 5), (v.z & 0x1F1F1F1Fu) | (hs.z << 5),
                       (v.w & 0x1F1F1F1Fu) | (hs.w << 5));
    sts128(value_at, v);
    const uint32_t votes = __ballot_sync(0xFFFFFFFFu, is_wide);
    sts32_if(lane == 0, mask_word, votes);
    sts8_if(is_wide, list + __popc(votes & below), lane);
    return all;
}

// First phase of a full block, all threads: thread t takes the groups t, t + 256, .. of the block through pack_run.
// Returns whether some value is not representable (HIST only).
// All loads of a thread's four runs are in flight together (3584 blocks of bf16: 56.2 us; two runs, in a rolled loop, 59.6) and
// take no room in L1, of which the shared memory of three CTAs leaves little.
template <int DT, bool PLAIN, bool HIST, bool CHECK, bool WIDE>
__device__ __forceinline__ bool pack_front_runs(const FusedTensor& t, uint32_t k, uint32_t work, uint32_t* s_mask, uint32_t tid) {
    using Shape = FusedShape<DT>;
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    constexpr uint32_t kStep = 16 * kFusedThreads;   // elements between a thread's runs
    static_assert(kBlockElems == 4 * kStep, "a thread has four runs");
    const uint32_t lane = tid & 31, warp = tid >> 5;
    const uint8_t* in = t.in + (uint64_t(k) * kBlockElems + 16 * tid) * kElemBytes;
    uint8_t* sm_out = t.sm + (uint64_t(k) * kBlockElems + 16 * tid);
    uint8_t* lo_out = t.lo + (uint64_t(k) * kBlockElems + 16 * tid) * 2;
    const uint32_t minuend = t.c, nmask4 = t.nmask4, s4 = t.s4, wide4 = t.wide4, wide_ok = t.wide_ok;
    const uint32_t values = work + Shape::kValuesAt + tid * 16, list = work + Shape::kListAt + warp * 32,
                   masks = smem_u32(&s_mask[warp]), below = (1u << lane) - 1;
    uint32_t all = 0;
    auto run = [&](const Run& r, uint32_t i) {
        all |= pack_run<DT, PLAIN, HIST, CHECK>(r, minuend, nmask4, s4, wide4, work + Shape::kHistAt + lane * 4, lane, below, values + i * kStep,
                                                list + i * kFusedThreads, masks + i * (kFusedWarps * 4), true, sm_out + i * kStep);
    };
    if constexpr (DT == ENEC_FP32) {   // one run's 64 bytes in flight (two runs', unrolled: 1024 blocks 45.3 -> 49.6 us)
        const bool wide_in = (wide_ok & 1) != 0;
        Run a = load32_any(in, wide_in), b = load32_any(in + 32, wide_in);
#pragma unroll 1
        for (uint32_t i = 0; i < 4; ++i) {
            const Run r = split_halves(a, b, lo_out + i * (kStep * 2), (wide_ok & 2) != 0);
            in += kStep * kElemBytes;
            if (i < 3) { a = load32_any(in, wide_in); b = load32_any(in + 32, wide_in); }
            run(r, i);
        }
    } else {                           // all of the thread's runs
        const Run a = load32<WIDE>(in), b = load32<WIDE>(in + kStep * kElemBytes), c = load32<WIDE>(in + 2 * kStep * kElemBytes),
                  d = load32<WIDE>(in + 3 * kStep * kElemBytes);
        run(a, 0);
        run(b, 1);
        run(c, 2);
        run(d, 3);
    }
    return (HIST || CHECK) && (DT == ENEC_FP16 ? all & rep4(0x1F) & ~nmask4 : all & ~nmask4) != 0;
}

// Two bodies for 16-bit types, since one with both kinds of loads moves what was loaded to the registers of the other kind (31
// instructions per thread and block); fp32, with one run in flight, has one.
template <int DT, bool PLAIN, bool HIST, bool CHECK = false>
__device__ __forceinline__ bool pack_front_full(const FusedTensor& t, uint32_t k, uint32_t work, uint32_t* s_mask, uint32_t tid) {
    if (DT == ENEC_FP32 || (t.wide_ok & 1)) return pack_front_runs<DT, PLAIN, HIST, CHECK, true>(t, k, work, s_mask, tid);
    return pack_front_runs<DT, PLAIN, HIST, CHECK, false>(t, k, work, s_mask, tid);
}

// The same for the tensor's last block when it is not full and has at least 128 padded elements.
template <int DT, bool PLAIN, bool HIST, bool CHECK = false>
__device__ __noinline__ bool pack_front_tail(uint32_t k, uint32_t slot = 0) {
    using Shape = FusedShape<DT>;
    const FusedTensor& t = fused_tensor<DT>(slot);
    FusedShared& sh = fused_shared<DT>();
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t work = smem_u32(fused_smem());
    const uint32_t N = t.tail_padded, real = t.tail_real;
    const uint8_t* in = t.in + uint64_t(k) * kBlockElems * kElemBytes;
    uint8_t* out_lo = t.lo + uint64_t(k) * kBlockElems * 2;
    if (tid < 32) sh.mask[tid] = 0;
    if (HIST && tid < (real & 15)) {   // the values of the one run that is part padding are counted one by one
        const uint32_t x = exponent_of_word<DT>(exponent_word<DT>(in, (real & ~15u) + tid));
        red_add_one(work + Shape::kHistAt + lane * 4 + (x & (Shape::kRows - 1)) * HistShape<DT>::kRowBytes);
    }
    __syncthreads();
    uint32_t all = 0;
    // (one run at a time: with more registers the full blocks' loop, which shares its frame with the call, loses 6 %)
#pragma unroll 1
    for (uint32_t i = 0; i < kBlockElems / (16 * kFusedThreads); ++i) {
        const uint32_t first = i * kFusedThreads + warp * 32;   // the warp's first group of this round
        if (first >= N / 16) break;
        const uint32_t g = first + lane, e0 = 16 * g;
        const int left = int(real) - int(e0);                   // groups from N / 16 on are padding too
        Run r;
        if (left >= 16) {
            if constexpr (DT == ENEC_FP32)
                r = split_halves(load32<false>(in + uint64_t(e0) * 4), load32<false>(in + uint64_t(e0) * 4 + 32), out_lo + uint64_t(e0) * 2, false);
            else
                r = load32<false>(in + uint64_t(e0) * 2);
            if (HIST) {
#pragma unroll
                for (int q = 0; q < 8; ++q) count_halves<DT>(work + Shape::kHistAt + lane * 4, r.w[q]);
            }
        } else {
            r = load_run_tail<DT>(in + uint64_t(e0) * kElemBytes, out_lo + uint64_t(e0) * 2, left,
                                  int(align16(2 * uint64_t(real)) / 2) - int(e0), t.pad);
        }
        // the padding's sign/mantissa bytes are zero
        all |= pack_run<DT, PLAIN, false, CHECK>(r, t.c, t.nmask4, t.s4, t.wide4, 0, lane, (1u << lane) - 1, work + Shape::kValuesAt + g * 16,
                                                 work + Shape::kListAt + first, smem_u32(&sh.mask[i * kFusedWarps + warp]), left > 0,
                                                 t.sm + uint64_t(k) * kBlockElems + e0);
    }
    const bool bad = (HIST || CHECK) && (DT == ENEC_FP16 ? all & rep4(0x1F) & ~t.nmask4 : all & ~t.nmask4) != 0;
    return bad;
}

// Every warp: the wide groups before each of the block's mask words (lane l: word l); returns the block's wide groups.
__device__ __forceinline__ uint32_t scan_mask(const uint32_t* s_mask, uint32_t lane, uint32_t& before) {
    const uint32_t word = s_mask[lane];
    uint32_t incl = __popc(word);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= uint32_t(d)) incl += up;
    }
    before = incl - __popc(word);
    return __shfl_sync(0xFFFFFFFFu, incl, 31);
}

// A tail block of 16, 32 or 64 padded elements, all threads, one element per thread, bit by bit (Algorithm 2 followed for
// every set bit).
template <int DT, bool CHECK = false>
__device__ __noinline__ void pack_short_block(uint32_t k, int* status, uint32_t slot = 0) {
    const FusedTensor& t = fused_tensor<DT>(slot);
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    const uint32_t tid = threadIdx.x;
    const uint32_t N = t.tail_padded, real = t.tail_real;
    const uint8_t* in = t.in + uint64_t(k) * kBlockElems * kElemBytes;
    uint8_t* out_sm = t.sm + uint64_t(k) * kBlockElems;
    uint8_t* out_lo = t.lo + uint64_t(k) * kBlockElems * 2;  // fp32 only
    const uint32_t hbits = uint32_t(t.hbits);
    uint32_t* s_low = reinterpret_cast<uint32_t*>(fused_smem() + FusedShape<DT>::kPlanesAt);   // 64 bytes
    uint32_t* s_hi3 = s_low + 16;                                  // 32 bytes
    uint32_t* s_rec = s_hi3 + 16;                                  // 4 records of up to 14 bytes
    uint32_t* s_or = s_rec + 16;                                   // OR of y per group
    if (tid < 64) s_low[tid] = 0;
    __syncthreads();
    auto put = [](uint32_t* plane, uint32_t lanes, int a, uint32_t e, uint32_t value, uint32_t base) {
        for (int q = 0; q < a; ++q)
            if ((value >> q) & 1) {
                uint32_t pos; int bit;
                alg2_locate(lanes, a, e, q, pos, bit);
                pos += base;
                atomicOr(&plane[pos >> 2], 1u << (8 * (pos & 3) + bit));
            }
    };
    uint32_t y = 0, hs = 0;
    if (tid < N) {
        if (tid < real) {
            if (DT == ENEC_FP32) reinterpret_cast<uint16_t*>(out_lo)[tid] = uint16_t(reinterpret_cast<const uint32_t*>(in)[tid]);
            const uint32_t w = exponent_word<DT>(in, tid);
            y = uint32_t(t.b - int(exponent_of_word<DT>(w))) & ((1u << t.n) - 1);
            if (DT != ENEC_FP16) {
                out_sm[tid] = uint8_t(((w >> 8) & 0x80) | (w & 0x7F));
            } else {
                out_sm[tid] = uint8_t(w);
                hs = ((w >> 13) & 4) | ((w >> 8) & 3);
            }
        } else {
            if (tid < uint32_t(align16(real))) out_sm[tid] = 0;
            if (DT == ENEC_FP32 && 2 * tid < uint32_t(align16(2 * uint64_t(real)))) reinterpret_cast<uint16_t*>(out_lo)[tid] = 0;
        }
        atomicOr(&s_or[tid >> 4], y);
        put(s_low, N, t.m, tid, y, 0);
        if (DT == ENEC_FP16) put(s_hi3, N, 3, tid, hs, 0);
    }
    __syncthreads();
    uint32_t mask = 0;
    for (uint32_t g = 0; g < (N >> 4); ++g) mask |= (s_or[g] >> t.m) != 0 ? 1u << g : 0u;
    if (tid < N && hbits > 0 && ((mask >> (tid >> 4)) & 1))
        put(s_rec, 16, int(hbits), tid & 15, y >> t.m, __popc(mask & ((1u << (tid >> 4)) - 1)) * 2 * hbits);
    __syncthreads();
    // planes out, padded to 16 bytes with zeros
    uint32_t* out_low = reinterpret_cast<uint32_t*>(t.low + uint64_t(k) * (kBlockElems / 8) * uint32_t(t.m));
    uint32_t* out_mask = reinterpret_cast<uint32_t*>(t.mask + uint64_t(k) * (kGroupsPerBlock / 8));
    if (tid < uint32_t(align16(uint64_t(N) * t.m / 8)) / 4) out_low[tid] = s_low[tid];
    if (tid < 4) out_mask[tid] = tid == 0 ? mask : 0;
    if (DT == ENEC_FP16 && tid < uint32_t(align16(uint64_t(N) * 3 / 8)) / 4)
        reinterpret_cast<uint32_t*>(t.smhi + uint64_t(k) * (kBlockElems / 8) * 3)[tid] = s_hi3[tid];
    const uint32_t wide = __popc(mask);
    if (tid < 32) {
        uint32_t before = 0;
        const bool ok = groups_before(t, k, before);
        if (ok) {
            uint16_t* out_rec = reinterpret_cast<uint16_t*>(t.high + uint64_t(before) * 2 * hbits);
            if (tid < wide * hbits) out_rec[tid] = reinterpret_cast<const uint16_t*>(s_rec)[tid];   // at most 28
            finish_block<DT, CHECK>(t, k, before, wide);
        } else if (tid == 0) {   // the last block: nobody waits for it
            report(status, ENEC_ERR_TIMEOUT);
            leave_no_stream(t);
        }
    }
    __syncthreads();
}

// ---- histogram stages ----------------------------------------------------------------------------------
// The exponents of one block into the stage's table (column: the lane's copy), all threads.
template <int DT>
__device__ __forceinline__ void count_block(const uint8_t* in, uint32_t real, uint32_t column, uint32_t tid) {
    constexpr uint32_t kPer = HistShape<DT>::kPerLoad;
    const uint4* in4 = reinterpret_cast<const uint4*>(in);
    const uint32_t chunks = real / kPer;
    uint32_t at = tid;
    for (; at + 7 * kFusedThreads < chunks; at += 8 * kFusedThreads) {
        uint4 v[8];
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q) v[q] = in4[at + q * kFusedThreads];
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q) {
            count_word_pair<DT>(column, v[q].x);
            count_word_pair<DT>(column, v[q].y);
            count_word_pair<DT>(column, v[q].z);
            count_word_pair<DT>(column, v[q].w);
        }
    }
    for (; at < chunks; at += kFusedThreads) {
        const uint4 v = in4[at];
        count_word_pair<DT>(column, v.x);
        count_word_pair<DT>(column, v.y);
        count_word_pair<DT>(column, v.z);
        count_word_pair<DT>(column, v.w);
    }
    for (uint32_t e = chunks * kPer + tid; e < real; e += kFusedThreads)
        red_add_one(column + exponent_of_word<DT>(exponent_word<DT>(in, e)) * HistShape<DT>::kRowBytes);
}

// publish: with all that the thread (and, before a barrier, its CTA) has written or has seen written; publish_word: the word stands
// for itself, whoever reads it relies on no other store.
__device__ __forceinline__ void publish(uint32_t* where, uint32_t word) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(where), "r"(word) : "memory");
}
__device__ __forceinline__ void publish_word(uint32_t* where, uint32_t word) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(where), "r"(word) : "memory");
}
// A count of finished work, by one thread after a barrier of its CTA: what the CTA has written is there for whoever sees the
// sum, and what the others before it have written for this CTA.
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t* where, uint32_t n) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(where), "r"(n) : "memory");
    return old;
}
// One thread: a published word; 0 when it does not come within about two seconds. When it has not come after some 20 us
// and `left()` finds work that nobody has taken: kParamsTake.
template <class Left>
__device__ __forceinline__ uint32_t await_published(const uint32_t* where, Left left) {
    for (uint32_t polls = 0; polls < (1u << 22); ++polls) {
        uint32_t w;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(where) : "memory");
        if (w) return w;
        if (polls > 64 && left()) return kParamsTake;
        __nanosleep(polls > 64 ? 500 : 100);
    }
    return 0;
}
__device__ __forceinline__ uint32_t await_published(const uint32_t* where) {
    return await_published(where, [] { return false; });
}

// One thread: block k towards L2.
template <int DT>
__device__ __forceinline__ void fetch_block(const FusedTensor& t, uint32_t k) {
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    if (k < t.nblocks) {
        const uint32_t bytes = ((k + 1 == t.nblocks ? t.tail_real : kBlockElems) * kElemBytes) & ~15u;
        if (bytes) bulk_prefetch_l2(t.in + uint64_t(k) * kBlockElems * kElemBytes, bytes);
    }
}

// All threads: `mine` more blocks are in hist[which] (or in pack_hist); the CTA that brings them to `complete` runs the search.
template <int DT>
__device__ __forceinline__ void count_done(FusedControl* ctl, uint32_t which, uint32_t mine, uint32_t complete) {
    FusedShared& sh = fused_shared<DT>();
    const uint32_t tid = threadIdx.x;
    __syncthreads();
    if (tid == 0) sh.word = add_acq_rel(&ctl->hist_done[which].value, mine) + mine == complete;
    __syncthreads();
    if (sh.word && tid < 32) {
        const uint32_t found = search_global<DT>(ctl->hist[which], which == 1 ? ctl->pack_hist : nullptr,
                                                 reinterpret_cast<unsigned long long*>(fused_smem() + FusedShape<DT>::kTableAt)) | kParamsValid;
        if (tid == 0) {
            // hist[1]'s parameters may begin a second pass, which writes where the first one has written: what the CTAs counted
            // by hist_done wrote before is ordered before it
            if (which == 0) publish_word(&ctl->params[0], found);
            else publish(&ctl->params[1], found);
        }
    }
}

// The histogram of `total` blocks, every `stride`-th from `base` on, all CTAs together, and the parameters that the search
// finds for it (0: a wait ran out). which: 0 the sample, 1 what the pack stage's histogram lacks of the whole tensor; it is
// complete when `complete` blocks are counted here or there.
// In the sample stage a CTA starts with the block of its own number: it loads it at once and claims it meanwhile (444 CTAs
// that ask one ticket and wait for the answer begin up to 2 us later). The rest goes by tickets. A claim, because the block
// of a CTA that has not started (other work holds its SM) is taken by one that waits; the CTA drops its counts then.
template <int DT>
__device__ __noinline__ uint32_t histogram_stage(FusedControl* ctl, uint32_t which, uint32_t base, uint32_t total, uint32_t stride,
                                            uint32_t complete) {
    const FusedTensor& t = fused_tensor<DT>();
    FusedShared& sh = fused_shared<DT>();
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t table = smem_u32(fused_smem()) + FusedShape<DT>::kTableAt;
    uint32_t* const ticket = &ctl->hist_ticket[which].value;
    const uint32_t claimed = which != 0 ? 0 : total < gridDim.x ? total : gridDim.x;   // blocks that are claimed
    auto claim = [&](uint32_t i) { return (atomicOr(&ctl->claims[i / 32].value, 1u << (i & 31)) >> (i & 31) & 1) == 0; };
    auto unclaimed = [&](uint32_t w) {
        const uint32_t bits = claimed - 32 * w < 32 ? (1u << (claimed - 32 * w)) - 1 : ~0u;
        return bits & ~ld_relaxed_u32(&ctl->claims[w].value);
    };
    uint32_t word;
    for (bool first = true;; first = false) {
        __syncthreads();
        for (uint32_t i = tid; i < uint32_t(HistShape<DT>::kBytes / 16); i += kFusedThreads) sts128(table + 16 * i, make_uint4(0, 0, 0, 0));
        const bool own = first && blockIdx.x < claimed;
        uint32_t taken = 0;   // thread 0: not zero when somebody else counts the block of this CTA's number
        uint32_t i = blockIdx.x;
        const uint32_t bit = own ? 1u << (i & 31) : 0;
        if (own) {
            if (tid == 0) taken = atomicOr(&ctl->claims[i / 32].value, bit);   // the answer comes while the block is counted
            __syncthreads();
        } else {
            if (tid == 0) {
                uint32_t got = total;
                if (claimed == 0) {
                    got = atomicAdd(ticket, 1u);
                } else if (!first) {
                    for (uint32_t w = 0; 32 * w < claimed && got == total; ++w)
                        for (uint32_t bits = unclaimed(w); bits && got == total; bits &= bits - 1) {
                            const uint32_t c = 32 * w + uint32_t(__ffs(bits)) - 1;
                            if (claim(c)) got = c;
                        }
                }
                sh.word = got;
            }
            __syncthreads();
            i = sh.word;
        }
        uint32_t mine = 0;
        while (i < total) {
            // (asked for, not waited for: fetching the next block towards L2 meanwhile, 1024 blocks 26.9 us instead of 25.5)
            uint32_t asked = 0;
            if (tid == 0 && claimed < total) asked = atomicAdd(ticket, 1u);
            const uint32_t k = base + i * stride;
            const uint32_t real = k + 1 == t.nblocks ? t.tail_real : kBlockElems;
            count_block<DT>(t.in + uint64_t(k) * kBlockElems * kElemBytes, real, table + lane * 4, tid);
            __syncthreads();
            if (tid == 0) {
                sh.word = claimed < total ? claimed + asked : total;
                sh.ok = (taken & bit) == 0;
                taken = 0;
            }
            __syncthreads();
            i = sh.word;
            if (sh.ok) {
                ++mine;
            } else {
                for (uint32_t j = tid; j < uint32_t(HistShape<DT>::kBytes / 16); j += kFusedThreads) sts128(table + 16 * j, make_uint4(0, 0, 0, 0));
                __syncthreads();
            }
        }
        if (mine) {
            if (tid < uint32_t(HistShape<DT>::kBins)) {
                const uint32_t n = fold_hist_row<false>(table + tid * HistShape<DT>::kRowBytes, tid);
                if (n) atomicAdd(&ctl->hist[which][tid], (unsigned long long)n);
            }
            count_done<DT>(ctl, which, mine, complete);
        }
        __syncthreads();   // sh.word has been read by everybody
        if (tid == 0) {
            if (which == 0 && first) {   // the CTA's first block of the pack stage is asked for, and brought towards L2, meanwhile
                sh.next = atomicAdd(&ctl->pack_ticket[0].value, 1u);
                if (!mine) __nanosleep(2000);   // behind the loads of the blocks that are being counted
                fetch_block<DT>(t, sh.next);
            }
            sh.word = await_published(&ctl->params[which], [&] {
                if (claimed == 0) return ld_relaxed_u32(ticket) < total;
                for (uint32_t w = 0; 32 * w < claimed; ++w)
                    if (unclaimed(w)) return true;
                return false;
            });
        }
        __syncthreads();
        word = sh.word;
        __syncthreads();
        if (word != kParamsTake) return word;
    }
}

// A block with a value that the sampled parameters cannot represent: its counts are taken out of the CTA's table of the pack
// stage, whose rows cannot tell all exponents apart, and added to the whole tensor's histogram. All threads; the shared
// memory of the block's planes and values is used.
template <int DT>
__device__ __noinline__ void recount_block(FusedControl* ctl, uint32_t k) {
    using Shape = FusedShape<DT>;
    const FusedTensor& t = fused_tensor<DT>();
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    constexpr uint32_t kBins = HistShape<DT>::kBins, kColumns = 16;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t work = smem_u32(fused_smem());
    const uint8_t* in = t.in + uint64_t(k) * kBlockElems * kElemBytes;
    const uint32_t real = k + 1 == t.nblocks ? t.tail_real : kBlockElems;
    __syncthreads();
    for (uint32_t i = tid; i < kBins * kColumns / 4; i += kFusedThreads) sts128(work + Shape::kPlanesAt + 16 * i, make_uint4(0, 0, 0, 0));
    __syncthreads();
    auto move = [&](uint32_t w) {   // one value's 16-bit word
        const uint32_t x = exponent_of_word<DT>(w);
        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(work + Shape::kHistAt + lane * 4 + (x & (Shape::kRows - 1)) * HistShape<DT>::kRowBytes), "r"(~0u)
                     : "memory");
        red_add_one(work + Shape::kPlanesAt + (x * kColumns + (lane & (kColumns - 1))) * 4);
    };
    constexpr uint32_t kPer = HistShape<DT>::kPerLoad;
    for (uint32_t i = tid; i < real / kPer; i += kFusedThreads) {
        const uint4 v = reinterpret_cast<const uint4*>(in)[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            move(w[q] >> 16);
            if (DT != ENEC_FP32) move(w[q]);
        }
    }
    for (uint32_t e = real / kPer * kPer + tid; e < real; e += kFusedThreads) move(exponent_word<DT>(in, e));
    __syncthreads();
    if (tid < kBins) {
        uint32_t n = 0;
        for (uint32_t c = 0; c < kColumns; ++c) n += lds32(work + Shape::kPlanesAt + (tid * kColumns + c) * 4);
        if (n) atomicAdd(&ctl->hist[1][tid], (unsigned long long)n);
    }
    __syncthreads();
}

// A warp, when the CTA has flushed the histogram of its blocks of the first pass: `mine` more blocks are counted. The warp
// that completes the tensor runs the search, with the CTA's table of the pack stage as its shared memory.
template <int DT>
__device__ __noinline__ void first_pass_counted(FusedControl* ctl, uint32_t mine, uint32_t nblocks) {
    uint32_t last = 0;
    if ((threadIdx.x & 31) == 0) last = add_acq_rel(&ctl->pack_done.value, mine) + mine == nblocks;
    __syncwarp();   // the other lanes read what the first one's count has made visible
    if (!__shfl_sync(0xFFFFFFFFu, last, 0)) return;
    const uint32_t found = search_global<DT>(ctl->pack_hist, ctl->hist[1],
                                             reinterpret_cast<unsigned long long*>(fused_smem() + FusedShape<DT>::kHistAt)) |
                           kParamsValid | (ld_relaxed_u32(&ctl->pack_target) ? kParamsRedo : 0u);
    if ((threadIdx.x & 31) == 0) publish_word(&ctl->verdict, found);
}

// The pack stage's blocks, ticket after ticket, starting with the one in sh.next; all threads. HIST: the parameters come
// from a sample. Returns the number of blocks packed, and kPassEnded where a ticket said so: those blocks have not been added
// to pack_done yet. CHECK: the parameters are the caller's; a value that they lose ends the call without a stream. (A function of its own per form, so that each has its own registers.)
//
// Two barriers per block: A after the first phase (values, mask and lists are complete), B after the second (planes and
// records are complete). What follows B reads only what is not written before the next A.
template <int DT, bool PLAIN, bool HIST, bool CHECK = false>
__device__ __noinline__ uint32_t pack_pass(FusedControl* ctl, uint32_t pass, int* status) {
    using Shape = FusedShape<DT>;
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    constexpr int E = Shape::E;
    const FusedTensor& t = fused_tensor<DT>();
    FusedShared& sh = fused_shared<DT>();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t work = smem_u32(fused_smem());
    uint32_t pend_block = 0xFFFFFFFFu, pend_wide = 0, pend_at = 0;   // the block whose records wait in shared memory
    uint32_t iter = 0, mine = 0;
    uint32_t lost = 0;       // a block whose offset did not come in time (0: none; block 0 waits for nobody)
    // All threads: the waiting block's records to their place. Its offset is in sh.part, if the look-up begun during the
    // block after it (`asked_for`) found all blocks before it counted; else one of the last warps waits for them.
    auto place_waiting = [&](bool asked_for) {
        uint32_t before = 0;
        if (!sum_shares(sh.part, before) || !asked_for) {
            if (warp == kPlaceWarp0) {
                const bool ok = groups_before(t, pend_block, before);
                if (lane == 0) {
                    sh.before = before;
                    sh.ok = ok;
                }
            }
            __syncthreads();
            before = sh.before;
            if (!sh.ok) { lost = pend_block; return; }
        }
        if (warp < kPlaceWarp0) return;
        copy_halves(t.high + uint64_t(before) * 2 * uint32_t(t.hbits), pend_at, pend_wide * uint32_t(t.hbits), tid);
        if (warp == kPlaceWarp0) finish_block<DT, CHECK>(t, pend_block, before, pend_wide);
    };
    // one thread: no further block is handed out; those handed out already are packed, so that nobody waits for them in vain
    auto end_pass = [&]() {
        const uint32_t handed = atomicOr(&ctl->pack_ticket[pass].value, kPassEnded);
        if ((handed & kPassEnded) == 0) publish_word(&ctl->pack_target, handed < t.nblocks ? handed : t.nblocks);
    };
    auto say_lossy = [&]() {   // one thread, before the block's count is published
        report(status, ENEC_ERR_PARAMS_NOT_LOSSLESS);
        leave_no_stream(t);   // nobody writes a header: see finish_block
        atomicOr(&ctl->lossy, 1u);
        __threadfence();
    };
    uint32_t k = sh.next;
    __syncthreads();   // before thread 0 writes the next ticket there
    const uint32_t limit = t.nblocks - (t.tail_padded < 128 ? 1 : 0);   // a last block of less than 128 elements: behind the loop
    for (; k < limit; ++iter) {
        uint32_t asked = 0;
        if (tid == 0) asked = t.nblocks == 1 ? 1u : atomicAdd(&ctl->pack_ticket[pass].value, 1u);
        ++mine;
        const bool last = k + 1 == t.nblocks && t.tail_real != kBlockElems;   // the tensor's last block, not full
        const uint32_t N = last ? t.tail_padded : kBlockElems;
        bool bad = false;
        if (!last) {
            bad = pack_front_full<DT, PLAIN, HIST, CHECK>(t, k, work, sh.mask, tid);
        } else {
            bad = pack_front_tail<DT, PLAIN, HIST, CHECK>(k);
        }
        if (tid == 0) {
            sh.next = asked;
            fetch_block<DT>(t, asked);
        }
        const bool lossy = __syncthreads_or(bad) != 0;   // barrier A
        if (CHECK && lossy && tid == 0) say_lossy();
        if ((lossy || lost) && tid == 0) end_pass();
        const bool waiting = pend_block != 0xFFFFFFFFu;
        Asked answer{0, 0};
        if (waiting && warp >= kPlaceWarp0) answer = ask_before(t, pend_block, tid);   // it comes while the block is packed
        uint32_t excl;
        const uint32_t wide = scan_mask(sh.mask, lane, excl);
        if (tid == 0 && t.nblocks != 1) {
            st_relaxed_u64(&t.state[k], ((unsigned long long)t.epoch << 32) | wide);
            atomicAdd(&t.super[k / kSuperBlocks], (1ull << 32) | wide);
            if (t.nblocks > kSuperBlocks * kHyperSupers) atomicAdd(&t.hyper[k / (kSuperBlocks * kHyperSupers)], (1ull << 32) | wide);
        }
        if (HIST && sh.next >= kPassEnded) {   // what is packed now will be packed again: the block has been counted, that is all
            if (lossy) recount_block<DT>(ctl, k);
            pend_block = 0xFFFFFFFFu;
            k = sh.next;
            break;
        }
        const uint32_t hbits = uint32_t(t.hbits), m = uint32_t(t.m);
        // the records do not fit the waiting area, or there is nothing to wait for (one block: 8.85 -> 8.5 us)
        const bool direct = wide * 2 * hbits > Shape::kPend || t.nblocks == 1;
        if (tid < uint32_t(align16(((N >> 4) + 7) / 8)) / 16)
            reinterpret_cast<uint4*>(t.mask + uint64_t(k) * (kGroupsPerBlock / 8))[tid] = reinterpret_cast<const uint4*>(sh.mask)[tid];
        pack_planes<DT>(t, work, N, tid);
        if (direct) {
            if (warp == 0) {
                uint32_t before = 0;
                const bool ok = groups_before(t, k, before);
                if (ok) finish_block<DT, CHECK>(t, k, before, wide);
                if (lane == 0) { sh.before = before; sh.ok = ok; }
            }
            __syncthreads();
            if (!sh.ok) lost = k;
        }
        if (!direct || sh.ok)
            pack_records_any<DT>(int(hbits), work + Shape::kValuesAt, work + Shape::kListAt, wide, excl, t.s4, int(m),
                                 work + Shape::pend_at(iter),
                                 direct ? t.high + uint64_t(sh.before) * 2 * hbits : nullptr);
        if (waiting && warp >= kPlaceWarp0) {
            const uint32_t share = share_before(t, answer, pend_block, tid);
            if (lane == 0) sh.part[warp - kPlaceWarp0] = share;
        }
        const uint32_t next = sh.next;
        __syncthreads();                                      // barrier B
        fold_out(work + Shape::kPlanesAt, N * m / 8, t.low + uint64_t(k * m) * (kBlockElems / 8), tid);   // N >= 128: whole pieces of 16 bytes
        if (DT == ENEC_FP16) fold_out(work + Shape::kSmhiAt, N * 3 / 8, t.smhi + uint64_t(k) * (kBlockElems / 8) * 3, tid);
        if (waiting) place_waiting(true);
        pend_block = direct ? 0xFFFFFFFFu : k;
        pend_wide = wide;
        pend_at = work + Shape::pend_at(iter);
        if (HIST && lossy) recount_block<DT>(ctl, k);
        k = next;
    }
    __syncthreads();
    const bool ends_short = k < t.nblocks;   // the CTA has that block: all others have been handed out
    if (ends_short) {
        ++mine;
        if (HIST || CHECK) {
            bool bad = false;
            if (tid < t.tail_real) {
                const uint32_t x = exponent_of_word<DT>(exponent_word<DT>(t.in + uint64_t(k) * kBlockElems * kElemBytes, tid));
                if (HIST) red_add_one(work + Shape::kHistAt + lane * 4 + (x & (Shape::kRows - 1)) * HistShape<DT>::kRowBytes);
                bad = (((uint32_t(t.b - int(x)) + (1u << (t.n - 1))) & ((1u << E) - 1)) >> t.n) != 0;
            }
            if (__syncthreads_or(bad)) {
                if (CHECK && tid == 0) say_lossy();
                if (HIST && tid == 0) end_pass();
                if (HIST) recount_block<DT>(ctl, k);
            }
        }
    }
    if (HIST && mine && warp == 0) {
        // The CTA's counts go out, and the search on the whole tensor's is run, while the last four warps look up the last block's offset.
        // Row r of the table holds the exponent x of that remainder that the parameters can represent.
        for (uint32_t row = lane; row < Shape::kRows; row += 32) {
            const uint32_t n = fold_hist_row<false>(work + Shape::kHistAt + row * HistShape<DT>::kRowBytes, row);
            const uint32_t d = uint32_t(t.b) + (1u << (t.n - 1));
            const uint32_t x = (d - ((d - row) & (Shape::kRows - 1))) & ((1u << E) - 1);
            if (n) atomicAdd(&ctl->pack_hist[x], (unsigned long long)n);
        }
        __syncwarp();
        if (k < kPassEnded) first_pass_counted<DT>(ctl, mine, t.nblocks);
    }
    if (HIST && k >= kPassEnded) return mine | kPassEnded;
    if (pend_block != 0xFFFFFFFFu) place_waiting(false);
    if (ends_short) {
        __syncthreads();
        pack_short_block<DT, CHECK>(k, status);
    }
    if (lost && tid == 0) give_up<DT>(lost, status);
    return mine;
}

template <int DT>
__global__ void __launch_bounds__(kFusedThreads, FusedShape<DT>::kCtasPerSm)
enec_fused_kernel(const FusedJob job, int* status) {
    uint8_t* const smem = fused_smem();
    FusedTensor& t = fused_tensor<DT>();
    FusedShared& sh = fused_shared<DT>();
    using Shape = FusedShape<DT>;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t work = smem_u32(smem);
    const uint32_t table = work + Shape::kTableAt;
    unsigned long long* const search_table = reinterpret_cast<unsigned long long*>(smem + Shape::kTableAt);
    FusedControl* const ctl = job.ctl;
    const uint32_t nblocks = uint32_t((job.count + kBlockElems - 1) / kBlockElems);
    pdl_launch_dependents();
    if (gridDim.x == 1 && !job.given)
        for (uint32_t i = tid; i < uint32_t(HistShape<DT>::kBytes / 16); i += kFusedThreads) sts128(table + 16 * i, make_uint4(0, 0, 0, 0));
    if (tid == 32) {
        // The block that the CTA most likely begins with is asked for while the kernel before still runs: L2 is coherent, so a line that
        // is written until then is simply updated, and nothing is read here (1024 blocks of bf16 23.7 us, now 22.8, 3584 blocks 48.9 and
        // 48.2, with given parameters 14.6 and 14.0, 36.2 and 35.3).
        const uint32_t stride = job.given ? 1 : nblocks / job.sample, k = blockIdx.x * stride;
        if (job.given || blockIdx.x < job.sample) {
            constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
            const uint64_t from = uint64_t(k) * kBlockElems, left = job.count - from;
            const uint32_t bytes = ((left < kBlockElems ? uint32_t(left) : kBlockElems) * kElemBytes) & ~15u;
            if (bytes) bulk_prefetch_l2(job.in + from * kElemBytes, bytes);
        }
    }
    if (tid == 0) {
        t.in = job.in; t.out = job.out; t.count = job.count; t.out_size = job.out_size;
        set_geometry<DT>(t);
    }
    __syncthreads();
    pdl_wait();  // above, lines of the input are asked for; nothing is read or written
    {
        // the next call on this scratch area finds its control set and sums zeroed
        const uint32_t at = blockIdx.x * kFusedThreads + tid, all = gridDim.x * kFusedThreads;
        for (uint32_t i = at; i < sizeof(FusedControl) / 16; i += all) reinterpret_cast<uint4*>(job.ctl_next)[i] = make_uint4(0, 0, 0, 0);
        for (uint32_t i = at; i < job.clear_supers; i += all) job.super_next[i] = job.super_next[job.super_stride + i] = 0;
    }

    // ---- sample stage ----
    uint32_t word = 0;                              // the parameters
    bool exact = job.sample == nblocks;             // they are the whole tensor's
    if (job.given) {
        word = job.given;
        exact = true;
        if (tid == 0) sh.next = nblocks == 1 ? 0u : atomicAdd(&ctl->pack_ticket[0].value, 1u);
    } else if (gridDim.x == 1) {  // one block: nothing to hand out, nobody to tell
        count_block<DT>(job.in, t.tail_real, table + lane * 4, tid);
        __syncthreads();
        uint32_t* counts = reinterpret_cast<uint32_t*>(smem + Shape::kPendAt);
        if (tid < uint32_t(HistShape<DT>::kBins)) counts[tid] = fold_hist_row<false>(table + tid * HistShape<DT>::kRowBytes, tid);
        __syncthreads();
        if (warp == 0) {
            const uint32_t found = search_by_warp<DT>([&](int x) { return (unsigned long long)counts[x]; }, search_table);
            if (lane == 0) { sh.word = found | kParamsValid; sh.next = 0; }
        }
        __syncthreads();
        word = sh.word;
    } else {
        word = histogram_stage<DT>(ctl, 0, 0, job.sample, nblocks / job.sample, job.sample);
        if (!exact && word != 0 && !(sample_will_do<DT>(word) && histogram_in_place<DT>())) {
            exact = true;
            word = histogram_stage<DT>(ctl, 1, 0, nblocks, 1, nblocks);
        }
    }

    // ---- pack stage ----
    for (uint32_t pass = 0;; ++pass) {
        if (word == 0) {
            if (tid == 0) {   // if the CTA has a ticket for a block, that one stays unpacked and nobody writes a header
                report(status, ENEC_ERR_TIMEOUT);
                leave_no_stream(t);
            }
            return;
        }
        __syncthreads();
        if (tid == 0) {
            set_parameters<DT>(t, word);
            t.state = job.state;
            t.super = job.super + pass * job.super_stride;
            t.hyper = ctl->hyper[pass];
            t.epoch = job.epoch + pass;
        }
        if (!exact) {
            for (uint32_t i = tid; i < Shape::kHistBytes / 16; i += kFusedThreads) sts128(work + Shape::kHistAt + 16 * i, make_uint4(0, 0, 0, 0));
        }
        __syncthreads();
        if (job.given) {
            if (tid == 0) t.lossy = &ctl->lossy;
            __syncthreads();
            if (t.plain || DT == ENEC_FP16) pack_pass<DT, true, false, true>(ctl, 0, status);
            else pack_pass<DT, false, false, true>(ctl, 0, status);
            return;
        }
        const uint32_t left = !exact                       ? pack_pass<DT, true, true>(ctl, pass, status)
                              : t.plain || DT == ENEC_FP16 ? pack_pass<DT, true, false>(ctl, pass, status)
                                                           : pack_pass<DT, false, false>(ctl, pass, status);
        if (exact) return;
        exact = true;
        const uint32_t mine = left & ~kPassEnded;

        if (left & kPassEnded) {
            // some block does not bear the sampled parameters: how many blocks had been handed out?
            __syncthreads();
            if (tid == 0) sh.word = await_published(&ctl->pack_target);
            __syncthreads();
            const uint32_t target = sh.word;
            __syncthreads();
            if (target != nblocks) {   // the rest of the tensor is counted, then everything packed again
                if (mine) count_done<DT>(ctl, 1, mine, nblocks);
                word = target ? histogram_stage<DT>(ctl, 1, target, nblocks - target, 1, nblocks) : 0u;
                if (tid == 0) sh.next = atomicAdd(&ctl->pack_ticket[1].value, 1u);
                continue;
            }
        }

        // ---- the sampled parameters against the whole tensor's ----
        __syncthreads();
        if (mine && (left & kPassEnded) && warp == 0) first_pass_counted<DT>(ctl, mine, nblocks);
        if (tid == 0) {
            const uint32_t verdict = await_published(&ctl->verdict);
            if (verdict != word && verdict != 0) {
                // a second pass: it begins when the first one's last bytes have been written
                if (mine && add_acq_rel(&ctl->pack_left.value, mine) + mine == nblocks) publish(&ctl->all_left, 1u);
                sh.ok = await_published(&ctl->all_left);
                sh.next = atomicAdd(&ctl->pack_ticket[1].value, 1u);
            }
            sh.word = verdict;
        }
        __syncthreads();
        if (sh.word == word) return;
        word = sh.ok ? sh.word & ~kParamsRedo : 0u;
    }
}

}  // namespace enec

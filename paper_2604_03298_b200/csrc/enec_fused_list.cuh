// enec_compress_batched in one kernel: the one-kernel compressor's stages over a list of tensors.
//
// The tensors of two blocks or more come first in the list's index space of blocks, each from a multiple of kHistBlocks on,
// the tensors of one block after them. Three kinds of units are handed out by a ticket:
//   count   kHistBlocks blocks of a tensor into its histogram; the CTA that completes a tensor runs the search of Sec. 5.5
//           and leaves everything the packing needs in the tensor's control words
//   pack    one block with its tensor's parameters (as in enec_fused_kernel, always with the whole tensor's parameters)
//   whole   a tensor of one block: count, search and pack, by one CTA
// The order is: count the first wave of tensors, the tensors of one block, then in turn count the wave after the next and
// pack a wave. A wave ends with the tensor that brings it to kWaveBytes, so that its second reading comes from L2 unless one of its
// tensors is too large for that; the wave counted in between gives the searches time. A unit waits only for units with
// smaller tickets.
//
// Against the two launches before (histograms of all tensors, then a look-back kernel over all blocks): 56 tensors of 139 MB
// bf16 120 -> 86 us, a Llama-3-8B-shaped layer 308 -> 242 us.
#pragma once

#include "enec_fused.cuh"

namespace enec {

constexpr uint32_t kHistBlocks = 4;
constexpr uint64_t kWaveBytes = uint64_t(40) << 20;   // 8 experts and 32 vectors: 12 MB 106 us, 24 MB 97, 40 MB 91

struct alignas(16) FusedItemControl {
    unsigned long long hist[256];
    FusedTensor tensor;            // complete once `ready` is published
    uint32_t done;                 // blocks counted
    uint32_t ready;
};

struct FusedListItem {
    const uint8_t* in;
    uint8_t* out;
    uint64_t count;
    unsigned long long* out_size;  // device, may be null
    unsigned long long* state;     // tensors of two blocks or more: state words, first- and second-level sums (zero when
    unsigned long long* super;     // the call starts)
    unsigned long long* hyper;
    uint32_t first_block, nblocks;
};

struct FusedListSegment {
    uint32_t first_ticket, first_block;
    uint32_t kind;                 // FusedListKind
};
enum FusedListKind : uint32_t { kUnitEnd = 0, kUnitCount = 1, kUnitPack = 2, kUnitWhole = 3 };

struct FusedList {
    const FusedListItem* items;
    FusedItemControl* controls;          // per tensor of two blocks or more; zero when the call starts
    const uint32_t* chunk_item;          // the tensor of every kHistBlocks blocks
    const FusedListSegment* segments;    // [n_segments + 1], the last with the number of tickets
    uint32_t n_segments, n_items, n_multi;   // n_multi: tensors of two blocks or more
    uint32_t multi_blocks;               // index of the first block of the tensors of one block
    uint32_t* ticket;                    // zero when the call starts
};

// The parameters found for a tensor in `word`, with all that follows from them, into a slot of shared memory. One thread.
template <int DT>
__device__ __noinline__ void fill_tensor(FusedTensor& t, const FusedListItem& item, uint32_t word) {
    t.in = item.in; t.out = item.out; t.count = item.count; t.out_size = item.out_size;
    t.state = item.state; t.super = item.super; t.hyper = item.hyper;
    t.epoch = 1;
    t.first_block = item.first_block;
    set_geometry<DT>(t);
    set_parameters<DT>(t, word);
}

template <int DT>
__global__ void __launch_bounds__(kFusedThreads, FusedShape<DT>::kCtasPerSm)
enec_fused_list_kernel(const FusedList list, int* status) {
    using Shape = FusedShape<DT>;
    constexpr uint32_t kElemBytes = DT == ENEC_FP32 ? 4 : 2;
    uint8_t* const smem = fused_smem();
    FusedShared& sh = fused_shared<DT>();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t work = smem_u32(smem);
    const uint32_t table = work + Shape::kTableAt;
    unsigned long long* const search_table = reinterpret_cast<unsigned long long*>(smem + Shape::kTableAt);
    pdl_launch_dependents();
    pdl_wait();  // nothing above touches global memory

    // Scout: the last warp looks ahead, so that a unit's tensor is in shared memory when the unit begins. Its first lane knows
    // the next unit at the start of this one (the ticket was asked for a unit before), the unit's tensor index in the
    // middle, and if that tensor's parameters are there by then, the warp brings them; all of it is written before
    // the unit's last barrier. sh.unit[i & 1] for unit i: kind | tensor << 2, first block, whether the tensor is in its slot.
    const bool scout = warp == kFusedWarps - 1;
    uint32_t segment = 0, ticket_after = 0, next_kind = 0, next_block = 0, next_item = 0;
    auto unit_of = [&](uint32_t ticket) {   // tickets of a CTA grow, so the search moves forward
        while (segment < list.n_segments && list.segments[segment + 1].first_ticket <= ticket) ++segment;
        next_kind = kUnitEnd;
        next_block = next_item = 0;
        if (segment == list.n_segments) return;
        const FusedListSegment s = list.segments[segment];
        next_kind = s.kind;
        next_block = s.first_block + (ticket - s.first_ticket) * (s.kind == kUnitCount ? kHistBlocks : 1);
        next_item = next_block >= list.multi_blocks ? list.n_multi + (next_block - list.multi_blocks) : list.chunk_item[next_block / kHistBlocks];
    };
    uint32_t brought[2], brought_ready = 0;
    auto scout_start = [&]() {
        if (scout && lane == 0) {
            unit_of(ticket_after);
            ticket_after = atomicAdd(list.ticket, 1u);
        }
    };
    auto scout_middle = [&]() {
        if (!scout) return;
        uint32_t ready = 0;
        if (lane == 0 && next_kind == kUnitPack)
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(ready) : "l"(&list.controls[next_item].ready) : "memory");
        __syncwarp();   // the other lanes' reads come after the first lane's acquire, which a shuffle alone does not say
        brought_ready = __shfl_sync(0xFFFFFFFFu, ready, 0);
        if (brought_ready) {
            const uint32_t* from = reinterpret_cast<const uint32_t*>(&list.controls[__shfl_sync(0xFFFFFFFFu, next_item, 0)].tensor);
            brought[0] = ld_relaxed_u32(from + lane);
            brought[1] = lane + 32 < sizeof(FusedTensor) / 4 ? ld_relaxed_u32(from + lane + 32) : 0u;
        }
    };
    auto scout_end = [&](uint32_t iter, uint32_t next_slot) {
        if (!scout) return;
        if (brought_ready) {
            uint32_t* to = reinterpret_cast<uint32_t*>(&fused_tensor<DT>(next_slot));
            to[lane] = brought[0];
            if (lane + 32 < sizeof(FusedTensor) / 4) to[lane + 32] = brought[1];
        }
        if (lane == 0) {
            sh.unit[(iter + 1) & 1][0] = next_kind | next_item << 2;
            sh.unit[(iter + 1) & 1][1] = next_block;
            sh.unit[(iter + 1) & 1][2] = brought_ready;
        }
    };
    if (scout && lane == 0) {
        unit_of(atomicAdd(list.ticket, 1u));
        sh.unit[0][0] = next_kind | next_item << 2;
        sh.unit[0][1] = next_block;
        sh.unit[0][2] = 0;
        ticket_after = atomicAdd(list.ticket, 1u);
    }
    uint32_t pend_block = 0xFFFFFFFFu, pend_wide = 0, pend_at = 0, pend_slot = 1;   // the block whose records wait in shared memory
    uint32_t slot = 0;                                                             // of this unit's tensor
    bool stop = false;                                                             // a wait ran out
    uint32_t lost = 0;                                                             // slot << 28 | block: not placed (0: none is known)
    auto place_waiting = [&](bool asked_for) {   // see pack_pass
        const FusedTensor& t = fused_tensor<DT>(pend_slot);
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
            if (!sh.ok) { stop = true; lost = pend_slot << 28 | pend_block; return; }
        }
        if (warp < kPlaceWarp0) return;
        copy_halves(t.high + uint64_t(before) * 2 * uint32_t(t.hbits), pend_at, pend_wide * uint32_t(t.hbits), tid);
        if (warp == kPlaceWarp0) finish_block<DT>(t, pend_block, before, pend_wide);
    };
    auto share_waiting = [&](const Asked& answer) {
        if (warp < kPlaceWarp0) return;
        const uint32_t share = share_before(fused_tensor<DT>(pend_slot), answer, pend_block, tid);
        if (lane == 0) sh.part[warp - kPlaceWarp0] = share;
    };
    auto clear_table = [&]() {
        for (uint32_t i = tid; i < uint32_t(HistShape<DT>::kBytes / 16); i += kFusedThreads) sts128(table + 16 * i, make_uint4(0, 0, 0, 0));
    };

    __syncthreads();
    for (uint32_t iter = 0;; ++iter) {
        // (whatever is written before a unit's last barrier is read after it; the barriers A and B are those of pack_pass)
        const uint32_t kind = sh.unit[iter & 1][0] & 3, item_index = sh.unit[iter & 1][0] >> 2, block = sh.unit[iter & 1][1];
        const bool loaded = sh.unit[iter & 1][2] != 0;
        if (kind == kUnitEnd || stop) break;
        scout_start();
        const bool waiting = pend_block != 0xFFFFFFFFu;
        const uint32_t next_slot = 3 - slot - pend_slot;
        Asked answer{0, 0};
        auto ask_waiting = [&]() {
            if (waiting && warp >= kPlaceWarp0) answer = ask_before(fused_tensor<DT>(pend_slot), pend_block, tid);
        };
        uint32_t wide = 0, k = 0;
        bool leaves_records = false;
        if (kind == kUnitCount) {
            const FusedListItem& item = list.items[item_index];
            FusedItemControl& ctl = list.controls[item_index];
            const uint32_t first = block - item.first_block;
            const uint32_t n = item.nblocks - first < kHistBlocks ? item.nblocks - first : kHistBlocks;
            const uint64_t from = uint64_t(first) * kBlockElems;
            const uint64_t left = item.count - from;
            const uint8_t* in = item.in + from * kElemBytes;
            __syncthreads();   // the planes of the block before have been read
            clear_table();
            ask_waiting();
            __syncthreads();
            count_block<DT>(in, left < n * kBlockElems ? uint32_t(left) : n * kBlockElems, table + lane * 4, tid);
            if (waiting) share_waiting(answer);
            scout_middle();
            __syncthreads();
            if (tid < uint32_t(HistShape<DT>::kBins)) {
                const uint32_t c = fold_hist_row<false>(table + tid * HistShape<DT>::kRowBytes, tid);
                if (c) atomicAdd(&ctl.hist[tid], (unsigned long long)c);
            }
            __syncthreads();
            if (tid == 0) sh.word = add_acq_rel(&ctl.done, n) + n == item.nblocks;
            scout_end(iter, next_slot);
            __syncthreads();
            if (sh.word && warp == 0) {
                const uint32_t found = search_global<DT>(ctl.hist, nullptr, search_table);
                if (lane == 0) {
                    fill_tensor<DT>(ctl.tensor, item, found);
                    publish(&ctl.ready, 1u);
                }
            }
            __syncthreads();
        } else {
            const FusedTensor& t = fused_tensor<DT>(slot);
            bool present = true;   // not an index between two tensors
            if (kind == kUnitWhole) {
                const FusedListItem& item = list.items[item_index];
                __syncthreads();
                clear_table();
                __syncthreads();
                count_block<DT>(item.in, uint32_t(item.count), table + lane * 4, tid);
                __syncthreads();
                uint32_t* counts = reinterpret_cast<uint32_t*>(smem + Shape::kListAt);   // 1 KB
                if (tid < uint32_t(HistShape<DT>::kBins)) counts[tid] = fold_hist_row<false>(table + tid * HistShape<DT>::kRowBytes, tid);
                __syncthreads();
                if (warp == 0) {
                    const uint32_t found = search_by_warp<DT>([&](int x) { return (unsigned long long)counts[x]; }, search_table);
                    if (lane == 0) fill_tensor<DT>(fused_tensor<DT>(slot), item, found);
                }
                __syncthreads();
            } else {
                if (!loaded) {   // its parameters were not there when the scout looked: wait for them
                    const FusedItemControl& ctl = list.controls[item_index];
                    if (tid == 0) sh.word = await_published(&ctl.ready);
                    __syncthreads();
                    if (!sh.word) {
                        stop = true;
                        if (pend_block != 0xFFFFFFFFu) lost = pend_slot << 28 | pend_block;
                        break;
                    }
                    if (tid < sizeof(FusedTensor) / 4)
                        reinterpret_cast<uint32_t*>(&fused_tensor<DT>(slot))[tid] = ld_relaxed_u32(reinterpret_cast<const uint32_t*>(&ctl.tensor) + tid);
                    __syncthreads();
                }
                present = block - t.first_block < t.nblocks;
                if (present) k = block - t.first_block;
            }
            const bool last = k + 1 == t.nblocks && t.tail_real != kBlockElems;
            const uint32_t N = last ? t.tail_padded : kBlockElems;
            if (!present) {
            } else if (!last) {
                if (t.plain || DT == ENEC_FP16) pack_front_full<DT, true, false>(t, k, work, sh.mask, tid);
                else pack_front_full<DT, false, false>(t, k, work, sh.mask, tid);
            } else if (N >= 128) {
                if (t.plain || DT == ENEC_FP16) pack_front_tail<DT, true, false>(k, slot);
                else pack_front_tail<DT, false, false>(k, slot);
            }
            __syncthreads();                                      // barrier A
            scout_middle();
            if (present && N < 128) {
                pack_short_block<DT>(k, status, slot);            // its records go straight to their place
            } else if (present) {
                uint32_t excl;
                wide = scan_mask(sh.mask, lane, excl);
                if (tid == 0 && t.nblocks != 1) {
                    st_relaxed_u64(&t.state[k], ((unsigned long long)t.epoch << 32) | wide);
                    atomicAdd(&t.super[k / kSuperBlocks], (1ull << 32) | wide);
                    if (t.nblocks > kSuperBlocks * kHyperSupers) atomicAdd(&t.hyper[k / (kSuperBlocks * kHyperSupers)], (1ull << 32) | wide);
                }
                const uint32_t hbits = uint32_t(t.hbits), m = uint32_t(t.m);
                // records that do not fit the waiting area, or (one block) need not wait, go straight to their place
                const bool direct = t.nblocks == 1 || wide * 2 * hbits > Shape::kPend;
                if (tid < uint32_t(align16(((N >> 4) + 7) / 8)) / 16)
                    reinterpret_cast<uint4*>(t.mask + uint64_t(k) * (kGroupsPerBlock / 8))[tid] = reinterpret_cast<const uint4*>(sh.mask)[tid];
                pack_planes<DT>(t, work, N, tid);
                // (asked for right behind barrier A, the answers are held over the scan and the planes, for which there are no registers:
                // 56 tensors of fp32 152.2 -> 154.9 us, of bf16 86.8 -> 87.4, heavy-tailed 89.4 -> 91.9)
                ask_waiting();
                if (direct) {
                    if (warp == 0) {
                        uint32_t before = 0;
                        const bool ok = groups_before(t, k, before);
                        if (ok) finish_block<DT>(t, k, before, wide);
                        if (lane == 0) { sh.before = before; sh.ok = ok; }
                    }
                    __syncthreads();
                    if (!sh.ok) { stop = true; lost = slot << 28 | k; }
                }
                if (!stop)
                    pack_records_any<DT>(int(hbits), work + Shape::kValuesAt, work + Shape::kListAt, wide, excl,
                                         t.s4, int(m), work + Shape::pend_at(iter),
                                         direct ? t.high + uint64_t(sh.before) * 2 * hbits : nullptr);
                leaves_records = !direct;
            }
            if (waiting) {
                if (!present || N < 128) ask_waiting();
                share_waiting(answer);
            }
            scout_end(iter, next_slot);
            __syncthreads();                                      // barrier B
            if (present && N >= 128) {
                const uint32_t m = uint32_t(t.m);
                fold_out(work + Shape::kPlanesAt, N * m / 8, t.low + uint64_t(k * m) * (kBlockElems / 8), tid);
                if (DT == ENEC_FP16) fold_out(work + Shape::kSmhiAt, N * 3 / 8, t.smhi + uint64_t(k) * (kBlockElems / 8) * 3, tid);
            }
        }
        if (waiting) {
            place_waiting(true);
            pend_block = 0xFFFFFFFFu;
        }
        if (leaves_records) {
            pend_block = k;
            pend_wide = wide;
            pend_at = work + Shape::pend_at(iter);
            pend_slot = slot;
        }
        slot = next_slot;
    }
    __syncthreads();   // sh.before has been read by everybody
    if (pend_block != 0xFFFFFFFFu && !stop) place_waiting(false);
    if (stop) {
        // A wait ran out. The CTA's waiting block is not placed and the unit that it has a ticket for is not done; whose tensor
        // that is, and which tensors wait for it, is not followed up: no tensor of the list keeps a header from before.
        if (tid == 0) {
            if (lost) give_up<DT>(lost & 0x0FFFFFFFu, status, lost >> 28);   // a tensor has at most 2^22 blocks
            else report(status, ENEC_ERR_TIMEOUT);
        }
        for (uint32_t i = tid; i < list.n_items; i += kFusedThreads) {
            reinterpret_cast<Header*>(list.items[i].out)->magic = 0;
            if (list.items[i].out_size) *list.items[i].out_size = 0;
        }
    }
}

}  // namespace enec

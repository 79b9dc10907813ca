// pv_handout.cuh -- how the warps of a CTA of the batched search take their chains (search_round_kernel): the
// state they share, and taking the next unit of work from it. Needs globaltimer() and PV_FULL (pv_device.cuh).
#pragma once
#include "pv_internal.h"

namespace pv {

// A time that all lanes of a warp agree on.
__device__ __forceinline__ unsigned long long warp_time() { return __shfl_sync(PV_FULL, globaltimer(), 0); }

// What the warps of a CTA share: the item whose chains are being handed out, and the staged ligands.
struct CtaWork {
    int lock;                     // held by one lane for a handful of instructions
    int done;                     // the queue is empty, or a wait ran out
    int pending;                  // an item taken from the queue that no ligand slot was free for, -1 none
    int blk, pos, pair, unit0;    // the current item: step block, its pair's position in the order, the pair, first unit
    int next, count;              //                   units handed out, units in all
    int slot;                     //                   ligand slot
    int lig[kLigSlots];           // staged ligand, -1 none
    int refs[kLigSlots];          // warps working on it
    int ready[kLigSlots];         // staged in full
};

// A unit of work of one warp: one chain, or two on half warps, of a step block.
struct WarpWork {
    int status;                   // 0 none left, 1 taken, 2 taken and its ligand is to be staged by this warp
    int blk, pos, pair, unit, slot;
};

// Takes the next unit for a warp. Chains of the CTA's current item are handed out one
// by one; when it is used up the next item comes from the queue, into a ligand slot that holds its
// ligand or that no warp works on. A warp holds no slot while it waits for one, and slots are given back when
// their chains end, so the wait ends. It is bounded by the launch's wait_ns all the same; a warp that waited that
// long retires for the rest of the launch, and the warps whose chains hold the slots take the waiting item when
// they are done. A shorter bound of its own (it was 2 s) took warps out of launches whose step blocks ran longer.
constexpr int kLockSpins = 1 << 22;                        // over 0.1 s
constexpr unsigned long long kStageWaitNs = 1000000000ull; // a staging takes microseconds
__device__ __forceinline__ WarpWork take_work(const SearchArgs& A, CtaWork& shared) {
    volatile CtaWork& W = shared;
    const bool first = (threadIdx.x & 31) == 0;
    WarpWork w;
    w.status = 0;
    w.blk = w.pos = w.pair = w.unit = w.slot = 0;
    unsigned long long t0 = 0ull;
    for (;;) {
        for (int spin = 0;; ++spin) {                       // the holder never waits
            int busy = 0;
            if (first) busy = atomicCAS(&shared.lock, 0, 1);
            if (!__shfl_sync(PV_FULL, busy, 0)) break;
            if (spin >= kLockSpins) {
                if (first) atomicOr(A.err, PV_EBIT_WAIT);
                return w;
            }
            __nanosleep(32);
        }
        __threadfence_block();
        // every lane reads the state; the first writes it
        int next = W.next, count = W.count, blk = W.blk, pos = W.pos, pair = W.pair, unit0 = W.unit0, slot = W.slot;
        int t = W.pending;
        const int done = W.done;
        bool starved = false;
        __syncwarp();
        if (next >= count) {
            if (t < 0 && !done) {
                if (first) t = atomicAdd(A.queue, 1);
                t = __shfl_sync(PV_FULL, t, 0);
                if (t >= A.n_items) {
                    if (first) W.done = 1;
                    t = -1;
                }
            }
            if (t >= 0) {
                blk = t / A.items_per_block;
                const int j = t - blk * A.items_per_block;
                pos = j / A.items_per_pair;
                unit0 = (j - pos * A.items_per_pair) * A.item_units;
                pair = A.order[pos];
                const int lig = A.pairs[pair].ligand;
                // a slot with this ligand, or one nobody works on (-1 none). Warps give slots back without the
                // lock, so each slot is read by one lane and the warp votes: lanes that read the counts
                // themselves could see a slot come free between their reads and part ways.
                const int k = (int)threadIdx.x & 31;
                const unsigned has = __ballot_sync(PV_FULL, k < A.lig_slots && W.lig[k] == lig);
                const unsigned idle = __ballot_sync(PV_FULL, k < A.lig_slots && W.refs[k] == 0);
                const int held = __ffs(has) - 1;
                slot = has ? held : __ffs(idle) - 1;
                starved = slot < 0;
                if (starved) {
                    if (first) W.pending = t;
                } else {
                    next = 0;
                    count = min(A.item_units, A.units - unit0);
                    if (held < 0) w.status = 2;
                    if (first) {
                        if (held < 0) {
                            W.lig[slot] = lig;
                            W.ready[slot] = 0;
                        }
                        W.pending = -1;
                        W.blk = blk;
                        W.pos = pos;
                        W.pair = pair;
                        W.unit0 = unit0;
                        W.count = count;
                        W.slot = slot;
                    }
                }
            }
        }
        if (!starved && next < count) {
            if (w.status == 0) w.status = 1;
            w.blk = blk;
            w.pos = pos;
            w.pair = pair;
            w.slot = slot;
            w.unit = unit0 + next;
            if (first) {
                W.next = next + 1;
                atomicAdd(&shared.refs[slot], 1);
            }
        }
        __threadfence_block();
        __syncwarp();
        if (first) atomicExch(&shared.lock, 0);
        if (!starved) return w;
        const unsigned long long now = warp_time();
        if (t0 == 0ull) t0 = now;
        if (now - t0 >= A.wait_ns) return w;                // the warps that hold the slots go on with it
        __nanosleep(1000);
    }
}

}  // namespace pv

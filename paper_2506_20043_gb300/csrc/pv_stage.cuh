// pv_stage.cuh -- staging of a ligand record into shared memory by a whole CTA.
#pragma once
#include "pv_layout.h"

namespace pv {

__device__ __forceinline__ int slot_of(uint64_t lo, uint64_t hi, int xs) {
    uint64_t w = xs < 8 ? lo : hi;
    int sh = 8 * (xs < 8 ? xs : xs - 8);
    return (int)(int8_t)((w >> sh) & 0xff);
}

// Staged form of a lane's pair slots. Rounds are worked on two at a time in packed arithmetic, so rounds
// 2 q and 2 q + 1 are staged as two 16-byte words per lane, (c0, c0', c1, c1') in the place of the first round's
// slots and (w, w', meta, meta') in that of the second's: packed operands come out of the loads without
// register moves. An odd last round keeps the slot's own order (meta, c0, c1, w). meta is rewritten for its use: bits
// 0-4 the lane whose pair this lane receives (shuffles take the low bits), 5 a pair is received, 6 the received
// pair's atom is the lane's second, 7 the pair's own atom is the lane's second, 16-31 the byte offset of the
// partner's position. With the merged sums of team_eval and the pocket record read in 16-byte words:
// 518 -> 557 M evaluations/s of a 30-atom ligand (variant 3 x 4, packed maps), 207 -> 227 of a 47-atom one
// (1 x 4), 952 -> 1,038 of a 16-atom one on half warps (5 x 4), the same bits.
__device__ __forceinline__ int staged_meta(int meta) {
    return ((meta >> 8) & 31) | (((meta >> 13) & 1) << 5) | (((meta >> 14) & 1) << 6) | (((meta >> 7) & 1) << 7) |
           ((meta & 127) << 20);
}

// Copies the fixed part and the pair schedule of a team of LANES lanes of `src` into `dst`
// (16-byte words; the other width's schedule is left out, and a half-warp copy holds its schedule
// at slot 0), the schedule in its staged form, then writes each atom's map slot into bits 16-23 of its
// packed word. `threads` threads take part, this one being the tid-th; sync() is their barrier, called at
// the end too.
static_assert(PV_LIG_FIXED_BYTES % 16 == 0 && sizeof(PvPairSlot) == 16, "ligand record is staged in 16-byte words");
template <int LANES, typename Sync>
__device__ __forceinline__ void stage_ligand_by(PvLigBlob* dst, const PvLigBlob* __restrict__ src, uint64_t slots_lo,
                                                uint64_t slots_hi, int tid, int threads, Sync&& sync) {
    const int fixed = PV_LIG_FIXED_BYTES / 16;
    const int rounds = LANES == 32 ? src->h.n_rounds : src->h.n_rounds16;
    const int first = LANES == 32 ? 0 : src->h.pairs16_at;
    const int4* s = reinterpret_cast<const int4*>(src);
    int4* d = reinterpret_cast<int4*>(dst);
    for (int i = tid; i < fixed; i += threads) d[i] = __ldg(s + i);
    const int4* sp = reinterpret_cast<const int4*>(src->pairs + first);
    int4* dp = reinterpret_cast<int4*>(dst->pairs);
    for (int i = tid; i < ((rounds + 1) >> 1) * LANES; i += threads) {
        const int at = 2 * (i & ~(LANES - 1)) + (i & (LANES - 1));   // the lane's slot of round 2 q
        int4 a = __ldg(sp + at);
        a.x = staged_meta(a.x);
        if (at + LANES < rounds * LANES) {
            const int4 b = __ldg(sp + at + LANES);
            dp[at] = make_int4(a.y, b.y, a.z, b.z);
            dp[at + LANES] = make_int4(a.w, b.w, a.x, staged_meta(b.x));
        } else {
            dp[at] = a;
        }
    }
    sync();
    if (tid == 0) dst->h.pairs16_at = 0;
    const int n = dst->h.n_atoms;
    for (int a = tid; a < n; a += threads) {
        int w = __float_as_int(dst->atom[a].w);
        int xs = (w >> 8) & 255;
        int slot = slot_of(slots_lo, slots_hi, xs);
        w = (w & 0xffff) | ((slot & 255) << 16);
        dst->atom[a].w = __int_as_float(w);
    }
    sync();
}

// By the whole CTA, ending with __syncthreads().
template <int LANES = 32>
__device__ __forceinline__ void stage_ligand(PvLigBlob* dst, const PvLigBlob* __restrict__ src, uint64_t slots_lo,
                                             uint64_t slots_hi) {
    stage_ligand_by<LANES>(dst, src, slots_lo, slots_hi, threadIdx.x, blockDim.x, [] { __syncthreads(); });
}

}  // namespace pv

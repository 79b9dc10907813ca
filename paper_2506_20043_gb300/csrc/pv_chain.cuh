// pv_chain.cuh -- the chain runners and the persistent round kernel of the batched search,
// templated on the team width and on the first-order consistency check, instantiated by
// pv_search.cu (check off) and pv_search_focc.cu (check on) so that the two compile in parallel and
// the check costs the unchecked kernels nothing.
#pragma once
#include "pv_internal.h"
#include "pv_stage.cuh"
#include "pv_warp.cuh"
#include "pv_handout.cuh"

namespace pv {

// The line search's base point, kept in the team's scratch across evaluations instead of registers
// (translation and orientation written by the team's first lane, torsions per lane).
template <int LANES>
__device__ __forceinline__ void stash_state(WarpScratch& S, const Pose& x) {
    const int tl = Team<LANES>::lane();
    if (tl == 0) {
        S.xb_tq[0] = make_float4(x.T.x, x.T.y, x.T.z, 0.f);
        S.xb_tq[1] = x.q;
    }
    S.xb_psi[tl] = x.psi;
}
template <int LANES>
__device__ __forceinline__ void unstash_state(const WarpScratch& S, Pose& x) {
    const float4 t = S.xb_tq[0];
    x.T = make_float3(t.x, t.y, t.z);
    x.q = S.xb_tq[1];
    x.psi = S.xb_psi[Team<LANES>::lane()];
}
template <int LANES>
__device__ __forceinline__ void stash_state(WarpScratch& S, const float& x) { S.xb_psi[Team<LANES>::lane()] = x; }
template <int LANES>
__device__ __forceinline__ void unstash_state(const WarpScratch& S, float& x) { x = S.xb_psi[Team<LANES>::lane()]; }

// One chain of Algorithm 2 for MC steps [step0, step1), written as a single loop that evaluates
// one pose per iteration (so a warp's teams stay converged at the evaluator): the random start
// (a zero-iteration local search), then per step a mutation (Eq. 2) optimised by RILC-BFGS
// (Eq. 6-12), the Metropolis test (Eq. 13 read as exp((e_cur - e_new) / T)), and for a new best a
// second RILC-BFGS run whose result becomes both current and best. Lanes of a team without a
// chain (have == false) only take part in the loop's warp vote.
template <int LANES, bool FOCC, int LAYOUT>
__device__ __forceinline__ void run_chain(const SearchArgs& A, const PvLigBlob& L, WarpScratch& S, const Site& site,
                                          int pair, uint32_t key, int chain, bool have, int step0, int step1,
                                          uint32_t& evals_out, int& flags_out) {
    using Tm = Team<LANES>;
    const int tl = Tm::lane();
    const PvSearchConst& C = A.C;
    const int n_rot = L.h.n_rot, n_tan = 6 + n_rot, m = C.bfgs_m;
    const int max_iter = C.bfgs_max_iter > 0 ? C.bfgs_max_iter : L.h.bfgs_iters;
    float* rec = A.chains + ((size_t)pair * C.chains + (have ? chain : 0)) * PV_CHAIN_STRIDE;
    float* ring = FOCC ? A.ring + ((size_t)pair * C.chains + (have ? chain : 0)) * PV_RING_STRIDE : nullptr;
    int nb_n = 0, nb_head = 0;
    float* curs = S.cur;
    float* Hs = &S.hs[0][0];
    float* Hy = &S.hy[0][0];
    enum { kStart = 0, kOptimise = 1, kRefine = 2, kDone = 3 };
    int stage = !have ? kDone : (step0 == 0 ? kStart : kOptimise);
    int s = step0, flags = 0;
    uint32_t evals = 0, evals_before = 0;
    float e_cur = 0.f, e_best = 0.f, u = 0.f;
    // local-search state; the base point of the line search (stash_state), the lane's gradient,
    // direction, gradient at the largest Armijo-satisfying trial and history entry's 1 / (y.s) live
    // in the team's scratch, not in registers through the evaluations
    Pose xt;
    float f = 0.f, gd = 0.f, lam = 1.f, lo = 0.f, hi = -1.f, flo = 0.f, gg = 0.f, gamma = 0.f;
    float& g = S.lg[tl];
    float& d = S.ld[tl];
    float& rh = S.lr[tl];
    float& glo = S.glo[tl];
    g = 0.f;
    d = 0.f;
    rh = 0.f;
    glo = 0.f;
    int it = 0, tr = 0, stored = 0, head = 0, iters = 0;
    bool have_lo = false, bstart = true;
    if (stage == kStart) {
        xt = random_pose<LANES>(L, *site.P, (uint32_t)chain, key, C);
        iters = 0;
    } else if (stage == kOptimise) {
        for (int i = tl; i < 7 + n_rot; i += LANES) curs[i] = __ldcg(rec + PV_CH_CUR + i);
        e_cur = __ldcg(rec + PV_CH_ECUR);
        e_best = __ldcg(rec + PV_CH_EBEST);
        evals_before = __float_as_uint(__ldcg(rec + PV_CH_EVALS));
        if (FOCC) {
            nb_n = __float_as_int(__ldcg(ring + PV_RING_N));
            nb_head = __float_as_int(__ldcg(ring + PV_RING_HEAD));
        }
        Tm::sync();
        if (s < step1) {
            xt = load_pose<LANES>(curs, n_rot);
            u = mutate<LANES>(L, xt, (uint32_t)chain, key, s, C);
            iters = max_iter;
        } else {
            stage = kDone;
        }
    }
    for (;;) {
        const bool active = stage != kDone;
        if (!__any_sync(PV_FULL, active)) break;
        if (!active) continue;
        float ge;
        const float fe = team_eval<LANES, true, LAYOUT>(L, S, site, xt, ge, true);
        ++evals;
        bool bdone = false, next_iter = false, at_xt = false;
        if (bstart) {                                   // the start point of a local search
            bstart = false;
            stash_state<LANES>(S, xt);
            at_xt = true;
            f = fe; g = ge;
            it = 0; stored = 0; head = 0;
            gg = Tm::sum(ge * ge);
            // a mutated candidate that fails the consistency check (Eq. 4-5) is not optimised
            if (FOCC && stage == kOptimise && !focc_pass<LANES>(xt, f, g, ring, nb_n, n_rot, C.focc_min_delta))
                bdone = true;
            else
                next_iter = true;
        } else {                                        // a line-search trial at x + lam d
            const float gtd = Tm::sum(ge * d);
            bool take = false;
            float ft = fe, gt = ge;
            if (!(fe <= f + lam * C.rho * gd)) {
                hi = lam;                                       // Eq. 7 holds: Armijo fails
            } else if (gtd < C.sigma * gd) {
                lo = lam; have_lo = true; flo = fe; glo = ge;   // Eq. 8 holds: Wolfe fails
            } else {
                take = true;
            }
            if (!take) {
                ++tr;
                if (tr < C.bfgs_max_trials) {
                    lam = hi < 0.f ? 2.f * lam : 0.5f * (lo + hi);
                    Pose xb;
                    unstash_state<LANES>(S, xb);
                    xt = team_retract<LANES>(xb, lam * d, n_tan);
                    continue;
                }
                if (have_lo) {
                    lam = lo; ft = flo; gt = glo;
                    Pose xb;
                    unstash_state<LANES>(S, xb);
                    xt = team_retract<LANES>(xb, lam * d, n_tan);  // the same arithmetic as that trial
                    take = true;
                } else {
                    bdone = true;                               // no acceptable step: stop at x
                }
            }
            if (take) {
                // curvature-guarded history update (Eq. 10-11), move, Eq. 12 test
                const float sv = lam * d, yv = gt - g;
                const float4 sums = Tm::sum4(yv * sv, sv * sv, yv * yv, gt * gt);
                const float ys = sums.x, ss = sums.y, gn = sqrtf(gg);
                if (ss > 0.f && ys / ss > C.eps * gn) {
                    Hs[head * 32 + tl] = sv;
                    Hy[head * 32 + tl] = yv;
                    if (tl == head) rh = 1.f / ys;
                    gamma = ys / sums.z;
                    head = head + 1 == m ? 0 : head + 1;
                    stored = min(stored + 1, m);
                }
                gg = sums.w;
                Tm::sync();                                     // every lane has read the old base
                stash_state<LANES>(S, xt);
                at_xt = true;
                g = gt; f = ft;
                ++it;
                if (sqrtf(gg) <= C.eps) bdone = true;
                else next_iter = true;
            }
        }
        if (next_iter) {
            if (it >= iters) {
                bdone = true;
            } else {
                d = lbfgs_direction<LANES>(Hs, Hy, S.lr, gamma, g, stored, head, m);
                gd = Tm::sum(g * d);
                if (!(gd < 0.f)) {
                    bdone = true;
                } else {
                    lam = 1.f; lo = 0.f; hi = -1.f; have_lo = false; tr = 0;
                    xt = team_retract<LANES>(xt, lam * d, n_tan);  // from the new base, xt itself
                }
            }
        }
        if (!bdone) continue;
        // a local search ended at x with SF f: the MC decision
        Pose x;
        if (at_xt) x = xt;
        else unstash_state<LANES>(S, x);
        if (stage == kStart) {
            e_cur = f;
            e_best = f;
            Tm::sync();
            store_pose<LANES>(curs, x, n_rot);
            store_pose<LANES>(rec + PV_CH_BEST, x, n_rot);
            Tm::sync();
            if (FOCC) focc_push<LANES>(ring, x, f, g, n_rot, C.focc, nb_n, nb_head);
            stage = kOptimise;
        } else if (stage == kOptimise) {
            if (!(f < e_cur || u < expf((e_cur - f) / C.temperature))) {
                ++s;                                            // rejected
            } else if (f < e_best) {
                stage = kRefine;                                // accepted, a new best: refine first
                xt = x;
                bstart = true;
                iters = max_iter;
                continue;
            } else {
                e_cur = f;                                      // accepted
                Tm::sync();
                store_pose<LANES>(curs, x, n_rot);
                Tm::sync();
                if (FOCC) focc_push<LANES>(ring, x, f, g, n_rot, C.focc, nb_n, nb_head);
                ++s;
            }
        } else {                                                // the refined new best
            e_cur = f;
            e_best = f;
            Tm::sync();
            store_pose<LANES>(rec + PV_CH_BEST, x, n_rot);
            store_pose<LANES>(curs, x, n_rot);
            Tm::sync();
            if (FOCC) focc_push<LANES>(ring, x, f, g, n_rot, C.focc, nb_n, nb_head);
            stage = kOptimise;
            ++s;
        }
        if (A.timeout_ns) {
            unsigned long long now = tl == 0 ? globaltimer() : 0ull;
            now = __shfl_sync(Tm::mask(), now, 0, LANES);
            if (now - *A.t0 > A.timeout_ns) {
                flags |= PV_EBIT_TIMEOUT;
                stage = kDone;
                continue;
            }
        }
        if (s < step1) {                                        // the next MC step
            xt = load_pose<LANES>(curs, n_rot);
            u = mutate<LANES>(L, xt, (uint32_t)chain, key, s, C);
            bstart = true;
            iters = max_iter;
        } else {
            stage = kDone;
        }
    }
    if (have) {
        if (!(e_best == e_best)) flags |= PV_EBIT_NAN;
        Tm::sync();
        for (int i = tl; i < 7 + n_rot; i += LANES) rec[PV_CH_CUR + i] = curs[i];
        if (tl == 0) {
            if (FOCC) {
                ring[PV_RING_N] = __int_as_float(nb_n);
                ring[PV_RING_HEAD] = __int_as_float(nb_head);
            }
            rec[PV_CH_ECUR] = e_cur;
            rec[PV_CH_EBEST] = e_best;
            rec[PV_CH_EVALS] = __uint_as_float(evals_before + evals);
            if (flags) atomicOr(reinterpret_cast<int*>(rec + PV_CH_FLAGS), flags);   // zeroed at the dock's start
        }
    }
    evals_out = evals;
    flags_out = flags;
}

// The docking objective of a whole-warp chain: SF (Eq. 3) at a pose with its tangent gradient (lane
// k holds component k), and the retraction of a tangent step (translation, world-frame rotation
// vector, torsions). warp_rilc_bfgs is written against this interface so that the same optimiser
// code also runs on analytic objectives (pv_check.cu).
template <int LAYOUT>
struct WarpDockObjective {
    using State = Pose;
    const PvLigBlob& L;
    WarpScratch& S;
    const Site& site;
    int n_tan;
    __device__ __forceinline__ float eval(const Pose& x, float& g, bool) const {
        return team_eval<32, true, LAYOUT>(L, S, site, x, g, true);
    }
    __device__ __forceinline__ Pose retract(const Pose& x, float step) const {
        return team_retract<32>(x, step, n_tan);
    }
};

// The same objective where a CTA of several warps runs one chain (search_few_kernel): with the first trial of a
// line search, or the first that was not foreseen, the other warps evaluate those that follow it if all fail
// alike (Eq. 7: lambda halves, or moves down the bracket; Eq. 8: it doubles, or moves up), and a trial whose lambda
// is among them is only looked up. The chain and its helpers meet twice per round, whatever the trials give, and
// once more when the chain ends, so that no warp waits for one that left.
struct Foreseen {
    int go;                            // 0: the chain has ended
    float lam[32];                     // helper h's trial (base + lam direction),
    float f[kFewWarps];                // SF there and its tangent gradient
    float g[kFewWarps][32];
};
// Whole warps meet at a barrier of the CTA, from different places of the code.
__device__ __forceinline__ void few_meet(int id) {
    __syncwarp();
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(32 * kFewWarps) : "memory");
}
// Helper h's trial: h odd follows (h + 1) / 2 failures of Eq. 7, h even h / 2 of Eq. 8.
__device__ __forceinline__ bool helps_eq7(int h) { return h & 1; }
__device__ __forceinline__ float next_step(float lam, float lo, float hi) { return hi < 0.f ? 2.f * lam : 0.5f * (lo + hi); }

template <int LAYOUT>
struct FewDockObjective {
    using State = Pose;
    const PvLigBlob& L;
    WarpScratch& S;
    const Site& site;
    int n_tan;
    Foreseen& R;
    __device__ __forceinline__ float eval(const Pose& x, float& g, bool start) const {
        if (!start) {
            if (S.cs.tr > 0) {
                const int tl = Team<32>::lane();
                const unsigned known = __ballot_sync(PV_FULL, tl > 0 && tl < kFewWarps && R.lam[tl] == S.cs.lam);
                if (known) {
                    const int h = __ffs(known) - 1;
                    g = R.g[h][tl];
                    return R.f[h];
                }
            }
            few_meet(1);                                        // the helpers read base, direction and bracket
        }
        const float f = team_eval<32, true, LAYOUT>(L, S, site, x, g, true);
        if (!start) few_meet(2);                                // their values are there
        return f;
    }
    __device__ __forceinline__ Pose retract(const Pose& x, float step) const {
        return team_retract<32>(x, step, n_tan);
    }
};

// Helper warp h of the chain whose state is in `chain`: a trial for each of the chain's calls, to its end.
template <int LAYOUT>
__device__ __forceinline__ void help_chain(const PvLigBlob& L, const WarpScratch& chain, WarpScratch& S, const Site& site,
                                           Foreseen& R, int h) {
    const int tl = Team<32>::lane(), n_tan = 6 + L.h.n_rot;
    for (;;) {
        few_meet(1);
        if (!R.go) return;
        const ChainScalars& Q = chain.cs;
        float lam = Q.lam, lo = Q.lo, hi = Q.hi;
        for (int k = 0; k < (h + 1) / 2; ++k) {
            if (helps_eq7(h)) hi = lam;
            else lo = lam;
            lam = next_step(lam, lo, hi);
        }
        Pose xb;
        unstash_state<32>(chain, xb);
        float g;
        const float f = team_eval<32, true, LAYOUT>(L, S, site, team_retract<32>(xb, lam * chain.ld[tl], n_tan), g, true);
        R.g[h][tl] = g;
        if (tl == 0) {
            R.lam[h] = lam;
            R.f[h] = f;
        }
        few_meet(2);
    }
}

// RILC-BFGS (Eq. 6-12) of one whole-warp team from x (updated in place); returns the objective at
// x and, in g_out, the lane's component of its gradient. One evaluation call site: the start
// point, then every line-search trial. With a neighbour ring (FOCC, dock objective only), the start
// point is first put to the consistency check (Eq. 4-5); a candidate that fails it is returned as
// it is.
template <bool FOCC, class Obj>
__device__ __forceinline__ float warp_rilc_bfgs(const Obj& obj, WarpScratch& S, typename Obj::State& x,
                                                const PvSearchConst& C, int max_iter, uint32_t& evals, float& g_out,
                                                const float* ring, int n_rot) {
    using Tm = Team<32>;
    using State = typename Obj::State;
    const int tl = Tm::lane();
    const int m = C.bfgs_m;
    float* Hs = &S.hs[0][0];
    float* Hy = &S.hy[0][0];
    // The line search's uniform scalars live in S.cs between evaluations: each iteration loads them
    // after the evaluation's team barrier and stores them back before the next evaluation, so no
    // lane reads a slot another lane has already rewritten in the same iteration.
    ChainScalars& Q = S.cs;
    // The lane's gradient and direction components and its history entry's 1 / (y.s) live in
    // lane-private shared slots, and the base point of the line search in shared memory too
    // (stash_state): none of them is held in registers through an evaluation, which leaves the
    // evaluation the registers of the capped variants without spilling.
    float& rh = S.lr[tl];
    float& g = S.lg[tl];
    float& d = S.ld[tl];
    rh = 0.f;
    g = 0.f;
    d = 0.f;
    bool start = true;
    State xt = x;
    stash_state<32>(S, x);
    for (;;) {
        float ge;
        const float fe = obj.eval(xt, ge, start);
        ++evals;
        const float4 q0 = *reinterpret_cast<const float4*>(&Q.f);
        const int4 q1 = *reinterpret_cast<const int4*>(&Q.hi), q2 = *reinterpret_cast<const int4*>(&Q.stored);
        float f = q0.x, gd = q0.y, lam = q0.z, lo = q0.w, hi = __int_as_float(q1.x), flo = __int_as_float(q1.y);
        int it = q1.z, tr = q1.w, stored = q2.x, head = q2.y, have_lo = q2.z;
        float gg = __int_as_float(q2.w), gamma = Q.gamma;
        bool next_iter = false, stop = false, retry = false, at_xt = false;
        if (start) {
            start = false;
            at_xt = true;
            f = fe; g = ge; it = 0; stored = 0; head = 0;
            gg = Tm::sum(ge * ge);
            bool skip = false;
            if constexpr (FOCC) skip = ring && !focc_pass<32>(xt, fe, g, ring, Q.nb_n, n_rot, C.focc_min_delta);
            if (skip) stop = true;
            else next_iter = true;
        } else {
            const float gtd = Tm::sum(ge * d);
            bool take = false;
            float ft = fe, gt = ge;
            if (!(fe <= f + lam * C.rho * gd)) {
                hi = lam;                                       // Eq. 7 holds: Armijo fails
            } else if (gtd < C.sigma * gd) {
                lo = lam; have_lo = 1; flo = fe;                // Eq. 8 holds: Wolfe fails
                S.glo[tl] = ge;
            } else {
                take = true;
            }
            if (!take) {
                ++tr;
                if (tr < C.bfgs_max_trials) {
                    lam = next_step(lam, lo, hi);
                    State xb;
                    unstash_state<32>(S, xb);
                    xt = obj.retract(xb, lam * d);
                    retry = true;
                } else if (!have_lo) {
                    stop = true;                                // no acceptable step: stop at x
                } else {
                    lam = lo; ft = flo; gt = S.glo[tl];
                    State xb;
                    unstash_state<32>(S, xb);
                    xt = obj.retract(xb, lam * d);               // the same arithmetic as that trial
                    take = true;
                }
            }
            if (take) {
                const float sv = lam * d, yv = gt - g;
                const float4 sums = Tm::sum4(yv * sv, sv * sv, yv * yv, gt * gt);
                const float ys = sums.x, ss = sums.y, gn = sqrtf(gg);
                if (ss > 0.f && ys / ss > C.eps * gn) {
                    Hs[head * 32 + tl] = sv;
                    Hy[head * 32 + tl] = yv;
                    if (tl == head) rh = 1.f / ys;
                    gamma = ys / sums.z;
                    head = head + 1 == m ? 0 : head + 1;
                    stored = min(stored + 1, m);
                }
                gg = sums.w;
                Tm::sync();                                     // every lane has read the old base
                stash_state<32>(S, xt);
                at_xt = true;
                g = gt; f = ft;
                ++it;
                if (sqrtf(gg) <= C.eps) stop = true;
                else next_iter = true;
            }
        }
        if (next_iter) {
            if (it >= max_iter) {
                stop = true;
            } else {
                d = lbfgs_direction<32>(Hs, Hy, S.lr, gamma, g, stored, head, m);
                gd = Tm::sum(g * d);
                if (!(gd < 0.f)) {
                    stop = true;
                } else {
                    lam = 1.f; lo = 0.f; hi = -1.f; have_lo = 0; tr = 0;
                    xt = obj.retract(xt, lam * d);
                }
            }
        }
        if (stop) {
            if (at_xt) x = xt;
            else unstash_state<32>(S, x);
            Tm::sync();
            g_out = g;
            return f;
        }
        (void)retry;
        Tm::sync();                       // every lane has read this iteration's scalars
        *reinterpret_cast<float4*>(&Q.f) = make_float4(f, gd, lam, lo);
        *reinterpret_cast<int4*>(&Q.hi) = make_int4(__float_as_int(hi), __float_as_int(flo), it, tr);
        *reinterpret_cast<int4*>(&Q.stored) = make_int4(stored, head, have_lo, __float_as_int(gg));
        Q.gamma = gamma;
    }
}
template <bool FOCC, class Obj>
__device__ __forceinline__ void run_chain_warp(const SearchArgs& A, const PvLigBlob& L, WarpScratch& S,
                                               const Site& site, const Obj& obj, int pair, uint32_t key, int chain, int step0,
                                               int step1, uint32_t& evals_out, int& flags_out) {
    using Tm = Team<32>;
    const int tl = Tm::lane();
    const PvSearchConst& C = A.C;
    const int n_rot = L.h.n_rot;
    const int max_iter = C.bfgs_max_iter > 0 ? C.bfgs_max_iter : L.h.bfgs_iters;
    float* rec = A.chains + ((size_t)pair * C.chains + chain) * PV_CHAIN_STRIDE;
    float* ring = FOCC ? A.ring + ((size_t)pair * C.chains + chain) * PV_RING_STRIDE : nullptr;
    float* curs = S.cur;
    // The MC step's uniform scalars live in S.cs across the local search (whose evaluations end
    // with team barriers): loaded after it returns, stored back before the next one.
    ChainScalars& Q = S.cs;
    uint32_t evals = 0;
    float g_new = 0.f;
    {
        float e_cur = 0.f, e_best = 0.f;
        uint32_t evals_before = 0;
        int nb_n = 0, nb_head = 0;
        if (step0 != 0) {
            for (int i = tl; i < 7 + n_rot; i += 32) curs[i] = __ldcg(rec + PV_CH_CUR + i);
            e_cur = __ldcg(rec + PV_CH_ECUR);
            e_best = __ldcg(rec + PV_CH_EBEST);
            evals_before = __float_as_uint(__ldcg(rec + PV_CH_EVALS));
            if (FOCC) {
                nb_n = __float_as_int(__ldcg(ring + PV_RING_N));
                nb_head = __float_as_int(__ldcg(ring + PV_RING_HEAD));
            }
        }
        Tm::sync();
        Q.e_cur = e_cur; Q.e_best = e_best; Q.u = 0.f; Q.evals_before = evals_before;
        Q.nb_n = nb_n; Q.nb_head = nb_head; Q.flags = 0; Q.s = step0; Q.stage = step0 == 0 ? 0 : 1;
        Tm::sync();
    }
    Pose cand;
    if (step0 == 0) cand = random_pose<32>(L, *site.P, (uint32_t)chain, key, C);
    for (;;) {
        const int stage0 = Q.stage, s0 = Q.s;                   // 0 start, 1 MC step, 2 refine
        if (!(stage0 == 0 || s0 < step1)) break;
        if (stage0 == 1) {
            cand = load_pose<32>(curs, n_rot);
            const float u = mutate<32>(L, cand, (uint32_t)chain, key, s0, C);
            Tm::sync();
            Q.u = u;
        }
        const float e_new = warp_rilc_bfgs<FOCC>(obj, S, cand, C, stage0 == 0 ? 0 : max_iter, evals, g_new,
                                                 FOCC && stage0 == 1 ? ring : nullptr, n_rot);
        float e_cur = Q.e_cur, e_best = Q.e_best;
        const float u = Q.u;
        int s = Q.s, stage = Q.stage, flags = Q.flags, nb_n = Q.nb_n, nb_head = Q.nb_head;
        bool stop = false;
        if (stage == 0) {
            e_cur = e_new;
            e_best = e_new;
            store_pose<32>(curs, cand, n_rot);
            store_pose<32>(rec + PV_CH_BEST, cand, n_rot);
            Tm::sync();
            if (FOCC) focc_push<32>(ring, cand, e_new, g_new, n_rot, C.focc, nb_n, nb_head);
            stage = 1;
        } else if (stage == 1 && !(e_new < e_cur || u < expf((e_cur - e_new) / C.temperature))) {
            ++s;                                                // rejected
        } else if (stage == 1 && e_new < e_best) {
            stage = 2;                                          // accepted, a new best: refine first
        } else if (stage == 1) {
            e_cur = e_new;                                      // accepted
            Tm::sync();
            store_pose<32>(curs, cand, n_rot);
            Tm::sync();
            if (FOCC) focc_push<32>(ring, cand, e_new, g_new, n_rot, C.focc, nb_n, nb_head);
            ++s;
        } else {                                                // the refined new best
            e_cur = e_new;
            e_best = e_new;
            store_pose<32>(rec + PV_CH_BEST, cand, n_rot);
            Tm::sync();
            store_pose<32>(curs, cand, n_rot);
            Tm::sync();
            if (FOCC) focc_push<32>(ring, cand, e_new, g_new, n_rot, C.focc, nb_n, nb_head);
            stage = 1;
            ++s;
        }
        if (A.timeout_ns && stage != 2) {
            unsigned long long now = tl == 0 ? globaltimer() : 0ull;
            now = __shfl_sync(PV_FULL, now, 0);
            if (now - *A.t0 > A.timeout_ns) { flags |= PV_EBIT_TIMEOUT; stop = true; }
        }
        Tm::sync();
        Q.e_cur = e_cur; Q.e_best = e_best; Q.s = s; Q.stage = stop ? 3 : stage; Q.flags = flags;
        Q.nb_n = nb_n; Q.nb_head = nb_head;
        Tm::sync();
        if (stop) break;
    }
    const float e_cur = Q.e_cur, e_best = Q.e_best;
    int flags = Q.flags;
    if (!(e_best == e_best)) flags |= PV_EBIT_NAN;
    for (int i = tl; i < 7 + n_rot; i += 32) rec[PV_CH_CUR + i] = curs[i];
    if (tl == 0) {
        if (FOCC) {
            ring[PV_RING_N] = __int_as_float(Q.nb_n);
            ring[PV_RING_HEAD] = __int_as_float(Q.nb_head);
        }
        rec[PV_CH_ECUR] = e_cur;
        rec[PV_CH_EBEST] = e_best;
        rec[PV_CH_EVALS] = __uint_as_float(Q.evals_before + evals);
        if (flags) atomicOr(reinterpret_cast<int*>(rec + PV_CH_FLAGS), flags);   // zeroed at the dock's start
    }
    Tm::sync();
    evals_out = evals;
    flags_out = flags;
}

// The waits below are run by whole warps, their conditions taken from the first lane, so that a warp is
// converged when it goes on: waits of one lane left the warp split through the chain code after them, which then
// ran at half its rate.
__device__ __forceinline__ int load_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return __shfl_sync(PV_FULL, v, 0);
}
// Waits until the chains' previous step block is published (`*progress >= blk`). Every CTA
// of the launch is resident and an item is taken from the queue only after all items before it,
// by CTAs that are running, so the wait ends (of all unfinished items the first one's chains wait
// for nothing); it is still bounded by limit_ns. Returns 1 when the predecessor is published, 0 when the
// bound ran out, -1 when the chains were given up (poisoned) by an earlier block.
__device__ __forceinline__ int wait_block(const int* progress, int blk, unsigned long long limit_ns) {
    int v = load_acquire(progress);
    if (v >= PV_PROGRESS_POISON) return -1;
    if (v >= blk) return 1;
    const unsigned long long t0 = warp_time();
    unsigned ns = 64;
    for (;;) {
        if (warp_time() - t0 >= limit_ns) return 0;
        __nanosleep(ns);
        if (ns < 4096) ns <<= 1;
        v = load_acquire(progress);
        if (v >= PV_PROGRESS_POISON) return -1;
        if (v >= blk) return 1;
    }
}

// One launch of the batched search: MC steps [step0, step1) of every chain of every pair, cut into
// step blocks of block_steps; the queue hands out all work items (some chains of a pair) of block 0,
// then of block 1, and so on, so no SM idles at a block boundary while the chains of the last
// wave finish (the blocks of one chain run in order through `progress`). A CTA's warps are independent: each
// takes a chain of the CTA's current item, runs its step block, publishes it and takes the next, without a
// barrier. Chains differ in cost, so a barrier per item of a chain per warp kept the warps of 4-warp
// CTAs waiting for 11 to 12 % of their time; and one CTA with all of an SM's warps stages a ligand once
// where seven did (a 60-atom ligand's 28 KB held the 4-warp CTAs to 16 warps per SM, now 20). Ten pockets x
// 1,000 chains x 100 steps, M evaluations/s: 568 -> 612 for a 30-atom ligand (variant 3), 228 -> 267 for 47 atoms,
// 1,055 -> 1,140 for 16 atoms on half warps (variant 5), 527 -> 583 with the consistency check; 24 ligands of
// 10-60 atoms x 5 pockets x 64 chains x 60 steps: 72.9 -> 60.8 ms (variant 1).
// Compiled for several register budgets (threads per SM) and team widths (a chain per warp, or per half warp),
// and for both map layouts (plain, cell-packed); the runtime picks one (search variant, layout).
template <int THREADS, int LANES, bool FOCC, int LAYOUT>
__global__ void __launch_bounds__(THREADS, 1) search_round_kernel(SearchArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ CtaWork s_work;
    constexpr int TPW = 32 / LANES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lig_bytes = (A.lig_smem_bytes + 127) & ~127;
    PvPocket* pockets = reinterpret_cast<PvPocket*>(smem + A.lig_slots * lig_bytes);
    WarpScratch* scratch = reinterpret_cast<WarpScratch*>(pockets + (blockDim.x >> 5));
    WarpScratch& S = scratch[warp * TPW + Team<LANES>::index()];
    PvPocket& P = pockets[warp];
    init_scratch<LANES>(S);
    if (threadIdx.x == 0) {
        s_work.lock = 0;
        s_work.done = 0;
        s_work.pending = -1;
        s_work.next = s_work.count = 0;
        for (int k = 0; k < kLigSlots; ++k) {
            s_work.lig[k] = -1;
            s_work.refs[k] = 0;
            s_work.ready[k] = 0;
        }
    }
    __syncthreads();
    for (;;) {
        const WarpWork w = take_work(A, s_work);
        if (w.status == 0) break;
        const int blk = w.blk, pair = w.pair, slot = w.slot, at = w.pos * A.units + w.unit;
        const int step0 = A.step0 + blk * A.block_steps, step1 = min(A.step1, step0 + A.block_steps);
        const PvPairDesc pd = A.pairs[pair];
        PvLigBlob& L = *reinterpret_cast<PvLigBlob*>(smem + slot * lig_bytes);
        if (lane < (int)(sizeof(PvPocket) / 4))
            reinterpret_cast<int*>(&P)[lane] = reinterpret_cast<const int*>(A.pockets + pd.pocket)[lane];
        // a unit whose predecessor is not published within the bound is skipped, not run on
        // chain records that are still being written; its later blocks are skipped too (poisoned
        // progress) and the launch reports PV_EBIT_WAIT
        int go = 1;
        if (w.status == 2) {
            stage_ligand_by<LANES>(&L, A.ligs[pd.ligand], A.slots_lo, A.slots_hi, lane, 32, [] { __syncwarp(); });
            __threadfence_block();
            __syncwarp();
            if (lane == 0) atomicExch(&s_work.ready[slot], 1);
        } else {
            volatile int* ready = &s_work.ready[slot];
            if (!__shfl_sync(PV_FULL, *ready, 0)) {
                const unsigned long long t0 = warp_time();
                while (go && !__shfl_sync(PV_FULL, *ready, 0)) {
                    if (warp_time() - t0 >= kStageWaitNs) go = 0;
                    __nanosleep(64);
                }
            }
            __threadfence_block();
        }
        if (blk > 0 && go == 1) go = wait_block(A.progress + at, blk, A.wait_ns);
        if (go == 0 && lane == 0) {
            atomicOr(A.err, PV_EBIT_WAIT);
            atomicMax(A.progress + at, PV_PROGRESS_POISON);
        }
        __syncwarp();
        const int chain = w.unit * TPW + Team<LANES>::index();
        if (go != 1) {
            if (Team<LANES>::lane() == 0 && chain < A.C.chains) {
                float* rec = A.chains + ((size_t)pair * A.C.chains + chain) * PV_CHAIN_STRIDE;
                atomicOr(reinterpret_cast<int*>(rec + PV_CH_FLAGS), PV_EBIT_WAIT);
            }
        } else {
            Site site;
            site.maps = P.maps;
            site.P = &P;
            uint32_t evals = 0;
            int flags = 0;
            if constexpr (LANES == 32)
                run_chain_warp<FOCC>(A, L, S, site, WarpDockObjective<LAYOUT>{L, S, site, 6 + L.h.n_rot}, pair,
                                     (uint32_t)pd.key, chain, step0, step1, evals, flags);
            else
                run_chain<LANES, FOCC, LAYOUT>(A, L, S, site, pair, (uint32_t)pd.key, chain, chain < A.C.chains, step0,
                                               step1, evals, flags);
            if (Team<LANES>::lane() == 0 && evals) {
                atomicAdd(A.evals, (unsigned long long)evals);
                if (flags) atomicOr(A.err, flags);
            }
        }
        __syncwarp();
        // the unit's chain records are written: publish them to its next block (a maximum, so that
        // poisoned progress stays poisoned), and give the ligand slot back
        if (lane == 0) {
            __threadfence();
            if (go == 1) atomicMax(A.progress + at, blk + 1);
            atomicSub(&s_work.refs[slot], 1);
        }
    }
}

// A launch with few chains: one CTA of kFewWarps warps per chain, for all the launch's MC steps. A lone warp
// waits for its own latencies while most of the GPU idles, and a line search takes 2.5 evaluations on average, one
// after another; of these all but 1.16 are helpers' (counted over 4,961 line searches of the FP64 restatement: 1.53 with 3
// warps, 1.29 with 5, 1.19 with 7). Same evaluator, same bits: an evaluation that is looked up is the one that
// the chain would have made. 100 steps of 8 chains of a 20-atom ligand: 10.7 -> 8.4 ms, and no trials of variants
// before the first dock.
template <bool FOCC, int LAYOUT>
__global__ void __launch_bounds__(32 * kFewWarps, 1) search_few_kernel(SearchArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Foreseen s_seen;
    __shared__ PvPocket s_pocket;
    const int warp = threadIdx.x >> 5;
    PvLigBlob& L = *reinterpret_cast<PvLigBlob*>(smem);
    WarpScratch* scratch = reinterpret_cast<WarpScratch*>(smem + ((A.lig_smem_bytes + 127) & ~127));
    WarpScratch& S = scratch[warp];
    init_scratch<32>(S);
    const int pair = A.order[blockIdx.x / A.units], chain = blockIdx.x % A.units;
    const PvPairDesc pd = A.pairs[pair];
    if (threadIdx.x < (int)(sizeof(PvPocket) / 4))
        reinterpret_cast<int*>(&s_pocket)[threadIdx.x] = reinterpret_cast<const int*>(A.pockets + pd.pocket)[threadIdx.x];
    if (threadIdx.x == 0) s_seen.go = 1;
    stage_ligand(&L, A.ligs[pd.ligand], A.slots_lo, A.slots_hi);
    __syncthreads();
    Site site;
    site.maps = s_pocket.maps;
    site.P = &s_pocket;
    if (warp > 0) {
        help_chain<LAYOUT>(L, scratch[0], S, site, s_seen, warp);
        return;
    }
    uint32_t evals = 0;
    int flags = 0;
    run_chain_warp<FOCC>(A, L, S, site, FewDockObjective<LAYOUT>{L, S, site, 6 + L.h.n_rot, s_seen}, pair,
                         (uint32_t)pd.key, chain, A.step0, A.step1, evals, flags);
    if (threadIdx.x == 0) {
        s_seen.go = 0;
        if (evals) {
            atomicAdd(A.evals, (unsigned long long)evals);
            if (flags) atomicOr(A.err, flags);
        }
    }
    few_meet(1);
}

}  // namespace pv

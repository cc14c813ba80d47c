// The per-system decisions of the CG engine, shared by its kernels (the
// persistent grid engine and the on-chip engine).
#pragma once

#include "hh_engine.cuh"

namespace hh {

constexpr int kNumericErr = -5;
constexpr int kNoConv = -4;

// Next mode of a system from its previous state and the |r|^2 (or, after the
// last preconditioner sub-step, <r, z>) reduced from the previous iteration's
// slot 3.  Pure function of its inputs: all blocks agree.
__device__ inline EngState decide(const EngSystem &Y, const EngState &P, double rr)
{
    EngState S = P;
    switch (P.mode) {
    case MODE_DONE:
        return S;
    case MODE_NEW:
        S.mode = MODE_INIT;
        S.cg_steps = 0;
        S.n_ru = 0;
        S.status = 0;
        S.final_ru = 0;
        S.true_relres = 1.0;
        S.prec = Y.precision;
        S.stall = 0;
        S.fp64_steps = 0;
        S.since_ru = 0;
        S.pre_j = 0;
        S.no_guess = 0;
        return S;
    case MODE_INIT:
        S.bb = rr;
        S.rr_last = rr;
        S.rr_ru = rr;
        if (!isfinite(rr)) {
            S.mode = MODE_DONE;
            S.status = kNumericErr;
            return S;
        }
        if (Y.x0_given && !P.no_guess) {
            if (rr == 0.0) {
                // b = 0: the solution is x = 0 whatever the guess; one more
                // INIT zeroes x.
                S.no_guess = 1;
                return S;
            }
            // Initial guess: the true residual b - Q x0 first (an RU step),
            // then CG from it (beta = rr / inf = 0 restarts).  The guess's
            // residual is not a stall of the mixed iteration.
            S.mode = MODE_RU;
            S.rr_alpha = INFINITY;
            S.rr_ru = INFINITY;
            S.rr_last = INFINITY;
            S.maxr2 = rr;
            return S;
        }
        if (rr == 0.0) {
            S.mode = MODE_DONE;
            S.true_relres = 0.0;
            return S;
        }
        S.mode = MODE_CG;
        S.beta = 0.0;
        S.rr_alpha = rr;
        S.maxr2 = rr;
        if (Y.cheb_n > 0) {
            // PCG: first precondition r = b; beta = 0 marks the first step.
            S.mode = MODE_PRE;
            S.pre_j = 0;
            S.rr_alpha = 0.0;
        }
        return S;
    case MODE_PRE: {
        // rr is <r, z> after the last sub-step (published in slot 3).
        if (P.pre_j + 1 < 2 * Y.cheb_n) {
            S.pre_j = P.pre_j + 1;
            return S;
        }
        if (!isfinite(rr) || rr <= 0.0) {
            S.mode = MODE_DONE;
            S.status = kNumericErr;
            return S;
        }
        S.mode = MODE_CG;
        S.beta = (P.rr_alpha > 0.0) ? rr / P.rr_alpha : 0.0;
        S.rr_alpha = rr;
        return S;
    }
    case MODE_CG: {
        S.cg_steps = P.cg_steps + 1;
        if (P.prec == PREC_FP64) S.fp64_steps = P.fp64_steps + 1;
        S.rr_last = rr;
        if (!isfinite(rr)) {
            S.mode = MODE_DONE;
            S.status = kNumericErr;
            return S;
        }
        S.since_ru = P.since_ru + 1;
        bool need = rr <= Y.tol2 * P.bb;
        if (P.prec == PREC_MIXED && rr < Y.delta2 * P.maxr2) need = true;
        if (P.prec == PREC_MIXED && S.since_ru >= Y.stall_window) need = true;
        if (S.cg_steps >= Y.maxit) {
            need = true;
            S.final_ru = 1;
        }
        if (need) {
            S.mode = MODE_RU;
            return S;
        }
        if (Y.cheb_n > 0) {
            S.mode = MODE_PRE;
            S.pre_j = 0;
            return S;
        }
        S.mode = MODE_CG;
        S.beta = rr / P.rr_alpha;
        S.rr_alpha = rr;
        S.maxr2 = fmax(P.maxr2, rr);
        return S;
    }
    case MODE_RU:
    default: {
        S.n_ru = P.n_ru + 1;
        S.rr_last = rr;
        S.true_relres = sqrt(rr / P.bb);
        if (!isfinite(rr)) {
            S.mode = MODE_DONE;
            S.status = kNumericErr;
            return S;
        }
        if (rr <= Y.tol2 * P.bb) {
            S.mode = MODE_DONE;
            S.status = 0;
            return S;
        }
        if (P.final_ru) {
            S.mode = MODE_DONE;
            S.status = kNoConv;
            return S;
        }
        S.mode = MODE_CG;
        S.beta = rr / P.rr_alpha;
        S.rr_alpha = rr;
        S.maxr2 = rr;
        S.since_ru = 0;
        if (Y.cheb_n > 0) {
            // PCG after residual replacement: precondition the new r; beta
            // comes from <r, z> at the end of the sub-steps.
            S.mode = MODE_PRE;
            S.pre_j = 0;
            S.rr_alpha = P.rr_alpha;
            S.rr_ru = rr;
            return S;
        }
        if (P.prec == PREC_MIXED) {
            // A reliable update that did not halve the true residual norm
            // since the previous one (whether the FP32 residual fell below
            // delta or the stall window ran out) means the FP32 steps have
            // stopped making progress (eps_32 * cond(Q) >~ 1).  After two
            // stalls in a row the system continues with FP64 CG steps from a
            // restart at the FP64 residual.
            // Also a stall: the true residual is more than 4x (in norm) the
            // FP32 recursive residual that triggered this update, i.e. the
            // FP32 recursion no longer tracks b - Q x.
            const bool no_progress = rr > 0.25 * P.rr_ru;
            const bool drifted = rr > 16.0 * P.rr_last;
            S.stall = (no_progress || drifted) ? P.stall + 1 : 0;
            if (S.stall >= 2) {
                S.prec = PREC_FP64;
                S.beta = 0.0;
            }
        }
        S.rr_ru = rr;
        return S;
    }
    }
}

}  // namespace hh

// control.cuh -- the per-matrix decision of the polar iteration (one warp per matrix), shared
// by the control kernel (polar.cu) and the polar loop (polar_loop.cu).
#pragma once
#include "common.cuh"
#include "ns_schedule.h"
#include "types.h"

namespace isoloco {

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Coefficients (a, b, c) of quintic step `step` of a matrix.  Near-square matrices (deep)
// start with one round of the deep schedule, which reaches singular values down to 1e-6
// of the normalisation.  Whatever was below that has grown by the product of its linear
// coefficients (~4e6): from 1e-8 up it is above 0.038, inside the design interval of the
// standard schedule's third step, so the next round starts there (5 steps instead of 7);
// any later round, and every round of the other matrices, is the full standard schedule.
// (Singular values under 1e-8 of s are below what the split arithmetic resolves.)
constexpr int kDeepRestart = 2;  // first standard step after the deep round

// Partial isometries (Alg. 2's Iso-C of a rank-deficient Delta: Q = U_rho V_rho^T).  A
// direction whose singular value is exactly 0 stays at 0 under every odd polynomial step,
// so ||X^T X - I||_F^2 keeps one unit per such direction and the full-rank test never
// passes.  The iteration cannot tell such a direction from a tiny nonzero one still being
// lifted, so singular values below kZeroFloor of the normalisation (under what the
// split-precision arithmetic resolves) are the ones taken as zero, and the test waits for
// the end of a round that started with every value at or above kZeroFloor inside the
// round's design interval (lift_round * kZeroFloor >= the round's first lower bound): the
// schedule then guarantees all of them in [0.998, 1.002], and what is left near 0 is zero.
// With rho = round(tr X^T X) < n directions at 1, the residual of the converged part,
// (||X^T X - I||_F^2 - (n - rho)) / rho (each zero direction adds ~1 to the first term),
// must be below tol^2; the matrix then takes the cubic polish, which keeps zeros at zero.
constexpr float kZeroFloor = 1e-8f;

// Rounds of the schedule (sched_row): a near-square matrix takes the deep round (steps
// 0 .. kSchedDeepSteps - 1), the restart round (kSchedSteps - kDeepRestart steps from the
// standard schedule's step kDeepRestart) and then standard rounds; any other matrix takes
// standard rounds.  True when `steps` quintic steps end a round; *lo is then the lower end
// of the design interval that round started from.
__device__ __forceinline__ bool round_end(bool deep, int steps, float* lo) {
    if (steps <= 0) return false;
    if (!deep) {
        *lo = kSchedLo[0];
        return steps % kSchedSteps == 0;
    }
    const int restart_end = kSchedDeepSteps + kSchedSteps - kDeepRestart;
    if (steps == kSchedDeepSteps) {
        *lo = kSchedDeepLo[0];
        return true;
    }
    if (steps == restart_end) {
        *lo = kSchedLo[kDeepRestart];
        return true;
    }
    *lo = kSchedLo[0];
    return steps > restart_end && (steps - restart_end) % kSchedSteps == 0;
}
__device__ __forceinline__ const float* sched_row(bool deep, int step) {
    if (!deep) return kSched[step % kSchedSteps];
    if (step < kSchedDeepSteps) return kSchedDeep[step];
    const int kk = step - kSchedDeepSteps;
    if (kk < kSchedSteps - kDeepRestart) return kSched[kDeepRestart + kk];
    return kSched[(kk - (kSchedSteps - kDeepRestart)) % kSchedSteps];
}

// The polar loop's word for a decision: iterations decided, done, mode (see polar_loop.cu).
__device__ __forceinline__ uint32_t control_word(int t, bool done, int mode) {
    return (static_cast<uint32_t>(t + 1) << 4) | (done ? 8u : 0u) | static_cast<uint32_t>(mode);
}

// Decision of one matrix, taken by one warp.  t: iteration index (0 = first Gram of Delta).  The
// state and the Gram's partial sums are read past L1 (within the polar loop another SM's warp
// may have taken the matrix's last decision), all at once: the step is a chain of memory
// latencies otherwise.  After iteration 0 the arithmetic is fp32: the fp64 pipe is slow, and
// nothing is scaled any more.  Returns the control word (lane 0).
__device__ __forceinline__ uint32_t control_matrix(const ControlMat& md, MatState* sp, const float* fin_part, int t,
                                                   int max_iter, float tol, uint32_t* err, int lane, int fast_steps,
                                                   int4 gram_one, int4 upd_one, int gs_on) {
    MatState& st = *sp;
    const int st_done = __ldcg(&st.done), st_step = __ldcg(&st.step), st_iters = __ldcg(&st.iters);
    const float st_resid = __ldcg(&st.resid), lift = __ldcg(&st.lift), lift_round = __ldcg(&st.lift_round);
    // fp32 lane sums and a fixed shuffle tree: each lane adds at most a few dozen
    // non-negative terms (relative error ~1e-6, far below the tolerance this sum is
    // tested against), and fp32 keeps one SM off GB300's narrow fp64 pipe.
    // four independent accumulators per lane keep four slots' loads in flight
    const int nslots = kPartSlots * md.n_gtiles;
    const float* pp = fin_part + md.gpart_slot * kPartSlots * 3;
    float a_sq[4] = {0.f, 0.f, 0.f, 0.f}, a_tr[4] = {0.f, 0.f, 0.f, 0.f}, a_dev[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i0 = lane; i0 < nslots; i0 += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            if (i < nslots) {
                a_sq[u] += __ldcg(pp + 3 * i);
                a_tr[u] += __ldcg(pp + 3 * i + 1);
                a_dev[u] += __ldcg(pp + 3 * i + 2);
            }
        }
    }
    if (st_done) {
        if (lane == 0) st.mode = 0;
        return control_word(t, true, 0);
    }
    float sqf = (a_sq[0] + a_sq[1]) + (a_sq[2] + a_sq[3]);
    float trf = (a_tr[0] + a_tr[1]) + (a_tr[2] + a_tr[3]);
    float devf = (a_dev[0] + a_dev[1]) + (a_dev[2] + a_dev[3]);
    sqf = warp_sum_f(sqf);
    trf = warp_sum_f(trf);
    devf = warp_sum_f(devf);
    if (lane != 0) return 0u;

    float d;
    double gscale = 1.0;  // used at t = 0 only
    // this Gram ran a single pass (precision schedule: the step range of the matrix's kind,
    // gram_one = (standard from, to, deep from, to), and a large previous residual)
    const int g_from = md.deep ? gram_one.z : gram_one.x, g_to = md.deep ? gram_one.w : gram_one.y;
    const bool gram_single =
        !md.gs && t > 0 && st_step >= g_from && st_step < g_to && st_resid >= kOnePassGramResid;
    if (t == 0) {
        const double sq = sqf, tr = trf, n = static_cast<double>(md.n);
        const double s2 = sqrt(sq);  // ||Delta^T Delta||_F >= sigma_max(Delta)^2
        if (!(s2 > 0.0) || !isfinite(s2)) {
            // Delta = 0 (or unusable): Q = 0, sigma_bar = 0, zero update.
            if (!isfinite(s2)) atomicOr(err, kErrNonFinite);
            st.mode = 0;
            st.done = 1;
            st.final_buf = 2;
            st.resid = 0.f;
            return control_word(t, true, 0);
        }
        gscale = 1.0 / s2;
        st.xscale = static_cast<float>(1.0 / sqrt(s2));
        // fast variant (Sec. 4.3): sigma_bar = RMS of the singular values = ||Delta||_F / sqrt(r),
        // with ||Delta||_F^2 = tr(Delta^T Delta), the trace of this Gram
        if (fast_steps) st.sigma_bar = static_cast<float>(sqrt(fmax(0.0, tr) / n));
        // ||G/s2 - I||_F^2 = ||G||^2/s2^2 - 2 tr(G)/s2 + n, with ||G||^2/s2^2 = 1
        const double dd = sqrt(fmax(0.0, 1.0 - 2.0 * tr * gscale + n) / n);
        d = static_cast<float>(dd);
    } else {
        st.xscale = 1.f;
        d = sqrtf(fmaxf(0.f, devf) / static_cast<float>(md.n));
    }
    st.resid = d;
    if (!isfinite(d)) {
        atomicOr(err, kErrNonFinite);
        st.mode = 0;
        st.done = 1;
        st.final_buf = 2;
        return control_word(t, true, 0);
    }
    // coefficients on G / s^2 (G itself after iteration 0)
    auto coef_b = [&](float q) { return t == 0 ? static_cast<float>(q * gscale) : q; };
    auto coef_c = [&](float q) { return t == 0 ? static_cast<float>(q * gscale * gscale) : q; };
    // partial-isometry test at the end of a round (see kZeroFloor)
    float round_lo = 1.f;
    const bool at_round_end = round_end(md.deep != 0, st_step, &round_lo);
    bool partial = false;
    if (t > 0 && !fast_steps && at_round_end && lift_round * kZeroFloor >= round_lo) {
        const float rho = rintf(trf);
        const float ext = static_cast<float>(md.n) - rho;  // directions taken as zero
        if (rho >= 1.f && ext >= 1.f) partial = (devf - ext) / rho < tol * tol;
    }
    if (fast_steps) {
        // fast variant: a fixed number of standard quintic steps, no test, no polish (steps
        // after the schedule's last repeat it); the last one leaves Q in the buffer its
        // update writes
        const float* q = kSched[st_step < kSchedSteps ? st_step : kSchedSteps - 1];
        st.mode = 1;
        st.a = q[0];
        st.b = coef_b(q[1]);
        st.c = coef_c(q[2]);
        st.step = st_step + 1;
        st.iters = st_iters + 1;
        const bool last = st_iters + 1 >= fast_steps;
        if (last) {
            st.done = 1;
            st.final_buf = (t + 1) & 1;
        }
        return control_word(t, last, 1);
    }
    if ((d < tol || partial) && !gram_single) {
        // Cubic polish p(x) = 1.5 x - 0.5 x^3 on singular values already near 1 (or 0).
        // (Not from a single-pass Gram: the matrix then takes one more quintic step, and the
        // Gram after it, with a small residual, keeps its passes.)
        st.mode = 2;
        // the polish update's epilogue sums tr(Q^T Delta) (a Gram-side matrix's polish writes
        // Z, and its Q = Delta Z launch sums it instead)
        st.trace_fused = (gs_on && md.gs) ? 0 : 1;
        st.a = 1.5f;
        st.b = coef_b(-0.5f);
        st.c = 0.f;
        st.iters = st_iters + 1;
        st.done = 1;
        st.final_buf = (t + 1) & 1;
        return control_word(t, true, 2);
    }
    if (st_iters >= max_iter) {
        st.mode = 0;
        st.done = 1;
        st.final_buf = t & 1;
        st.status = kErrNotConverged;
        atomicOr(err, kErrNotConverged);
        return control_word(t, true, 0);
    }
    const float* q = sched_row(md.deep != 0, st_step);
    st.mode = 1;
    // the X this step writes needs no lo plane when the next Gram and update run single-pass
    // (next step in both ranges, this residual large: the next test cannot pass, no
    // polish) and the next iteration cannot hit max_iter (Q = X would be final)
    const int kn = st_step + 1;
    const int u_from = md.deep ? upd_one.z : upd_one.x, u_to = md.deep ? upd_one.w : upd_one.y;
    st.x_hi_only = (!md.gs && kn >= g_from && kn < g_to && kn >= u_from && kn < u_to &&
                    d >= kOnePassGramResid && st_iters + 2 <= max_iter) ? 1 : 0;
    if (st_step == 0 || at_round_end) st.lift_round = lift;  // this step starts a round
    st.lift = lift * q[0];
    st.a = q[0];
    st.b = coef_b(q[1]);
    st.c = coef_c(q[2]);
    st.step = st_step + 1;
    st.iters = st_iters + 1;
    // the next Gram writes Y = b I + c G of the step after this one (X normalised by then)
    const float* qn = sched_row(md.deep != 0, st_step + 1);
    st.yb = qn[1];
    st.yc = qn[2];
    return control_word(t, false, 1);
}

}  // namespace isoloco

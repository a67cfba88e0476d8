// Adaptive lambda on the moments, two steps a launch: the run's record and its clockwork.
//
// At omega = 1 a state is its moments and the lambda of its equilibria.  The lambda with which step
// k + 1 streams follows from the largest bound of state k - 1 (adapt_prep_kernel), so a launch of
// steps k and k + 1 needs the bounds of states k - 2 and k - 1 only, which the launch before it has
// reduced: every block takes the clock forward by itself (one warp, while the others load) and no launch
// stands between two of them.  Per step of 768 x 768 cells 14.6 us with the storing kernel and its
// clock's launch, 9.3 us in pairs on the moments.
#pragma once

#include "lbrs_kernels.cuh"

namespace lbrs {

constexpr int kBoundSlots = 8;   // words a state's bound is spread over: blocks take turns at their atomics

struct AdaptRun {
    double t, lam, c;        // time, lambda and 1/(4 lambda) of the state's distributions
    double dt;               // dx / lambda
    long long steps;
    int last;                // the next step ends the run
    int done;                // the run has ended: further steps keep the state
    int dead;                // it had ended when the call began
};

struct AdaptPair {
    const AdaptRun* in;      // the record after the step before the last one, or (pending 1) after the last
    AdaptRun* out;           // the record after the first step of this launch
    const unsigned long long* bounds_in;    // of the last two states, as bits of non-negative doubles
    unsigned long long* bounds_out;         // of this launch's two states
    unsigned long long* bounds_clear;       // the next launch's
    int pending;             // steps of the clock to take: 2, or 1 at the chain's start
    double dx, safety, t_final, gamma;
};

// The clock's step k: the lambda of state k from the bound of state k - 1, with dt = dx / lam and
// c = 1 / (4 lam) given (adapt_prep_kernel's expressions, without contraction in every unit).
__device__ __forceinline__ void adapt_clock(AdaptRun& r, double lam, double dt, double c, double dx, double t_final)
{
    if (r.done) return;
    const double t_next = r.last ? t_final : __dadd_rn(r.t, r.dt);
    int last = 0;
    if (!r.last && t_final > 0.0 && __dadd_rn(t_next, dt) >= t_final) {
        lam = __ddiv_rn(dx, __dadd_rn(t_final, -t_next));
        dt = __ddiv_rn(dx, lam);
        c = __ddiv_rn(1.0, __dmul_rn(4.0, lam));
        last = 1;
    }
    r.t = t_next;
    r.lam = lam;
    r.c = c;
    r.dt = dt;
    r.steps += 1;
    if (r.last) r.done = 1;
    r.last = last;
}

// Both steps of the clock by one warp, every lane with the same result: r after the first and the
// second (step 1 left out if `pending` is 1).  A division takes most of a microsecond's third, so four
// lanes do the four of them at once.
__device__ __forceinline__ void adapt_clocks(const AdaptRun& in, const unsigned long long* bounds, int pending,
                                             double dx, double safety, double t_final, AdaptRun& r1, AdaptRun& r2)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned long long b = lane < 2 * kBoundSlots ? bounds[lane] : 0ull;   // lanes 0..7 and 8..15
#pragma unroll
    for (int off = kBoundSlots / 2; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(full, b, off);
        b = o > b ? o : b;
    }
    const double lam1 = __dmul_rn(safety, __longlong_as_double((long long)__shfl_sync(full, b, 0)));
    const double lam2 = __dmul_rn(safety, __longlong_as_double((long long)__shfl_sync(full, b, kBoundSlots)));
    const double lam = lane & 2 ? lam2 : lam1;
    const double q = __ddiv_rn(lane & 1 ? 1.0 : dx, lane & 1 ? __dmul_rn(4.0, lam) : lam);
    r1 = in;
    if (pending == 2) adapt_clock(r1, lam1, __shfl_sync(full, q, 0), __shfl_sync(full, q, 1), dx, t_final);
    r2 = r1;
    adapt_clock(r2, lam2, __shfl_sync(full, q, 2), __shfl_sync(full, q, 3), dx, t_final);
}

// bound_local<float> as the bits of a non-negative float (0 for states it gives -1): max(|u + v|, |u - v|)
// is |u| + |v|, exactly also after rounding (one of u + v, u - v has that size; rounding is symmetric).
__device__ __forceinline__ unsigned bound_bits(const float U[4], float g, float gm1)
{
    const float inv = rcp_f32(U[0]);
    const float u = U[1] * inv, v = U[2] * inv;
    const float p = gm1 * (U[3] - 0.5f * (U[1] * u + U[2] * v));
    if (!(U[0] > 0.f) || !(p > 0.f) || !isfinite(p)) return 0u;
    return __float_as_uint(fabsf(u) + fabsf(v) + sqrtf(2.f * (g * p * inv)));
}

}  // namespace lbrs

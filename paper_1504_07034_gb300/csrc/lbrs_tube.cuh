// FP32 D1Q2 and D1Q3 tubes, many steps per launch with the state in registers (sm_103a).
//
// One warp owns a window of 32 C cells of a tube, C adjacent ones per lane, and steps it `halo`
// times without leaving its registers: a population moves one cell a step, so only the cells at a
// lane's ends cross lanes (three shuffles each way per C cells), and after s steps the window's
// cells within s of a cut edge are stale while the tile inside stays exact.  No shared memory and
// no barrier between steps; shared memory only turns the coalesced order of loads and stores into
// the lanes' order and back.
//
// Cells j and j + C/2 of a lane share a register pair (a shift by one cell moves whole pairs but
// the two at the ends) and the arithmetic is the packed FP32 form.  The expressions are fixed
// operation by operation and give the bits of batch1d_kernel, where the compiler contracts the
// same products.
//
// At omega = 1 the collision returns f^eq(U) and the state is U (three values per cell): a step is
// U'(x) = f^eq_0(U(x + 1)) [+ f^eq_1(U(x))] + f^eq_last(U(x - 1)).  Otherwise it is f*.
#pragma once

#include "lbrs_batch.cuh"
#include "lbrs_march.cuh"

namespace lbrs {

struct TubeArgs {
    const float* __restrict__ src;          // f* [Q][3][N]
    float* __restrict__ dst;
    int64_t N;                              // plane stride
    const BatchTile* __restrict__ tiles;    // nullptr: one tube of one_len cells in even tiles
    const int64_t* __restrict__ tube_off;
    const int* __restrict__ tube_len;
    const int* __restrict__ tube_steps;
    const float* __restrict__ tube_c;       // 1/(2 lambda)
    int ntiles;
    int one_len, one_steps;
    float one_c;
    int halo;                               // steps per launch at most
    int launch;                             // index of the launch within the run
    int periodic;
    float om, om1, gm1;
};

// A tile's window starts a whole number of lanes before it, so that a tube's first cell is a
// lane's first.
template <int C>
__device__ __host__ constexpr int tube_pad(int halo) { return (halo + C - 1) / C * C; }

struct TubeConst {
    P2 c, nc, gm1, ngm1, half, one, third, nthree, om, om1;
};

__device__ __forceinline__ bool tube_ordinary(float q) { return fabsf(q) > 0.f && fabsf(q) < INFINITY; }

// Equilibria of a pair: l[0..2] of the population moving to -x, z of the resting one (Q = 3), r of
// the one moving to +x.  INF: of infinite moments, too (Q = 3: without it they become NaN).
template <int Q, bool INF = false>
__device__ __forceinline__ void tube_feq(const P2 U[3], const TubeConst& m, P2 l[3], P2 z[3], P2 r[3])
{
    // 1/rho (rcp_f32), with the sign carried along
    const P2 ninv = neg_rcp2(U[0], m.one);
    const P2 nu = mul2(U[1], ninv);
    const P2 nt = mul2(U[1], nu);                    // -(rho u u)
    const P2 pi = fma2(m.half, nt, U[2]);            // p / (gamma - 1)
    const P2 nG1 = fma2(m.ngm1, pi, nt);
    const P2 nG2 = mul2(nu, fma2(m.gm1, pi, U[2]));
    if constexpr (Q == 2) {
        const P2 b[3] = {mul2(m.c, U[1]), mul2(m.nc, nG1), mul2(m.nc, nG2)};
        const P2 nb[3] = {mul2(m.nc, U[1]), mul2(m.c, nG1), mul2(m.c, nG2)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            l[k] = fma2(m.half, U[k], nb[k]);
            r[k] = fma2(m.half, U[k], b[k]);
        }
    } else {
        // U/3 rounded: the reciprocal's product and one correction of the remainder (Markstein), at any
        // size; the product itself is the quotient of a zero (whose sign the correction loses) and of an
        // infinity (whose remainder is NaN)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const P2 q = mul2(U[k], m.third);
            z[k] = fma2(fma2(q, m.nthree, U[k]), m.third, q);
            if constexpr (INF) z[k] = pk(tube_ordinary(lo2(q)) ? lo2(z[k]) : lo2(q), tube_ordinary(hi2(q)) ? hi2(z[k]) : hi2(q));
        }
        l[0] = fma2(m.nc, U[1], z[0]);
        r[0] = fma2(m.c, U[1], z[0]);
        l[1] = fma2(m.c, nG1, z[1]);
        r[1] = fma2(m.nc, nG1, z[1]);
        l[2] = fma2(m.c, nG2, z[2]);
        r[2] = fma2(m.nc, nG2, z[2]);
    }
}

// What a warp's window holds of the tube's ends (transmissive).
struct TubeEnds {
    bool first;          // this lane's first cell is the tube's first
    bool last;           // this lane's last cell is the tube's last
    int ghost;           // place in the lane of the cell after the tube's last, where that is not a
                         // lane's first; -1 elsewhere
    bool any_ghost;      // some lane of the warp has one
};

// Of a window whose tube begins (first) in lane pad / C and, after g cells of the window, ends (last).
template <int C>
__device__ __forceinline__ TubeEnds tube_ends(int lane, int pad, bool first, bool last, int g)
{
    TubeEnds w;
    w.first = first && lane == pad / C;
    w.last = last && g % C == 0 && lane == g / C - 1;
    w.ghost = last && lane == g / C && g % C ? g % C : -1;
    w.any_ghost = last && g % C && g < 32 * C;
    return w;
}

__device__ __forceinline__ TubeConst tube_const(const TubeArgs& a, float c)
{
    TubeConst m;
    m.c = pk(c, c);
    m.nc = pk(-c, -c);
    m.gm1 = pk(a.gm1, a.gm1);
    m.ngm1 = pk(-a.gm1, -a.gm1);
    m.half = pk(0.5f, 0.5f);
    m.one = pk(1.f, 1.f);
    m.third = pk(1.f / 3.f, 1.f / 3.f);
    m.nthree = pk(-3.f, -3.f);
    m.om = pk(a.om, a.om);
    m.om1 = pk(a.om1, a.om1);
    return m;
}

// Cell j of a lane's C cells kept in pairs (j, j + C/2).
template <int C>
__device__ __forceinline__ float tube_cell(const P2 (*v)[3], int j, int k)
{
    return j < C / 2 ? lo2(v[j][k]) : hi2(v[j - C / 2][k]);
}

// The cell beyond the tube's end repeats the last one.
template <int C>
__device__ __forceinline__ void tube_ghost(P2 (*v)[3], const TubeEnds& w)
{
    constexpr int P = C / 2;
    float from[C][3];
#pragma unroll
    for (int j = 1; j < C; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) from[j][k] = tube_cell<C>(v, j - 1, k);
#pragma unroll
    for (int j = 0; j < P; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float lo = j && w.ghost == j ? from[j ? j : 1][k] : lo2(v[j][k]);
            v[j][k] = pk(lo, w.ghost == j + P ? from[j + P][k] : hi2(v[j][k]));
        }
}

// One step at omega = 1 on the moments of the lane's pairs:
// U'(j) = (l(j + 1) [+ z(j)]) + r(j - 1), pair by pair, in place.
template <int Q, int C>
__device__ __forceinline__ void tube_step_u(P2 U[C / 2][3], const TubeConst& m, const TubeEnds& w)
{
    constexpr int P = C / 2;
    if (w.any_ghost) tube_ghost<C>(U, w);
    P2 first_l[3], r0[3], l[3], z[3], r[3], zp[3], rp[3], rpp[3];
#pragma unroll
    for (int j = 0; j < P; ++j) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            rpp[k] = rp[k];
            rp[k] = r[k];
            zp[k] = z[k];
        }
        tube_feq<Q>(U[j], m, l, z, r);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (j == 0) {
                first_l[k] = l[k];
                r0[k] = r[k];
            } else {
                const P2 s = Q == 3 ? add2(l[k], zp[k]) : l[k];
                U[j - 1][k] = j == 1 ? s : add2(s, rpp[k]);      // pair 0 waits for the lane before
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float up = __shfl_up_sync(0xffffffffu, hi2(r[k]), 1);
        float down = __shfl_down_sync(0xffffffffu, lo2(first_l[k]), 1);
        up = w.first ? lo2(r0[k]) : up;                          // the ends pull their own values
        down = w.last ? hi2(l[k]) : down;
        const P2 lP = pk(hi2(first_l[k]), down);
        U[0][k] = add2(U[0][k], pk(up, lo2(r[k])));
        U[P - 1][k] = add2(Q == 3 ? add2(lP, z[k]) : lP, rp[k]);
    }
}

// One step of the general collision on the stored populations: L moves to -x, Z rests, R moves to
// +x.
template <int Q, int C>
__device__ __forceinline__ void tube_step_f(P2 L[C / 2][3], P2 Z[C / 2][3], P2 R[C / 2][3], const TubeConst& m,
                                            const TubeEnds& w)
{
    constexpr int P = C / 2;
    if (w.any_ghost) tube_ghost<C>(L, w);
    P2 rprev[3], lend[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float up = __shfl_up_sync(0xffffffffu, hi2(R[P - 1][k]), 1);
        float down = __shfl_down_sync(0xffffffffu, lo2(L[0][k]), 1);
        up = w.first ? lo2(R[0][k]) : up;
        down = w.last ? hi2(L[P - 1][k]) : down;
        rprev[k] = pk(up, lo2(R[P - 1][k]));
        lend[k] = pk(hi2(L[0][k]), down);
    }
#pragma unroll
    for (int j = 0; j < P; ++j) {
        P2 gl[3], gr[3], U[3], l[3], z[3], r[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            gl[k] = j + 1 < P ? L[j + 1 < P ? j + 1 : 0][k] : lend[k];
            gr[k] = rprev[k];
            rprev[k] = R[j][k];
            U[k] = Q == 3 ? add2(add2(gl[k], Z[j][k]), gr[k]) : add2(gl[k], gr[k]);
        }
        tube_feq<Q>(U, m, l, z, r);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            L[j][k] = fma2(m.om1, gl[k], mul2(m.om, l[k]));
            if constexpr (Q == 3) Z[j][k] = fma2(m.om1, Z[j][k], mul2(m.om, z[k]));
            R[j][k] = fma2(m.om1, gr[k], mul2(m.om, r[k]));
        }
    }
}

// From the coalesced order (a value every 32 cells) to the lane's cells and back, through
// shared memory with one word of padding per lane.
template <int C>
__device__ __forceinline__ P2 tube_pair(const float* sm, int lane, int j)
{
    return pk(sm[lane * (C + 1) + j], sm[lane * (C + 1) + j + C / 2]);
}

// Some cell of the warp is not finite.  In D1Q3 the steps above turn an infinite moment into NaN, which then
// stays in its cell's moments and resting population, so that their end shows whether they met one.
template <int C>
__device__ __forceinline__ bool tube_not_finite(const P2 (*v)[3])
{
    bool bad = false;
#pragma unroll
    for (int j = 0; j < C / 2; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) bad |= !(fabsf(lo2(v[j][k])) < INFINITY) || !(fabsf(hi2(v[j][k])) < INFINITY);
    return __any_sync(0xffffffffu, bad);
}

// Where cell x of a tube lies in memory: wrapped, or clamped to its ends.
__device__ __forceinline__ int64_t tube_place(int64_t off, int len, int periodic, int x)
{
    if (periodic) {
        x %= len;
        return off + (x < 0 ? x + len : x);
    }
    return off + min(max(x, 0), len - 1);
}

// A window's steps once more with infinities kept (D1Q3), cell by cell in thread-local memory.  Such a state is
// garbage soon, so this need not be fast.  1024 tubes of 200 to 15000 cells: 16.0 ms without any care, 17.4
// with it in every step, 15.0 with this call (whose presence also changes the steps' registers, 128 a lane
// instead of 159); at omega = 1.2, up to 9000 cells: 11.4 without, 12.3 in every step, 11.7 so.
template <int C>
__device__ __noinline__ void tube_redo(const TubeArgs& a, float c, bool first, bool last, int64_t off, int len, int x0,
                                       int ns, int t0, int tlen)
{
    const int lane = threadIdx.x & 31, xl = x0 + lane * C;
    const TubeEnds w = tube_ends<C>(lane, tube_pad<C>(a.halo), first, last, len - x0);
    const TubeConst m = tube_const(a, c);
    float f[C][9];                                        // [q * 3 + k]
#pragma unroll 1
    for (int j = 0; j < C; ++j) {
        const int64_t at = tube_place(off, len, a.periodic, xl + j);
        for (int n = 0; n < 9; ++n) f[j][n] = a.src[LBRS_IX(n * a.N + at, 9 * a.N, 53)];
    }
#pragma unroll 1
    for (int s = 0; s < ns; ++s) {
        if (w.ghost > 0)
            for (int k = 0; k < 3; ++k) f[w.ghost][k] = f[w.ghost - 1][k];
        float right[3], end[3];                           // what the cell before handed on; what follows the lane
        for (int k = 0; k < 3; ++k) {
            const float up = __shfl_up_sync(0xffffffffu, f[C - 1][6 + k], 1);
            const float down = __shfl_down_sync(0xffffffffu, f[0][k], 1);
            right[k] = w.first ? f[0][6 + k] : up;
            end[k] = w.last ? f[C - 1][k] : down;
        }
#pragma unroll 1
        for (int j = 0; j < C; ++j) {
            float g[3][3];
            P2 U[3], e[3][3];
            for (int k = 0; k < 3; ++k) {
                g[0][k] = j + 1 < C ? f[j + 1 < C ? j + 1 : 0][k] : end[k];
                g[1][k] = f[j][3 + k];
                g[2][k] = right[k];
                right[k] = f[j][6 + k];
                const float u = __fadd_rn(__fadd_rn(g[0][k], g[1][k]), g[2][k]);
                U[k] = pk(u, u);
            }
            tube_feq<3, true>(U, m, e[0], e[1], e[2]);
            for (int q = 0; q < 3; ++q)
                for (int k = 0; k < 3; ++k)
                    f[j][q * 3 + k] = a.om1 == 0.f ? lo2(e[q][k])
                                                   : lo2(fma2(m.om1, pk(g[q][k], g[q][k]), mul2(m.om, e[q][k])));
        }
    }
#pragma unroll 1
    for (int j = 0; j < C; ++j) {
        if (xl + j < t0 || xl + j >= t0 + tlen) continue;
        for (int n = 0; n < 9; ++n) a.dst[LBRS_IX(n * a.N + off + xl + j, 9 * a.N, 54)] = f[j][n];
    }
}

constexpr int kTubeWarps = 4;

// One warp per tile, up to a.halo steps.  UFORM: omega = 1, on the moments.
template <int Q, int C, bool UFORM>
__global__ void __launch_bounds__(32 * kTubeWarps) tube_kernel(const __grid_constant__ TubeArgs a)
{
    constexpr int P = C / 2, WIN = 32 * C, SM = 32 * (C + 1);
    __shared__ float s_turn[kTubeWarps][3][SM];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile = blockIdx.x * kTubeWarps + warp;
    if (tile >= a.ntiles) return;                         // whole warps only: no block barrier follows
    float(*sm)[SM] = s_turn[warp];

    int len, steps, t0, tlen;
    int64_t off = 0;
    float c;
    if (a.tiles) {
        const int4 t = __ldg(reinterpret_cast<const int4*>(a.tiles) + tile);   // {tube, t0, len, pad}
        len = a.tube_len[t.x];
        steps = a.tube_steps[t.x];
        off = a.tube_off[t.x];
        c = a.tube_c[t.x];
        t0 = t.y;
        tlen = t.z;
    } else {
        len = a.one_len;
        steps = a.one_steps;
        c = a.one_c;
        t0 = (int)((int64_t)tile * len / a.ntiles);
        tlen = (int)((int64_t)(tile + 1) * len / a.ntiles) - t0;
    }
    const int ns = min(a.halo, steps - a.launch * a.halo);                     // >= 1 for an active tile
    const int pad = tube_pad<C>(a.halo);
    // the window: the tube's first cell on a lane's first, else its last cell on a lane's last, if
    // they matter to the tile
    const bool first = !a.periodic && t0 == 0, end = !a.periodic && t0 + tlen + a.halo > len;
    const int x0 = end && !first ? len - (WIN - pad) : t0 - pad;
    const TubeEnds w = tube_ends<C>(lane, pad, first, end, len - x0);
    const TubeConst m = tube_const(a, c);

    auto place = [&](int x) { return tube_place(off, len, a.periodic, x); };
    auto turn_in = [&](P2(*v)[3]) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < P; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) v[j][k] = tube_pair<C>(sm[k], lane, j);
        __syncwarp();
    };
    auto load3 = [&](int q, P2(*v)[3]) {
#pragma unroll 4
        for (int i = lane; i < WIN; i += 32) {
            const int64_t at = place(x0 + i);
#pragma unroll
            for (int k = 0; k < 3; ++k) sm[k][i + i / C] = __ldg(a.src + LBRS_IX((q * 3 + k) * a.N + at, 3 * Q * a.N, 53));
        }
        turn_in(v);
    };
    auto store3 = [&](int q, P2(*v)[3]) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < P; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                sm[k][lane * (C + 1) + j] = lo2(v[j][k]);
                sm[k][lane * (C + 1) + j + P] = hi2(v[j][k]);
            }
        __syncwarp();
#pragma unroll 4
        for (int i = t0 - x0 + lane; i < t0 - x0 + tlen; i += 32) {
            const int64_t at = off + x0 + i;
#pragma unroll
            for (int k = 0; k < 3; ++k) a.dst[LBRS_IX((q * 3 + k) * a.N + at, 3 * Q * a.N, 54)] = sm[k][i + i / C];
        }
    };

    if constexpr (UFORM) {
        P2 U[P][3];
        // the first step's pull, straight into moments
#pragma unroll 4
        for (int i = lane; i < WIN; i += 32) {
            const int x = x0 + i;
            const int64_t xp = place(x + 1), xm = place(x - 1), xc = Q == 3 ? place(x) : 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float u = __ldg(a.src + LBRS_IX(k * a.N + xp, 3 * Q * a.N, 53));
                if constexpr (Q == 3) u = __fadd_rn(u, __ldg(a.src + LBRS_IX((3 + k) * a.N + xc, 3 * Q * a.N, 53)));
                sm[k][i + i / C] =
                    __fadd_rn(u, __ldg(a.src + LBRS_IX((3 * (Q - 1) + k) * a.N + xm, 3 * Q * a.N, 53)));
            }
        }
        turn_in(U);
        for (int s = 1; s < ns; ++s) tube_step_u<Q, C>(U, m, w);
        if constexpr (Q == 3)
            if (tube_not_finite<C>(U)) return tube_redo<C>(a, c, first, end, off, len, x0, ns, t0, tlen);
        P2 v[P][3];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
#pragma unroll
            for (int j = 0; j < P; ++j) {
                P2 l[3], z[3], r[3];
                tube_feq<Q>(U[j], m, l, z, r);
#pragma unroll
                for (int k = 0; k < 3; ++k) v[j][k] = q == 0 ? l[k] : (q == Q - 1 ? r[k] : z[k]);
            }
            store3(q, v);
        }
    } else {
        P2 L[P][3], Z[P][3], R[P][3];
        load3(0, L);
        if constexpr (Q == 3) load3(1, Z);
        load3(Q - 1, R);
        for (int s = 0; s < ns; ++s) tube_step_f<Q, C>(L, Z, R, m, w);
        if constexpr (Q == 3)
            if (tube_not_finite<C>(Z)) return tube_redo<C>(a, c, first, end, off, len, x0, ns, t0, tlen);
        store3(0, L);
        if constexpr (Q == 3) store3(1, Z);
        store3(Q - 1, R);
    }
}

}  // namespace lbrs

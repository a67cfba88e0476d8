// D2Q4 steps at omega = 1 on the moments alone, several steps per launch, the state of the
// steps in between in registers (sm_103a).
//
// At omega = 1 the collision returns f* = f^eq(U) (Section II.A), so a step is
//   U'(x) = sum_q f^eq_q(U(x - c_q)),
// the populations added in the order q = 0..3 as the storing kernels do.  One warp owns a
// strip of 64 columns, two adjacent ones per lane, and marches down the rows.  Processing
// source row r of a step computes its equilibria once, hands each to the two columns beside
// it (in the lane's registers, or by a warp shuffle at the lane's ends) and
//   * finishes row r + 1: U' = (S + f_2) + f_3 with the S that row r + 2 left there;
//   * starts row r - 1: S = f_0 + f_1, the populations that move down.
// So a step keeps two rows of partial sums (16 registers a lane), its finished row is the
// next step's source row in the same iteration, and K steps need no shared memory, no
// barrier and no reload: memory is read and written once per K steps.
//
// A lane's two columns share a register pair and the arithmetic is the packed FP32 form
// (fma.rn.f32x2 and its kin), which rounds each half as the scalar instruction does.  The
// expressions are fixed operation by operation and give the bits of the storing kernels'
// collide_2d, where the compiler contracts the same products.
#pragma once

#include "lbrs_chain.cuh"
#include "lbrs_kernels.cuh"

namespace lbrs {

// ---------------------------------------------------------------- packed FP32 pairs

using P2 = unsigned long long;

__device__ __forceinline__ P2 pk(float lo, float hi)
{
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo2(P2 v)
{
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a;
}
__device__ __forceinline__ float hi2(P2 v)
{
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return b;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c)
{
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b)
{
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ P2 add2(P2 a, P2 b)
{
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// -(1/x) of both halves: rcp_f32 of lbrs_kernels.cuh with the sign carried along.
__device__ __forceinline__ P2 neg_rcp2(P2 x, P2 one)
{
    float a, b;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(-lo2(x)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(-hi2(x)));
    const P2 r = pk(a, b);
    const P2 e = fma2(x, r, one);
    return fma2(r, e, r);
}

// ---------------------------------------------------------------- arguments

constexpr int kMarchWin = 64;                             // columns of a warp's window, two per lane
template <int K>
struct MarchShape {
    static constexpr int halo = (K + 1) / 2 * 2;          // window columns beyond the own ones, each side
    static constexpr int own = kMarchWin - 2 * halo;      // columns a warp stores
};

struct MarchArgs {
    const float* src;                 // U [4][N]
    float* dst;                       // U [4][N], not src; RECORD: the moments of each step, [K][4][N]
    float ghost[4][GHOST_STRIDE];     // f^eq of each Dirichlet side's state, [q * 4 + k]
    int64_t N;                        // plane stride
    int nx, ny;
    int bc[4];                        // x-lo, x-hi, y-lo, y-hi
    float c, gm1;                     // 1/(4 lambda), gamma - 1
    int strips, chunks;               // warps side by side, one above the other
    int rows, end_rows;               // rows a warp stores; those of the first and the last (0: as all)
};

struct MarchConst {
    P2 c, nc, gm1, ngm1, half, quarter, one;
};

// The factors of a pair's equilibria, signs as they fall out of -1/rho.
struct MarchPrim {
    P2 nu, nv, nF1, nF2, nG1, nG2, H;
};

__device__ __forceinline__ MarchPrim march_prim(const P2 U0, const P2 U1, const P2 U2, const P2 U3, const MarchConst& m)
{
    MarchPrim r;
    const P2 ninv = neg_rcp2(U0, m.one);
    r.nu = mul2(U1, ninv);
    r.nv = mul2(U2, ninv);
    const P2 q2 = mul2(U2, r.nv);                    // -(rho v v)
    const P2 nt = fma2(U1, r.nu, q2);                // -(rho |u|^2)
    const P2 pi = fma2(m.half, nt, U3);              // p / (gamma - 1)
    const P2 np = mul2(m.ngm1, pi);
    r.H = fma2(m.gm1, pi, U3);                       // rho E + p
    r.nF1 = fma2(U1, r.nu, np);
    r.nF2 = mul2(U1, r.nv);
    r.nG1 = mul2(U2, r.nu);
    r.nG2 = fma2(m.ngm1, pi, q2);
    return r;
}

// f^eq_q of field k of a pair, q = (-,-), (+,-), (+,+), (-,+).
template <int K>
__device__ __forceinline__ void march_feq(const P2 U[4], const MarchPrim& p, const MarchConst& m, P2 e[4])
{
    P2 ap, am, g;
    if constexpr (K == 0) {
        const P2 b = mul2(m.c, U[1]), nb = mul2(m.nc, U[1]);
        ap = fma2(m.quarter, U[0], b);
        am = fma2(m.quarter, U[0], nb);
        e[0] = fma2(m.nc, U[2], am);
        e[1] = fma2(m.nc, U[2], ap);
        e[2] = fma2(m.c, U[2], ap);
        e[3] = fma2(m.c, U[2], am);
        return;
    } else {
        P2 nf;
        if constexpr (K == 1) {
            nf = p.nF1;
            g = p.nG1;
        } else if constexpr (K == 2) {
            nf = p.nF2;
            g = p.nG2;
        } else {
            nf = mul2(p.nu, p.H);
            g = mul2(p.nv, p.H);
        }
        const P2 b = mul2(m.nc, nf), nb = mul2(m.c, nf);
        ap = fma2(m.quarter, U[K], b);
        am = fma2(m.quarter, U[K], nb);
        e[0] = fma2(m.c, g, am);                     // g is -G: c g = -(c G)
        e[1] = fma2(m.c, g, ap);
        e[2] = fma2(m.nc, g, ap);
        e[3] = fma2(m.nc, g, am);
    }
}

// What a warp knows of its place.  Column 0 lies in a lane's first place; column nx - 1 in the
// second, or (nx odd) in the first.  The flags are false where the x sides are periodic.
struct MarchPlace {
    int lane;
    bool left, right0, right1;         // this lane holds column 0; column nx - 1 in its first, second place
    bool dleft, dright0, dright1;      // the same beside a Dirichlet side
};

// The populations of one field of a source row as the columns beside receive them, f_q for the
// lane's first (l) and second (h) column.
struct MarchIn {
    float l[4], h[4];
};

// EDGE: the warp's window reaches an x side, and the end column takes its own value (clamped, EDGE = 1)
// or, beside a Dirichlet side, the side's ghost (EDGE = 2), by selects: a branch or a load here would
// cut the row's code into pieces that wait for one shuffle each.  ODD: column nx - 1 may be the first of
// a lane (nx odd), and memory is accessed by single words.
template <int EDGE, bool ODD, int K>
__device__ __forceinline__ void march_shift(const P2 e[4], const MarchArgs& a, const MarchPlace& w, MarchIn& n)
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (q == 1 || q == 2) {                          // to the right
            float in = __shfl_up_sync(0xffffffffu, hi2(e[q]), 1);
            if constexpr (EDGE >= 1) in = w.left ? lo2(e[q]) : in;
            if constexpr (EDGE == 2) in = w.dleft ? a.ghost[0][q * 4 + K] : in;
            n.l[q] = in;
            n.h[q] = lo2(e[q]);
        } else {                                         // to the left
            float in = __shfl_down_sync(0xffffffffu, lo2(e[q]), 1);
            float l = hi2(e[q]);
            if constexpr (EDGE >= 1) in = w.right1 ? hi2(e[q]) : in;
            if constexpr (EDGE == 2) in = w.dright1 ? a.ghost[1][q * 4 + K] : in;
            if constexpr (EDGE >= 1 && ODD) l = w.right0 ? lo2(e[q]) : l;
            if constexpr (EDGE == 2 && ODD) l = w.dright0 ? a.ghost[1][q * 4 + K] : l;
            n.l[q] = l;
            n.h[q] = in;
        }
    }
}

// Finish row q + 1 and start row q - 1 of one field: both share the partial sum S (rows of the
// same parity take turns in it).
__device__ __forceinline__ void march_sum(const MarchIn& n, P2& S, P2& out)
{
    out = pk(__fadd_rn(__fadd_rn(lo2(S), n.l[2]), n.l[3]), __fadd_rn(__fadd_rn(hi2(S), n.h[2]), n.h[3]));
    S = pk(__fadd_rn(n.l[0], n.l[1]), __fadd_rn(n.h[0], n.h[1]));
}

// The same where y sides are walls, whose relations need the row's own populations: the two that
// enter row ny - 1 (f_0, f_1; top: q = ny - 2) or row 0 (f_2, f_3; bottom: q = 1, which finishes the
// row at once) are the other two mirrored, rho v negated.  By selects, as at the x sides.
template <int K>
__device__ __forceinline__ void march_sum_wall(const MarchIn& n, bool top, bool bottom, P2& S, P2& out)
{
    float C[2] = {lo2(S), hi2(S)}, start[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float n0 = h ? n.h[0] : n.l[0], n1 = h ? n.h[1] : n.l[1], n2 = h ? n.h[2] : n.l[2], n3 = h ? n.h[3] : n.l[3];
        C[h] = top ? (K == 2 ? __fadd_rn(-n3, -n2) : __fadd_rn(n3, n2)) : C[h];
        C[h] = __fadd_rn(__fadd_rn(C[h], n2), n3);
        const float s = __fadd_rn(n0, n1);
        const float t = K == 2 ? __fadd_rn(__fadd_rn(s, -n1), -n0) : __fadd_rn(__fadd_rn(s, n1), n0);
        start[h] = bottom ? t : s;
    }
    out = pk(C[0], C[1]);
    S = pk(start[0], start[1]);
}

// Dirichlet y sides (an x side's ghost goes before a y side's): the partial sum f_0 + f_1 of row
// ny - 1, and row 0 finished from its partial sum.
template <int K>
__device__ __forceinline__ P2 march_top(const MarchArgs& a, const MarchPlace& w)
{
    const float l0 = w.dright0 ? a.ghost[1][K] : a.ghost[3][K], h0 = w.dright1 ? a.ghost[1][K] : a.ghost[3][K];
    const float l1 = w.dleft ? a.ghost[0][4 + K] : a.ghost[3][4 + K];
    return pk(__fadd_rn(l0, l1), __fadd_rn(h0, a.ghost[3][4 + K]));
}
template <int K>
__device__ __forceinline__ P2 march_bottom(P2 S, const MarchArgs& a, const MarchPlace& w)
{
    const float l2 = w.dleft ? a.ghost[0][8 + K] : a.ghost[2][8 + K], h2 = a.ghost[2][8 + K];
    const float l3 = w.dright0 ? a.ghost[1][12 + K] : a.ghost[2][12 + K];
    const float h3 = w.dright1 ? a.ghost[1][12 + K] : a.ghost[2][12 + K];
    return pk(__fadd_rn(__fadd_rn(lo2(S), l2), l3), __fadd_rn(__fadd_rn(hi2(S), h2), h3));
}

// Two columns x[0], x[1] (adjacent on an 8-byte boundary unless ODD) of the row at offset `row` of an
// array of n values.  The offset is the same for all lanes, which leaves the address arithmetic to
// the uniform data path.  CHAINED: the launch before may still be writing the array (lbrs_chain.cuh).
template <bool ODD, bool CHAINED>
__device__ __forceinline__ P2 march_load2(const float* p, int64_t n, int64_t row, const int x[2])
{
    if constexpr (CHAINED) {
        if constexpr (ODD) return pk(chain_load(p + LBRS_IX(row + x[0], n, 51)), chain_load(p + LBRS_IX(row + x[1], n, 51)));
        else return chain_load(reinterpret_cast<const P2*>(p + LBRS_IX(row + x[0], n - 1, 51)));
    } else {
        if constexpr (ODD) return pk(__ldg(p + LBRS_IX(row + x[0], n, 51)), __ldg(p + LBRS_IX(row + x[1], n, 51)));
        else return __ldg(reinterpret_cast<const P2*>(p + LBRS_IX(row + x[0], n - 1, 51)));
    }
}

template <bool ODD>
__device__ __forceinline__ void march_store2(float* p, int64_t n, int64_t row, int x, int nx, P2 v)
{
    if constexpr (ODD) {
        p[LBRS_IX(row + x, n, 52)] = lo2(v);
        if (x + 1 < nx) p[LBRS_IX(row + x + 1, n, 52)] = hi2(v);
    } else {
        *reinterpret_cast<P2*>(p + LBRS_IX(row + x, n - 1, 52)) = v;
    }
}

// Source row q of one step: from its moments U the finished row q + 1 of the next state.
template <int EDGE, bool WALL, bool ODD>
__device__ __forceinline__ void march_level(const P2 U[4], P2 S[4], P2 out[4], int q, const MarchArgs& a,
                                            const MarchPlace& w, const MarchConst& m)
{
    P2 e[4];
    MarchIn n;
    const MarchPrim p = march_prim(U[0], U[1], U[2], U[3], m);
    const bool top = WALL && a.bc[3] == BC_WALL && q == a.ny - 2, bottom = WALL && a.bc[2] == BC_WALL && q == 1;
#define LBRS_MARCH_FIELD(F)                                               \
    march_feq<F>(U, p, m, e);                                             \
    march_shift<EDGE, ODD, F>(e, a, w, n);                                \
    if constexpr (WALL) march_sum_wall<F>(n, top, bottom, S[F], out[F]);  \
    else march_sum(n, S[F], out[F]);
    LBRS_MARCH_FIELD(0)
    LBRS_MARCH_FIELD(1)
    LBRS_MARCH_FIELD(2)
    LBRS_MARCH_FIELD(3)
#undef LBRS_MARCH_FIELD
}

// The march of one warp over its rows [ya, yb) and the rows its steps need around them: in
// iteration r step s takes source row r + s, which step s - 1 has just finished.  Rows outside what
// a step needs are computed too (a branch costs more than the two or four rows) and never stored.
//
// SIDE: the warp's rows reach a y side (1: clamped or Dirichlet; 2: a wall among them).  A clamped
// side's row beyond it is a copy: row ny starts row ny - 1 with the sum that row ny - 1 hands to row
// ny - 2, and row -1 repeats row 0 (the input is loaded clamped, a step's finished row 0 is handed on
// twice).  The code of a row is the same as elsewhere, so that the loop stays in the instruction
// cache (a second copy of it for the rows beside a side cost 40 % of the march).
template <int EDGE, int SIDE, bool ODD, int K, bool RECORD>
__device__ __forceinline__ void march_rows(const MarchArgs& a, const MarchPlace& w, int ya, int yb, int xl, const int x[2])
{
    constexpr int HL = MarchShape<K>::halo / 2;
    const bool own = w.lane >= HL && w.lane < 32 - HL && xl < a.nx;
    const bool yper = a.bc[2] == BC_PERIODIC;
    MarchConst m;
    m.c = pk(a.c, a.c);
    m.nc = pk(-a.c, -a.c);
    m.gm1 = pk(a.gm1, a.gm1);
    m.ngm1 = pk(-a.gm1, -a.gm1);
    m.half = pk(0.5f, 0.5f);
    m.quarter = pk(0.25f, 0.25f);
    m.one = pk(1.f, 1.f);

    P2 S[K][2][4];                                       // partial sums: step; parity of the row; field
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
        for (int k = 0; k < 4; ++k) S[s][0][k] = S[s][1][k] = 0ull;

    int r = yb + K - 1;
    if (SIDE) r = min(r, a.ny - 1);
    const int rlast = ya - K;
    // the input row that the next load brings: clamped at sides, wrapped on periodic grids
    int fetch = yper ? r % a.ny : r;
    auto fetch_row = [&]() {
        const int j = SIDE ? max(fetch, 0) : fetch;
        if (--fetch < 0 && yper) fetch = a.ny - 1;
        return (int64_t)j * a.nx;
    };
    P2 nxt[2][4];                                        // the next two source rows, loads in flight
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        const int64_t row = fetch_row();
#pragma unroll
        for (int k = 0; k < 4; ++k) nxt[n][k] = march_load2<ODD, !RECORD>(a.src, 4 * a.N, k * a.N + row, x);
    }
    auto iteration = [&](auto parity) {
        constexpr int p = decltype(parity)::value;
        P2 U[4];
        const int64_t in = fetch_row();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            U[k] = nxt[p][k];
            nxt[p][k] = march_load2<ODD, !RECORD>(a.src, 4 * a.N, k * a.N + in, x);
        }
#pragma unroll
        for (int s = 0; s < K; ++s) {
            const int q = r + s;                         // this step's source row
            const int t = (p + s) & 1;                   // the partial sums' turn (static once unrolled)
            P2 out[4];
            // below row 0 the partial sum of the row to finish holds row 0 itself, finished before
            if (SIDE != 0 && q < (a.bc[2] == BC_TRANSMISSIVE ? -1 : 0)) {
#pragma unroll
                for (int k = 0; k < 4; ++k) out[k] = S[s][t][k];
            } else {
                march_level<EDGE, SIDE == 2, ODD>(U, S[s][t], out, q, a, w, m);
            }
            if constexpr (SIDE != 0) {
                if (q == a.ny - 1) {
                    if (a.bc[3] == BC_DIRICHLET) {
                        S[s][t ^ 1][0] = march_top<0>(a, w);
                        S[s][t ^ 1][1] = march_top<1>(a, w);
                        S[s][t ^ 1][2] = march_top<2>(a, w);
                        S[s][t ^ 1][3] = march_top<3>(a, w);
                    } else if (a.bc[3] == BC_TRANSMISSIVE) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) S[s][t ^ 1][k] = S[s][t][k];
                    }
                }
                if (q == 0 && a.bc[2] == BC_DIRICHLET) {
                    S[s][t ^ 1][0] = march_bottom<0>(S[s][t ^ 1][0], a, w);
                    S[s][t ^ 1][1] = march_bottom<1>(S[s][t ^ 1][1], a, w);
                    S[s][t ^ 1][2] = march_bottom<2>(S[s][t ^ 1][2], a, w);
                    S[s][t ^ 1][3] = march_bottom<3>(S[s][t ^ 1][3], a, w);
                }
                if (q < 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) S[s][t ^ 1][k] = out[k];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) U[k] = out[k];
            // U is the finished row q + 1 of step s + 1
            if ((RECORD || s == K - 1) && own && q + 1 >= ya && q + 1 < yb) {
                const int64_t row = (int64_t)(q + 1) * a.nx + (RECORD ? 4 * s * a.N : 0);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    march_store2<ODD>(a.dst, (RECORD ? 4 * K : 4) * a.N, k * a.N + row, xl, a.nx, U[k]);
            }
        }
        --r;
    };
    while (r >= rlast) {
        iteration(std::integral_constant<int, 0>());
        iteration(std::integral_constant<int, 1>());
    }
}

// K steps a launch, one warp a block.  RECORD: every step's moments are stored; such launches are never links
// of a chain and read by __ldg (backward pass of 2048^2, 400 steps: 23.7 ms, 24.1 with a chain's loads).
template <int K, bool ODD, bool RECORD>
__global__ void __launch_bounds__(32, 16) march2d_kernel(const __grid_constant__ MarchArgs a)
{
    chain_begin();
    const int strip = blockIdx.x % a.strips;
    const int chunk = blockIdx.x / a.strips;
    int ya = chunk * a.rows, yb = min(ya + a.rows, a.ny);
    if (a.end_rows) {
        const bool last = chunk == a.chunks - 1;
        ya = chunk == 0 ? 0 : (last ? a.ny - a.end_rows : a.end_rows + (chunk - 1) * a.rows);
        yb = chunk == 0 ? a.end_rows : (last ? a.ny : min(ya + a.rows, a.ny - a.end_rows));
    }
    const int x0 = strip * MarchShape<K>::own - MarchShape<K>::halo;

    MarchPlace w;
    w.lane = threadIdx.x;
    const int xl = x0 + 2 * w.lane;                      // the lane's first column
    const bool xper = a.bc[0] == BC_PERIODIC;
    w.left = !xper && xl == 0;
    w.right0 = !xper && a.nx - 1 == xl;
    w.right1 = !xper && a.nx - 1 == xl + 1;
    w.dleft = w.left && a.bc[0] == BC_DIRICHLET;
    w.dright0 = w.right0 && a.bc[1] == BC_DIRICHLET;
    w.dright1 = w.right1 && a.bc[1] == BC_DIRICHLET;

    // where the lane's columns lie in memory: wrapped beyond periodic sides, any column of the row
    // beyond others (nothing reads what such a column computes)
    int x[2];
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        int i = xl + n;
        if (xper) {
            i %= a.nx;
            if (i < 0) i += a.nx;
        } else {
            i = min(max(i, 0), a.nx - 1);
        }
        x[n] = i;
    }
    if (!ODD && !xper) x[0] = min(max(xl, 0), a.nx - 2);
    const bool edge = !xper && (x0 < 0 || x0 + kMarchWin >= a.nx);
    const int xs = !edge ? 0 : (a.bc[0] == BC_DIRICHLET || a.bc[1] == BC_DIRICHLET ? 2 : 1);
    // the rows loaded lie in [ya - K - 3, yb + K - 1] (two ahead, and one more iteration)
    const bool side = a.bc[2] != BC_PERIODIC && (ya < K + 4 || yb + K > a.ny);
    const int ys = !side ? 0 : (a.bc[2] == BC_WALL || a.bc[3] == BC_WALL ? 2 : 1);
#define LBRS_MARCH_ROWS(X, Y) \
    if (xs == X && ys == Y) march_rows<X, Y, ODD, K, RECORD>(a, w, ya, yb, xl, x);
    LBRS_MARCH_ROWS(0, 0)
    LBRS_MARCH_ROWS(1, 0)
    LBRS_MARCH_ROWS(2, 0)
    LBRS_MARCH_ROWS(0, 1)
    LBRS_MARCH_ROWS(1, 1)
    LBRS_MARCH_ROWS(2, 1)
    LBRS_MARCH_ROWS(0, 2)
    LBRS_MARCH_ROWS(1, 2)
    LBRS_MARCH_ROWS(2, 2)
#undef LBRS_MARCH_ROWS
}

}  // namespace lbrs

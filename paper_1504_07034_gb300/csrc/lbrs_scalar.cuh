// Scalar D2Q4 steps (2-D inviscid Burgers) at omega = 1, FP32, many steps per launch on the field u in
// shared memory (sm_103a).
//
// At omega = 1 the collision returns f^eq(u), so the state is u alone (4 B per cell) and a step is
// u'(x) = sum_q f^eq_q(u(x - c_q)).  A block holds a window of the grid twice in shared memory and
// takes up to K steps there, one barrier each; a thread owns two columns (a packed FP32 pair) and R
// rows, reads each source row's neighbours once and keeps what two target rows share.  A window
// that holds the whole grid has no stale edge and takes all steps of a call; otherwise the cells
// within K of a cut edge go stale and the launch stores the tile inside.
//
// Beyond a side the window holds what the single-step pull resolves there: a Dirichlet side's profile
// value (constant), a transmissive side's clamped cell (copied by the thread that steps it), the
// wrapped cells of a periodic one (stepped like any others).  The expressions are fixed operation by
// operation and give the bits of collide_2ds, where the compiler contracts the same products.
#pragma once

#include "lbrs_march.cuh"

namespace lbrs {

struct ScalarArgs {
    const float* __restrict__ src;    // u [N], or f* [4][N] (LOADF: the first step's pull comes on top)
    float* __restrict__ dst;          // u [N], or f* [4][N] (STOREF)
    StepArgs<float> f;                // geometry, sides, ghosts; its src for LOADF
    int wx, wy;                       // window: columns (even), rows
    int hx, hy;                       // columns and rows beyond the tile, each side (hx even)
    int tx, ty;                       // tile
    int steps;
    int loadf, storef;
};

struct ScalarConst {
    P2 c, nc, half, quarter;
};

// f^eq of two sources: the populations moving right (up: f_2, down: f_1) or left (f_3, f_0), the
// products of the two directions shared.
__device__ __forceinline__ void scalar_right(P2 u, const ScalarConst& m, P2& down, P2& up)
{
    const P2 b = mul2(m.c, mul2(mul2(m.half, u), u));
    const P2 ap = fma2(m.quarter, u, b);
    down = fma2(m.nc, u, ap);
    up = fma2(m.c, u, ap);
}
__device__ __forceinline__ void scalar_left(P2 u, const ScalarConst& m, P2& down, P2& up)
{
    const P2 nb = mul2(m.nc, mul2(mul2(m.half, u), u));
    const P2 am = fma2(m.quarter, u, nb);
    down = fma2(m.nc, u, am);
    up = fma2(m.c, u, am);
}

// Value beyond the domain's sides at cell (i, j), -1 <= i <= nx, -1 <= j <= ny, where it is a constant
// of the run: a Dirichlet profile, the x side first.  False where it is a copy of a cell.
__device__ __forceinline__ bool scalar_ghost(const StepArgs<float>& a, int i, int j, float& v)
{
    const bool ox = i < 0 || i >= a.nx, oy = j < 0 || j >= a.ny;
    const int kx = i < 0 ? a.bc[0] : a.bc[1], ky = j < 0 ? a.bc[2] : a.bc[3];
    if (ox && kx == BC_DIRICHLET) {
        v = profile_value<float>(a.ghost + (i < 0 ? 0 : 1) * GHOST_STRIDE, j);
        return true;
    }
    if (oy && ky == BC_DIRICHLET) {
        int m = i;
        if (ox) m = kx == BC_PERIODIC ? (i < 0 ? i + a.nx : i - a.nx) : (i < 0 ? 0 : a.nx - 1);
        v = profile_value<float>(a.ghost + (j < 0 ? 2 : 3) * GHOST_STRIDE, m);
        return true;
    }
    return false;
}

template <int R>
__global__ void __launch_bounds__(1024) step2ds_window_kernel(const __grid_constant__ ScalarArgs a)
{
    extern __shared__ __align__(16) float s_u[];          // two buffers of wy x wx
    const StepArgs<float>& g = a.f;
    const int wx = a.wx, wy = a.wy, n = wx * wy;
    const int i0 = blockIdx.x * a.tx - a.hx, j0 = blockIdx.y * a.ty - a.hy;
    const bool px = g.bc[0] == BC_PERIODIC, py = g.bc[2] == BC_PERIODIC;

    // the window: cells of the grid, wrapped beyond periodic sides, ghosts beyond the others
    for (int w = threadIdx.x; w < n; w += blockDim.x) {
        int i = i0 + w % wx, j = j0 + w / wx;
        if (px) {
            i %= g.nx;
            if (i < 0) i += g.nx;
        }
        if (py) {
            j %= g.ny;
            if (j < 0) j += g.ny;
        }
        float u = 0.f;
        const int ic = min(max(i, 0), g.nx - 1), jc = min(max(j, 0), g.ny - 1);
        if (i < -1 || i > g.nx || j < -1 || j > g.ny || !scalar_ghost(g, i, j, u)) {
            if (a.loadf) {
                float f[4];
                if (ic > 0 && ic < g.nx - 1 && jc > 0 && jc < g.ny - 1) {
                    const int64_t c = (int64_t)jc * g.nx + ic;
                    const int64_t s[4] = {c + g.nx + 1, c + g.nx - 1, c - g.nx - 1, c - g.nx + 1};
#pragma unroll
                    for (int q = 0; q < 4; ++q) f[q] = g.src[LBRS_IX(q * g.N + s[q], 4 * g.N, 56)];
                } else {
                    pull_edge_2ds<float>(g, ic, jc, f);
                }
                u = __fadd_rn(__fadd_rn(__fadd_rn(f[0], f[1]), f[2]), f[3]);
            } else {
                u = a.src[LBRS_IX((int64_t)jc * g.nx + ic, g.N, 56)];
            }
        }
        s_u[w] = u;
        s_u[n + w] = u;
    }
    __syncthreads();

    // this thread's columns 2 p, 2 p + 1 and rows r0 .. r0 + R - 1 of the window
    const int pairs = wx / 2, p = threadIdx.x % pairs, r0 = threadIdx.x / pairs * R;
    const int cl = max(2 * p - 1, 0), cr = min(2 * p + 2, wx - 1);
    const int i = i0 + 2 * p;
    const bool lo = px || (i >= 0 && i < g.nx), hi = px || (i + 1 >= 0 && i + 1 < g.nx);
    // clamped columns -1 and nx that this pair feeds (transmissive): their place beside the pair
    const bool gl = !px && g.bc[0] == BC_TRANSMISSIVE && i == 0;
    const bool gr0 = !px && g.bc[1] == BC_TRANSMISSIVE && i == g.nx - 1 && 2 * p + 1 < wx;
    const bool gr1 = !px && g.bc[1] == BC_TRANSMISSIVE && i + 1 == g.nx - 1 && 2 * p + 2 < wx;
    const bool bot = !py && g.bc[2] == BC_TRANSMISSIVE, top = !py && g.bc[3] == BC_TRANSMISSIVE;
    ScalarConst m;
    m.c = pk(g.c, g.c);
    m.nc = pk(-g.c, -g.c);
    m.half = pk(0.5f, 0.5f);
    m.quarter = pk(0.25f, 0.25f);

    // the rows that this thread may write, and whether any of its cells is copied beyond a side
    unsigned rows = 0;
    bool copies = gl || gr0 || gr1;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int y = r0 + t, j = j0 + y;
        if (y < wy && (py || (j >= 0 && j < g.ny)) && (lo || hi)) rows |= 1u << t;
        copies |= (bot && j == 0) || (top && j == g.ny - 1);
    }
    const bool whole = rows == (1u << R) - 1 && lo && hi;

    int cur = 0;
    for (int s = 0; s < a.steps; ++s) {
        const float* in = s_u + cur * n;
        float* out = s_u + (cur ^ 1) * n;
        // every load before the first store: the two buffers alias for the compiler
        P2 own[R + 2];
        float lf[R + 2], rt[R + 2];
#pragma unroll
        for (int t = 0; t < R + 2; ++t) {
            const float* row = in + min(max(r0 + t - 1, 0), wy - 1) * wx;
            own[t] = *reinterpret_cast<const P2*>(row + 2 * p);
            lf[t] = row[cl];
            rt[t] = row[cr];
        }
        P2 v[R], up_r[2], up_l[2];                         // up: of the last two source rows
#pragma unroll
        for (int t = 0; t < R + 2; ++t) {
            P2 dr, ur, dl, ul;
            scalar_right(pk(lf[t], lo2(own[t])), m, dr, ur);   // f_1, f_2
            scalar_left(pk(hi2(own[t]), rt[t]), m, dl, ul);    // f_0, f_3
            // target row r0 + t - 2: f_0 and f_1 of the row above it, f_2 and f_3 of the one below
            if (t >= 2) v[t - 2] = add2(add2(add2(dl, dr), up_r[t & 1]), up_l[t & 1]);
            up_r[t & 1] = ur;
            up_l[t & 1] = ul;
        }
        float* o = out + r0 * wx + 2 * p;
        if (whole) {
#pragma unroll
            for (int t = 0; t < R; ++t) *reinterpret_cast<P2*>(o + t * wx) = v[t];
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (rows >> t & 1) {
                    if (lo) o[t * wx] = lo2(v[t]);
                    if (hi) o[t * wx + 1] = hi2(v[t]);
                }
        }
        if (copies) {
            // beyond transmissive sides; a corner is a copy only if both sides are
#pragma unroll
            for (int t = 0; t < R; ++t) {
                if (!(rows >> t & 1)) continue;
                const int y = r0 + t, j = j0 + y;
#pragma unroll
                for (int e = -1; e <= 1; ++e) {
                    if (e < 0 && !(bot && j == 0 && y > 0)) continue;
                    if (e > 0 && !(top && j == g.ny - 1 && y + 1 < wy)) continue;
                    float* w = o + (t + e) * wx;
                    if (e && lo) w[0] = lo2(v[t]);
                    if (e && hi) w[1] = hi2(v[t]);
                    if (gl) w[-1] = lo2(v[t]);
                    if (gr0) w[1] = lo2(v[t]);
                    if (gr1) w[2] = hi2(v[t]);
                }
            }
        }
        __syncthreads();
        cur ^= 1;
    }

    // the tile
    const float* fin = s_u + cur * n;
    for (int w = threadIdx.x; w < a.tx * a.ty; w += blockDim.x) {
        const int x = w % a.tx, y = w / a.tx;
        const int ii = i0 + a.hx + x, jj = j0 + a.hy + y;
        if (ii >= g.nx || jj >= g.ny) continue;
        const float u = fin[(a.hy + y) * wx + a.hx + x];
        const int64_t c = (int64_t)jj * g.nx + ii;
        if (a.storef) {
            P2 dr, ur, dl, ul;
            scalar_right(pk(u, u), m, dr, ur);
            scalar_left(pk(u, u), m, dl, ul);
            a.dst[LBRS_IX(c, 4 * g.N, 57)] = lo2(dl);
            a.dst[LBRS_IX(g.N + c, 4 * g.N, 57)] = lo2(dr);
            a.dst[LBRS_IX(2 * g.N + c, 4 * g.N, 57)] = lo2(ur);
            a.dst[LBRS_IX(3 * g.N + c, 4 * g.N, 57)] = lo2(ul);
        } else {
            a.dst[LBRS_IX(c, g.N, 57)] = u;
        }
    }
}

}  // namespace lbrs

// FP32 D2Q4 steps at omega = 1 on the moments (lbrs_march.cuh): the launchers and the kernels
// that lead from stored distributions into the moments and back.
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "lbrs_adapt.cuh"
#include "lbrs_march.cuh"
#include "lbrs_launch.h"

namespace lbrs {

namespace {

constexpr int kWarpsPerSM = 16;   // the march's registers allow 16 one-warp blocks per SM

// Moments of the next step's pull from stored distributions: U = sum_q f*_q(x - c_q).  WALLS: with
// internal walls (solid cells: the moments of what they hold).
template <bool WALLS>
__global__ void __launch_bounds__(256) pull_moments_2d_kernel(const StepArgs<float> a, float* __restrict__ U)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= a.nx || j >= a.ny) return;
    const int64_t c = (int64_t)j * a.nx + i;
    float f[4][4];
    bool plain = i > 0 && i < a.nx - 1 && j > 0 && j < a.ny - 1;
    int64_t s[4] = {c + a.nx + 1, c + a.nx - 1, c - a.nx - 1, c - a.nx + 1};
    if constexpr (WALLS) {
        if (a.solid[LBRS_IX(c, a.N, 50)]) {
            plain = true;
            s[0] = s[1] = s[2] = s[3] = c;
        } else if (plain) {
            for (int q = 0; q < 4; ++q) plain &= !a.solid[LBRS_IX(s[q], a.N, 50)];
        }
    }
    if (plain) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) f[q][k] = a.src[LBRS_IX((q * 4 + k) * a.N + s[q], 16 * a.N, 50)];
    } else if constexpr (WALLS) {
        pull_obstacle_2d<float>(a, i, j, f);
    } else {
        pull_edge_2d<float, false>(a, i, j, f);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        U[LBRS_IX(k * a.N + c, 4 * a.N, 50)] =
            __fadd_rn(__fadd_rn(__fadd_rn(f[0][k], f[1][k]), f[2][k]), f[3][k]);
}

// The code of launch_wall_codes, by the rule of pull_obstacle_2d.
__global__ void __launch_bounds__(256) wall_code_2d_kernel(const StepArgs<float> a, uint8_t* __restrict__ codes)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    if (i >= a.nx || j >= a.ny) return;
    const int SX[4] = {-1, 1, 1, -1}, SY[4] = {-1, -1, 1, 1};
    const int64_t c = (int64_t)j * a.nx + i;
    unsigned code = 0;
    if (!a.solid[LBRS_IX(c, a.N, 58)]) {
        for (int q = 0; q < 4; ++q) {
            const int si = i - SX[q], sj = j - SY[q];
            // a wall side's own relation and a Dirichlet ghost go before; solid_at takes both for fluid
            const bool out_x = si < 0 || si >= a.nx, out_y = sj < 0 || sj >= a.ny;
            if (out_y && (sj < 0 ? a.bc[2] : a.bc[3]) == BC_WALL) continue;
            if (out_x && (si < 0 ? a.bc[0] : a.bc[1]) == BC_DIRICHLET) continue;
            if (!solid_at(a, si, sj)) continue;
            const bool xn = solid_at(a, si, j), yn = solid_at(a, i, sj);
            code |= ((yn && !xn ? 0u : 1u) | (xn && !yn ? 0u : 2u)) << (2 * q);
        }
    }
    codes[LBRS_IX(c, a.N, 58)] = (uint8_t)code;
}

// An adaptive step's moments and their bound (adapt_prep_kernel has run).
__global__ void __launch_bounds__(256) adapt_pull_kernel(const StepArgs<float> a, float* __restrict__ U, AdaptState* st,
                                                         double gamma)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    float bnd = -1.f;
    if (i < a.nx && j < a.ny) {
        const int64_t c = (int64_t)j * a.nx + i;
        float f[4][4], u[4];
        pull_edge_2d<float, false>(a, i, j, f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u[k] = __fadd_rn(__fadd_rn(__fadd_rn(f[0][k], f[1][k]), f[2][k]), f[3][k]);
            U[LBRS_IX(k * a.N + c, 4 * a.N, 60)] = u[k];
        }
        bnd = bound_local<float>(u, gamma);
    }
    block_max_into<256>(bnd, &st->bound_bits[st->slot_cur]);
}

__global__ void adapt_enter_kernel(const AdaptState* st, AdaptRun* run, unsigned long long* bounds, double dx)
{
    for (int n = threadIdx.x; n < 6 * kBoundSlots; n += 32)
        bounds[n] = n == kBoundSlots ? st->bound_bits[st->slot_cur] : 0ull;
    if (threadIdx.x != 0) return;
    run->t = st->t;
    run->lam = st->lam_cur;
    run->c = st->c_new;
    run->dt = __ddiv_rn(dx, st->lam_cur);
    run->steps = st->steps;
    run->last = st->last;
    run->done = st->done;
    run->dead = st->skip;
}

__global__ void adapt_leave_kernel(AdaptState* st, AdaptRun* run, const unsigned long long* last, double dx,
                                   double safety, double t_final)
{
    AdaptRun r, unused;
    adapt_clocks(*run, last, 2, dx, safety, t_final, r, unused);     // the last state's own clock step
    if (threadIdx.x != 0) return;
    unsigned long long b = 0ull;
    for (int n = 0; n < kBoundSlots; ++n) b = last[kBoundSlots + n] > b ? last[kBoundSlots + n] : b;
    *run = r;
    st->t = r.t;
    st->lam_cur = r.lam;
    st->c_new = r.c;
    st->steps = r.steps;
    st->last = r.last;
    st->done = r.done;
    st->bound_bits[st->slot_cur] = b;
}

// f* = f^eq(U) into the populations' planes, two cells a thread; solid cells keep theirs.  run: the
// adaptive record whose lambda the distributions take (nothing is written if its run had ended).
__global__ void __launch_bounds__(256) equilibria_2d_kernel(const float* __restrict__ U, float* __restrict__ f,
                                                            const uint8_t* __restrict__ solid,
                                                            const AdaptRun* __restrict__ run, int64_t N, float c,
                                                            float gm1)
{
    if (run) {
        if (run->dead) return;
        c = (float)run->c;
    }
    const int64_t i = 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= N) return;
    const bool two = i + 1 < N;
    const bool keep0 = solid && solid[LBRS_IX(i, N, 64)], keep1 = !two || (solid && solid[LBRS_IX(i + 1, N, 64)]);
    const bool vec = (N & 1) == 0 && !keep0 && !keep1;   // every plane starts on 8 bytes
    MarchConst m;
    m.c = pk(c, c);
    m.nc = pk(-c, -c);
    m.gm1 = pk(gm1, gm1);
    m.ngm1 = pk(-gm1, -gm1);
    m.half = pk(0.5f, 0.5f);
    m.quarter = pk(0.25f, 0.25f);
    m.one = pk(1.f, 1.f);
    P2 u[4], e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float* p = U + LBRS_IX(k * N + i, 4 * N, 64);
        u[k] = pk(p[0], two ? p[1] : p[0]);
    }
    const MarchPrim pr = march_prim(u[0], u[1], u[2], u[3], m);
    auto store = [&](int k) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float* p = f + LBRS_IX((q * 4 + k) * N + i, 16 * N, 64);
            if (vec) {
                *reinterpret_cast<P2*>(p) = e[q];
            } else {
                if (!keep0) p[0] = lo2(e[q]);
                if (!keep1) p[1] = hi2(e[q]);
            }
        }
    };
    march_feq<0>(u, pr, m, e);
    store(0);
    march_feq<1>(u, pr, m, e);
    store(1);
    march_feq<2>(u, pr, m, e);
    store(2);
    march_feq<3>(u, pr, m, e);
    store(3);
}

// Time of an iteration (K source rows) with w warps per SM sub-partition, in us (periodic, K = 2: 768^2
// 0.34 at one on the fullest, 900^2 0.44 at two, 2048 x 512 0.63 at three, 1200^2 0.81 at four), full waves and
// a rest beyond.  A wave of one more warp measured 0.22 on top; taken as 0.32, because the rest starts late:
// with 0.22 the rule picks 38 rows instead of 42 at 2400^2 (26.7 us a step instead of 21.0) and 64 instead of
// 50 at 6144 x 2048 (49.1 instead of 44.7).
double march_iteration(double w)
{
    static const double t[5] = {0.34, 0.34, 0.44, 0.63, 0.80};
    if (w <= 4.0) return t[(int)ceil(w)];
    double sum = 0.0;
    for (; w > 4.0; w -= 4.0) sum += t[4];
    return sum + 0.12 + 0.2 * w;
}

// Rows a warp stores.  Fewer rows mean more warps to hide latencies, and more rows recomputed around
// each warp's own (2 K of them): a launch takes about 1.5 us and (rows + 2 K) iterations, and the rule
// takes the minimum over the rows (us per step, K = 2: 1024^2 with clamped sides 16 rows 5.4, 10 rows
// 6.2, 30 rows 7.1; 2048^2 30 rows in one full wave 16.2, 16 rows 17.5, 20 rows 18.0, 40 rows 17.3).
// The warps beside y sides that are not periodic take longer per row (0.40 us by themselves, 0.60 beside
// a wall, 0.4 more with another warp) and get as many rows, an even number, as keep them from ending
// last (1024^2, 16 rows, 8 of them 5.4, 9 5.6, 12 6.2).  Returns that time without the 1.5 us.
double march_rows_for(MarchArgs& a, int own, int steps)
{
    a.strips = (a.nx + own - 1) / own;
    const bool per = a.bc[2] == BC_PERIODIC;
    const double lone = a.bc[2] == BC_WALL || a.bc[3] == BC_WALL ? 0.60 : 0.40;
    double best = 0.0;
    for (int rows = 4; rows <= 64; rows += 2) {
        int end = 0;
        int64_t chunks = (a.ny + rows - 1) / rows;
        const int64_t per_sm = (a.strips * chunks + kSMs - 1) / kSMs;
        const double w = (double)per_sm / 4.0, resident = fmin(w, kWarpsPerSM / 4);
        double t = (rows + 2 * steps) * march_iteration(w);
        if (!per) {
            const double iteration = lone + 0.36 * fmin(fmax(ceil(resident) - 1.0, 0.0), 1.67);   // beside a y side
            end = (int)((rows + 2 * steps) * march_iteration(resident) / iteration) - steps;
            end = end < 2 ? 2 : (end > rows ? rows : end & ~1);
            if (a.ny > 2 * end) {
                chunks = 2 + (a.ny - 2 * end + rows - 1) / rows;
                t = (rows + 2 * steps) * march_iteration((double)((a.strips * chunks + kSMs - 1) / kSMs) / 4.0);
            } else {
                end = 0;
                t = fmax(t, (rows + steps) * iteration);
            }
        }
        if (best == 0.0 || t < best) {
            best = t;
            a.rows = rows;
            a.end_rows = end;
            a.chunks = (int)chunks;
        }
    }
    return best;
}

template <int K, bool RECORD>
cudaError_t launch_k(MarchArgs a, bool chained, cudaStream_t s)
{
    march_rows_for(a, MarchShape<K>::own, K);
    const int64_t blocks = (int64_t)a.strips * a.chunks;
    // pairs of columns move as 8-byte words where every row starts on one: nx even, and (moments recorded into
    // a caller's buffer) the buffers themselves on 8 bytes
    const bool words = (a.nx & 1) || (((uintptr_t)a.src | (uintptr_t)a.dst) & 7);
    chained = chained && !RECORD;
    if (words) return launch_in_chain(chained, march2d_kernel<K, true, RECORD>, (unsigned)blocks, 32, s, a);
    return launch_in_chain(chained, march2d_kernel<K, false, RECORD>, (unsigned)blocks, 32, s, a);
}

}  // namespace

static int march_mode()
{
    static const int v = [] {
        const char* e = getenv("LBRS_F32_MARCH");
        return e ? atoi(e) : 1;
    }();
    return v;
}

bool march_enabled() { return march_mode() != 0; }
bool march_always() { return march_mode() >= 2; }

// The tile kernel's two-step launch (step2d_u2_kernel, 32 x 16 tiles, four blocks per SM) starts
// faster than a march and wins on small grids: about 2.7 us and 1.05 us per tile of an SM against the
// march's 1.5 us and its iterations, 1 us and a quarter more of them beside sides that are not periodic
// (us per launch, in a graph, tiles and march, periodic and then with clamped sides: 128^2 3.1, 4.1 and 2.9, 4.9;
// 256^2 3.1, 5.1 and 3.0, 6.0; 384^2 4.4, 4.9 and 4.2, 6.9; 448^2 5.1, 4.9 and 5.0, 6.9; 512^2 6.4, 5.0 and 6.2,
// 6.3; 1531 x 200 6.7, 5.9 and 6.7, 8.5; 640^2 8.4, 5.9 and 8.2, 6.8; 768^2 10.3, 7.6 and 10.2, 7.8.  Of 54 grids
// and side sets from 64^2 to 1531 x 973 the choice is at most 4 % slower than the other kernel.)
bool march_prefers_tiles(int nx, int ny, const int bc[4])
{
    if (march_always()) return false;
    MarchArgs a;
    a.nx = nx;
    a.ny = ny;
    for (int s = 0; s < 4; ++s) a.bc[s] = bc[s];
    const bool per = bc[2] == BC_PERIODIC;
    const double march = (per ? 1.5 : 2.5) + march_rows_for(a, MarchShape<2>::own, 2) * (per ? 1.0 : 1.25);
    const double tiles = (double)((nx + 31) / 32) * (double)((ny + 15) / 16);
    return 2.7 + 1.05 * tiles / kSMs < march;
}

// f^eq of the Dirichlet sides' states in FP64, rounded: the values of the device's ghost table
// (the same operations in the same order; no contraction on either side).
void march_ghosts(const GhostSpec& g, double gamma, double c, float out[4][16])
{
    for (int s = 0; s < 4; ++s) {
        for (int n = 0; n < 16; ++n) out[s][n] = 0.f;
        if (g.kind[s] != BC_DIRICHLET) continue;
        const double rho = g.prim[s][0], u0 = g.prim[s][1], v0 = g.prim[s][2], p0 = g.prim[s][3];
        const double U[4] = {rho, rho * u0, rho * v0, p0 / (gamma - 1.0) + 0.5 * rho * (u0 * u0 + v0 * v0)};
        const double u = U[1] / U[0], v = U[2] / U[0];
        const double p = (gamma - 1.0) * (U[3] - 0.5 * (U[1] * u + U[2] * v));
        const double F[4] = {U[1], U[1] * u + p, U[1] * v, u * (U[3] + p)};
        const double G[4] = {U[2], U[2] * u, U[2] * v + p, v * (U[3] + p)};
        for (int k = 0; k < 4; ++k) {
            const double a = 0.25 * U[k], b = c * F[k], d = c * G[k];
            out[s][k] = (float)((a - b) - d);
            out[s][4 + k] = (float)((a + b) - d);
            out[s][8 + k] = (float)((a + b) + d);
            out[s][12 + k] = (float)((a - b) + d);
        }
    }
}

cudaError_t launch_march_f32(const MarchStep& st, int steps, bool record, cudaStream_t s)
{
    MarchArgs a;
    a.src = st.src;
    a.dst = st.dst;
    memcpy(a.ghost, st.ghost, sizeof a.ghost);
    a.N = st.N;
    a.nx = st.nx;
    a.ny = st.ny;
    for (int n = 0; n < 4; ++n) a.bc[n] = st.bc[n];
    a.c = st.c;
    a.gm1 = st.gm1;
    if (record) return steps == 2 ? launch_k<2, true>(a, st.chained, s) : launch_k<1, true>(a, st.chained, s);
    return steps == 2 ? launch_k<2, false>(a, st.chained, s) : launch_k<1, false>(a, st.chained, s);
}

cudaError_t launch_pull_moments_f32(const StepArgs<float>& a, float* U, cudaStream_t s)
{
    const dim3 block(64, 4);
    const dim3 grid((unsigned)((a.nx + 63) / 64), (unsigned)((a.ny + 3) / 4));
    if (a.solid) pull_moments_2d_kernel<true><<<grid, block, 0, s>>>(a, U);
    else pull_moments_2d_kernel<false><<<grid, block, 0, s>>>(a, U);
    return cudaGetLastError();
}

cudaError_t launch_wall_codes(const StepArgs<float>& a, uint8_t* codes, cudaStream_t s)
{
    const dim3 grid((unsigned)((a.nx + 63) / 64), (unsigned)((a.ny + 3) / 4));
    wall_code_2d_kernel<<<grid, dim3(64, 4), 0, s>>>(a, codes);
    return cudaGetLastError();
}

cudaError_t launch_equilibria_f32(const float* U, float* f, const uint8_t* solid, int64_t N, float c, float gm1,
                                  cudaStream_t s)
{
    const int64_t threads = (N + 1) / 2;
    equilibria_2d_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(U, f, solid, nullptr, N, c, gm1);
    return cudaGetLastError();
}

bool adapt_moments_enabled()
{
    static const int v = [] {
        const char* e = getenv("LBRS_F32_ADAPT_MOMENTS");
        return (e && !strcmp(e, "0")) ? 0 : 1;
    }();
    return v != 0;
}

cudaError_t launch_adapt_enter_f32(const StepArgs<float>& a, float* U, void* st, void* run0,
                                   unsigned long long* bounds, double gamma, double dx, cudaStream_t s)
{
    const dim3 grid((unsigned)((a.nx + 63) / 64), (unsigned)((a.ny + 3) / 4));
    adapt_pull_kernel<<<grid, dim3(64, 4), 0, s>>>(a, U, (AdaptState*)st, gamma);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    adapt_enter_kernel<<<1, 32, 0, s>>>((const AdaptState*)st, (AdaptRun*)run0, bounds, dx);
    return cudaGetLastError();
}

cudaError_t launch_adapt_leave_f32(const float* U, float* f, int64_t N, float gm1, void* st, void* run,
                                   const unsigned long long* last_bounds, double dx, double safety, double t_final,
                                   cudaStream_t s)
{
    adapt_leave_kernel<<<1, 32, 0, s>>>((AdaptState*)st, (AdaptRun*)run, last_bounds, dx, safety, t_final);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t threads = (N + 1) / 2;
    equilibria_2d_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(U, f, nullptr, (const AdaptRun*)run, N, 0.f, gm1);
    return cudaGetLastError();
}

LBRS_DEBUG_WORD(debug_word_march)

}  // namespace lbrs

// FP32 D2Q4 steps of the distribution form at omega != 1, two per launch, the state in between in
// registers (sm_103a).
//
// A warp owns 30 columns (a lane each, one more on either side) and marches up its rows.  At row r it
// pulls row r's populations of the input state, collides (step 1), hands them to the columns beside by
// shuffles, and finishes row r - 1 of step 2 from them: f_0, f_1 come from row r, f_2, f_3 from row
// r - 2, which two sets of eight registers keep.  No shared memory, no barrier and no tensor copies
// (whose strides must be multiples of 16 bytes): every grid takes it as it is.
//
// A launch reads and writes the state once (128 B per cell for two steps).  Bound by that traffic from a
// full wave of warps on (5.2 TB/s; 1001 x 777 periodic, 100 MB of state in both buffers: 8.6 us per step,
// the direct-load two-step tile kernel 11.9), by the latency of an iteration (0.6 us) below.  Three steps
// a launch on the same plan needed 100 to 114 registers a lane and took as long or longer (8.6 us there at
// its best, with clamped sides 11.3 against 9.8); so did the fields two to a register pair in packed
// arithmetic (the pairs cost as many moves as it saves).
#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "lbrs_chain.cuh"
#include "lbrs_kernels.cuh"
#include "lbrs_launch.h"

namespace lbrs {
namespace {

constexpr int kFMOwn = 30;            // columns a warp stores
constexpr int kFMBlocks = 24;         // warps of an SM (80 registers a lane)

struct FMarchArgs {
    const float* src;
    float* dst;
    float* Uout;                      // recording: the moments of both steps, [2][4][N]
    float ghost[4][GHOST_STRIDE];     // f^eq of each Dirichlet side's state
    int64_t N;
    int nx, ny, rows;
    int bc[4];
    float om, om1, c, gm1;
};

// U of the pulled populations, then what the collision makes of them (collide_2d's operations).
__device__ __forceinline__ void fm_collide(const FMarchArgs& a, const float f[4][4], float U[4], float out[4][4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) U[k] = ((f[0][k] + f[1][k]) + f[2][k]) + f[3][k];
    float e[4][4];
    equilibria2d<float>(U, a.gm1, a.c, e);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) out[q][k] = a.om1 * f[q][k] + a.om * e[q][k];
}

// Row j's populations that sides replace: a Dirichlet y side's ghosts, over them a Dirichlet x side's
// (left, right: this lane's column lies beside one), over both the walls' mirror images.
__device__ __forceinline__ void fm_sides(const FMarchArgs& a, int j, bool left, bool right, float f[4][4])
{
    if (j == a.ny - 1 && a.bc[3] == BC_DIRICHLET) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[0][k] = a.ghost[3][k];
            f[1][k] = a.ghost[3][4 + k];
        }
    }
    if (j == 0 && a.bc[2] == BC_DIRICHLET) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[2][k] = a.ghost[2][8 + k];
            f[3][k] = a.ghost[2][12 + k];
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        f[0][k] = right ? a.ghost[1][k] : f[0][k];
        f[3][k] = right ? a.ghost[1][12 + k] : f[3][k];
        f[1][k] = left ? a.ghost[0][4 + k] : f[1][k];
        f[2][k] = left ? a.ghost[0][8 + k] : f[2][k];
    }
    if (j == a.ny - 1 && a.bc[3] == BC_WALL) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float s = k == 2 ? -1.f : 1.f;
            f[0][k] = s * f[3][k];
            f[1][k] = s * f[2][k];
        }
    }
    if (j == 0 && a.bc[2] == BC_WALL) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float s = k == 2 ? -1.f : 1.f;
            f[3][k] = s * f[0][k];
            f[2][k] = s * f[1][k];
        }
    }
}

// SIDES: not all four sides are periodic.
template <bool SIDES, bool RECORD>
__global__ void __launch_bounds__(32, kFMBlocks) fmarch_kernel(const FMarchArgs a)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x, i = (int)blockIdx.x * kFMOwn - 1 + lane;
    const int ja = (int)blockIdx.y * a.rows, jb = min(ja + a.rows, a.ny);
    const bool own = lane >= 1 && lane <= kFMOwn && i < a.nx;
    const bool xper = !SIDES || a.bc[0] == BC_PERIODIC, yper = !SIDES || a.bc[2] == BC_PERIODIC;
    // the lane's column and the ones its populations come from
    int x, xm, xp;
    if (xper) {
        x = i < 0 ? a.nx - 1 : i % a.nx;
        xm = x == 0 ? a.nx - 1 : x - 1;
        xp = x == a.nx - 1 ? 0 : x + 1;
    } else {
        x = min(max(i, 0), a.nx - 1);
        xm = max(x - 1, 0);
        xp = min(x + 1, a.nx - 1);
    }
    const bool left = SIDES && !xper && i == 0, right = SIDES && !xper && i == a.nx - 1;
    const bool dleft = left && a.bc[0] == BC_DIRICHLET, dright = right && a.bc[1] == BC_DIRICHLET;

    // Beyond a clamped side a row is the side's own, computed once more.
    auto row_of = [&](int j) { return yper ? (j < 0 ? j + a.ny : (j >= a.ny ? j - a.ny : j)) : min(max(j, 0), a.ny - 1); };
    chain_begin();
    float f[4][4];
    auto load = [&](int r) {
        const int j = row_of(r);
        const int64_t up = (int64_t)row_of(j + 1) * a.nx, down = (int64_t)row_of(j - 1) * a.nx;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[0][k] = chain_load(a.src + LBRS_IX((0 + k) * a.N + up + xp, 16 * a.N, 61));
            f[1][k] = chain_load(a.src + LBRS_IX((4 + k) * a.N + up + xm, 16 * a.N, 61));
            f[2][k] = chain_load(a.src + LBRS_IX((8 + k) * a.N + down + xm, 16 * a.N, 61));
            f[3][k] = chain_load(a.src + LBRS_IX((12 + k) * a.N + down + xp, 16 * a.N, 61));
        }
    };
    float h1[2][4], h2[2][4];           // f_2, f_3 of the rows r - 1 and r - 2, as their receivers see them
#pragma unroll
    for (int k = 0; k < 4; ++k) h1[0][k] = h1[1][k] = h2[0][k] = h2[1][k] = 0.f;
    load(ja - 1);
#pragma unroll 1
    for (int r = ja - 1; r <= jb; ++r) {
        float U[4], o[4][4];
        if constexpr (SIDES) fm_sides(a, row_of(r), dleft, dright, f);
        fm_collide(a, f, U, o);
        if (RECORD && own && r >= ja && r < jb) {
#pragma unroll
            for (int k = 0; k < 4; ++k) a.Uout[LBRS_IX(k * a.N + (int64_t)r * a.nx + i, 8 * a.N, 62)] = U[k];
        }
        if (r < jb) load(r + 1);        // its latency passes under step 2
        float g[4][4];                  // row r - 1 of step 2
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float n0 = __shfl_down_sync(full, o[0][k], 1), n1 = __shfl_up_sync(full, o[1][k], 1);
            const float n2 = __shfl_up_sync(full, o[2][k], 1), n3 = __shfl_down_sync(full, o[3][k], 1);
            g[0][k] = SIDES && right ? o[0][k] : n0;
            g[1][k] = SIDES && left ? o[1][k] : n1;
            g[2][k] = h2[0][k];
            g[3][k] = h2[1][k];
            h2[0][k] = h1[0][k];
            h2[1][k] = h1[1][k];
            h1[0][k] = SIDES && left ? o[2][k] : n2;
            h1[1][k] = SIDES && right ? o[3][k] : n3;
        }
        if (r <= ja) continue;
        const int j = r - 1;
        if constexpr (SIDES) fm_sides(a, j, dleft, dright, g);
        fm_collide(a, g, U, o);
        if (own) {
            const int64_t row = (int64_t)j * a.nx;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < 4; ++k) a.dst[LBRS_IX((q * 4 + k) * a.N + row + i, 16 * a.N, 63)] = o[q][k];
            if constexpr (RECORD) {
#pragma unroll
                for (int k = 0; k < 4; ++k) a.Uout[LBRS_IX((4 + k) * a.N + row + i, 8 * a.N, 62)] = U[k];
            }
        }
    }
}

}  // namespace

bool fmarch_enabled()
{
    static const int v = [] {
        const char* e = getenv("LBRS_F32_FMARCH");
        return (e && !strcmp(e, "0")) ? 0 : 1;
    }();
    return v != 0;
}

// Rows of a warp: as few as leave one wave of warps (64 x 64 periodic 1.41 us per step at 1 row, 1.67 at 2,
// 1.92 at 3; 1000 x 1000 at 10 rows 11.6, at 8 in two waves 13.2), 8 where a wave would take more than 12.
static int64_t fmarch_wave_rows(int nx, int ny)
{
    const int64_t slots = kSMs * kFMBlocks;
    return ((int64_t)((nx + kFMOwn - 1) / kFMOwn) * ny + slots - 1) / slots;
}

static int fmarch_rows(int nx, int ny)
{
    const int64_t n = fmarch_wave_rows(nx, ny);
    return n > 12 ? 8 : (int)std::max<int64_t>(n, 1);
}

// The marching kernel rather than the tile kernel's two steps a launch?  While one wave takes at most 10 rows
// (1024^2, calls of two: 30.8 us against 34.8, recording 38.9 against 43.0).  Grids that the tiles' tensor
// copies cannot take march at any size (2047^2: two steps on tiles by plain loads 57.8 us a step, march 52.0).
bool fmarch_beats_pairs(int nx, int ny) { return fmarch_wave_rows(nx, ny) <= 10; }

// Rather than three steps a launch on tiles?  Up to about a million cells, whose two buffers the second-level
// cache holds in good part (us per step, periodic, tiles against march: 128^2 3.99, 2.91; 512^2 6.19, 5.21;
// 800^2 9.07, 7.41; 960^2 12.1, 11.5; 1000^2 13.35, 12.65; 1008^2 13.4, 13.1; 2048 x 500 12.9, 13.1; 1024^2 13.2,
// 13.4; 2048^2 37, 50).  The march has no work beside sides of other kinds where the tiles do (clamped, 1024^2
// 14.5, 13.5).  Recording adds 32 B a cell to every two steps of either, which costs the march more (800^2
// 10.4, 10.3; 896^2 12.5, 13.5; 1024^2 15.1, 17.8).
bool fmarch_beats_threes(int nx, int ny, bool periodic, bool record)
{
    const int64_t rows = fmarch_wave_rows(nx, ny);
    if (record) return rows <= 6;
    return rows <= 10 && (!periodic || (int64_t)nx * ny <= 1020000);
}

cudaError_t launch_fmarch_f32(const StepArgs<float>& s, const float ghost[4][GHOST_STRIDE], bool chained,
                              cudaStream_t st)
{
    FMarchArgs a;
    a.src = s.src;
    a.dst = s.dst;
    a.Uout = s.Uout;
    memcpy(a.ghost, ghost, sizeof a.ghost);
    a.N = s.N;
    a.nx = s.nx;
    a.ny = s.ny;
    bool sides = false;
    for (int n = 0; n < 4; ++n) {
        a.bc[n] = s.bc[n];
        sides = sides || s.bc[n] != BC_PERIODIC;
    }
    a.om = s.om;
    a.om1 = s.om1;
    a.c = s.c;
    a.gm1 = s.gm1;
    const int64_t strips = (s.nx + kFMOwn - 1) / kFMOwn;
    a.rows = fmarch_rows(s.nx, s.ny);
    const dim3 grid((unsigned)strips, (unsigned)((s.ny + a.rows - 1) / a.rows));
    if (s.Uout) {
        if (sides) return launch_in_chain(chained, fmarch_kernel<true, true>, grid, 32, st, a);
        return launch_in_chain(chained, fmarch_kernel<false, true>, grid, 32, st, a);
    }
    if (sides) return launch_in_chain(chained, fmarch_kernel<true, false>, grid, 32, st, a);
    return launch_in_chain(chained, fmarch_kernel<false, false>, grid, 32, st, a);
}

LBRS_DEBUG_WORD(debug_word_fmarch)

}  // namespace lbrs

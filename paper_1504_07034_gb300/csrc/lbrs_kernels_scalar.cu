// Launchers of the scalar D2Q4 window kernel (lbrs_scalar.cuh).
#include <stdlib.h>
#include <string.h>

#include "lbrs_scalar.cuh"
#include "lbrs_launch.h"

namespace lbrs {

namespace {

constexpr size_t kSmemPerSM = 227 * 1024;

template <int R>
cudaError_t launch_r(const ScalarArgs& a, dim3 grid, int threads, size_t smem, cudaStream_t s)
{
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(step2ds_window_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)kSmemPerSM);
        if (e != cudaSuccess) return e;
    }
    step2ds_window_kernel<R><<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

int threads_for(int wx, int wy, int r) { return wx / 2 * ((wy + r - 1) / r); }

}  // namespace

bool scalar_windows_enabled()
{
    static const int v = [] {
        const char* e = getenv("LBRS_F32S_WINDOW");
        return (e && !strcmp(e, "0")) || getenv("LBRS_F32S_TILE_Y") ? 0 : 1;   // (the two-step kernel's tile height)
    }();
    return v != 0;
}

// A grid that one window holds takes all its steps in one launch, up to 6,400 cells (64^2: 1.05 us a step;
// 1.42 with eight rows a thread, 1.33 in 32 x 32 windows of eight steps a launch.  400 steps: 76^2 in one
// window 514 us, 84 x 86 631, 125 x 62 605; 96^2 in windows of 64 x 32 568).  Larger grids: eight steps a
// launch, windows and rows per thread growing with the grid as the SMs fill (us a step: 256^2 in 64 x 32
// windows 1.58, 64 x 64 1.84, 128 x 64 2.88; 512^2 2.13, 1.87, 3.16; 2048^2 17.4, 13.7, and 12.0 in 128 x 64
// with eight rows a thread).
//
// A window costs its loads and stores whatever the steps, so short calls keep the two-step kernel (us for
// 2, 3, .. steps by windows and by that kernel: 64^2 17 17 18 and 11 16 20; 76^2 21 21 23 24 and 12 15 19 24;
// 256^2 13 15 and 11 16; 1024^2 34 36 40 42 44 48 and 17 25 31 39 45 54; 4096^2 230 252 273 296 317 340 and 93
// 184 184 275 274 365), and so do the last steps of a call that would leave a window mostly unused (4096^2,
// the last launch of 1, 2, 3, 4 steps 175, 197, 217, 240 by a window and 91, 92, 183, 184 by two steps, beside
// 30 for distributions to start them from; 2048^2 45, 51, 57, 65 and 31, 31, 62, 62 beside 7).
ScalarPlan scalar_plan(int nx, int ny, const int bc[4])
{
    const int64_t cells = (int64_t)nx * ny;
    ScalarPlan p{};
    if (bc[0] != BC_PERIODIC && bc[2] != BC_PERIODIC && cells <= 6400) {
        p.wx = (nx + 3 + 1) / 2 * 2;
        p.wy = ny + 2;
        p.hx = 2;
        p.hy = 1;
        p.tx = nx;
        p.ty = ny;
        p.rows = 4;
        p.steps = 512;
        p.min_steps = cells <= 5200 ? 4 : 5;
        if (threads_for(p.wx, p.wy, p.rows) <= 1024) return p;
        p = ScalarPlan{};
    }
    // Flat grids keep the low windows, whose rows they fill better (40 steps, us, low and high ones: 20000 x 8 89,
    // 150; 65536 x 12 207, 392; 200000 x 16 563, 935; 65536 x 20 374, 338), and the flattest large ones the two-step
    // kernel (10 steps, us, windows and that kernel: 200000 x 4 187, 147; 65536 x 4 71, 65; 200000 x 6 153, 157).
    if (ny < 6 && cells >= 100000) return p;
    const bool flat = ny <= 16, wide = cells >= 1000000 && !flat;
    p.wx = wide ? 128 : 64;
    p.wy = cells < 150000 || flat ? 32 : 64;
    p.rows = wide ? 8 : 4;
    p.hx = p.hy = p.steps = 8;
    p.tx = p.wx - 16;
    p.ty = p.wy - 16;
    p.min_steps = cells < 1000000 ? 3 : 7;
    p.tail = cells < 1000000 ? 0 : (cells < 8000000 ? 2 : 4);
    return p;
}

cudaError_t launch_scalar_window(const StepArgs<float>& f, const ScalarPlan& p, const float* u, float* dst, int steps,
                                 bool loadf, bool storef, cudaStream_t s)
{
    ScalarArgs a;
    a.src = u;
    a.dst = dst;
    a.f = f;
    a.wx = p.wx;
    a.wy = p.wy;
    a.hx = p.hx;
    a.hy = p.hy;
    a.tx = p.tx;
    a.ty = p.ty;
    a.steps = steps;
    a.loadf = loadf;
    a.storef = storef;
    const dim3 grid((unsigned)((f.nx + p.tx - 1) / p.tx), (unsigned)((f.ny + p.ty - 1) / p.ty));
    const size_t smem = 2 * sizeof(float) * (size_t)p.wx * p.wy;
    const int threads = threads_for(p.wx, p.wy, p.rows);
    if (p.rows == 4) return launch_r<4>(a, grid, threads, smem, s);
    return launch_r<8>(a, grid, threads, smem, s);
}

LBRS_DEBUG_WORD(debug_word_scalar)

}  // namespace lbrs

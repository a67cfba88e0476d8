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

// A grid that one window holds at four rows a thread (about 5,900 cells) takes all its steps in one
// launch (64^2: 1.05 us a step; 1.42 with eight rows a thread, 1.33 in 32 x 32 windows of eight steps a
// launch).  Larger grids: eight steps a launch, windows and rows per thread growing with the grid as
// the SMs fill (us a step: 256^2 in 64 x 32 windows 1.58, 64 x 64 1.84, 128 x 64 2.88; 512^2 2.13, 1.87,
// 3.16; 2048^2 17.4, 13.7, and 12.0 in 128 x 64 with eight rows a thread).
ScalarPlan scalar_plan(int nx, int ny, const int bc[4])
{
    ScalarPlan p{};
    if (bc[0] != BC_PERIODIC && bc[2] != BC_PERIODIC && (int64_t)nx * ny <= 16384) {
        p.wx = (nx + 3 + 1) / 2 * 2;
        p.wy = ny + 2;
        p.hx = 2;
        p.hy = 1;
        p.tx = nx;
        p.ty = ny;
        p.rows = 4;
        p.steps = 512;
        if (threads_for(p.wx, p.wy, p.rows) <= 1024) return p;
    }
    const int64_t cells = (int64_t)nx * ny;
    p.wx = cells < 1000000 ? 64 : 128;
    p.wy = cells < 150000 ? 32 : 64;
    p.rows = cells < 1000000 ? 4 : 8;
    p.hx = p.hy = p.steps = 8;
    p.tx = p.wx - 16;
    p.ty = p.wy - 16;
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

// Launchers of the FP32 1-D kernel (lbrs_tube.cuh): batched tubes and single ones.
#include "lbrs_tube.cuh"
#include "lbrs_launch.h"

namespace lbrs {

namespace {

template <int Q, int C, bool UFORM>
cudaError_t launch_q(const TubeArgs& a, cudaStream_t s)
{
    tube_kernel<Q, C, UFORM><<<(unsigned)((a.ntiles + kTubeWarps - 1) / kTubeWarps), 32 * kTubeWarps, 0, s>>>(a);
    return cudaGetLastError();
}

template <int C, bool UFORM>
cudaError_t launch_c(const TubeArgs& a, int q, cudaStream_t s)
{
    return q == 3 ? launch_q<3, C, UFORM>(a, s) : launch_q<2, C, UFORM>(a, s);
}

// Cells per lane of the batched windows: as many as the registers hold, since the halo is
// recomputed once per window (16 on the moments, 8 on the populations).
constexpr int kBatchCellsU = 16, kBatchCellsF = 8;

TubeArgs tube_args(const BatchArgs<float>& b)
{
    TubeArgs a;
    a.src = b.src;
    a.dst = b.dst;
    a.N = b.N;
    a.tiles = b.tiles;
    a.tube_off = b.tube_off;
    a.tube_len = b.tube_len;
    a.tube_steps = b.tube_steps;
    a.tube_c = b.tube_c;
    a.ntiles = 0;
    a.one_len = b.one_len;
    a.one_steps = b.one_steps;
    a.one_c = b.one_c;
    a.halo = b.halo;
    a.launch = b.launch;
    a.periodic = b.periodic;
    a.om = b.om;
    a.om1 = b.om1;
    a.gm1 = b.gm1;
    return a;
}

}  // namespace

int tube_tile_cells(int halo, bool omega1)
{
    if (halo > kTubeMaxHalo) return 0;
    return omega1 ? 32 * kBatchCellsU - 2 * tube_pad<kBatchCellsU>(halo)
                  : 32 * kBatchCellsF - 2 * tube_pad<kBatchCellsF>(halo);
}

cudaError_t launch_tubes_f32(const BatchArgs<float>& b, int ntiles, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    TubeArgs a = tube_args(b);
    a.ntiles = ntiles;
    return b.om1 == 0.f ? launch_c<kBatchCellsU, true>(a, b.q, s) : launch_c<kBatchCellsF, false>(a, b.q, s);
}

// A tube by itself, one_steps <= halo steps in one launch.
//
// Four cells a lane (tiles of 64 cells at 32 steps a launch), which spreads a short tube over more SMs; tubes
// that fill them use no more halo than the launch has steps.  The batched windows, which recompute less, take
// over in launches of more than 16 steps of long tubes (32 steps, four cells a lane and batched windows, us:
// D1Q2 at omega = 1 200,000 cells 19, 21; 300,000 23, 27; 500,000 33, 27; 4,000,000 224, 134; D1Q3 300,000 29,
// 32, 500,000 42, 33; omega != 1 D1Q2 140,000 23, 25; 200,000 29, 25; D1Q3 140,000 27, 31; 200,000 35, 31.
// 16 steps: 1,000,000 cells 28, 28; 35, 33; 44, 40; 56, 60).
//
// At omega != 1, where a lane holds the populations and they turn through shared memory once each, launches of
// few steps stay with the shared-memory kernel (four cells a lane and that kernel, us: D1Q2 1,000,000 cells
// 1 step 17, 13; 2 steps 18, 15; 4 steps 21, 19; 6 steps 23, 25; 4,000,000 cells 60, 50; 64, 57; 72, 69; 87,
// 83; D1Q3 4,000,000 cells 89, 78; 94, 91; 4 steps 105, 124; 20,000 cells 11, 9; 11, 11), and so do tubes of a
// few warps (100 steps: D1Q2 64 cells 35, 31; 128 cells 38, 31; 200 cells 40, 37; 320 cells 40, 44; 8 steps: D1Q3
// 64 cells 10, 9; 200 cells 11, 9).
cudaError_t launch_one_tube_f32(const BatchArgs<float>& b, cudaStream_t s)
{
    const bool u = b.om1 == 0.f;
    const int len = b.one_len, m = b.one_steps;
    const bool shared = !u && (b.q == 2 ? len < 256 || m <= 4 : m <= (len < 256 ? 8 : (len < 1000 ? 4 : 1)));
    if (shared) {
        constexpr int kBlock = 256, kCells = 4;
        BatchArgs<float> a = b;
        a.tile_cells = kBlock * kCells - 2 * a.halo;
        const cudaError_t e = prepare_batch_f32(kBlock, b.q);
        if (e != cudaSuccess) return e;
        return launch_batch_f32(a, (len + a.tile_cells - 1) / a.tile_cells, kBlock, s);
    }
    TubeArgs a = tube_args(b);
    if (len >= 150000 && m < a.halo) a.halo = m;
    const bool wide = m > 16 && len >= (u ? 400000 : 170000);
    const int tile = wide ? tube_tile_cells(a.halo, u) : 32 * 4 - 2 * tube_pad<4>(a.halo);
    a.ntiles = (len + tile - 1) / tile;
    if (wide) return u ? launch_c<kBatchCellsU, true>(a, b.q, s) : launch_c<kBatchCellsF, false>(a, b.q, s);
    return u ? launch_c<4, true>(a, b.q, s) : launch_c<4, false>(a, b.q, s);
}

LBRS_DEBUG_WORD(debug_word_tube)

}  // namespace lbrs

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

// A tube by itself: four cells a lane (tiles of 64 cells at 32 steps a launch), which spreads a
// short tube over more SMs, until the chip has as many warps as it can use (8 per SM); then the
// batched windows, which recompute less.
cudaError_t launch_one_tube_f32(const BatchArgs<float>& b, cudaStream_t s)
{
    TubeArgs a = tube_args(b);
    const bool u = b.om1 == 0.f;
    const int small = 32 * 4 - 2 * tube_pad<4>(a.halo), large = tube_tile_cells(a.halo, u);
    const bool wide = a.one_len > 152 * 8 * small;
    const int tile = wide ? large : small;
    a.ntiles = (a.one_len + tile - 1) / tile;
    if (wide) return u ? launch_c<kBatchCellsU, true>(a, b.q, s) : launch_c<kBatchCellsF, false>(a, b.q, s);
    return u ? launch_c<4, true>(a, b.q, s) : launch_c<4, false>(a, b.q, s);
}

LBRS_DEBUG_WORD(debug_word_tube)

}  // namespace lbrs

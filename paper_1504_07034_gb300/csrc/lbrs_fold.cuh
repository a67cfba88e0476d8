// Folding of the diagnostics' partial records (sm_103a): one block, in a fixed order.
//
// One thread that loads a record and adds it waits a trip to memory per record (608 records 0.3 ms).
// Here the block brings them to shared memory together and eight lanes fold each field, every eighth
// record each, then their eight results pairwise: bound by 76 dependent FP64 additions of 60 ns (one
// lane a field: 40 us; lbrs_diagnostics of 64 x 64 cells 376 us with one thread in all, 80 with one lane
// a field, 53 now).
#pragma once

#include "lbrs_kernels.cuh"

namespace lbrs {

constexpr int kFoldThreads = 256;
constexpr int kFoldChunk = 512;          // records in shared memory at a time

constexpr int kFoldLanes = 8;

// Totals (fields 0..3), minima (4, 5), maximum (6) and counts (7, 8) of nrec records of DIAG_W words;
// the totals times `scale` (all by the kFoldThreads threads of one block).
__device__ __forceinline__ void fold_diag_records(const double* rec, int nrec, double scale, double* out)
{
    const unsigned full = 0xffffffffu;
    __shared__ double s[kFoldChunk * DIAG_W];
    // warp 0 adds the totals, warp 1 the counts, warp 2 takes the minima, warp 3 the maximum
    const int warp = threadIdx.x / 32, group = threadIdx.x % 32 / kFoldLanes, lane = threadIdx.x % kFoldLanes;
    const int field = warp == 0 ? group : (warp == 1 ? 7 + group : (warp == 2 ? 4 + group : 6));
    const bool mine = warp == 0 || (warp < 3 && group < 2) || (warp == 3 && group == 0);
    double acc = warp == 2 ? INFINITY : 0.0;
    for (int r0 = 0; r0 < nrec; r0 += kFoldChunk) {
        const int n = min(kFoldChunk, nrec - r0);
        __syncthreads();
        for (int k = threadIdx.x; k < n * DIAG_W; k += kFoldThreads) s[k] = rec[(int64_t)r0 * DIAG_W + k];
        __syncthreads();
        if (!mine) continue;
        const double* p = s + field;
        if (warp < 2) {
#pragma unroll 8
            for (int r = lane; r < n; r += kFoldLanes) acc += p[r * DIAG_W];
        } else if (warp == 2) {
#pragma unroll 8
            for (int r = lane; r < n; r += kFoldLanes) acc = fmin(acc, p[r * DIAG_W]);
        } else {
#pragma unroll 8
            for (int r = lane; r < n; r += kFoldLanes) acc = fmax(acc, p[r * DIAG_W]);
        }
    }
    if (warp > 3) return;
#pragma unroll
    for (int off = 1; off < kFoldLanes; off *= 2) {
        const double o = __shfl_xor_sync(full, acc, off);
        acc = warp < 2 ? acc + o : (warp == 2 ? fmin(acc, o) : fmax(acc, o));
    }
    if (mine && lane == 0) out[field] = field < 4 ? acc * scale : acc;
    if (threadIdx.x == 127) out[9] = 0.0;
}

// The sum of one word a record, valid in thread 0.
__device__ __forceinline__ double fold_sum(const double* rec, int nrec)
{
    double acc = 0.0;
    if (threadIdx.x >= 32) return acc;
#pragma unroll 4
    for (int r = threadIdx.x; r < nrec; r += 32) acc += rec[r];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    return acc;
}

}  // namespace lbrs

// lll_paths_block.cuh -- the time-blocked path kernel of one simulation and its
// choice by node count, paths per thread and path count.  Caplets
// (lll_paths_block.cu) and swaptions (lll_paths_swaption.cu) are compiled apart.
#pragma once

#include <cuda_runtime.h>

#include "lll_device.cuh"
#include "lll_internal.h"
#include "lll_sweep.cuh"

namespace lll {

typedef void (*BlockFn)(const PathArgs);
// lll_paths_swaption.cu
BlockFn pick_swaption_kernel(int scheme, int QP, int R, uint64_t paths);
int launch_wide_swaptions(int scheme, int QP, int R, int grid, int threads, cudaStream_t st, const PathArgs &a);

namespace {

// Steps per block for QP nodes and R paths per thread.  N = 120 (20 nodes, four
// steps a period), 2^17 paths: 14.7 ms with two steps, 13.4 with four.
__host__ __device__ constexpr int steps_of(int QP, int R)
{
    return R == 2 ? (QP <= 4 ? 8 : QP <= 8 ? 4 : QP <= 24 ? 2 : 1) : (QP <= 8 ? 8 : QP <= 20 ? 4 : 2);
}

// Blocks of 256 threads per SM the registers are budgeted for.  (With 20 nodes
// and four steps the Picard kernel gains by 128 registers, 15.6 -> 14.0 ms; the
// full one from kManyPaths on.)
__host__ __device__ constexpr int blocks_of(int scheme, int QP, int R)
{
    return R * steps_of(QP, R) * QP <= 64 || (scheme == PICARD && R == 1 && QP == 20) ? 2 : 1;
}

template <int PRICES, int SCHEME, int QP, int R, int BL = blocks_of(SCHEME, QP, R)>
__global__ void __launch_bounds__(kMaxThreads, BL) block_kernel(const PathArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int B = steps_of(QP, R), NST = (SCHEME == PICARD) ? 2 : 1;
    const int T = blockDim.x, tid = threadIdx.x;
    const BlockSmem sm = block_carve(smem_raw, QP, B, R, a.n, T, a.chunk_rows);
    for (int e = tid; e < a.n; e += T) sm.c0[e] = -1.4426950408889634f * a.c0[e];
    for (int e = tid; e < QP; e += T) reinterpret_cast<float *>(sm.cn)[e] = a.cn[e];
    State<NST * R> *st = reinterpret_cast<State<NST * R> *>(a.state) + (size_t)blockIdx.x * a.n * T + tid;
    const size_t nout = (size_t)a.n * a.ns * 2;
    double *acc = a.partials + blockIdx.x * nout, *comp = a.partials + (gridDim.x + blockIdx.x) * nout;
    const uint64_t TP = (uint64_t)T * R, ntiles = (a.paths + TP - 1) / TP;
    __shared__ int beyond; // (of the swaptions' kernels only)
    if (PRICES == SWAPTIONS && tid == 0) beyond = 0; // ordered by the tile's first barrier
    for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
        block_tile<SCHEME, QP, B, R, PRICES>(a, sm, st, tile, acc, comp, tile == blockIdx.x, &beyond);
    // a mark for wide_kernel, which runs next
    if (PRICES == SWAPTIONS) {
        __syncthreads();
        if (tid == 0 && beyond) comp[0] = nan("");
    }
}

// The full scheme on 20 nodes runs as well in two blocks of 128 threads an SM at
// 192 registers as in four at 128 (a wave of 38,912 paths 3.9 ms, of 77,824 paths
// 7.4); the two differ by how many paths the last wave is short of, and from here
// on the larger wave wins throughout: N = 120, 140,000 paths 14.8 ms at 128
// registers, 15.5 at 192, 2^20 paths 99.7 and 108.7.  Below, 192 registers are
// taken, which is not always the better: 116,000 paths 11.6 ms (12.9 at 128), but
// 55,000 paths 7.7 (6.0).  Other node counts were not measured for it.
constexpr uint64_t kManyPaths = 140000;

template <int PRICES, int SCHEME, int R>
BlockFn pick_qp(int QP)
{
    switch (QP) {
    case 4: return block_kernel<PRICES, SCHEME, 4, R>;
    case 8: return block_kernel<PRICES, SCHEME, 8, R>;
    case 12: return block_kernel<PRICES, SCHEME, 12, R>;
    case 16: return block_kernel<PRICES, SCHEME, 16, R>;
    case 20: return block_kernel<PRICES, SCHEME, 20, R>;
    case 24: return block_kernel<PRICES, SCHEME, 24, R>;
    case 32: return block_kernel<PRICES, SCHEME, 32, R>;
    default: return nullptr;
    }
}

template <int PRICES>
BlockFn pick(int scheme, int QP, int R, uint64_t paths)
{
    if (scheme == FULL && QP == 20 && R == 1 && paths >= kManyPaths) return block_kernel<PRICES, FULL, 20, 1, 2>;
    if (scheme == FULL) return R == 1 ? pick_qp<PRICES, FULL, 1>(QP) : R == 2 ? pick_qp<PRICES, FULL, 2>(QP) : nullptr;
    if (scheme == PICARD) return R == 1 ? pick_qp<PRICES, PICARD, 1>(QP) : R == 2 ? pick_qp<PRICES, PICARD, 2>(QP) : nullptr;
    return nullptr;
}

}  // namespace
}  // namespace lll

// lll_paths_block.cu -- the path kernels for rules with a shorter equivalent
// (shorter_rule in lll_quadrature.cpp): full and Picard schemes, time-blocked
// rate sweep (lll_sweep.cuh), one simulation or a batch of instances.
//
// With 4 to 32 nodes in place of the given 32 to 128 a unit (path, rate, step)
// is 1.5 QP packed FP32 instructions and about ten others, so what a unit costs
// besides the nodes decides: R = 2 paths a thread share each table load, and
// the block length B keeps R B QP near 64 registers of node products.
//
// Measured on a GB300 (whole call, prices read) against the step-by-step sweep
// of the rule as given (lll_paths.cu): Picard, N = 40, 64 -> 8 nodes, 2^20
// paths 59.8 -> 15.0 ms, of which the shorter rule alone in that sweep gave
// 29.7; full, N = 120, 96 -> 24 nodes, 2^17 paths 63.1 -> 18.3 ms (27.1); full,
// N = 40, 4096 paths 2.11 -> 0.66 ms (1.02).
#include <cuda_runtime.h>

#include "lll_device.cuh"
#include "lll_internal.h"
#include "lll_sweep.cuh"

namespace lll {
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

template <int SCHEME, int QP, int R, int BL = blocks_of(SCHEME, QP, R)>
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
    for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
        block_tile<SCHEME, QP, B, R>(a, sm, st, tile, acc, comp, tile == blockIdx.x);
}

// A batch: the blocks claim items as in batch_kernel (lll_paths.cu), and take
// each instance at its own rule's length, up to QMAX nodes.
template <int SCHEME, int QP, int R>
__device__ __forceinline__ void batch_item(const PathArgs &a, unsigned char *smem, float *state, uint2 tiles, double *acc,
                                           double *comp)
{
    constexpr int B = steps_of(QP, R), NST = (SCHEME == PICARD) ? 2 : 1;
    const int T = blockDim.x, tid = threadIdx.x;
    const BlockSmem sm = block_carve(smem, QP, B, R, a.n, T, a.chunk_rows);
    for (int e = tid; e < a.n; e += T) sm.c0[e] = -1.4426950408889634f * a.c0[e];
    for (int e = tid; e < QP; e += T) reinterpret_cast<float *>(sm.cn)[e] = a.cn[e];
    State<NST * R> *st = reinterpret_cast<State<NST * R> *>(state) + tid;
    for (uint32_t t = tiles.x; t < tiles.y; ++t)
        block_tile<SCHEME, QP, B, R>(a, sm, st, t, acc, comp, t == tiles.x);
}

template <int SCHEME, int QMAX, int R>
__global__ void __launch_bounds__(kMaxThreads, blocks_of(FULL, QMAX > 8 ? 24 : 8, R)) batch_block_kernel(const BatchArgs b)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NST = (SCHEME == PICARD) ? 2 : 1;
    const int T = blockDim.x, tid = threadIdx.x;
    float *state = b.state + (size_t)blockIdx.x * R * NST * b.n_max * T;
    __shared__ PathArgs sa; // the current instance's arguments
    __shared__ int claimed;
    int cur = -1;
    for (;;) {
        __syncthreads(); // the previous item's readers of sa and shared memory are done
        if (tid == 0) claimed = atomicAdd(b.next, 1);
        __syncthreads();
        const int it = claimed;
        if (it >= b.n_items) break;
        const int q = b.item_inst[it];
        if (q != cur) {
            cur = q;
            if (tid == 0) sa = b.desc[q];
            __syncthreads();
        }
        const uint2 tr = b.item_tiles[it];
        double *acc = b.partials + b.seg_off[it], *comp = b.comps + b.seg_off[it];
        switch (sa.qr) {
        case 4: batch_item<SCHEME, 4, R>(sa, smem_raw, state, tr, acc, comp); break;
        case 8: batch_item<SCHEME, 8, R>(sa, smem_raw, state, tr, acc, comp); break;
        default:
            if constexpr (QMAX > 8) {
                if (sa.qr == 12) batch_item<SCHEME, 12, R>(sa, smem_raw, state, tr, acc, comp);
                else if (sa.qr == 16) batch_item<SCHEME, 16, R>(sa, smem_raw, state, tr, acc, comp);
                else if (sa.qr == 20) batch_item<SCHEME, 20, R>(sa, smem_raw, state, tr, acc, comp);
                else if (sa.qr == 24) batch_item<SCHEME, 24, R>(sa, smem_raw, state, tr, acc, comp);
                else batch_item<SCHEME, 32, R>(sa, smem_raw, state, tr, acc, comp);
            }
        }
    }
}

typedef void (*KernelFn)(const PathArgs);

// The full scheme on 20 nodes runs as well in two blocks of 128 threads an SM at
// 192 registers as in four at 128 (a wave of 38,912 paths 3.9 ms, of 77,824 paths
// 7.4); the two differ by how many paths the last wave is short of, and from here
// on the larger wave wins throughout: N = 120, 140,000 paths 14.8 against 15.5 ms,
// 2^20 paths 99.7 against 108.7.  (Below, either may: 116,000 paths 12.9 against
// 11.6, 55,000 paths 6.0 against 7.7.)
constexpr uint64_t kManyPaths = 140000;
typedef void (*BatchFn)(const BatchArgs);

template <int SCHEME, int R>
KernelFn pick_qp(int QP)
{
    switch (QP) {
    case 4: return block_kernel<SCHEME, 4, R>;
    case 8: return block_kernel<SCHEME, 8, R>;
    case 12: return block_kernel<SCHEME, 12, R>;
    case 16: return block_kernel<SCHEME, 16, R>;
    case 20: return block_kernel<SCHEME, 20, R>;
    case 24: return block_kernel<SCHEME, 24, R>;
    case 32: return block_kernel<SCHEME, 32, R>;
    default: return nullptr;
    }
}

KernelFn pick(int scheme, int QP, int R, uint64_t paths)
{
    if (scheme == FULL && QP == 20 && R == 1 && paths >= kManyPaths) return block_kernel<FULL, 20, 1, 2>;
    if (scheme == FULL) return R == 1 ? pick_qp<FULL, 1>(QP) : R == 2 ? pick_qp<FULL, 2>(QP) : nullptr;
    if (scheme == PICARD) return R == 1 ? pick_qp<PICARD, 1>(QP) : R == 2 ? pick_qp<PICARD, 2>(QP) : nullptr;
    return nullptr;
}

BatchFn pick_batch(int scheme, int QMAX, int R)
{
    if (QMAX == 8) {
        if (scheme == FULL) return R == 1 ? batch_block_kernel<FULL, 8, 1> : batch_block_kernel<FULL, 8, 2>;
        return R == 1 ? batch_block_kernel<PICARD, 8, 1> : batch_block_kernel<PICARD, 8, 2>;
    }
    if (scheme == FULL) return R == 1 ? batch_block_kernel<FULL, 32, 1> : batch_block_kernel<FULL, 32, 2>;
    return R == 1 ? batch_block_kernel<PICARD, 32, 1> : batch_block_kernel<PICARD, 32, 2>;
}

template <class F>
int prepare(F f, size_t smem, size_t most, int threads, int *blocks_per_sm)
{
    if (!f) return (int)cudaErrorInvalidValue;
    const cudaError_t e = allow_smem(f, smem, most);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, f, threads, smem);
}

}  // namespace

// Rates per staged chunk: `rows` (0: all) as far as the double-buffered rows
// stay near 24 KB, so that shared memory does not limit the resident blocks.
int block_chunk_rates(int QP, int R, int n, int rows)
{
    const int fit = (24 * 1024) / (2 * steps_of(QP, R) * (QP * 4 + 16));
    return max(1, min(rows > 0 ? min(rows, n) : n, fit));
}

size_t block_kernel_smem(int QP, int R, int n, int threads, int chunk_rates)
{
    return block_smem_bytes(QP, steps_of(QP, R), R, n, threads, chunk_rates);
}

int block_kernel_prepare(int scheme, int QP, int R, uint64_t paths, size_t smem, int threads, int *blocks_per_sm)
{
    return prepare(pick(scheme, QP, R, paths), smem, kMaxSmem, threads, blocks_per_sm);
}

int launch_block_kernel(int scheme, int QP, int R, int grid, int threads, size_t smem, cudaStream_t st, const PathArgs &a)
{
    KernelFn f = pick(scheme, QP, R, a.paths);
    if (!f) return (int)cudaErrorInvalidValue;
    f<<<grid, threads, smem, st>>>(a);
    return (int)cudaGetLastError();
}

int batch_block_prepare(int scheme, int QMAX, int R, size_t smem, int threads, int *blocks_per_sm)
{
    // less its static shared memory
    return prepare(pick_batch(scheme, QMAX, R), smem, kMaxSmem - 1024, threads, blocks_per_sm);
}

int launch_batch_block_kernel(int scheme, int QMAX, int R, int grid, int threads, size_t smem, cudaStream_t st,
                              const BatchArgs &b)
{
    BatchFn f = pick_batch(scheme, QMAX, R);
    f<<<grid, threads, smem, st>>>(b);
    return (int)cudaGetLastError();
}

}  // namespace lll

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
// paths 59.8 -> 12.7 ms; full, N = 120, 96 -> 20 nodes, 2^17 paths 63.1 -> 13.6
// ms; full, N = 40, 4096 paths 2.11 -> 0.60 ms (the pipeline: 0.15).
#include <algorithm>

#include <cuda_runtime.h>

#include "lll_paths_block.cuh"

namespace lll {
namespace {

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
        block_tile<SCHEME, QP, B, R, CAPLETS>(a, sm, st, t, acc, comp, t == tiles.x);
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

typedef void (*BatchFn)(const BatchArgs);

BatchFn pick_batch(int scheme, int QMAX, int R)
{
    if (QMAX == 8) {
        if (scheme == FULL) return R == 1 ? batch_block_kernel<FULL, 8, 1> : batch_block_kernel<FULL, 8, 2>;
        return R == 1 ? batch_block_kernel<PICARD, 8, 1> : batch_block_kernel<PICARD, 8, 2>;
    }
    if (scheme == FULL) return R == 1 ? batch_block_kernel<FULL, 32, 1> : batch_block_kernel<FULL, 32, 2>;
    return R == 1 ? batch_block_kernel<PICARD, 32, 1> : batch_block_kernel<PICARD, 32, 2>;
}

BlockFn pick_kernel(int scheme, int product, int QP, int R, uint64_t paths)
{
    return product == 0 ? pick<CAPLETS>(scheme, QP, R, paths) : pick_swaption_kernel(scheme, QP, R, paths);
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

// Time of a launch on default shape in us (see step_as_path): one tile's latency, or all
// tiles' throughput, by (rate, step block) and by unit.
double block_estimate_us(int QP, int n, int s, uint64_t paths)
{
    const int B = steps_of(QP, 1);
    const double pairs = 0.5 * n * (n + 1.0), blocks = pairs * ((s + B - 1) / B), units = pairs * s;
    return 10.0 + std::max(0.25 * blocks + 0.045 * units + 0.4 * n * s, (double)paths * (8e-6 * blocks + 1.3e-6 * units));
}

int block_kernel_prepare(int scheme, int product, int QP, int R, uint64_t paths, size_t smem, int threads,
                         int *blocks_per_sm)
{
    // less its static shared memory
    return prepare(pick_kernel(scheme, product, QP, R, paths), smem, kMaxSmem - 1024, threads, blocks_per_sm);
}

int launch_block_kernel(int scheme, int QP, int R, int grid, int threads, size_t smem, cudaStream_t st, const PathArgs &a)
{
    BlockFn f = pick_kernel(scheme, a.product, QP, R, a.paths);
    if (!f) return (int)cudaErrorInvalidValue;
    if (a.product == 0 || !a.wide_strikes) f<<<grid, threads, smem, st>>>(a);
    if (a.product != 0) {
        const int e = launch_wide_swaptions(scheme, QP, R, grid, threads, st, a);
        if (e != 0) return e;
    }
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

// lll_paths_swaption.cu -- the time-blocked path kernels (lll_paths_block.cuh) of
// co-terminal swaptions.
//
// Payoffs are formed in pairs of FP32 numbers (maturity_values): FP64 has a 64th of
// the FP32 rate.  The pairs have FP32's exponents, so a block that meets a value
// beyond their range (beyond_pairs) marks its sums, and wide_kernel, launched behind,
// runs that block's tiles again with FP64 payoffs: 300,007 paths of N = 40, 3.89 ms a
// call in pairs (3.87 without the check), 9.8 ms where every block goes to wide_kernel.
// Without a mark wide_kernel ends at once: 9 rates, 8000 paths 131 us a call, 128
// without its launch.  (Formed in FP64 within the first kernel instead, the code for it
// alone cost 2.5 % there; the mark kept in a register until the end, N = 120 on 60,000
// paths took 8.98 ms, 8.62 with the word in shared memory, 8.49 without a check.)
#include "lll_paths_block.cuh"

namespace lll {
namespace {

// The tiles of the marked ones of `blocks` blocks with R paths a thread, as R tiles
// each of one path a thread.  Strikes beyond the range are known on the host: then
// every block.  One block an SM (kWideBlocks).
constexpr int kWideBlocks = 152;

template <int SCHEME, int QP>
__global__ void __launch_bounds__(kMaxThreads, 1) wide_kernel(const PathArgs a, int R, int blocks)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int B = steps_of(QP, 1), NST = (SCHEME == PICARD) ? 2 : 1;
    const int T = blockDim.x, tid = threadIdx.x;
    const size_t nout = (size_t)a.n * a.ns * 2;
    const double *marks = a.partials + blocks * nout; // comp[0] of each block: + b nout
    bool any = a.wide_strikes;
    for (int b = blockIdx.x + tid * gridDim.x; b < blocks; b += T * gridDim.x) any = any || isnan(marks[b * nout]);
    if (!__syncthreads_or(any)) return;
    const BlockSmem sm = block_carve(smem_raw, QP, B, 1, a.n, T, a.chunk_rows);
    for (int e = tid; e < a.n; e += T) sm.c0[e] = -1.4426950408889634f * a.c0[e];
    for (int e = tid; e < QP; e += T) reinterpret_cast<float *>(sm.cn)[e] = a.cn[e];
    State<NST> *st = reinterpret_cast<State<NST> *>(a.state) + (size_t)blockIdx.x * a.n * T + tid;
    const uint64_t TP = (uint64_t)T * R, ntiles = (a.paths + TP - 1) / TP;
    for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
        double *acc = a.partials + b * nout, *comp = a.partials + (blocks + b) * nout;
        if (!a.wide_strikes && !isnan(comp[0])) continue; // the same for all threads
        __syncthreads();                                  // before the mark is written over
        bool first = true;
        for (uint64_t tile = b; tile < ntiles; tile += blocks)
            for (int q = 0; q < R; ++q) {
                block_tile<SCHEME, QP, B, 1, WIDE_SWAPTIONS>(a, sm, st, tile * R + q, acc, comp, first);
                first = false;
            }
    }
}

typedef void (*WideFn)(const PathArgs, int, int);

template <int SCHEME>
WideFn pick_wide(int QP)
{
    switch (QP) {
    case 4: return wide_kernel<SCHEME, 4>;
    case 8: return wide_kernel<SCHEME, 8>;
    case 12: return wide_kernel<SCHEME, 12>;
    case 16: return wide_kernel<SCHEME, 16>;
    case 20: return wide_kernel<SCHEME, 20>;
    case 24: return wide_kernel<SCHEME, 24>;
    case 32: return wide_kernel<SCHEME, 32>;
    default: return nullptr;
    }
}

}  // namespace

BlockFn pick_swaption_kernel(int scheme, int QP, int R, uint64_t paths) { return pick<SWAPTIONS>(scheme, QP, R, paths); }

int launch_wide_swaptions(int scheme, int QP, int R, int grid, int threads, cudaStream_t st, const PathArgs &a)
{
    WideFn f = scheme == FULL ? pick_wide<FULL>(QP) : scheme == PICARD ? pick_wide<PICARD>(QP) : nullptr;
    if (!f) return (int)cudaErrorInvalidValue;
    PathArgs w = a;
    w.chunk_rows = block_chunk_rates(QP, 1, a.n, 0);
    const size_t smem = block_kernel_smem(QP, 1, a.n, threads, w.chunk_rows);
    const cudaError_t e = allow_smem(f, smem);
    if (e != cudaSuccess) return (int)e;
    f<<<grid < kWideBlocks ? grid : kWideBlocks, threads, smem, st>>>(w, R, grid);
    return (int)cudaGetLastError();
}

}  // namespace lll

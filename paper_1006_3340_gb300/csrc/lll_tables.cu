// lll_tables.cu -- FP64 precomputation on the GPU and the final reduction.
//
// tables_kernel: for every step k and rate l, the node table of the jump
//   compensator of Eq. (LIBOR-drift-PT): E_lj = e^{lambda_l(t_k) x_j} - 1
//   (rounded to FP32), the per-node factors c_j = W_j / x_j^2 (FP32), and the
//   constant K_l = C_l - sum_j fl32(E_lj c_j) with
//   C_l = sum_j W_j (E_lj - lambda_l x_j) / x_j^2, so that
//   A_l = K_l + sum_j E_lj (c_j P_j) reproduces C_l when P = 1 up to the FP32
//   sum.  C_l itself (the compensator with all later weights zero) is kept too.
// frozen_drift_kernel: the drift b(t_k, T_l; Z(0)) of Eq. (Picard-2), i.e.
//   Eq. (LIBOR-drift-PT) with L frozen at L(0).
// prefix_kernel: D0_l(t_k) = sum_{m<k} b0_l(t_m) h, the deterministic drift
//   integral of Z^(1).
// finalize_kernel: sum of the per-block payoff partials in a fixed order.
#include <cuda_runtime.h>

#include "lll_internal.h"
#include "lll_sweep.cuh"

namespace lll {
namespace {

// One block per Euler step k, one warp per live rate: lanes over the nodes.
// FP64 runs at about 2 lanes per SM and clock, so the expm1 of every (rate,
// node) pair is the cost; only the rates live at the step are built (rows of
// rates already fixed hold lambda alone, nothing reads the rest), and the
// warps of a block and the blocks are independent.
__global__ void tables_kernel(const double *lam, const double *x, const double *W, int Q, const double *xr,
                              const double *Wr, int Qr, int n, int s, int QP, double scale, float4 *tab, float *cn,
                              float4 *row, float4 *brow, double *Cs, float *Ctab)
{
    const int k = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int imin = k / s + 1;
    if (k == 0)
        for (int j = threadIdx.x; j < QP; j += blockDim.x)
            cn[j] = (j < Qr) ? (float)(scale * (Wr[j] / (xr[j] * xr[j]))) : 0.0f;
    for (int i = warp + 1; i <= n; i += nw) {
        const size_t idx = (size_t)k * n + (i - 1);
        const double li = lam[idx];
        double C = 0.0, sa = 0.0;
        float *out = reinterpret_cast<float *>(tab + idx * (QP / 4));
        if (i >= imin)
            for (int j = lane; j < Q; j += 32) {
                const double xj = x[j];
                C += W[j] / (xj * xj) * (expm1(li * xj) - li * xj);
            }
        for (int j = lane; j < QP; j += 32) {
            float e = 0.0f;
            if (i >= imin && j < Qr) {
                e = (float)expm1(li * xr[j]);
                sa += (double)__fmul_rn(e, (float)(scale * (Wr[j] / (xr[j] * xr[j]))));
            }
            out[j] = e;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            C += __shfl_xor_sync(0xffffffffu, C, o);
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
        }
        if (lane == 0) {
            *reinterpret_cast<float2 *>(&row[idx]) = make_float2((float)li, (float)(C - sa / scale));
            if (brow) {
                brow[idx].x = (float)li;
                brow[idx].w = 0.0f;
                Cs[idx] = scale * C;
            }
            Ctab[idx] = (float)C;
        }
    }
}

// K' = -h C less the dot product at zero weights, formed by the sweeps' own FP32
// operations.  One thread a row.
template <int QP>
__global__ void close_kernel(const float4 *tab, const float *cn, const double *Cs, int rows, float4 *brow)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    float4 E[QP / 4];
    float2 P[QP / 2];
#pragma unroll
    for (int j = 0; j < QP / 4; ++j) E[j] = tab[(size_t)r * (QP / 4) + j];
#pragma unroll
    for (int j = 0; j < QP / 2; ++j) P[j] = reinterpret_cast<const float2 *>(cn)[j];
    brow[r].z = (float)(Cs[r] - (double)sweep_dot<QP>(E, P));
}

// One block per step, one thread per node carrying its product P_j down the
// live rates; the contributions of kDriftRates rates at a time go through
// shared memory, where one warp sums each rate over the nodes.
constexpr int kDriftRates = 16;

__global__ void frozen_drift_kernel(const double *lam, const double *x, const double *W,
                                    const double *w0, int n, int s, int Q, double c, double *b0)
{
    __shared__ double contrib[kDriftRates][kMaxQP + 1];
    __shared__ double cont[kDriftRates]; // sum of w_l lambda_l over the rates above
    const int k = blockIdx.x, j = threadIdx.x, lane = j & 31, warp = j >> 5, nw = blockDim.x >> 5;
    const int imin = k / s + 1;
    double P = 1.0, scont = 0.0;
    const double xj = (j < Q) ? x[j] : 0.0;
    const double inv = (j < Q) ? W[j] / (xj * xj) : 0.0;
    for (int i0 = n; i0 >= imin; i0 -= kDriftRates) {
        const int cnt = min(kDriftRates, i0 - imin + 1);
        for (int u = 0; u < cnt; ++u) {
            const int i = i0 - u;
            const double li = lam[(size_t)k * n + (i - 1)], wi = w0[i - 1];
            if (j < Q) {
                const double e = expm1(li * xj);
                contrib[u][j] = inv * (e * P - li * xj);
                P *= 1.0 + wi * e;
            }
            if (j == 0) cont[u] = scont;
            scont += wi * li;
        }
        __syncthreads();
        for (int u = warp; u < cnt; u += nw) {
            double A = 0.0;
            for (int t = lane; t < Q; t += 32) A += contrib[u][t];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) A += __shfl_xor_sync(0xffffffffu, A, o);
            const int i = i0 - u;
            const double li = lam[(size_t)k * n + (i - 1)];
            if (lane == 0) b0[(size_t)k * n + (i - 1)] = -A - 0.5 * c * li * li - c * li * cont[u];
        }
        __syncthreads();
    }
}

// Thread per rate: the running integral over the steps it lives, eight steps'
// loads ahead of their additions.
__global__ void prefix_kernel(const double *b0, int n, int s, double h, const double *L0, double delta, float4 *row,
                              float4 *brow)
{
    constexpr int U = 8;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int K = (l + 1) * s;
    const double c0 = brow ? log(delta * L0[l + 1]) : 0.0;
    double D = 0.0;
    for (int k0 = 0; k0 < K; k0 += U) {
        double b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) b[u] = k0 + u < K ? b0[(size_t)(k0 + u) * n + l] : 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k0 + u >= K) break;
            const double bh = b[u] * h;
            float2 *out = reinterpret_cast<float2 *>(&row[(size_t)(k0 + u) * n + l].z);
            *out = make_float2((float)D, (float)bh);
            if (brow) brow[(size_t)(k0 + u) * n + l].y = (float)(-1.4426950408889634 * (c0 + D));
            D += bh;
        }
    }
}

// Sum of the per-block partials of kOutPer outputs a block: kSlices threads an
// output, each Kahan-summing every kSlices-th block, then a fixed tree over the
// slices.  (One thread an output took 110 us for 608 blocks: a chain of FP64
// additions and their loads; this takes a few.)
constexpr int kOutPer = 4, kSlices = 32;

__global__ void __launch_bounds__(kOutPer *kSlices) finalize_kernel(const double *partials, int grid, int n_out,
                                                                    double *sums)
{
    __shared__ double ps[kSlices][kOutPer], pc[kSlices][kOutPer];
    const int x = threadIdx.x % kOutPer, y = threadIdx.x / kOutPer;
    const int e = blockIdx.x * kOutPer + x;
    double s = 0.0, c = 0.0;
    if (e < n_out)
        for (int b = y; b < grid; b += kSlices) {
            const double v = partials[(size_t)b * n_out + e] - c;
            const double t = s + v;
            c = (t - s) - v;
            s = t;
        }
    ps[y][x] = s;
    pc[y][x] = c;
    __syncthreads();
    for (int o = kSlices / 2; o > 0; o >>= 1) {
        if (y < o) {
            const double v = ps[y + o][x] - (pc[y][x] + pc[y + o][x]);
            const double t = ps[y][x] + v;
            pc[y][x] = (t - ps[y][x]) - v;
            ps[y][x] = t;
        }
        __syncthreads();
    }
    if (y == 0 && e < n_out) sums[e] = ps[0][x];
}

// Per instance of a batch: add the partials of its work items in tile order.
__global__ void batch_finalize_kernel(const double *partials, const size_t *seg_off, const int *inst_seg_ptr,
                                      const int *inst_segs, const size_t *out_off, const int *out_count,
                                      double *sums)
{
    const int q = blockIdx.x;
    for (int e = threadIdx.x; e < out_count[q]; e += blockDim.x) {
        double s = 0.0, c = 0.0;
        for (int k = inst_seg_ptr[q]; k < inst_seg_ptr[q + 1]; ++k) {
            const double y = partials[seg_off[inst_segs[k]] + e] - c;
            const double t = s + y;
            c = (t - s) - y;
            s = t;
        }
        sums[out_off[q] + e] = s;
    }
}

}  // namespace

int batch_finalize(const double *partials, const size_t *seg_off, const int *inst_seg_ptr, const int *inst_segs,
                   const size_t *out_off, int n_inst, const int *out_count, double *sums, cudaStream_t st)
{
    batch_finalize_kernel<<<n_inst, 128, 0, st>>>(partials, seg_off, inst_seg_ptr, inst_segs, out_off, out_count,
                                                  sums);
    return (int)cudaGetLastError();
}

int launch_tables(const double *lam, const double *x, const double *W, int Q, const double *xr, const double *Wr,
                  int Qr, int n, int S, int QP, double h, float4 *tab, float *cn, float4 *row, float4 *brow,
                  double *Cs, float *Ctab, cudaStream_t st)
{
    const int warps = n < 8 ? n : 8;
    tables_kernel<<<S, 32 * warps, 0, st>>>(lam, x, W, Q, xr, Wr, Qr, n, S / n, QP, brow ? -h : 1.0, tab, cn, row,
                                            brow, Cs, Ctab);
    if (brow) {
        const int rows = S * n, blocks = (rows + 127) / 128;
        switch (QP) {
        case 4: close_kernel<4><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 8: close_kernel<8><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 12: close_kernel<12><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 16: close_kernel<16><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 20: close_kernel<20><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 24: close_kernel<24><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        case 32: close_kernel<32><<<blocks, 128, 0, st>>>(tab, cn, Cs, rows, brow); break;
        default: return (int)cudaErrorInvalidValue;
        }
    }
    return (int)cudaGetLastError();
}

int launch_frozen_drift(const double *lam, const double *x, const double *W, const double *w0,
                        int n, int S, int Q, double c, double h, const double *L0, double delta, double *b0,
                        float4 *row, float4 *brow, cudaStream_t st)
{
    const int threads = Q <= 0 ? 32 : (Q + 31) / 32 * 32;
    frozen_drift_kernel<<<S, threads, 0, st>>>(lam, x, W, w0, n, S / n, Q, c, b0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    prefix_kernel<<<(n + 31) / 32, 32, 0, st>>>(b0, n, S / n, h, L0, delta, row, brow);
    return (int)cudaGetLastError();
}

int launch_finalize(const double *partials, int grid, int n_out, double *sums, cudaStream_t st)
{
    finalize_kernel<<<(n_out + kOutPer - 1) / kOutPer, kOutPer * kSlices, 0, st>>>(partials, grid, n_out, sums);
    return (int)cudaGetLastError();
}

}  // namespace lll

// lll_tables.cu -- FP64 precomputation on the GPU and the final reduction.
//
// tables_kernel: for every step k and rate l, the node table of the jump
//   compensator of Eq. (LIBOR-drift-PT): E_lj = e^{lambda_l(t_k) x_j} - 1
//   (rounded to FP32), the per-node factors c_j = W_j / x_j^2 (FP32), and the
//   constant K_l = C_l - sum_j fl32(E_lj c_j) with
//   C_l = sum_j W_j (E_lj - lambda_l x_j) / x_j^2, so that
//   A_l = K_l + sum_j E_lj (c_j P_j) reproduces C_l when P = 1 up to the FP32
//   sum.  C_l itself (the compensator with all later weights zero) is kept too,
//   and the drift b(t_k, T_l; Z(0)) of Eq. (Picard-2), i.e. Eq. (LIBOR-drift-PT)
//   with L frozen at L(0).
// prefix_kernel: D0_l(t_k) = sum_{m<k} b0_l(t_m) h, the deterministic drift
//   integral of Z^(1).
// finalize_kernel: sum of the per-block payoff partials in a fixed order.
#include <cuda_runtime.h>

#include "lll_internal.h"

namespace lll {
namespace {

// One block per Euler step k, over the rates live at it (rows of rates already
// fixed hold lambda alone; nothing reads the rest) in chunks of kTabRates:
//   1. E_ij of every (rate, node) pair, a thread a pair: FP64 runs at about 2
//      lanes per SM and clock, so these expm1 are the cost, and they are formed
//      once for the table, C, the frozen drift and K;
//   2. a thread a node carries P_j down the rates and leaves the drift's terms;
//   3. a thread a rate adds up its terms over the nodes.
// C and the frozen drift are formed with the sweeps' rule, like the table: both
// are integrals of its generating function (lll_quadrature.cpp), C over [0,
// lambda] alone.  short_rule: the sweeps' rule is a shorter one; its rows brow
// then hold K' = -h C less the dot product at zero weights as sweep_dot forms it.
// w0, b0 null: the table and C alone (of another rule of the same model).
constexpr int kTabRates = 32;

__global__ void tables_kernel(const double *lam, const double *x, const double *W, int Q, int n, int s, int QP, double h,
                              double c, const double *w0, float4 *tab, float *cn, float4 *row, float4 *brow, float *Ctab,
                              double *b0)
{
    extern __shared__ double sm_tab[];
    double *E = sm_tab, *term = E + kTabRates * Q, *P = term + kTabRates * Q, *cj = P + Q; // [kTabRates][Q] twice, [Q] twice
    const int k = blockIdx.x, tid = threadIdx.x, T = blockDim.x;
    const int imin = k / s + 1;
    const double scale = brow ? -h : 1.0;
    for (int j = tid; j < QP; j += T) {
        if (j < Q) {
            P[j] = 1.0;
            cj[j] = W[j] / (x[j] * x[j]);
        }
        if (k == 0) cn[j] = j < Q ? (float)(scale * cj[j]) : 0.0f;
    }
    for (int i = tid + 1; i < imin; i += T) {
        const size_t idx = (size_t)k * n + (i - 1);
        row[idx] = make_float4((float)lam[idx], 0.0f, 0.0f, 0.0f);
        if (brow) brow[idx] = make_float4((float)lam[idx], 0.0f, 0.0f, 0.0f);
        Ctab[idx] = 0.0f;
    }
    double scont = 0.0; // sum of w_l lambda_l over the rates above (every thread)
    for (int i0 = n; i0 >= imin; i0 -= kTabRates) {
        const int cnt = min(kTabRates, i0 - imin + 1);
        for (int e = tid; e < cnt * Q; e += T) E[e] = expm1(lam[(size_t)k * n + (i0 - e / Q - 1)] * x[e % Q]);
        __syncthreads();
        for (int e = tid; e < cnt * QP; e += T) {
            const int u = e / QP, j = e % QP;
            reinterpret_cast<float *>(tab)[((size_t)k * n + (i0 - u - 1)) * QP + j] = j < Q ? (float)E[u * Q + j] : 0.0f;
        }
        if (b0)
            for (int j = tid; j < Q; j += T) {
                double p = P[j];
                const double cc = cj[j], xj = x[j];
                for (int u = 0; u < cnt; ++u) {
                    const int i = i0 - u;
                    const double e = E[u * Q + j];
                    term[u * Q + j] = cc * (e * p - lam[(size_t)k * n + (i - 1)] * xj);
                    p *= 1.0 + w0[i - 1] * e;
                }
                P[j] = p;
            }
        __syncthreads();
        for (int u = tid; u < cnt; u += T) {
            const int i = i0 - u;
            const size_t idx = (size_t)k * n + (i - 1);
            const double li = lam[idx];
            double C = 0.0, sa = 0.0, A = 0.0;
            float2 a = make_float2(0.0f, 0.0f), b = make_float2(0.0f, 0.0f); // the sums of sweep_dot
            for (int j = 0; j < Q; ++j) {
                const double e = E[u * Q + j];
                const float ef = (float)e, cf = (float)(scale * cj[j]);
                C += cj[j] * (e - li * x[j]);
                if (b0) A += term[u * Q + j];
                if (!brow) sa += (double)__fmul_rn(ef, cf);
                float &acc = (j & 3) == 0 ? a.x : (j & 3) == 1 ? a.y : (j & 3) == 2 ? b.x : b.y;
                acc = fmaf(ef, cf, acc);
            }
            row[idx] = make_float4((float)li, (float)(C - sa), 0.0f, 0.0f);
            if (brow) {
                const float dot = __fadd_rn(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
                brow[idx] = make_float4((float)li, 0.0f, (float)(scale * C - (double)dot), 0.0f);
            }
            Ctab[idx] = (float)C;
            if (b0) {
                double sc = scont;
                for (int v = 0; v < u; ++v) sc += w0[i0 - v - 1] * lam[(size_t)k * n + (i0 - v - 1)];
                b0[idx] = -A - 0.5 * c * li * li - c * li * sc;
            }
        }
        if (b0 && c != 0.0)
            for (int v = 0; v < cnt; ++v) scont += w0[i0 - v - 1] * lam[(size_t)k * n + (i0 - v - 1)];
        __syncthreads();
    }
}

// Warp per rate: the running integral over the steps it lives, 32 steps at a
// time by a scan over the lanes.
__global__ void prefix_kernel(const double *b0, int n, int s, double h, const double *L0, double delta, float4 *row,
                              float4 *brow)
{
    const int l = blockIdx.x, lane = threadIdx.x;
    const int K = (l + 1) * s;
    const double c0 = brow ? log(delta * L0[l + 1]) : 0.0;
    double D = 0.0;
    for (int k0 = 0; k0 < K; k0 += 32) {
        const int k = k0 + lane;
        const double bh = k < K ? b0[(size_t)k * n + l] * h : 0.0;
        double t = bh;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += v;
        }
        if (k < K) {
            float2 *out = reinterpret_cast<float2 *>(&row[(size_t)k * n + l].z);
            *out = make_float2((float)(D + (t - bh)), (float)bh);
            if (brow) brow[(size_t)k * n + l].y = (float)(-1.4426950408889634 * (c0 + D + (t - bh)));
        }
        D += __shfl_sync(0xffffffffu, t, 31);
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

int launch_tables(const double *lam, const double *x, const double *W, int Q, int n, int S, int QP, double h, double c,
                  const double *w0, float4 *tab, float *cn, float4 *row, float4 *brow, float *Ctab, double *b0,
                  cudaStream_t st)
{
    const size_t smem = sizeof(double) * ((size_t)2 * kTabRates * Q + 2 * (size_t)Q);
    if (smem > 48 * 1024) {
        // always the need of the longest rule: the limit is the kernel's, and another
        // thread's launch (a context of its own) may need more than this one
        constexpr int most = sizeof(double) * (2 * kTabRates * kMaxQP + 2 * kMaxQP);
        const cudaError_t e = cudaFuncSetAttribute(tables_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return (int)e;
    }
    tables_kernel<<<S, 128, smem, st>>>(lam, x, W, Q, n, S / n, QP, h, c, w0, tab, cn, row, brow, Ctab, b0);
    return (int)cudaGetLastError();
}

int launch_prefix(const double *b0, int n, int S, double h, const double *L0, double delta, float4 *row, float4 *brow,
                  cudaStream_t st)
{
    prefix_kernel<<<n, 32, 0, st>>>(b0, n, S / n, h, L0, delta, row, brow);
    return (int)cudaGetLastError();
}

int launch_finalize(const double *partials, int grid, int n_out, double *sums, cudaStream_t st)
{
    finalize_kernel<<<(n_out + kOutPer - 1) / kOutPer, kOutPer * kSlices, 0, st>>>(partials, grid, n_out, sums);
    return (int)cudaGetLastError();
}

}  // namespace lll

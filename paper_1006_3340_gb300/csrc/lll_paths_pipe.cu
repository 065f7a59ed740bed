// lll_paths_pipe.cu -- the time-blocked sweep for few paths: a pipeline of
// warps over the rates (full and Picard, shorter rules, caplets).
//
// With few paths one thread per path leaves the GPU idle: 4096 paths are 128
// warps for 608 schedulers, and each of them runs the 6240 units of an N = 40
// path one after the other.  The triangle of lll_sweep.cuh has a second
// parallel direction: a block of steps is handed down the rates, so while the
// lower rates finish one block of steps, the upper rates can start the next.
// A block carries 32 paths (lane = path) through G warps.  At tick t warp g
// takes the step block t - g through its share of the live rates,
//     rates n - floor(L g / G) .. n - floor(L (g+1) / G) + 1,  L live rates,
// and hands the node products of the block's B steps (and, at a maturity, the
// numeraire product of Eq. (caplet)) to warp g + 1 through shared memory.  The
// shares are of equal size in every period; a rate whose owner changes moves to
// a later warp, whose tick comes after its last update.  Every unit is
// the arithmetic of sweep_dot, sweep_weight and sweep_grow on the same
// operands, so a path's rates and payoffs are those of the block kernel bit for
// bit.  Increments are drawn ahead by all warps; a warp's table rows of the next
// tick arrive by cp.async while it sweeps; the payoff sums of all maturities
// are formed at the end, a thread a (maturity, strike).
#include <cuda_runtime.h>

#include "lll_device.cuh"
#include "lll_internal.h"
#include "lll_sweep.cuh"

namespace lll {
namespace {

constexpr int kPipeWarps = 8; // warps at most; a power of two, so that shares are shifts

struct PipeSmem {
    float *dh;     // [S][32]
    float2 *P;     // [G][B][QP/2][32]: node products handed to the next warp
    float *Pf;     // [G][32]: numeraire products
    float *state;  // [n][32][NST]
    float4 *tab;   // [G][2][rates][B][QP/4]
    float4 *row;   // [G][2][rates][B]
    float2 *pay;   // [n][32]: (delta B(0,T_N) P, L_m)
    float2 *cn;    // [QP/2]
    float *c0;     // [n]: -log2(e) log(delta L(0, T_l))
    float *L0;     // [n]
};

__host__ __device__ inline size_t pipe_smem_bytes(int QP, int B, int nst, int n, int S, int G)
{
    const int rates = (n + G - 1) / G;
    return (size_t)S * 128 + (size_t)G * B * QP * 128 + (size_t)G * 128 + (size_t)n * 128 * nst +
           2 * (size_t)G * rates * B * (QP * 4 + 16) + (size_t)n * 256 + (size_t)QP * 4 + (size_t)n * 8;
}

__device__ inline PipeSmem pipe_carve(unsigned char *p, int QP, int B, int nst, int n, int S, int G)
{
    const int rates = (n + G - 1) / G;
    PipeSmem s;
    s.tab = reinterpret_cast<float4 *>(p);
    p += 2 * (size_t)G * rates * B * QP * 4;
    s.row = reinterpret_cast<float4 *>(p);
    p += 2 * (size_t)G * rates * B * 16;
    s.dh = reinterpret_cast<float *>(p);
    p += (size_t)S * 128;
    s.P = reinterpret_cast<float2 *>(p);
    p += (size_t)G * B * QP * 128;
    s.Pf = reinterpret_cast<float *>(p);
    p += (size_t)G * 128;
    s.state = reinterpret_cast<float *>(p);
    p += (size_t)n * 128 * nst;
    s.pay = reinterpret_cast<float2 *>(p);
    p += (size_t)n * 256;
    s.cn = reinterpret_cast<float2 *>(p);
    p += (size_t)QP * 4;
    s.c0 = reinterpret_cast<float *>(p);
    s.L0 = s.c0 + n;
    return s;
}

// Warp g's share [lo, hi] of the live rates m .. n (empty: lo > hi), G = 2^lg.
__device__ __forceinline__ void share_of(int n, int m, int g, int lg, int &hi, int &lo)
{
    const int L = n - m + 1;
    hi = n - ((L * g) >> lg);
    lo = n - ((L * (g + 1)) >> lg) + 1;
}

// Stage the rows of rates hi .. lo for the steps kb .. of period m.
template <int QP, int B>
__device__ __forceinline__ void pipe_stage(const PathArgs &a, float4 *dt, float4 *dr, int m, int kb, int hi, int lo)
{
    constexpr int Q4 = QP / 4;
    const int n = a.n, lane = threadIdx.x & 31, nb = min(B, a.s - kb), cnt = hi - lo + 1;
    const size_t r0 = ((size_t)(m - 1) * a.s + kb) * n + (lo - 1);
    for (int e = lane; e < cnt * B * Q4; e += 32) {
        const int j = e % Q4, s = e / Q4 % B, r = e / (Q4 * B);
        if (s < nb) cp_async16(dt + e, a.tab + (r0 + (size_t)s * n + r) * Q4 + j);
    }
    for (int e = lane; e < cnt * B; e += 32) {
        const int s = e % B, r = e / B;
        if (s < nb) cp_async16(dr + e, a.brow + r0 + (size_t)s * n + r);
    }
}

// One rate through H of the steps of a block, from step b0: all the steps' dot
// products first, then the rate's own chain, then the weights, then the
// products' growth, so that one warp keeps the pipes busy.
template <int SCHEME, int QP, int B, int H, bool TAIL>
__device__ __forceinline__ void pipe_steps_of_rate(const float4 *tr, const float4 *rr, float c0, int b0, int nb,
                                                   const float (&dH)[B], float (&z)[2], float2 (&P)[B][QP / 2])
{
    constexpr int Q4 = QP / 4;
    float4 E[H][Q4], rc[H];
    float bh[H], w[H];
#pragma unroll
    for (int u = 0; u < H; ++u) {
        if (TAIL && b0 + u >= nb) break;
        rc[u] = rr[b0 + u];
#pragma unroll
        for (int j = 0; j < Q4; ++j) E[u][j] = tr[(b0 + u) * Q4 + j];
        bh[u] = sweep_dot<QP>(E[u], P[b0 + u]) + rc[u].z;
    }
#pragma unroll
    for (int u = 0; u < H; ++u) {
        if (TAIL && b0 + u >= nb) break;
        w[u] = z[0];
        if constexpr (SCHEME == PICARD) {
            z[0] = fmaf(rc[u].x, dH[b0 + u], z[0]); // int lambda dH
            z[1] += bh[u];                          // Picard drift integral
        } else {
            z[0] = z[0] + fmaf(rc[u].x, dH[b0 + u], bh[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < H; ++u) {
        if (TAIL && b0 + u >= nb) break;
        w[u] = sweep_weight(SCHEME == PICARD ? rc[u].y : c0, w[u]);
    }
#pragma unroll
    for (int u = 0; u < H; ++u) {
        if (TAIL && b0 + u >= nb) break;
        sweep_grow<QP>(E[u], P[b0 + u], w[u]);
    }
}

// Steps whose rows are held in registers at a time.
__host__ __device__ constexpr int pipe_half(int QP, int B) { return QP >= 8 && B == 8 ? 4 : B; }

template <int SCHEME, int QP, int B>
__global__ void __launch_bounds__(32 * kPipeWarps, QP <= 8 && B == 4 ? 2 : 1) pipe_kernel(const PathArgs a, int lg)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int Q2 = QP / 2, Q4 = QP / 4, NST = (SCHEME == PICARD) ? 2 : 1, H = pipe_half(QP, B);
    const int G = 1 << lg, g = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = a.n, s = a.s, S = a.S, ns = a.ns, rates = (n + G - 1) >> lg;
    const PipeSmem sm = pipe_carve(smem_raw, QP, B, NST, n, S, G);
    const uint64_t lp = (uint64_t)blockIdx.x * 32 + lane;
    float4 *tab = sm.tab + (size_t)g * 2 * rates * B * Q4, *row = sm.row + (size_t)g * 2 * rates * B;

    int hi, lo; // the share of the step block in work
    share_of(n, 1, g, lg, hi, lo);
    pipe_stage<QP, B>(a, tab, row, 1, 0, hi, lo);
    cp_commit();
    for (int e = threadIdx.x; e < QP; e += blockDim.x) reinterpret_cast<float *>(sm.cn)[e] = a.cn[e];
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
        sm.c0[e] = -1.4426950408889634f * a.c0[e];
        sm.L0[e] = a.L0[e];
    }
    for (int e = threadIdx.x; e < n * 32 * NST; e += blockDim.x) sm.state[e] = 0.0f;
#pragma unroll 2
    for (int k = g; k < S; k += G) sm.dh[k * 32 + lane] = draw_increment(a, a.first_path + lp, (uint32_t)k);
    __syncthreads();

    const int NB = n * ((s + B - 1) / B); // step blocks in all
    int m = 1, kb = 0, buf = 0;           // period, first step and row buffer of this warp's block
    for (int t = 0; t < NB + G - 1; ++t) {
        const bool active = t >= g && t - g < NB;
        float2 P[B][Q2];
        float Pf = 1.0f;
        if (active) {
            if (g == 0) {
#pragma unroll
                for (int j = 0; j < Q2; ++j) {
                    const float2 c = sm.cn[j];
#pragma unroll
                    for (int u = 0; u < B; ++u) P[u][j] = c;
                }
            } else {
                const float2 *in = sm.P + (size_t)(g - 1) * B * Q2 * 32 + lane;
#pragma unroll
                for (int u = 0; u < B; ++u)
#pragma unroll
                    for (int j = 0; j < Q2; ++j) P[u][j] = in[(u * Q2 + j) * 32];
                Pf = sm.Pf[(g - 1) * 32 + lane];
            }
        }
        __syncthreads(); // every warp has taken what the warp above it handed down
        if (active) {
            const int nb = min(B, s - kb), k0 = (m - 1) * s + kb;
            const bool mat = kb + nb == s;
            const int mn = mat ? m + 1 : m, kn = mat ? 0 : kb + B; // the next block
            int hn = 0, ln = 1;
            if (mn <= n) {
                share_of(n, mn, g, lg, hn, ln);
                pipe_stage<QP, B>(a, tab + (size_t)(buf ^ 1) * rates * B * Q4, row + (size_t)(buf ^ 1) * rates * B, mn, kn, hn, ln);
            }
            cp_commit();
            float dH[B];
#pragma unroll
            for (int u = 0; u < B; ++u) dH[u] = u < nb ? sm.dh[(k0 + u) * 32 + lane] : 0.0f;
            cp_wait_1();
            __syncwarp();
            const float4 *tr = tab + ((size_t)buf * rates + (hi - lo)) * (B * Q4);
            const float4 *rr = row + ((size_t)buf * rates + (hi - lo)) * B;
            for (int i = hi; i >= lo; --i, tr -= B * Q4, rr -= B) {
                float *st = sm.state + ((size_t)(i - 1) * 32 + lane) * NST;
                float z[2] = {st[0], NST == 2 ? st[NST - 1] : 0.0f};
                const float c0 = sm.c0[i - 1];
                if (nb == B) {
#pragma unroll
                    for (int b0 = 0; b0 < B; b0 += H)
                        pipe_steps_of_rate<SCHEME, QP, B, H, false>(tr, rr, c0, b0, nb, dH, z, P);
                } else {
#pragma unroll
                    for (int b0 = 0; b0 < B; b0 += H)
                        pipe_steps_of_rate<SCHEME, QP, B, H, true>(tr, rr, c0, b0, nb, dH, z, P);
                }
                st[0] = z[0];
                if (NST == 2) st[NST - 1] = z[1];
                if (mat) {
                    const float off = NST == 2 ? z[0] + z[1] : z[0], L = sm.L0[i - 1] * expf(off);
                    if (i > m) Pf *= fmaf(a.delta, L, 1.0f);
                    else sm.pay[(m - 1) * 32 + lane] = lp < a.paths ? make_float2(a.dBN * Pf, L) : make_float2(0.0f, 0.0f);
                    if (a.snap != nullptr && lp < a.paths && lp % a.snap_stride == 0 && lp / a.snap_stride < a.n_snap)
                        a.snap[((size_t)(m - 1) * n + (i - 1)) * a.snap_pitch + lp / a.snap_stride] = off + a.Z0[i - 1];
                }
            }
            if (g + 1 < G) {
                float2 *out = sm.P + (size_t)g * B * Q2 * 32 + lane;
#pragma unroll
                for (int u = 0; u < B; ++u)
#pragma unroll
                    for (int j = 0; j < Q2; ++j) out[(u * Q2 + j) * 32] = P[u][j];
                sm.Pf[g * 32 + lane] = Pf;
            }
            m = mn;
            kb = kn;
            hi = hn;
            lo = ln;
            buf ^= 1;
        }
        __syncthreads(); // the products and states of this tick are written
    }
    cp_wait_0();

    double *out = a.partials + (size_t)blockIdx.x * n * ns * 2;
    for (int e = threadIdx.x; e < n * ns; e += blockDim.x) {
        const float K = a.strikes[e];
        const float2 *pay = sm.pay + e / ns * 32;
        DFloat s1{0.0f, 0.0f}, s2{0.0f, 0.0f};
        for (int p = 0; p < 32; ++p) {
            const float2 v = pay[p];
            const float x = v.x * fmaxf(v.y - K, 0.0f);
            s1 = df_add(s1, DFloat{x, 0.0f});
            s2 = df_add(s2, df_square(x));
        }
        out[2 * e] = (double)s1.hi + (double)s1.lo;
        out[2 * e + 1] = (double)s2.hi + (double)s2.lo;
    }
}

typedef void (*PipeFn)(const PathArgs, int);

template <int SCHEME>
PipeFn pick_pipe(int QP, int B)
{
    switch (QP) {
    case 4: return B == 8 ? pipe_kernel<SCHEME, 4, 8> : B == 5 ? pipe_kernel<SCHEME, 4, 5> : pipe_kernel<SCHEME, 4, 4>;
    case 8: return B == 8 ? pipe_kernel<SCHEME, 8, 8> : B == 5 ? pipe_kernel<SCHEME, 8, 5> : pipe_kernel<SCHEME, 8, 4>;
    case 12: return B == 4 ? pipe_kernel<SCHEME, 12, 4> : pipe_kernel<SCHEME, 12, 2>;
    case 16: return B == 4 ? pipe_kernel<SCHEME, 16, 4> : pipe_kernel<SCHEME, 16, 2>;
    case 20: return pipe_kernel<SCHEME, 20, 2>;
    case 24: return pipe_kernel<SCHEME, 24, 2>;
    case 32: return pipe_kernel<SCHEME, 32, 2>;
    default: return nullptr;
    }
}

}  // namespace

// The pipeline's shape for `tiles` blocks of 32 paths: B steps per block and 2^lg
// warps, as B | lg << 8; 0 where the block kernel is the better one or shared
// memory does not hold the pipeline.  Full scheme, ms:
//  * One block an SM: eight warps and as many steps as the registers of the
//    products and of the rows in work allow (8 or 5 up to 8 nodes, 4 up to 16,
//    else 2), preferring a divisor of the steps per period: 4096 paths of N = 40
//    0.119 with 8 steps, 0.158 with 4, and 0.56 in the block kernel.
//  * More blocks, 24 rates and more: 4 steps leave room for two blocks an SM (up
//    to 8 nodes), 9000 paths 0.209 (0.233 with 8 steps, 0.231 with four warps);
//    up to three waves: 29,000 paths 0.59 against 0.65, 38,000 paths 0.78 against
//    0.66; N = 120 (one block an SM), 4096 paths 0.74 against 2.74, 9000 paths
//    1.45, 16,000 paths 2.88 against 2.74.
//  * Fewer rates: fewer warps a block, and more blocks an SM, in one wave.  N = 10
//    (8 nodes), 10,000 paths: 0.083 with eight warps, 0.053 with four, against
//    0.098; 20,000 paths 0.073 with two against 0.103; 30,000 paths 0.090 against
//    0.107; 40,000 paths 0.128 against 0.120.  The heavy-tailed example (32
//    nodes): 5000 paths 0.081, 0.045 with four, against 0.086; 10,000 paths 0.054
//    with two against 0.087; 20,000 paths 0.095 against 0.102.
int pipe_shape(int scheme, int QP, int n, int s, int S, uint64_t tiles, int sms, size_t *smem)
{
    const int nst = scheme == PICARD ? 2 : 1;
    const uint64_t per_sm = (tiles + sms - 1) / sms; // blocks an SM
    int B = QP <= 8 ? (per_sm > 1 ? 4 : s % 8 == 0 ? 8 : s % 5 == 0 ? 5 : 4) : QP <= 16 ? 4 : 2;
    int most = 8; // warps
    if (n < 24 && per_sm > 1) {
        most = per_sm <= (QP <= 8 ? 4 : 2) ? 4 : 2;
        if (per_sm > (QP <= 8 ? 8 : 6)) return 0;
    }
    int lg = 0;
    while ((2 << lg) <= n && (2 << lg) <= most) ++lg;
    *smem = pipe_smem_bytes(QP, B, nst, n, S, 1 << lg);
    if (QP > 8 && B == 4 && *smem > 227 * 1024) {
        B = 2;
        *smem = pipe_smem_bytes(QP, B, nst, n, S, 1 << lg);
    }
    const uint64_t room = 227 * 1024 / *smem; // blocks an SM by shared memory
    if (room < 1 || (n < 24 && per_sm > room)) return 0;
    if (n >= 24 && per_sm > 3 * (QP <= 8 && B == 4 && room >= 2 ? 2 : 1)) return 0;
    return B | lg << 8;
}

// Time of such a launch in us, for the choice of lll_set_mapping(LLL_MAP_STEP): its
// ticks by the rates a warp takes through one (see step_as_path).
double pipe_estimate_us(int QP, int shape, size_t smem, int n, int s, uint64_t tiles, int sms)
{
    const int B = shape & 255, G = 1 << (shape >> 8);
    const double ticks = (double)n * ((s + B - 1) / B) + G - 1, rates = (n + G - 1) / G;
    const uint64_t per_sm = (tiles + sms - 1) / sms;
    const uint64_t at_once = n < 24 ? per_sm : QP <= 8 && B == 4 && 227 * 1024 / smem >= 2 ? 2 : 1;
    return 10.0 + (double)((per_sm + at_once - 1) / at_once) * ticks * (1.0 + rates * (0.08 + 0.003 * (s < B ? s : B) * QP));
}

int launch_pipe_kernel(int scheme, int QP, int shape, size_t smem, uint64_t paths, cudaStream_t st, const PathArgs &a)
{
    const int B = shape & 255, lg = shape >> 8;
    PipeFn f = scheme == FULL ? pick_pipe<FULL>(QP, B) : scheme == PICARD ? pick_pipe<PICARD>(QP, B) : nullptr;
    if (!f) return (int)cudaErrorInvalidValue;
    const cudaError_t e = allow_smem(f, smem);
    if (e != cudaSuccess) return (int)e;
    f<<<(unsigned)((paths + 31) / 32), 32 << lg, smem, st>>>(a, lg);
    return (int)cudaGetLastError();
}

}  // namespace lll

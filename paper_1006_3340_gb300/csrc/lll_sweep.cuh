// lll_sweep.cuh -- the time-blocked rate sweep of the path kernels.
//
// One path's Euler steps of Eq. (log-LIB-SDE-2) form a triangle: the drift of
// rate i at t_k reads the weights of the rates above it at the same t_k (Eq.
// (LIBOR-drift-PT)), and its own log-rate only through its own weight.  So a
// block of B consecutive steps can be swept rate by rate from the top: rate i
// is carried through all B steps while the node products of the B steps,
//     P~_j(k) = c_j prod_{l > i} (1 + w_l(t_k) E_lj(k)),   k = k0 .. k0 + B - 1,
// wait in registers, and then the next rate.  Against sweeping the rates step
// by step:
//  * a rate's state is loaded and stored once per B steps, not once per step;
//  * the B dot products of a rate do not depend on one another, and only B
//    additions and the weights of the rate's own chain are serial, so one warp
//    per scheduler already hides most of the latency;
//  * the table rows of B steps are staged behind one barrier.
// Every unit (path, rate, step) is the arithmetic of sweep_dot / sweep_grow
// below, whatever the block length and the mapping.
#pragma once

#include "lll_device.cuh"
#include "lll_internal.h"

namespace lll {

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// delta L / (1 + delta L) for x = log(delta L) (approximate ex2 and rcp: w only
// scales the state-dependent part of the compensator).
__device__ __forceinline__ float weight_of(float x)
{
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(-1.4426950408889634f * x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
    return r;
}

__device__ __forceinline__ void kahan_add(double *s, double *c, double x)
{
    const double y = x - *c;
    const double t = *s + y;
    *c = (t - *s) - y;
    *s = t;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Rows of the sweeps' rule: (lambda, x, K', 0) with x = -log2(e) (log(delta
// L(0,T_i)) + D0), the constant part of the weight's exponent under Picard.
// The node factors are scaled, -h c_j, so that the dot product and K' together
// are the drift's contribution b_i h to the step itself; K' closes the sum at
// zero weights (P~_j = -h c_j) as FP32 forms it, -h C_i less that sum, so that
// its rounding leaves no bias common to all paths (lll_tables.cu).
//
// sum_j E_ij P~_j for one row E of QP nodes (P~ as pairs).
template <int QP>
__device__ __forceinline__ float sweep_dot(const float4 (&E)[QP / 4], const float2 (&P)[QP / 2])
{
    float2 a, b;
#pragma unroll
    for (int j4 = 0; j4 < QP / 4; ++j4) {
        const float2 e0 = make_float2(E[j4].x, E[j4].y), e1 = make_float2(E[j4].z, E[j4].w);
        a = j4 == 0 ? __fmul2_rn(e0, P[0]) : __ffma2_rn(e0, P[2 * j4], a);
        b = j4 == 0 ? __fmul2_rn(e1, P[1]) : __ffma2_rn(e1, P[2 * j4 + 1], b);
    }
    a = __fadd2_rn(a, b);
    return a.x + a.y;
}

// w = delta L / (1 + delta L) = 1 / (1 + 2^(x - log2(e) z)) for the offset z of
// log L from x's constant (approximate ex2 and rcp, as weight_of).
__device__ __forceinline__ float sweep_weight(float x, float z)
{
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fmaf(-1.4426950408889634f, z, x)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
    return r;
}

// P~_j *= 1 + w E_ij.
template <int QP>
__device__ __forceinline__ void sweep_grow(const float4 (&E)[QP / 4], float2 (&P)[QP / 2], float w)
{
    const float2 w2 = make_float2(w, w);
#pragma unroll
    for (int j4 = 0; j4 < QP / 4; ++j4) {
        P[2 * j4] = __ffma2_rn(__fmul2_rn(w2, make_float2(E[j4].x, E[j4].y)), P[2 * j4], P[2 * j4]);
        P[2 * j4 + 1] = __ffma2_rn(__fmul2_rn(w2, make_float2(E[j4].z, E[j4].w)), P[2 * j4 + 1], P[2 * j4 + 1]);
    }
}

// ---- A tile of T R paths of one simulation ----------------------------------

// Shared memory of a block: table rows of CH rates for B steps, double-buffered.
struct BlockSmem {
    float4 *tab;  // [2][CH][B][QP/4]: the B steps of a rate side by side, at immediate offsets
    float4 *row;  // [2][CH][B]
    float2 *cn;   // [QP/2]: -h c_j
    float *c0;    // [n]: -log2(e) log(delta L(0, T_l))
    float *dh;    // [B][R][T]: increments on their way to registers
    float4 *pay;  // [R][T]: maturity_values of the block's paths
    float4 *part; // [T]: payoff sums of slices of them
};

__host__ __device__ inline size_t up16(size_t v) { return (v + 15) & ~size_t(15); }

// Bytes of each part, in the order of BlockSmem.
__host__ __device__ inline size_t block_smem_bytes(int QP, int B, int R, int n, int T, int CH)
{
    return 2 * (size_t)B * CH * QP * 4 + 2 * (size_t)B * CH * 16 + up16((size_t)QP * 4) + up16((size_t)n * 4) +
           up16((size_t)B * R * T * 4) + (size_t)(R + 1) * T * 16;
}

__device__ inline BlockSmem block_carve(unsigned char *p, int QP, int B, int R, int n, int T, int CH)
{
    BlockSmem s;
    s.tab = reinterpret_cast<float4 *>(p);
    p += 2 * (size_t)B * CH * QP * 4;
    s.row = reinterpret_cast<float4 *>(p);
    p += 2 * (size_t)B * CH * 16;
    s.cn = reinterpret_cast<float2 *>(p);
    p += up16((size_t)QP * 4);
    s.c0 = reinterpret_cast<float *>(p);
    p += up16((size_t)n * 4);
    s.dh = reinterpret_cast<float *>(p);
    p += up16((size_t)B * R * T * 4);
    s.pay = reinterpret_cast<float4 *>(p);
    s.part = s.pay + (size_t)R * T;
    return s;
}

// The steps of a tile in order: period m (rates m .. n live), blocks of B steps
// within the period, chunks of CH rates from the top within the block.
struct BlockPos {
    int m, kb, c; // period, first step within it, chunk
};

// Stage the rows of position `at` into buffer b.
template <int QP, int B>
__device__ __forceinline__ void stage_rows(const PathArgs &a, const BlockSmem &sm, const BlockPos &at, int b)
{
    constexpr int Q4 = QP / 4;
    const int n = a.n, CH = a.chunk_rows;
    const int itop = n - at.c * CH;
    const int ibot = max(at.m, itop - CH + 1);
    const int cnt = itop - ibot + 1;
    const int nb = min(B, a.s - at.kb);
    const size_t r0 = ((size_t)(at.m - 1) * a.s + at.kb) * n + (ibot - 1);
    float4 *dt = sm.tab + (size_t)b * B * CH * Q4, *dr = sm.row + (size_t)b * B * CH;
    for (int e = threadIdx.x; e < cnt * B * Q4; e += blockDim.x) {
        const int j = e % Q4, s = e / Q4 % B, r = e / (Q4 * B);
        if (s < nb) cp_async16(dt + e, a.tab + (r0 + (size_t)s * n + r) * Q4 + j);
    }
    for (int e = threadIdx.x; e < cnt * B; e += blockDim.x) {
        const int s = e % B, r = e / B;
        if (s < nb) cp_async16(dr + e, a.brow + r0 + (size_t)s * n + r);
    }
}

// A thread's state of one rate: its R paths' offsets of log L from log L(0)
// (full), or int lambda dH and the drift integral per path (Picard).
template <int N>
struct alignas(4 * N) State {
    float v[N];
};

// What a kernel prices: caplets; swaptions in pairs of FP32 numbers; swaptions in
// FP64 (values beyond the pairs' range, see beyond_pairs).
enum { CAPLETS = 0, SWAPTIONS = 1, WIDE_SWAPTIONS = 2 };

// Payoffs of the block's paths at T_m into the block's FP64 Kahan sums
// acc[(m-1) ns + q][2] with compensations comp[..][2].  Every thread leaves its
// paths' values in shared memory; then thread (strike q, slice g) adds up the
// payoffs of every G-th path in double-float pairs (FP64: WIDE_SWAPTIONS), and
// thread q the G slices.  (Reducing each strike over the warp's lanes instead, by
// shuffles, took 0.25 of 2.08 ms on the N = 40 workload and three times the
// latency.)  beyond (SWAPTIONS): a word in shared memory, set where a swaption of the
// block's paths is beyond the pairs.
template <int NST, int R, int PRICES>
__device__ __forceinline__ void block_maturity(const PathArgs &a, const BlockSmem &sm, const State<NST * R> *st, int T,
                                               int m, const uint64_t (&lp)[R], double *acc, double *comp, bool first,
                                               int *beyond)
{
    constexpr bool WIDE = PRICES == WIDE_SWAPTIONS;
    const int n = a.n, ns = a.ns, tid = threadIdx.x;
    // (the caplets' kernels keep the run-time product: with a constant in its place the
    // N = 40 Picard kernel took 12.88 ms for 2^20 paths, not 12.74)
    const int product = PRICES == CAPLETS ? a.product : 1;
    double2 *const values = reinterpret_cast<double2 *>(sm.pay), *const sums = reinterpret_cast<double2 *>(sm.part);
#pragma unroll
    for (int u = 0; u < R; ++u) {
        auto z = [&](int i) {
            const State<NST * R> v = st[(size_t)(i - 1) * T];
            float x = v.v[NST * u];
            if constexpr (NST == 2) x += v.v[2 * u + 1];
            return x;
        };
        if constexpr (WIDE) {
            auto rate = [&](int i) { return __ldg(a.L0 + i - 1) * expf(z(i)); };
            values[u * T + tid] = lp[u] < a.paths ? swaption_values(a.delta, n, m, rate) : make_double2(0.0, 0.0);
        } else {
            float4 v = maturity_values(a, product, m, z);
            if (lp[u] >= a.paths) v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if constexpr (PRICES == SWAPTIONS) {
                if (beyond_pairs(v)) *beyond = 1;
            }
            sm.pay[u * T + tid] = v;
        }
        if (a.snap != nullptr && lp[u] < a.paths && lp[u] % a.snap_stride == 0 && lp[u] / a.snap_stride < a.n_snap)
            for (int i = n; i >= m; --i)
                a.snap[((size_t)(m - 1) * n + (i - 1)) * a.snap_pitch + lp[u] / a.snap_stride] = z(i) + a.Z0[i - 1];
    }
    __syncthreads();
    for (int q0 = 0; q0 < ns; q0 += T) { // one pass unless there are more strikes than threads
        const int nq = min(ns - q0, T);
        // slices: about the square root of the paths, which balances the two sums
        const int G = min(T / nq, R * T >= 256 ? 16 : R * T >= 64 ? 8 : 6);
        const int q = tid % nq, g = tid / nq;
        if (g < G) {
            const float K = a.strikes[(size_t)(m - 1) * ns + q0 + q];
            if constexpr (WIDE) {
                const double scale = payoff_scale(a);
                double s1 = 0.0, s2 = 0.0;
                for (int p = g; p < R * T; p += G) {
                    const double X = values[p].x - (double)K * values[p].y, v = X > 0.0 ? scale * X : 0.0;
                    s1 += v;
                    s2 += v * v;
                }
                sums[g * nq + q] = make_double2(s1, s2);
            } else {
                DFloat s1{0.0f, 0.0f}, s2{0.0f, 0.0f};
                for (int p = g; p < R * T; p += G) {
                    const DFloat v = payoff_of(product, sm.pay[p], K);
                    s1 = df_add(s1, v);
                    s2 = df_add(s2, df_square_pair(v));
                }
                sm.part[g * nq + q] = make_float4(s1.hi, s1.lo, s2.hi, s2.lo);
            }
        }
        __syncthreads();
        if (tid < nq) {
            double v1, v2;
            if constexpr (WIDE) {
                v1 = sums[tid].x;
                v2 = sums[tid].y;
                for (int k = 1; k < G; ++k) {
                    v1 += sums[k * nq + tid].x;
                    v2 += sums[k * nq + tid].y;
                }
            } else {
                float4 r = sm.part[tid];
                DFloat x{r.x, r.y}, y{r.z, r.w};
                for (int k = 1; k < G; ++k) {
                    r = sm.part[k * nq + tid];
                    x = df_add(x, DFloat{r.x, r.y});
                    y = df_add(y, DFloat{r.z, r.w});
                }
                const double c = payoff_scale(a);
                v1 = c * ((double)x.hi + (double)x.lo);
                v2 = c * c * ((double)y.hi + (double)y.lo);
            }
            const size_t e = 2 * ((size_t)(m - 1) * ns + q0 + tid);
            if (first) {
                acc[e] = v1;
                acc[e + 1] = v2;
                comp[e] = comp[e + 1] = 0.0;
            } else {
                kahan_add(acc + e, comp + e, v1);
                kahan_add(acc + e + 1, comp + e + 1, v2);
            }
        }
        if (q0 + T < ns) __syncthreads();
    }
}

// Rates itop .. ibot through the nb <= B steps staged in buffer `buf` (TAIL:
// nb < B).  P: node products of each step; dH: increments.
template <int SCHEME, int QP, int B, int R, bool TAIL>
__device__ __forceinline__ void sweep_chunk(const PathArgs &a, const BlockSmem &sm, State<(SCHEME == PICARD ? 2 : 1) * R> *st,
                                            int T, int itop, int ibot, int buf, int nb, const float (&dH)[R][B],
                                            float2 (&P)[R][B][QP / 2])
{
    constexpr int Q4 = QP / 4, NST = (SCHEME == PICARD) ? 2 : 1;
    const int CH = a.chunk_rows;
    const float4 *tr = sm.tab + ((size_t)buf * CH + (itop - ibot)) * (B * Q4);
    const float4 *rr = sm.row + ((size_t)buf * CH + (itop - ibot)) * B;
    State<NST * R> next = st[(size_t)(itop - 1) * T];
    for (int i = itop; i >= ibot; --i, tr -= B * Q4, rr -= B) {
        State<NST * R> cur = next;
        if (i > ibot) next = st[(size_t)(i - 2) * T];
        const float c0 = sm.c0[i - 1];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (TAIL && b >= nb) break;
            const float4 rc = rr[b];
            float4 E[Q4];
#pragma unroll
            for (int j = 0; j < Q4; ++j) E[j] = tr[b * Q4 + j];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const float w = sweep_weight(SCHEME == PICARD ? rc.y : c0, cur.v[NST * q]);
                const float bh = sweep_dot<QP>(E, P[q][b]) + rc.z;
                if constexpr (SCHEME == PICARD) {
                    cur.v[2 * q] = fmaf(rc.x, dH[q][b], cur.v[2 * q]); // int lambda dH
                    cur.v[2 * q + 1] += bh;                            // Picard drift integral
                } else {
                    cur.v[q] = cur.v[q] + fmaf(rc.x, dH[q][b], bh);
                }
                sweep_grow<QP>(E, P[q][b], w);
            }
        }
        st[(size_t)(i - 1) * T] = cur;
    }
}

// One tile: all Euler steps and payoffs.  st: this thread's column of the
// block's state slot [n][T]; acc, comp: the block's payoff sums; first: they
// hold nothing yet; beyond: see block_maturity.
template <int SCHEME, int QP, int B, int R, int PRICES>
__device__ __forceinline__ void block_tile(const PathArgs &a, const BlockSmem &sm, State<(SCHEME == PICARD ? 2 : 1) * R> *st,
                                           uint64_t tile, double *acc, double *comp, bool first, int *beyond = nullptr)
{
    constexpr int NST = (SCHEME == PICARD) ? 2 : 1;
    const int T = blockDim.x, tid = threadIdx.x;
    const int n = a.n, s = a.s, CH = a.chunk_rows;
    uint64_t lp[R];
#pragma unroll
    for (int q = 0; q < R; ++q) lp[q] = tile * ((uint64_t)T * R) + (uint64_t)q * T + tid;
    State<NST * R> zero;
#pragma unroll
    for (int q = 0; q < NST * R; ++q) zero.v[q] = 0.0f;
    for (int l = 0; l < n; ++l) st[(size_t)l * T] = zero;

    __syncthreads(); // the previous tile's readers of both buffers are done
    BlockPos at{1, 0, 0};
    stage_rows<QP, B>(a, sm, at, 0);
    cp_commit();
    int buf = 0;
    for (int m = 1; m <= n; ++m) {
        const int nch = (n - m + CH) / CH; // ceil((n - m + 1) / CH)
        for (int kb = 0; kb < s; kb += B) {
            const int k0 = (m - 1) * s + kb, nb = min(B, s - kb);
            // the draws stay a loop (their code is long), two at a time to overlap their
            // latencies; registers take them afterwards
#pragma unroll 2
            for (int e = 0; e < nb * R; ++e) {
                const int b = e / R, q = e % R;
                sm.dh[(size_t)e * T + tid] =
                    draw_increment(a, a.first_path + tile * ((uint64_t)T * R) + (uint64_t)q * T + tid, (uint32_t)(k0 + b));
            }
            float dH[R][B];
#pragma unroll
            for (int b = 0; b < B; ++b)
#pragma unroll
                for (int q = 0; q < R; ++q) dH[q][b] = b < nb ? sm.dh[(size_t)(b * R + q) * T + tid] : 0.0f;
            float2 P[R][B][QP / 2]; // P~ = c_j above the top rate
#pragma unroll
            for (int j = 0; j < QP / 2; ++j) {
                const float2 cj = sm.cn[j];
#pragma unroll
                for (int q = 0; q < R; ++q)
#pragma unroll
                    for (int b = 0; b < B; ++b) P[q][b][j] = cj;
            }
            for (int c = 0; c < nch; ++c) {
                // the position after this one
                BlockPos nx{m, kb, c + 1};
                if (nx.c == nch) { nx.c = 0; nx.kb += B; }
                if (nx.kb >= s) { nx.kb = 0; nx.m += 1; }
                if (nx.m <= n) stage_rows<QP, B>(a, sm, nx, buf ^ 1);
                cp_commit();
                cp_wait_1();
                __syncthreads();
                const int itop = n - c * CH, ibot = max(m, itop - CH + 1);
                if (nb == B) sweep_chunk<SCHEME, QP, B, R, false>(a, sm, st, T, itop, ibot, buf, nb, dH, P);
                else sweep_chunk<SCHEME, QP, B, R, true>(a, sm, st, T, itop, ibot, buf, nb, dH, P);
                __syncthreads(); // buffer `buf` is staged into next
                buf ^= 1;
            }
        }
        block_maturity<NST, R, PRICES>(a, sm, st, T, m, lp, acc, comp, first, beyond);
    }
    cp_wait_0();
}

}  // namespace lll

// lll_capi.cpp -- the C ABI declared in include/lll.h.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/lll.h"
#include "lll_ctx.h"
#include "lll_internal.h"

namespace lll {
int build_nig_rule(double alpha, double beta, double dbar, double a, int Q, double *nodes,
                   double *weights);
int simulate_mlp(lll_ctx *ctx, uint64_t first_path, uint64_t paths, uint64_t seed);
int simulate_expand(lll_ctx *ctx, int order, uint64_t first_path, uint64_t paths, uint64_t seed);
}

namespace lll {
void dev_free(lll_ctx *ctx, void *p)
{
    const char *q = static_cast<const char *>(p);
    if (q && !(ctx->arena && q >= ctx->arena && q < ctx->arena + ctx->arena_bytes)) cudaFree(p);
}
}

using namespace lll;

namespace {

thread_local std::string g_err;

int fail(lll_ctx *ctx, int code, const std::string &msg)
{
    if (ctx) ctx->err = msg;
    g_err = msg;
    return code;
}

int cuda_fail(lll_ctx *ctx, cudaError_t e, const char *what)
{
    return fail(ctx, LLL_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define CUDA_TRY(ctx, expr)                                                                        \
    do {                                                                                           \
        cudaError_t e_ = (expr);                                                                   \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #expr);                                   \
    } while (0)

bool isfin(double v) { return std::isfinite(v); }

int padded_q(int Q)
{
    if (Q <= 0) return 0;
    const int opts[] = {16, 32, 64, 96, 128};
    for (int o : opts)
        if (Q <= o) return o;
    return -1;
}

template <class T>
cudaError_t dalloc(T **p, size_t count)
{
    return cudaMalloc((void **)p, sizeof(T) * std::max<size_t>(count, 1));
}

void free_all(lll_ctx *c)
{
    for (void *p : {(void *)c->d_partials, (void *)c->d_sums, (void *)c->d_state, (void *)c->d_snap,
                    (void *)c->d_err, (void *)c->d_K1, (void *)c->d_K2, (void *)c->d_K3})
        dev_free(c, p);
    cudaFree(c->arena);
    mlp_free(c->mlp);
    c->mlp = nullptr;
    for (auto &e : c->ev)
        if (e) cudaEventDestroy(e);
}

// Payoff scratch in the arena (doubles, 256 KB): short curves on a few thousand paths
// need no more (a pipeline of 4,864 paths, 9 rates, 11 strikes), and their fresh
// contexts, priced once, then allocate nothing else; a larger call allocates its own.
constexpr size_t kArenaPartials = size_t(1) << 15;

int default_chunk_rows(int n, int QP)
{
    if (QP == 0) return std::min(n, 64);
    // Keep the double-buffered node tables near 24 KB (room for five blocks per SM).
    const int rows = (24 * 1024) / (2 * (QP / 4) * (int)sizeof(float4));
    return std::max(1, std::min(n, rows));
}

}  // namespace

namespace lll {

int record_error(lll_ctx *ctx, int code, const char *msg) { return fail(ctx, code, msg); }

// In the room that lll_init keeps for them: no allocation, so the selections
// that need them may come at any time, also while the stream is captured (the
// two kernels are then part of the graph, and the next call outside builds them).
int ensure_full_tables(lll_ctx *ctx)
{
    if (ctx->QR == ctx->QP || ctx->full_built) return LLL_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess) cudaGetLastError();
    cudaError_t e = (cudaError_t)launch_tables(ctx->d_lam, ctx->d_x, ctx->d_W, ctx->Q, ctx->n, ctx->S, ctx->QP, ctx->h,
                                               ctx->c, nullptr, ctx->d_tab_full, ctx->d_cn_full, ctx->d_row_full, nullptr,
                                               ctx->d_C_full, nullptr, ctx->stream);
    if (e == cudaSuccess)
        e = (cudaError_t)launch_prefix(ctx->d_b0, ctx->n, ctx->S, ctx->h, nullptr, ctx->delta, ctx->d_row_full, nullptr,
                                       ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "tables of the given rule");
    ctx->full_built = cap == cudaStreamCaptureStatusNone;
    return LLL_OK;
}

int use_full_tables(lll_ctx *ctx)
{
    const int rc = ensure_full_tables(ctx);
    if (rc != LLL_OK || ctx->QR == ctx->QP) return rc;
    ctx->d_tab = ctx->d_tab_full;
    ctx->d_row = ctx->d_row_full;
    ctx->d_cn = ctx->d_cn_full;
    ctx->d_brow = nullptr;
    ctx->QR = ctx->QP;
    return LLL_OK;
}

int launch_plan(const LaunchPlan &plan, const PathArgs &a)
{
    if (plan.tenor > 0) return launch_tenor_kernel(plan.scheme, plan.qp, plan.tenor, plan.grid, plan.smem, plan.stream, a);
    if (plan.lpp > 1)
        return launch_group_kernel(plan.scheme, plan.qp, plan.lpp, plan.grid, plan.threads, plan.smem, plan.stream, a);
    if (plan.pipe) return launch_pipe_kernel(plan.scheme, plan.qp, plan.pipe, plan.smem, a.paths, plan.stream, a);
    if (plan.block)
        return launch_block_kernel(plan.scheme, plan.qp, plan.ppt, plan.grid, plan.threads, plan.smem, plan.stream, a);
    return launch_path_kernel(plan.scheme, plan.qp, plan.ppt, plan.grid, plan.threads, plan.smem, plan.stream, a);
}

// Paths per thread and threads per block of the time-blocked kernel where the
// caller has not set them.  128 threads share a block's staged rows (32-thread
// blocks fill shared memory with copies of them: N = 120 Picard, 16,384 paths
// 5.8 against 3.05 ms).  Two paths a thread pay up to 8 nodes once they leave no
// scheduler short of warps: N = 40, 90,000 paths 1.42 ms (one: 1.38), 130,000
// paths 1.81 (1.85), 2^20 paths 12.3 (12.6); with 20 nodes (N = 120, 2^17 paths)
// 16.4 against 14.7.
static void block_shape(const lll_ctx *ctx, uint64_t paths, int *R, int *T)
{
    if (ctx->ppt == 0) *R = ctx->QR <= 8 && paths >= 640ull * ctx->sm_count ? 2 : 1;
    if (ctx->threads == 0) *T = 128;
}

// Whether a default launch of caplets may take the pipeline (pipe_shape).
static bool pipe_allowed(const lll_ctx *ctx)
{
    return ctx->threads == 0 && ctx->blocks_per_sm == 0 && ctx->ppt == 0 && ctx->chunk_rows == 0 &&
           ctx->product == LLL_PRODUCT_CAPLET;
}

// Scratch that smaller calls of this context, on other kernels than this plan's, may
// need more of: a call with fewer paths than an earlier one then never changes the
// buffers.  The pipeline's many small blocks have more payoff sums than the block
// kernel's on more paths; and where the pipeline's shape for one block an SM does not
// fit shared memory, the block kernel serves fewer paths than the pipeline.
static void smaller_calls(const lll_ctx *ctx, const LaunchPlan &plan, size_t *state_floats, size_t *partial_doubles)
{
    if (!plan.block || !pipe_allowed(ctx)) return;
    const uint64_t now_per_sm = ((plan.args.paths + 31) / 32 + ctx->sm_count - 1) / ctx->sm_count;
    const int now = (int)std::min<uint64_t>(now_per_sm, kMaxPipePerSm);
    for (int scheme : {LLL_FULL, LLL_PICARD})
        for (int per_sm = 1; per_sm <= now; ++per_sm) {
            size_t smem;
            const uint64_t tiles = (uint64_t)per_sm * ctx->sm_count; // of 32 paths
            const bool pipe = pipe_shape(scheme, ctx->QR, ctx->n, ctx->s, ctx->S, tiles, ctx->sm_count, &smem) != 0;
            if (pipe && !plan.pipe) *partial_doubles = std::max(*partial_doubles, tiles * plan.n_out);
            if (!pipe && plan.pipe && per_sm < now)
                *state_floats = std::max(*state_floats, (tiles + 3) / 4 * ctx->n * 128 * (scheme == LLL_PICARD ? 2 : 1));
        }
}

// Same launch shape and arguments as lll_simulate, with no allocation: the
// per-block scratch sizes are returned for the caller to place.
int plan_launch(lll_ctx *ctx, int scheme, uint64_t first_path, uint64_t paths, uint64_t seed,
                LaunchPlan *plan, bool allow_tenor, bool given_rule, bool allow_pipe)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (!plan) return fail(ctx, LLL_EINVAL, "plan is NULL");
    if (scheme == LLL_MLP || scheme == LLL_EXPAND1 || scheme == LLL_EXPAND2)
        return fail(ctx, LLL_EUNSUPPORTED, "LLL_MLP and LLL_EXPAND1/2 run through lll_simulate only");
    if (scheme != LLL_FULL && scheme != LLL_PICARD && scheme != LLL_FROZEN)
        return fail(ctx, LLL_EINVAL, "unknown scheme");
    if (ctx->ns == 0) return fail(ctx, LLL_ESTATE, "lll_set_strikes must come before simulating");
    if (paths == 0) return fail(ctx, LLL_EINVAL, "paths must be > 0");
    if (first_path + paths < first_path) return fail(ctx, LLL_EINVAL, "path range overflows");
    // What a launch supports follows the rule as given (QPk nodes); the one-lane
    // kernels sweep its shorter equivalent, where there is one, in time blocks.
    const int QPk = (scheme == LLL_FROZEN) ? 0 : ctx->QP;
    // Tenor-parallel mapping (lll_set_mapping): G lanes per path, full and
    // Picard with a node table and caplet payoffs; other schemes keep the
    // path mapping.
    const int G = (allow_tenor && ctx->tenor_lanes > 0 && (scheme == LLL_FULL || scheme == LLL_PICARD))
                      ? ctx->tenor_lanes : 0;
    if (G > 0) {
        if (QPk == 0 || ctx->product != LLL_PRODUCT_CAPLET || !tenor_kernel_supported(scheme, QPk, G))
            return fail(ctx, LLL_EUNSUPPORTED, "the tenor-parallel mapping needs a node table and caplet payoffs");
    }
    // Lanes per group of paths: 1 (one lane sweeps all nodes of its path) or
    // 2 / 4 (lane groups share the node sweep); the default is 1.
    const int lpp = G > 0 ? 1 : (ctx->lpp > 0 ? ctx->lpp : 1);
    int R = (lpp > 1 || G > 0) ? 1 : (ctx->ppt > 0 ? ctx->ppt : 1);
    if (lpp > 1 && !group_kernel_supported(scheme, QPk, lpp))
        return fail(ctx, LLL_EUNSUPPORTED, "lane groups need a node table (NIG, full or Picard)");
    if (G == 0 && lpp == 1 && !path_kernel_supported(scheme, QPk, R))
        return fail(ctx, LLL_EUNSUPPORTED, "no kernel for this Q and paths per thread");
    int T = G > 0 ? tenor_kernel_threads() : ctx->threads > 0 ? ctx->threads : 128;
    int CH = ctx->chunk_rows > 0 ? ctx->chunk_rows : default_chunk_rows(ctx->n, ctx->QP);
    size_t smem = G > 0 ? tenor_kernel_smem(QPk, ctx->n, ctx->ns, G)
                : lpp > 1 ? group_kernel_smem(QPk, ctx->n, ctx->ns, T, CH)
                          : path_kernel_smem(QPk, ctx->n, ctx->ns, T, CH);
    if (smem > 227 * 1024) return fail(ctx, LLL_EUNSUPPORTED, "shared memory need exceeds 227 KB");
    const bool block = !given_rule && G == 0 && lpp == 1 && QPk > 0 && ctx->QR < ctx->QP;
    if (block) {
        block_shape(ctx, paths, &R, &T);
        CH = block_chunk_rates(ctx->QR, R, ctx->n, ctx->chunk_rows);
        smem = block_kernel_smem(ctx->QR, R, ctx->n, T, CH);
    }
    // The pipeline serves a default launch of caplets on few paths.
    size_t pipe_smem = 0;
    const int pipe = allow_pipe && block && pipe_allowed(ctx)
                         ? pipe_shape(scheme, ctx->QR, ctx->n, ctx->s, ctx->S, (paths + 31) / 32, ctx->sm_count, &pipe_smem)
                         : 0;
    int occ = 0;
    cudaError_t e;
    if (pipe) {
        R = 1;
        T = 32; // paths a block
        smem = pipe_smem;
        occ = 1;
    } else if (G > 0) {
        e = (cudaError_t)tenor_kernel_prepare(scheme, QPk, G, smem, &occ);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "tenor kernel attributes");
    } else if (lpp > 1) {
        e = (cudaError_t)group_kernel_prepare(scheme, QPk, lpp, smem, T, &occ);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "group kernel attributes");
    } else if (block) {
        e = (cudaError_t)block_kernel_prepare(scheme, ctx->product, ctx->QR, R, paths, smem, T, &occ);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "block kernel attributes");
    } else {
        e = (cudaError_t)path_kernel_prepare(scheme, QPk, R, paths, T, smem);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute");
        e = (cudaError_t)path_kernel_occupancy(scheme, QPk, R, paths, T, smem, &occ);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "occupancy");
    }
    if (occ < 1) return fail(ctx, LLL_EUNSUPPORTED, "launch shape does not fit on an SM");
    const int bps = ctx->blocks_per_sm > 0 ? std::min(ctx->blocks_per_sm, occ) : occ;
    const uint64_t per_tile = G > 0 ? (uint64_t)(T / G) : (uint64_t)T * R; // paths per block tile
    const uint64_t tiles = (paths + per_tile - 1) / per_tile;
    const int grid = (int)(pipe ? tiles : std::min<uint64_t>(tiles, (uint64_t)bps * ctx->sm_count));
    const int nst = (scheme == LLL_PICARD) ? 2 : 1;
    PathArgs a{};
    const bool other = !given_rule && !block && QPk > 0 && ctx->QR < ctx->QP; // the rule as given (lane groups, tenor mapping)
    if (other) {
        const int rc = ensure_full_tables(ctx);
        if (rc != LLL_OK) return rc;
    }
    a.tab = other ? ctx->d_tab_full : ctx->d_tab;
    a.cn = other ? ctx->d_cn_full : ctx->d_cn;
    a.brow = ctx->d_brow;
    a.row = other ? ctx->d_row_full : ctx->d_row;
    a.Z0 = ctx->d_Z0; a.L0 = ctx->d_L0; a.c0 = ctx->d_c0;
    a.strikes = ctx->d_strikes; a.partials = nullptr; a.state = nullptr;
    a.snap = nullptr; a.n_snap = 0; a.snap_stride = 1; a.snap_pitch = 0;
    a.first_path = first_path; a.paths = paths;
    a.n = ctx->n; a.s = ctx->s; a.S = ctx->S; a.ns = ctx->ns; a.chunk_rows = CH;
    a.key0 = (uint32_t)seed; a.key1 = (uint32_t)(seed >> 32); a.inst = 0;
    a.driver = ctx->driver; a.qr = block ? ctx->QR : QPk;
    a.h = (float)ctx->h; a.sqrt_h = (float)std::sqrt(ctx->h); a.delta = (float)ctx->delta;
    a.dBN = (float)(ctx->delta * ctx->BN);
    a.product = ctx->product;
    a.wide_strikes = ctx->wide_strikes;
    if (ctx->driver == LLL_DRIVER_NIG) {
        const double m = ctx->nig.delta * ctx->h / ctx->gam;
        const double l = (ctx->nig.delta * ctx->h) * (ctx->nig.delta * ctx->h);
        a.ig_m = (float)m; a.ig_m2 = (float)(m * m); a.ig_hl = (float)(m / (2.0 * l));
        a.ig_fl = (float)(4.0 * m * l); a.ig_md = m; a.ig_ld = l;
        a.nig_beta = (float)ctx->nig.beta; a.nig_muh = (float)(ctx->mu * ctx->h);
    }
    plan->args = a;
    plan->scheme = scheme; plan->qp = block ? ctx->QR : QPk; plan->block = block; plan->pipe = pipe; plan->ppt = R; plan->lpp = lpp; plan->threads = T; plan->grid = grid;
    plan->tenor = G;
    plan->smem = smem;
    // the tenor-parallel kernel keeps its path state in shared memory
    plan->state_floats_per_block = G > 0 || pipe ? 0 : (size_t)R * nst * ctx->n * T;
    plan->partial_doubles_per_block = (size_t)ctx->n * ctx->ns * 2 * (block && !pipe ? 2 : 1);
    plan->n_out = ctx->n * ctx->ns * 2;
    plan->stream = ctx->stream;
    plan->device = ctx->device;
    return LLL_OK;
}

}  // namespace lll

extern "C" {

const char *lll_last_error(const lll_ctx *ctx) { return ctx ? ctx->err.c_str() : g_err.c_str(); }

int lll_build_nig_quadrature(lll_nig nig, double xmax, int Q, double *nodes, double *weights)
{
    if (!nodes || !weights || Q < 1) return fail(nullptr, LLL_EINVAL, "null output or Q < 1");
    if (Q > kMaxQP) return fail(nullptr, LLL_EUNSUPPORTED, "Q > 128");
    if (!(nig.alpha > std::fabs(nig.beta)) || !(nig.delta > 0) || !(xmax > 0) || !isfin(xmax))
        return fail(nullptr, LLL_EINVAL, "need alpha > |beta|, delta > 0, xmax > 0");
    if (build_nig_rule(nig.alpha, nig.beta, nig.delta, xmax, Q, nodes, weights) != 0)
        return fail(nullptr, LLL_EINVAL, "quadrature construction failed");
    return LLL_OK;
}

int lll_sweep_rule(int Q, const double *nodes, const double *weights, double lo, double hi, int *count,
                   int *padded, double *x, double *w)
{
    if (!nodes || !weights || !count || !padded || !x || !w || Q < 1 || !(lo <= 0.0) || !(hi >= 0.0))
        return fail(nullptr, LLL_EINVAL, "null argument, Q < 1, or not lo <= 0 <= hi");
    const int QP = padded_q(Q);
    if (QP < 0) return fail(nullptr, LLL_EUNSUPPORTED, "Q > 128");
    for (int j = 0; j < Q; ++j)
        if (!isfin(nodes[j]) || nodes[j] == 0.0 || !isfin(weights[j]))
            return fail(nullptr, LLL_EINVAL, "nodes must be finite and non-zero");
    *padded = QP;
    *count = shorter_rule(nodes, weights, Q, QP, lo, hi, x, w, padded);
    return LLL_OK;
}

int lll_init(lll_ctx **out, int N, double tenor_delta, const double *L0, int steps_per_period,
             const double *lambda, int driver, lll_nig nig, int Q, const double *nodes,
             const double *weights, void *cuda_stream)
{
    if (!out) return fail(nullptr, LLL_EINVAL, "out is NULL");
    *out = nullptr;
    if (N < 2 || N > 4096) return fail(nullptr, LLL_EINVAL, "N must be in [2, 4096]");
    if (!(tenor_delta > 0) || !isfin(tenor_delta)) return fail(nullptr, LLL_EINVAL, "delta <= 0");
    if (steps_per_period < 1 || (long long)(N - 1) * steps_per_period > (1 << 24))
        return fail(nullptr, LLL_EINVAL, "steps_per_period out of range");
    if (!L0 || !lambda) return fail(nullptr, LLL_EINVAL, "L0 or lambda is NULL");
    if (driver != LLL_DRIVER_NIG && driver != LLL_DRIVER_BROWNIAN)
        return fail(nullptr, LLL_EINVAL, "unknown driver");
    const int n = N - 1, S = n * steps_per_period;
    double up = 0, down = 0; // largest sums of the live positive and negative volatilities over the steps
    for (int m = 0; m < N; ++m)
        if (!(L0[m] > 0) || !isfin(L0[m])) return fail(nullptr, LLL_EINVAL, "L0 must be finite and > 0");
    for (long long e = 0; e < (long long)S * n; ++e)
        if (!isfin(lambda[e])) return fail(nullptr, LLL_EINVAL, "lambda has NaN/Inf");
    int QP = 0;
    double mu = 0, gam = 0;
    bool domain_warn = false;
    if (driver == LLL_DRIVER_NIG) {
        if (!(nig.alpha > std::fabs(nig.beta)) || !(nig.delta > 0) || !isfin(nig.alpha) ||
            !isfin(nig.beta) || !isfin(nig.delta))
            return fail(nullptr, LLL_EINVAL, "NIG needs alpha > |beta| and delta > 0");
        if (Q < 1 || !nodes || !weights) return fail(nullptr, LLL_EINVAL, "NIG needs Q >= 1 nodes");
        QP = padded_q(Q);
        if (QP < 0) return fail(nullptr, LLL_EUNSUPPORTED, "Q > 128");
        for (int j = 0; j < Q; ++j)
            if (!isfin(nodes[j]) || nodes[j] == 0.0 || !isfin(weights[j]))
                return fail(nullptr, LLL_EINVAL, "nodes must be finite and non-zero");
        gam = std::sqrt(nig.alpha * nig.alpha - nig.beta * nig.beta);
        mu = std::isnan(nig.mu) ? -nig.delta * nig.beta / gam : nig.mu;
        if (!isfin(mu)) return fail(nullptr, LLL_EINVAL, "mu is Inf");
        for (int k = 0; k < S; ++k) {
            double sum = 0, pos = 0, neg = 0;
            for (int l = 0; l < n; ++l) {
                const double v = lambda[(size_t)k * n + l];
                sum += std::fabs(v);
                if (l >= k / steps_per_period) (v > 0 ? pos : neg) += v;
            }
            up = std::max(up, pos);
            down = std::min(down, neg);
            if (sum >= nig.alpha - std::fabs(nig.beta)) domain_warn = true;
        }
    } else {
        Q = 0;
    }

    int QR = QP, Qr = 0;
    double xr[32], wr[32];
    if (QP > 0) Qr = shorter_rule(nodes, weights, Q, QP, down, up, xr, wr, &QR);
    lll_ctx *c = new lll_ctx();
    c->QR = QR;
    c->N = N; c->n = n; c->s = steps_per_period; c->S = S; c->Q = Q; c->QP = QP;
    c->driver = driver; c->delta = tenor_delta; c->h = tenor_delta / steps_per_period;
    c->c = (driver == LLL_DRIVER_BROWNIAN) ? 1.0 : 0.0;
    c->nig = nig; c->mu = mu; c->gam = gam;
    c->stream = (cudaStream_t)cuda_stream;
    c->L0.assign(L0, L0 + N);
    c->lam.assign(lambda, lambda + (size_t)S * n);
    double BN = 1.0;
    for (int m = 0; m < N; ++m) BN /= 1.0 + tenor_delta * L0[m]; // Eq. (i-val) inverted
    c->BN = BN;

    auto bail = [&](int code) {
        std::string m = c->err;
        free_all(c);
        delete c;
        g_err = m;
        return code;
    };
    cudaError_t e;
    if ((e = cudaGetDevice(&c->device)) != cudaSuccess) { cuda_fail(c, e, "cudaGetDevice"); return bail(LLL_ECUDA); }
    if ((e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess) {
        cuda_fail(c, e, "cudaDeviceGetAttribute"); return bail(LLL_ECUDA);
    }
    // One arena: the inputs (one host image, one copy), then the tables, then
    // strikes, sums and payoff scratch for the usual sizes, and last room for the
    // tables of a rule as given beside its shorter one's.
    const size_t rows = (size_t)S * n;
    size_t bytes = 0;
    auto place = [&](size_t size) {
        const size_t at = bytes;
        bytes += (size + 255) & ~size_t(255);
        return at;
    };
    const size_t at_lam = place(8 * rows), at_x = place(8 * (size_t)Q), at_W = place(8 * (size_t)Q),
                 at_xr = place(8 * (size_t)Qr), at_wr = place(8 * (size_t)Qr), at_w0 = place(8 * (size_t)n),
                 at_Ld = place(8 * (size_t)N), at_Z0 = place(4 * (size_t)n), at_L0 = place(4 * (size_t)n),
                 at_c0 = place(4 * (size_t)n);
    const size_t in_bytes = bytes;
    const size_t at_b0 = place(8 * rows), at_tab = place(4 * rows * std::max(QR, 4)), at_cn = place(4 * std::max(QR, 4)),
                 at_row = place(16 * rows), at_brow = place(Qr > 0 ? 16 * rows : 0), at_C = place(4 * rows),
                 at_strikes = place(4 * (size_t)n * 64), at_sums = place(16 * (size_t)n * 64),
                 at_part = place(kArenaPartials * 8);
    const bool two = QR < QP;
    const size_t at_tabf = place(two ? 4 * rows * QP : 0), at_rowf = place(two ? 16 * rows : 0),
                 at_cnf = place(two ? 4 * (size_t)QP : 0), at_Cf = place(two ? 4 * rows : 0);
    std::vector<char> in(in_bytes);
    auto host = [&](size_t at) { return reinterpret_cast<double *>(in.data() + at); };
    std::memcpy(host(at_lam), lambda, 8 * rows);
    std::memcpy(host(at_Ld), L0, 8 * (size_t)N);
    if (Q > 0) {
        std::memcpy(host(at_x), nodes, 8 * (size_t)Q);
        std::memcpy(host(at_W), weights, 8 * (size_t)Q);
    }
    if (Qr > 0) {
        std::memcpy(host(at_xr), xr, 8 * (size_t)Qr);
        std::memcpy(host(at_wr), wr, 8 * (size_t)Qr);
    }
    for (int l = 1; l <= n; ++l) {
        host(at_w0)[l - 1] = tenor_delta * L0[l] / (1.0 + tenor_delta * L0[l]);
        reinterpret_cast<float *>(in.data() + at_Z0)[l - 1] = (float)std::log(L0[l]);
        reinterpret_cast<float *>(in.data() + at_L0)[l - 1] = (float)L0[l];
        reinterpret_cast<float *>(in.data() + at_c0)[l - 1] = (float)(std::log(L0[l]) + std::log(tenor_delta));
    }
    if (cudaMalloc((void **)&c->arena, bytes) != cudaSuccess) {
        c->arena = nullptr;
        fail(c, LLL_ENOMEM, "cudaMalloc of model tables failed");
        return bail(LLL_ENOMEM);
    }
    c->arena_bytes = bytes;
    auto dev = [&](size_t at) { return c->arena + at; };
    c->d_lam = (double *)dev(at_lam); c->d_x = (double *)dev(at_x); c->d_W = (double *)dev(at_W);
    c->d_w0 = (double *)dev(at_w0); c->d_b0 = (double *)dev(at_b0); c->d_tab = (float4 *)dev(at_tab);
    c->d_cn = (float *)dev(at_cn); c->d_row = (float4 *)dev(at_row); c->d_brow = Qr > 0 ? (float4 *)dev(at_brow) : nullptr;
    c->d_C = (float *)dev(at_C); c->d_Z0 = (float *)dev(at_Z0); c->d_L0 = (float *)dev(at_L0);
    c->d_c0 = (float *)dev(at_c0); c->d_strikes = (float *)dev(at_strikes); c->d_sums = (double *)dev(at_sums);
    c->sums_cap = 2 * (size_t)n * 64;
    c->d_partials = (double *)dev(at_part);
    c->partials_cap = kArenaPartials;
    if (two) {
        c->d_tab_full = (float4 *)dev(at_tabf); c->d_row_full = (float4 *)dev(at_rowf);
        c->d_cn_full = (float *)dev(at_cnf); c->d_C_full = (float *)dev(at_Cf);
    }
    for (auto &ev : c->ev)
        if ((e = cudaEventCreate(&ev)) != cudaSuccess) { cuda_fail(c, e, "cudaEventCreate"); return bail(LLL_ECUDA); }
    cudaStream_t st = c->stream;
#define INIT_TRY(expr)                                                                             \
    do {                                                                                           \
        cudaError_t e2 = (expr);                                                                   \
        if (e2 != cudaSuccess) { cuda_fail(c, e2, #expr); return bail(LLL_ECUDA); }               \
    } while (0)
    INIT_TRY(cudaMemcpyAsync(c->arena, in.data(), in_bytes, cudaMemcpyHostToDevice, st));
    INIT_TRY((cudaError_t)launch_tables(c->d_lam, Qr > 0 ? (double *)dev(at_xr) : c->d_x,
                                        Qr > 0 ? (double *)dev(at_wr) : c->d_W, Qr > 0 ? Qr : Q, n, S, QR, c->h, c->c,
                                        c->d_w0, c->d_tab, c->d_cn, c->d_row, c->d_brow, c->d_C, c->d_b0, st));
    INIT_TRY((cudaError_t)launch_prefix(c->d_b0, n, S, c->h, (double *)dev(at_Ld), tenor_delta, c->d_row, c->d_brow, st));
    // The host image goes out of scope: wait for the copy.
    INIT_TRY(cudaStreamSynchronize(st));
#undef INIT_TRY
    *out = c;
    if (domain_warn)
        return fail(c, LLL_EDOMAIN,
                    "sum |lambda| >= alpha - |beta|: the compensator uses the measure truncated to the rule");
    return LLL_OK;
}

int lll_set_product(lll_ctx *ctx, int product)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (product != LLL_PRODUCT_CAPLET && product != LLL_PRODUCT_SWAPTION)
        return fail(ctx, LLL_EINVAL, "unknown product");
    ctx->product = product;
    return LLL_OK;
}

int lll_set_strikes(lll_ctx *ctx, int n_strikes, const double *strikes)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (n_strikes < 1 || n_strikes > 64 || !strikes) return fail(ctx, LLL_EINVAL, "need 1..64 strikes");
    const size_t cnt = (size_t)ctx->n * n_strikes;
    std::vector<float> f(cnt);
    bool wide = false;
    for (size_t e = 0; e < cnt; ++e) {
        if (!isfin(strikes[e])) return fail(ctx, LLL_EINVAL, "strike is NaN/Inf");
        f[e] = (float)strikes[e];
        wide = wide || !(std::fabs(strikes[e]) < kPairStrike);
    }
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->d_strikes, f.data(), sizeof(float) * cnt, cudaMemcpyHostToDevice,
                                  ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    ctx->ns = n_strikes;
    ctx->wide_strikes = wide;
    ctx->simulated = false;
    return LLL_OK;
}

int lll_set_snapshots(lll_ctx *ctx, uint64_t count, uint64_t stride)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (stride < 1) return fail(ctx, LLL_EINVAL, "stride must be >= 1");
    ctx->snap_stride = stride;
    cudaFree(ctx->d_snap);
    ctx->d_snap = nullptr;
    ctx->n_snap = 0;
    if (count == 0) return LLL_OK;
    const size_t cells = (size_t)ctx->n * ctx->n * count;
    if (count > (1ull << 24)) return fail(ctx, LLL_EINVAL, "snapshot count too large");
    if (dalloc(&ctx->d_snap, cells) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "snapshot buffer");
    ctx->n_snap = count;
    return LLL_OK;
}

int lll_set_launch(lll_ctx *ctx, int threads_per_block, int blocks_per_sm, int chunk_rows,
                   int paths_per_thread, int lanes_per_path)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (threads_per_block != 0 &&
        (threads_per_block < 32 || threads_per_block > kMaxThreads || threads_per_block % 32))
        return fail(ctx, LLL_EINVAL, "threads_per_block must be a multiple of 32 in [32, 256]");
    if (blocks_per_sm < 0 || chunk_rows < 0) return fail(ctx, LLL_EINVAL, "negative launch value");
    if (paths_per_thread < 0 || paths_per_thread > 2)
        return fail(ctx, LLL_EINVAL, "paths_per_thread must be 0 (automatic), 1 or 2");
    if (lanes_per_path != 0 && lanes_per_path != 1 && lanes_per_path != 2 && lanes_per_path != 4)
        return fail(ctx, LLL_EINVAL, "lanes_per_path must be 0 (default), 1, 2 or 4");
    ctx->ppt = paths_per_thread;
    ctx->lpp = lanes_per_path;
    ctx->threads = threads_per_block;
    ctx->blocks_per_sm = blocks_per_sm;
    ctx->chunk_rows = std::min(chunk_rows, ctx->n);
    return LLL_OK;
}

int lll_set_mapping(lll_ctx *ctx, int mapping, int lanes)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (mapping == LLL_MAP_PATH) {
        ctx->tenor_lanes = 0;
        ctx->step_map = false;
        return LLL_OK;
    }
    if (mapping == LLL_MAP_STEP) {
        ctx->tenor_lanes = 0;
        ctx->step_map = true;
        return LLL_OK;
    }
    if (mapping != LLL_MAP_TENOR) return fail(ctx, LLL_EINVAL, "unknown mapping");
    if (lanes != 4 && lanes != 8 && lanes != 16 && lanes != 32)
        return fail(ctx, LLL_EINVAL, "lanes must be 4, 8, 16 or 32");
    ctx->tenor_lanes = lanes;
    ctx->step_map = false;
    return LLL_OK;
}

}  // extern "C"

namespace {

// Whether the step mapping of a default launch runs the path mapping's kernels
// instead (the same log-rates bit for bit): where they are the faster by the three
// kernels' estimates.  The step kernels' time is nearly the same from 32 to 1000
// paths and then grows by the unit; the pipeline's is its ticks, the block kernel's a
// path's latency, until the paths fill the GPU.  N = 40 (8 nodes), us: 32 paths 121
// in the pipeline, 102 in the step kernels; 4096 paths 127 and 232; 64,000 paths 977
// (block) and 2543.  N = 120: 20 nodes 1000 paths 741 and 372, 4096 paths 744 and
// 902; 8 nodes and 8 steps a period, where the pipeline does not fit shared memory,
// 2000 paths 4062 (block) and 775.  Over 20 curves (1 to 299 rates, 1 to 500 steps a
// period, 4 to 32 nodes) and 32 to 130,000 paths the estimates cost 0.4 % against the
// better choice, 29 % at worst.
bool step_as_path(const lll_ctx *ctx, uint64_t paths)
{
    if (ctx->QR >= ctx->QP || ctx->lpp > 1 || ctx->ppt > 0 || ctx->threads > 0 || ctx->blocks_per_sm > 0 ||
        ctx->chunk_rows > 0)
        return false;
    const uint64_t tiles = (paths + 31) / 32;
    size_t smem = 0;
    const int shape = ctx->product == LLL_PRODUCT_CAPLET
                          ? pipe_shape(LLL_PICARD, ctx->QR, ctx->n, ctx->s, ctx->S, tiles, ctx->sm_count, &smem)
                          : 0;
    const double path_us = shape ? pipe_estimate_us(ctx->QR, shape, smem, ctx->n, ctx->s, tiles, ctx->sm_count)
                                 : block_estimate_us(ctx->QR, ctx->n, ctx->s, paths);
    return path_us <= step_estimate_us(ctx->n, ctx->s, paths);
}

// The Picard scheme with its Euler steps in parallel (lll_paths_step.cu):
// chunks of paths through the five kernels, then the fixed-order block sum.
int simulate_step(lll_ctx *ctx, uint64_t first_path, uint64_t paths, uint64_t seed)
{
    LaunchPlan plan;
    int rc = plan_launch(ctx, LLL_PICARD, first_path, paths, seed, &plan, false);
    if (rc != LLL_OK) return rc;
    if (plan.qp == 0 || !step_kernels_supported(plan.qp, plan.block, ctx->ns))
        return fail(ctx, LLL_EUNSUPPORTED, "the step-parallel mapping needs a node table and at most 64 strikes");
    const int n = ctx->n, S = ctx->S;
    // intermediate arrays of about 4 (S + 2 S n + n^2) bytes per path: chunks within 2 GiB
    const size_t per_path = step_bytes_per_path(n, S);
    uint64_t Pc = std::max<uint64_t>(128, ((size_t(1) << 31) / per_path) / 128 * 128);
    Pc = std::min<uint64_t>(Pc, paths);
    const size_t floats = per_path / 4 * Pc;
    if (floats > ctx->state_cap) {
        dev_free(ctx, ctx->d_state);
        ctx->d_state = nullptr;
        ctx->state_cap = 0;
        if (dalloc(&ctx->d_state, floats) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "step-parallel scratch");
        ctx->state_cap = floats;
    }
    int blocks = 0;
    for (uint64_t c0 = 0; c0 < paths; c0 += Pc) blocks += step_blocks_per_chunk((int)std::min<uint64_t>(Pc, paths - c0));
    const size_t nout = (size_t)plan.n_out;
    if ((size_t)blocks * nout > ctx->partials_cap) {
        dev_free(ctx, ctx->d_partials);
        ctx->d_partials = nullptr;
        ctx->partials_cap = 0;
        if (dalloc(&ctx->d_partials, (size_t)blocks * nout) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "partials");
        ctx->partials_cap = (size_t)blocks * nout;
    }
    if (nout > ctx->sums_cap) {
        dev_free(ctx, ctx->d_sums);
        ctx->d_sums = nullptr;
        ctx->sums_cap = 0;
        if (dalloc(&ctx->d_sums, nout) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "sums");
        ctx->sums_cap = nout;
    }
    PathArgs a = plan.args;
    a.snap = ctx->d_snap; a.snap_stride = ctx->snap_stride; a.snap_pitch = ctx->n_snap;
    a.n_snap = ctx->d_snap ? std::min<uint64_t>(ctx->n_snap, (paths + ctx->snap_stride - 1) / ctx->snap_stride) : 0;
    float *dH = ctx->d_state, *Y = dH + (size_t)S * Pc, *Bh = Y + (size_t)S * n * Pc, *Zm = Bh + (size_t)S * n * Pc;
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[0], ctx->stream));
    int block0 = 0;
    for (uint64_t c0 = 0; c0 < paths; c0 += Pc) {
        const int pc = (int)std::min<uint64_t>(Pc, paths - c0);
        const cudaError_t e = (cudaError_t)launch_step_chunk(plan.qp, plan.block, a, c0, pc, dH, Y, Bh, Zm, block0,
                                                             ctx->d_partials, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "step-parallel kernels");
        block0 += step_blocks_per_chunk(pc);
    }
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[1], ctx->stream));
    const cudaError_t e = (cudaError_t)launch_finalize(ctx->d_partials, blocks, (int)nout, ctx->d_sums, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "finalize launch");
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[2], ctx->stream));
    ctx->simulated = true;
    ctx->err_pending = false;
    ctx->gemm_err_pending = false;
    ctx->last_paths = paths;
    ctx->last_snap_paths = a.n_snap;
    return LLL_OK;
}

}  // namespace

extern "C" {

int lll_simulate(lll_ctx *ctx, int scheme, uint64_t first_path, uint64_t paths, uint64_t seed)
{
    if (ctx && scheme == LLL_MLP) {
        if (ctx->ns == 0) return fail(ctx, LLL_ESTATE, "lll_set_strikes must come before lll_simulate");
        return simulate_mlp(ctx, first_path, paths, seed);
    }
    if (ctx && (scheme == LLL_EXPAND1 || scheme == LLL_EXPAND2)) {
        if (ctx->ns == 0) return fail(ctx, LLL_ESTATE, "lll_set_strikes must come before lll_simulate");
        if (paths == 0) return fail(ctx, LLL_EINVAL, "paths must be > 0");
        return simulate_expand(ctx, scheme == LLL_EXPAND1 ? 1 : 2, first_path, paths, seed);
    }
    if (ctx && ctx->step_map && (scheme == LLL_PICARD || scheme == LLL_FULL)) {
        if (scheme == LLL_FULL)
            return fail(ctx, LLL_EUNSUPPORTED,
                        "the step-parallel mapping is Picard's: the full scheme's drift reads the simulated rates");
        if (ctx->ns == 0) return fail(ctx, LLL_ESTATE, "lll_set_strikes must come before lll_simulate");
        if (paths == 0) return fail(ctx, LLL_EINVAL, "paths must be > 0");
        if (!step_as_path(ctx, paths)) return simulate_step(ctx, first_path, paths, seed);
    }
    LaunchPlan plan;
    int rc = plan_launch(ctx, scheme, first_path, paths, seed, &plan);
    if (rc != LLL_OK) return rc;
    const int grid = plan.grid;
    size_t state_need = plan.state_floats_per_block * grid, part_need = plan.partial_doubles_per_block * grid;
    smaller_calls(ctx, plan, &state_need, &part_need);
    if (state_need > ctx->state_cap) {
        dev_free(ctx, ctx->d_state);
        ctx->d_state = nullptr;
        ctx->state_cap = 0;
        if (dalloc(&ctx->d_state, state_need) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "state scratch");
        ctx->state_cap = state_need;
    }
    const size_t nout = (size_t)plan.n_out;
    if (part_need > ctx->partials_cap) {
        dev_free(ctx, ctx->d_partials);
        ctx->d_partials = nullptr;
        ctx->partials_cap = 0;
        if (dalloc(&ctx->d_partials, part_need) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "partials");
        ctx->partials_cap = part_need;
    }
    if (nout > ctx->sums_cap) {
        dev_free(ctx, ctx->d_sums);
        ctx->d_sums = nullptr;
        ctx->sums_cap = 0;
        if (dalloc(&ctx->d_sums, nout) != cudaSuccess) return fail(ctx, LLL_ENOMEM, "sums");
        ctx->sums_cap = nout;
    }
    PathArgs a = plan.args;
    a.partials = ctx->d_partials;
    a.state = ctx->d_state;
    a.snap = ctx->d_snap; a.snap_stride = ctx->snap_stride; a.snap_pitch = ctx->n_snap;
    a.n_snap = ctx->d_snap ? std::min<uint64_t>(ctx->n_snap, (paths + ctx->snap_stride - 1) / ctx->snap_stride) : 0;
    const int QPk = plan.qp, T = plan.threads;
    const size_t smem = plan.smem;
    cudaError_t e;
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[0], ctx->stream));
    e = (cudaError_t)launch_plan(plan, a);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "path kernel launch");
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[1], ctx->stream));
    e = (cudaError_t)launch_finalize(ctx->d_partials, grid, (int)nout, ctx->d_sums, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "finalize launch");
    CUDA_TRY(ctx, cudaEventRecord(ctx->ev[2], ctx->stream));
    ctx->simulated = true;
    ctx->err_pending = false;
    ctx->gemm_err_pending = false;
    ctx->last_paths = paths;
    ctx->last_snap_paths = a.n_snap;
    return LLL_OK;
}

int lll_get_sums(lll_ctx *ctx, double *sum, double *sumsq, uint64_t *count)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (!ctx->simulated) return fail(ctx, LLL_ESTATE, "no simulation to read");
    if (!sum || !sumsq) return fail(ctx, LLL_EINVAL, "null output");
    const size_t cnt = (size_t)ctx->n * ctx->ns;
    std::vector<double> buf(2 * cnt);
    CUDA_TRY(ctx, cudaMemcpyAsync(buf.data(), ctx->d_sums, sizeof(double) * 2 * cnt,
                                  cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    if (ctx->gemm_err_pending) {
        int word = 0;
        const cudaError_t e = (cudaError_t)mlp_gemm_take_error(&word, ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "GEMM error word");
        ctx->gemm_err_pending = false;
        if (word != 0) {
            ctx->simulated = false;
            return fail(ctx, LLL_ETIMEOUT, "a bounded wait of the tensor-core GEMM gave up; results discarded");
        }
    }
    if (ctx->err_pending && ctx->d_err) {
        int word = 0;
        CUDA_TRY(ctx, cudaMemcpy(&word, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost));
        if (word != 0) {
            ctx->simulated = false;
            return fail(ctx, LLL_ETIMEOUT, "a bounded wait of the tensor-core MLP kernel gave up; results discarded");
        }
    }
    for (size_t e = 0; e < cnt; ++e) {
        sum[e] = buf[2 * e];
        sumsq[e] = buf[2 * e + 1];
    }
    if (count) *count = ctx->last_paths;
    return LLL_OK;
}

int lll_price_caplets(lll_ctx *ctx, double *prices, double *stderr_)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (!prices) return fail(ctx, LLL_EINVAL, "prices is NULL");
    const size_t cnt = (size_t)ctx->n * ctx->ns;
    std::vector<double> s1(cnt), s2(cnt);
    uint64_t P = 0;
    int rc = lll_get_sums(ctx, s1.data(), s2.data(), &P);
    if (rc != LLL_OK) return rc;
    const double Pd = (double)P;
    for (size_t e = 0; e < cnt; ++e) {
        const double mean = s1[e] / Pd;
        prices[e] = mean;
        if (stderr_) {
            const double var = std::max(s2[e] / Pd - mean * mean, 0.0) * Pd / std::max(Pd - 1.0, 1.0);
            stderr_[e] = std::sqrt(var / Pd);
        }
    }
    return LLL_OK;
}

int lll_get_paths(lll_ctx *ctx, uint64_t first, uint64_t count, float *out)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (!ctx->simulated || !ctx->d_snap) return fail(ctx, LLL_ESTATE, "no snapshots recorded");
    if (!out) return fail(ctx, LLL_EINVAL, "out is NULL");
    if (first + count > ctx->last_snap_paths) return fail(ctx, LLL_EINVAL, "range beyond recorded snapshots");
    const int n = ctx->n;
    const uint64_t ns = ctx->n_snap; // row pitch of the device buffer
    std::vector<float> buf((size_t)n * n * ns);
    CUDA_TRY(ctx, cudaMemcpyAsync(buf.data(), ctx->d_snap, sizeof(float) * buf.size(),
                                  cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    for (uint64_t p = 0; p < count; ++p)
        for (int m = 1; m <= n; ++m)
            for (int l = 1; l <= n; ++l)
                out[((size_t)p * n + (m - 1)) * n + (l - 1)] =
                    (l >= m) ? buf[((size_t)(m - 1) * n + (l - 1)) * ns + first + p] : NAN;
    return LLL_OK;
}

int lll_kernel_ms(lll_ctx *ctx, float *path_kernel_ms, float *simulate_ms)
{
    if (!ctx) return fail(nullptr, LLL_EINVAL, "ctx is NULL");
    if (!ctx->simulated) return fail(ctx, LLL_ESTATE, "no simulation timed");
    CUDA_TRY(ctx, cudaEventSynchronize(ctx->ev[2]));
    float a = 0, b = 0;
    CUDA_TRY(ctx, cudaEventElapsedTime(&a, ctx->ev[0], ctx->ev[1]));
    CUDA_TRY(ctx, cudaEventElapsedTime(&b, ctx->ev[0], ctx->ev[2]));
    if (path_kernel_ms) *path_kernel_ms = a;
    if (simulate_ms) *simulate_ms = b;
    return LLL_OK;
}

void lll_destroy(lll_ctx *ctx)
{
    if (!ctx) return;
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    else cudaDeviceSynchronize();
    free_all(ctx);
    delete ctx;
}

}  // extern "C"

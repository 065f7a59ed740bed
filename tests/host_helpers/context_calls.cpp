// Test helper: the host code of the C ABI's contexts (lll_capi.cpp) on a fake
// CUDA runtime and fake kernel launchers that record what they are asked, on the
// CPU.  Built and run by tests/test_context_calls.py only; the first argument
// names the check.  Exit code 0: as expected; otherwise a message on stderr.
#include "../../paper_1006_3340_gb300/csrc/lll_capi.cpp"
#include "../../paper_1006_3340_gb300/csrc/lll_batch.cpp"
#include "../../paper_1006_3340_gb300/csrc/lll_quadrature.cpp"

#include <cstdlib>

namespace {
struct Tables {
    const void *tab, *Ctab;
    int QP;
};
std::vector<Tables> g_tables;              // launches of the table kernel
struct Need {
    int QP, n, ns, threads, rows;
};
std::vector<Need> g_need;                  // shared memory that was asked for
const void *g_path_tab = nullptr;          // table of the last path kernel
long g_mallocs = 0, g_frees = 0, g_launches = 0, g_copies = 0;
bool g_capturing = false;
uint64_t g_pipe_tiles = 0, g_pipe_hole = 0; // blocks an SM up to which the pipeline is chosen, and but one

int check(bool ok, const char *what)
{
    if (!ok) std::fprintf(stderr, "%s\n", what);
    return ok ? 0 : 1;
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t bytes)
{
    ++g_mallocs;
    *p = std::calloc(bytes, 1);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p)
{
    g_frees += p != nullptr;
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t bytes, cudaMemcpyKind, cudaStream_t)
{
    ++g_copies;
    std::memcpy(dst, src, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t bytes, cudaMemcpyKind k) { return cudaMemcpyAsync(dst, src, bytes, k, nullptr); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t bytes) { return *p = std::calloc(bytes, 1), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t bytes, cudaStream_t) { return std::memset(p, v, bytes), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
}

namespace lll {
void mlp_free(MlpState *) {}
bool path_kernel_supported(int, int, int) { return true; }
size_t path_kernel_smem(int QP, int n, int ns, int threads, int rows)
{
    g_need.push_back({QP, n, ns, threads, rows});
    return 1024;
}
int path_kernel_prepare(int, int, int, uint64_t, int, size_t) { return 0; }
int path_kernel_occupancy(int, int, int, uint64_t, int, size_t, int *b) { return *b = 4, 0; }
int launch_path_kernel(int, int, int, int, int, size_t, cudaStream_t, const PathArgs &a) { return ++g_launches, g_path_tab = a.tab, 0; }
int block_chunk_rates(int, int, int n, int) { return n; }
size_t block_kernel_smem(int, int, int, int, int) { return 1024; }
int block_kernel_prepare(int, int, int, int, uint64_t, size_t, int, int *b) { return *b = 4, 0; }
int launch_block_kernel(int, int, int, int, int, size_t, cudaStream_t, const PathArgs &a) { return ++g_launches, g_path_tab = a.tab, 0; }
int pipe_shape(int, int, int, int, int, uint64_t tiles, int sms, size_t *) 
{
    const uint64_t per_sm = (tiles + sms - 1) / sms;
    return per_sm <= g_pipe_tiles && per_sm != g_pipe_hole;
}
int launch_pipe_kernel(int, int, int, size_t, uint64_t, cudaStream_t, const PathArgs &) { return ++g_launches, 0; }
bool group_kernel_supported(int, int, int) { return true; }
size_t group_kernel_smem(int, int, int, int, int) { return 1024; }
int group_kernel_prepare(int, int, int, size_t, int, int *b) { return *b = 4, 0; }
int launch_group_kernel(int, int, int, int, int, size_t, cudaStream_t, const PathArgs &a) { return ++g_launches, g_path_tab = a.tab, 0; }
bool tenor_kernel_supported(int, int, int) { return true; }
size_t tenor_kernel_smem(int, int, int, int) { return 1024; }
int tenor_kernel_threads() { return 128; }
int tenor_kernel_prepare(int, int, int, size_t, int *b) { return *b = 4, 0; }
int launch_tenor_kernel(int, int, int, int, size_t, cudaStream_t, const PathArgs &a) { return ++g_launches, g_path_tab = a.tab, 0; }
int launch_tables(const double *, const double *, const double *, int, int, int, int QP, double, double, const double *,
                  float4 *tab, float *, float4 *, float4 *, float *Ctab, double *, cudaStream_t)
{
    ++g_launches;
    g_tables.push_back({tab, Ctab, QP});
    return 0;
}
int launch_prefix(const double *, int, int, double, const double *, double, float4 *, float4 *, cudaStream_t) { return ++g_launches, 0; }
int batch_block_prepare(int, int, int, size_t, int, int *b) { return *b = 4, 0; }
int batch_kernel_prepare(int, int, int, size_t, int, int *b) { return *b = 4, 0; }
int launch_batch_block_kernel(int, int, int, int, int, size_t, cudaStream_t, const BatchArgs &) { return ++g_launches, 0; }
int launch_batch_kernel(int, int, int, int, int, size_t, cudaStream_t, const BatchArgs &) { return ++g_launches, 0; }
int batch_finalize(const double *, const size_t *, const int *, const int *, const size_t *, int, const int *, double *, cudaStream_t) { return ++g_launches, 0; }
int launch_finalize(const double *, int, int, double *, cudaStream_t) { return ++g_launches, 0; }
}  // namespace lll

namespace {
// A 9-rate model whose 32-node rule has a shorter equivalent.
lll_ctx *model()
{
    const int N = 10, s = 2, n = N - 1, S = n * s, Q = 32;
    std::vector<double> L0(N, 0.03), lam((size_t)S * n, 0.05), x(Q), W(Q), K(n * 3, 0.03);
    const lll_nig nig{12.0, -3.0, 0.8, NAN};
    lll_ctx *c = nullptr;
    if (lll_build_nig_quadrature(nig, 1.5, Q, x.data(), W.data()) != LLL_OK ||
        lll_init(&c, N, 0.5, L0.data(), s, lam.data(), LLL_DRIVER_NIG, nig, Q, x.data(), W.data(), (void *)&g_launches) != LLL_OK ||
        lll_set_strikes(c, 3, K.data()) != LLL_OK || c->QR >= c->QP)
        std::abort();
    return c;
}

// The compensators that LLL_MLP reads are written by lll_init alone.
int compensators()
{
    lll_ctx *c = model();
    int bad = check(g_tables.size() == 1 && g_tables[0].Ctab == c->d_C, "lll_init writes C once");
    for (int lanes : {8, 0}) {
        if (lanes) lll_set_mapping(c, LLL_MAP_TENOR, lanes);
        else lll_set_launch(c, 0, 0, 0, 0, 2);
        bad += check(lll_simulate(c, LLL_PICARD, 0, 1000, 1) == LLL_OK, "simulate");
        lll_set_mapping(c, LLL_MAP_PATH, 0);
    }
    bad += check(g_tables.size() > 1, "the rule as given has tables of its own");
    for (size_t q = 1; q < g_tables.size(); ++q) bad += check(g_tables[q].Ctab != c->d_C, "C written by a selection");
    lll_destroy(c);
    return bad;
}
// Selecting lane groups or a mapping makes no CUDA call; the first simulation
// under the selection builds the tables that it needs without allocating, and
// once.  Built in a capture they belong to the graph: the next call builds them.
int selections()
{
    int bad = 0;
    for (int capture = 0; capture < 2; ++capture)
        for (int lanes : {8, 0}) {
            lll_ctx *c = model();
            bad += check(lll_simulate(c, LLL_PICARD, 0, 100000, 1) == LLL_OK, "scratch of a larger call");
            const void *sweeps = g_path_tab;
            const long mallocs = g_mallocs, launches = g_launches, copies = g_copies;
            g_tables.clear();
            g_capturing = capture;
            const int rc = lanes ? lll_set_mapping(c, LLL_MAP_TENOR, lanes) : lll_set_launch(c, 0, 0, 0, 0, 2);
            bad += check(rc == LLL_OK && g_mallocs == mallocs && g_launches == launches && g_copies == copies, "a selection called CUDA");
            for (int call = 0; call < 2; ++call) {
                bad += check(lll_simulate(c, LLL_PICARD, 0, 1000, 1) == LLL_OK, "simulate");
                bad += check(g_mallocs == mallocs, "a simulation under a selection allocated");
                bad += check(!g_tables.empty() && g_path_tab == g_tables[0].tab && g_path_tab != sweeps, "not the given rule's table");
                bad += check((int)g_tables.size() == (capture ? call + 1 : 1), "table launches");
            }
            g_capturing = false;
            bad += check(lll_simulate(c, LLL_PICARD, 0, 1000, 1) == LLL_OK && g_path_tab == g_tables[0].tab, "simulate");
            bad += check((int)g_tables.size() == (capture ? 3 : 1), "tables of a capture taken as built");
            lll_set_mapping(c, LLL_MAP_PATH, 0);
            lll_set_launch(c, 0, 0, 0, 0, 0);
            bad += check(lll_simulate(c, LLL_PICARD, 0, 1000, 1) == LLL_OK && g_path_tab == sweeps, "set back");
            lll_destroy(c);
        }
    return bad;
}
// A call with fewer paths than an earlier one allocates and frees nothing,
// whichever kernel it takes (its launches may be captured, and an earlier capture
// may hold the buffers).
int fewer_paths()
{
    int bad = 0;
    for (g_pipe_tiles = 1; g_pipe_tiles <= 8; ++g_pipe_tiles)
        for (g_pipe_hole = 0; g_pipe_hole < 3; ++g_pipe_hole)
        for (uint64_t most : {300000ull, 30000ull, 5000ull}) {
            lll_ctx *c = model();
            bad += check(lll_simulate(c, LLL_PICARD, 0, most, 1) == LLL_OK, "simulate");
            const long mallocs = g_mallocs, frees = g_frees;
            for (uint64_t paths = most; paths > 0; paths = paths * 9 / 10)
                for (int scheme : {LLL_PICARD, LLL_FULL}) bad += check(lll_simulate(c, scheme, 0, paths, 1) == LLL_OK, "simulate");
            if (g_mallocs != mallocs || g_frees != frees) std::fprintf(stderr, "pipeline to %d, but %d, from %llu paths: ", (int)g_pipe_tiles, (int)g_pipe_hole, (unsigned long long)most);
            bad += check(g_mallocs == mallocs && g_frees == frees, "a call with fewer paths changed its buffers");
            lll_destroy(c);
        }
    g_pipe_tiles = 0;
    return bad;
}
// The shared memory by which a call is refused is that of the rule as given and of
// 128 threads where none are set: 24 KB of staged rows of that rule, and as many rows
// under the frozen drift.
int limits()
{
    int bad = 0;
    lll_ctx *c = model();
    const int rows = 24 * 1024 / (2 * (32 / 4) * 16); // of 32 nodes
    for (int scheme : {LLL_FULL, LLL_PICARD, LLL_FROZEN}) {
        g_need.clear();
        bad += check(lll_simulate(c, scheme, 0, 5000, 1) == LLL_OK, "simulate");
        for (const Need &q : g_need) bad += check(q.threads == 128 && q.rows == std::min(rows, 9), "context");
    }
    lll_destroy(c);
    for (int N : {60, 400}) { // more rates than rows
        const int n = N - 1, Q = 128;
        std::vector<double> L0(N, 0.03), lam((size_t)n * n, 0.001), x(Q), W(Q), K(n, 0.03);
        const lll_nig nig{12.0, -3.0, 0.8, NAN};
        lll_build_nig_quadrature(nig, 1.5, Q, x.data(), W.data());
        bad += check(lll_init(&c, N, 0.25, L0.data(), 1, lam.data(), LLL_DRIVER_NIG, nig, Q, x.data(), W.data(), nullptr) == LLL_OK &&
                     lll_set_strikes(c, 1, K.data()) == LLL_OK, "init");
        for (int scheme : {LLL_FULL, LLL_FROZEN}) {
            g_need.clear();
            bad += check(lll_simulate(c, scheme, 0, 5000, 1) == LLL_OK, "simulate");
            for (const Need &q : g_need) bad += check(q.rows == 24 * 1024 / (2 * 32 * 16), "rows of a longer curve");
        }
        lll_destroy(c);
    }
    return bad;
}
// The same of a batch, with 48 KB of staged rows.
int batch_limits()
{
    int bad = 0;
    for (int N : {60, 400}) {
        const int n = N - 1, Q = 128;
        std::vector<double> L0(N, 0.03), lam((size_t)n * n, 0.001), x(Q), W(Q), K(n, 0.03);
        const lll_nig nig{12.0, -3.0, 0.8, NAN};
        lll_build_nig_quadrature(nig, 1.5, Q, x.data(), W.data());
        const lll_instance inst{N, 0.25, L0.data(), 1, lam.data(), LLL_DRIVER_NIG, nig, Q, x.data(), W.data(), 1, K.data(), 5000};
        lll_batch *b = nullptr;
        g_need.clear();
        bad += check(lll_batch_init(&b, 1, &inst, nullptr) == LLL_OK && b->QK > 0 && lll_batch_simulate(b, LLL_FULL, 1) == LLL_OK, "batch");
        for (const Need &q : g_need) bad += check(q.threads == 128, "threads of a batch");
        bad += check(!g_need.empty() && g_need[0].rows == 48, "rows of a batch");
        lll_batch_destroy(b);
    }
    return bad;
}
}  // namespace

int main(int argc, char **argv)
{
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "compensators") return compensators();
    if (what == "selections") return selections();
    if (what == "fewer_paths") return fewer_paths();
    if (what == "limits") return limits();
    if (what == "batch_limits") return batch_limits();
    return 2;
}

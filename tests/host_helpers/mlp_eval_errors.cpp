// Test helper: lll_mlp_eval's host code on a fake CUDA runtime, on the CPU.
// Every CUDA call and kernel launcher that it makes can be told to fail; the
// fake keeps, per stream, whether work was enqueued since the stream was last
// waited for.  Built and run by tests/test_mlp_eval_errors.py only.
//   mlp_eval_errors events N : event creation N fails in the first call, nothing in the second
//   mlp_eval_errors calls    : call after call, the next fallible call fails, to the last
// Exit code 0: as expected; otherwise a message on stderr.
#include "../../paper_1006_3340_gb300/csrc/lll_mlp_host.cpp"

#include <cstdlib>
#include <set>

namespace {
long g_calls = 0, g_fail = -1;       // fallible calls so far; the one that fails
long g_events = 0, g_fail_event = -1; // event creations
long g_live_events = 0;
std::set<void *> g_pending;          // streams with work nobody has waited for
std::set<std::pair<void *, void *>> g_after; // (event, stream whose work it follows)

bool fails() { return ++g_calls == g_fail; }

int launched(cudaStream_t st)
{
    if (fails()) return (int)cudaErrorUnknown;
    g_pending.insert(st);
    return 0;
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t bytes)
{
    if (fails()) return cudaErrorMemoryAllocation;
    *p = std::malloc(bytes);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t st) { return (cudaError_t)launched(st); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t st) { return (cudaError_t)launched(st); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    if (fails()) return cudaErrorUnknown;
    *s = (cudaStream_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    g_pending.erase(s);
    std::free(s);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    if (++g_events == g_fail_event || fails()) return cudaErrorUnknown;
    ++g_live_events;
    *e = (cudaEvent_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e)
{
    --g_live_events;
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st)
{
    if (fails()) return cudaErrorUnknown;
    g_after.insert({e, st});
    return cudaSuccess;
}
// Waiting for a stream that waits for an event's stream waits for both.
std::set<std::pair<void *, void *>> g_joined;
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned)
{
    if (fails()) return cudaErrorUnknown;
    for (auto &a : g_after)
        if (a.first == (void *)e) g_joined.insert({st, a.second});
    g_pending.insert(st);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st)
{
    if (fails()) return cudaErrorUnknown;
    g_pending.erase(st);
    for (auto &j : g_joined)
        if (j.first == (void *)st) g_pending.erase(j.second);
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
}

namespace lll {
int record_error(lll_ctx *, int code, const char *) { return code; }
int mlp_gemm(int, int, int, const void *, int, const void *, int, int, int, int, int, float *, const float *,
             const float *, float *, void *, cudaStream_t st) { return launched(st); }
int mlp_splits_used(int, int splits) { return splits; }
int mlp_gemm_kind() { return LLL_GEMM_TC; }
int mlp_out_loss(const void *, int, const void *, const float *, const float *, int, float *, float *, double *,
                 cudaStream_t st) { return launched(st); }
int mlp_vec_loss(float *, const float *, const float *, const int *, int, int, int, int, float *, void *, double *,
                 double *, cudaStream_t st) { return launched(st); }
int mlp_out_backward(const float *, const void *, const float *, int, int, float *, void *, cudaStream_t st) { return launched(st); }
int mlp_colsum_chunks(int) { return 1; }
int mlp_out_weight_grad(const float *, const void *, int, int, float *, float *, float *, cudaStream_t st) { return launched(st); }
int mlp_column_sums(const float *, int, int, float *, float *, cudaStream_t st) { return launched(st); }
int mlp_transpose_weights(const void *, void *, const size_t *, const int *, const int *, int, cudaStream_t st) { return launched(st); }
int mlp_reduce_splits(const float *, int, size_t, float *, cudaStream_t st) { return launched(st); }
int mlp_to_bf16(const float *, size_t, void *, cudaStream_t st) { return launched(st); }
int mlp_pack_rows(const float *, int, int, int, void *, cudaStream_t st) { return launched(st); }
}  // namespace lll

namespace {
int rows = 64;
std::vector<float> x, y, out, grads;

lll_ctx *model(int head)
{
    lll_ctx *c = new lll_ctx();
    c->N = 10;
    c->n = 9;
    c->s = 2;
    c->S = 18;
    c->delta = 0.5;
    c->driver = LLL_DRIVER_NIG;
    c->lam.assign(c->S * c->n, 0.1);
    c->stream = (cudaStream_t)std::malloc(1);
    if (lll_mlp_init_head(c, 128, 3, head, 1) != LLL_OK) std::abort();
    x.assign((size_t)rows * c->mlp->in_dim, 0.0f);
    y.assign((size_t)rows * c->mlp->outputs, 0.0f);
    out = y;
    grads.assign(c->mlp->n_params, 0.0f);
    return c;
}

int eval(lll_ctx *c, bool want_loss)
{
    double loss = 0;
    return lll_mlp_eval(c, x.data(), y.data(), rows, out.data(), grads.data(), want_loss ? &loss : nullptr);
}

void drop(lll_ctx *c)
{
    mlp_free(c->mlp);
    std::free(c->stream);
    delete c;
}
}  // namespace

int main(int argc, char **argv)
{
    const std::string what = argc > 1 ? argv[1] : "";
    for (int head = 0; head < 2; ++head) {
        if (what == "events") {
            lll_ctx *c = model(head);
            g_events = 0;
            g_fail_event = std::atol(argv[2]);
            const int first = eval(c, true);
            g_fail_event = -1;
            const int second = eval(c, true);
            const bool all = c->mlp->ready.size() == 5;
            drop(c);
            if (first == LLL_OK || second != LLL_OK || !all || g_live_events != 0) {
                std::fprintf(stderr, "head %d: first %d second %d, all events %d, left %ld\n", head, first, second, all,
                             g_live_events);
                return 1;
            }
        } else {
            for (int want_loss = 0; want_loss < 2; ++want_loss)
                for (long k = 1;; ++k) { // the k-th call of a network's first evaluation fails
                    lll_ctx *c = model(head);
                    g_pending.clear();
                    g_after.clear();
                    g_joined.clear();
                    g_calls = 0;
                    g_fail = k;
                    const int rc = eval(c, want_loss);
                    const bool failed = g_calls >= k;
                    g_fail = -1;
                    const size_t left = g_pending.size();
                    drop(c);
                    if ((rc == LLL_OK) == failed || left != 0) {
                        std::fprintf(stderr, "head %d loss %d call %ld: returned %d with %zu streams not waited for\n", head,
                                     want_loss, k, rc, left);
                        return 1;
                    }
                    if (!failed) break;
                }
        }
    }
    return 0;
}

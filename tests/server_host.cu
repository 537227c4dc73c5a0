// The request server's host side (server.cu) on a CPU: the CUDA runtime calls it
// makes are replaced by the fakes below. A solve "runs" until the scenario lets it
// complete; pool allocations above a size that it sets fail.
// Usage: server_host SCENARIO; exits 0 when the scenario holds.
#include "../paper_2001_02765_gb300/csrc/server.cu"

#include <stdio.h>
#include <stdlib.h>

static std::mutex g_mu;
static std::vector<std::pair<cudaHostFn_t, void *>> g_pending;  // solves in flight, in the order of their launch
static std::vector<const void *> g_started;                     // sigma of every solve launched alone
static int g_groups = 0;
static std::unordered_map<void *, size_t> g_live;               // pool allocations
static bool g_at_once = false;                                  // solves complete within their launch
static size_t g_largest = SIZE_MAX;                             // the largest pool allocation that succeeds

#ifndef __CUDA_ARCH__
extern "C" {
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t)
{
    std::lock_guard<std::mutex> lock(g_mu);
    if (n > g_largest) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    g_live[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t)
{
    std::lock_guard<std::mutex> lock(g_mu);
    g_live.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t fn, void *arg)
{
    if (g_at_once) return fn(arg), cudaSuccess;
    std::lock_guard<std::mutex> lock(g_mu);
    g_pending.push_back({fn, arg});
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *, const cudaMemPoolProps *) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return *p = calloc(n, 1), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
}
#endif

// what server.cu takes from the rest of the library
void sg_set_last_cuda_error(cudaError_t, const char *) {}
void sg_set_last_error_message(const char *) {}
void sg_tune_shape(sg_precision, int, int *shape) { memset(shape, 0, SG_TUNE_KNOBS * sizeof(int)); }
int64_t sg_workspace_bytes(const sg_plan *plan) { return plan->ws_fwd_bytes; }
sg_status sg_force_ws(sg_plan *, const sg_workspace *, const void *sigma, const void *, const void *, void *, void *,
                      cudaStream_t, void *)
{
    std::lock_guard<std::mutex> lock(g_mu);
    g_started.push_back(sigma);
    return SG_OK;
}
namespace sgk {
template <typename T>
sg_status rows_fwd(int, int, const row_fwd_args<T> &, int, const cplx_t<T> *, cudaStream_t, const row_fwd_args<T> *,
                   batch_shape, int, const edge_args<T> *, const edge_args<T> *)
{
    ++g_groups;
    return SG_OK;
}
template <typename T>
sg_status edge_cols(int, const edge_args<T> &, const cplx_t<T> *, cudaStream_t, const edge_args<T> *, batch_shape)
{
    return SG_OK;
}
template <typename T>
sg_status cols(int, int, int, const col_args<T> &, int, int, const cplx_t<T> *, int *, cudaStream_t, const col_args<T> *,
               batch_shape)
{
    return SG_OK;
}
template <typename T>
sg_status cols_central(int, int, int, const col_args<T> &, int, const cplx_t<T> *, int *, cudaStream_t,
                       const col_args<T> *, batch_shape)
{
    return SG_OK;
}
template <typename T>
sg_status rows_inv(int, int, const row_inv_args<T> &, int, const cplx_t<T> *, cudaStream_t, const row_inv_args<T> *,
                   batch_shape)
{
    return SG_OK;
}
}  // namespace sgk

#define CHECK(x)                                                              \
    do {                                                                      \
        if (!(x)) {                                                           \
            fprintf(stderr, "%s:%d: %s does not hold\n", __FILE__, __LINE__, #x); \
            exit(1);                                                          \
        }                                                                     \
    } while (0)

template <typename F>
static bool soon(F f)
{
    for (int k = 0; k < 5000; ++k) {
        if (f()) return true;
        std::this_thread::sleep_for(std::chrono::milliseconds(1));
    }
    return false;
}
static size_t in_flight()
{
    std::lock_guard<std::mutex> lock(g_mu);
    return g_pending.size();
}
static void complete_first()
{
    std::pair<cudaHostFn_t, void *> p;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        CHECK(!g_pending.empty());
        p = g_pending.front();
        g_pending.erase(g_pending.begin());
    }
    p.first(p.second);
}

static sg_plan make_plan(int side, int64_t bytes)
{
    sg_plan p;
    memset(&p, 0, sizeof(p));
    p.prec = SG_FP32;
    p.npatches = 1;
    p.pp = new sg_patch_plan[1]();
    p.pp[0].d.nx = p.pp[0].d.ny = side;
    p.pp[0].d.px = p.pp[0].d.py = sg_pad_length(side);
    p.geom.slope_mode = SG_SLOPES_NONE;
    p.ws_fwd_bytes = bytes;
    return p;
}

// A group whose workspaces do not fit goes back to its members' places in the queue:
// a request of another kind between them is not passed, and memory that was never
// held is not reported as the peak.
static void failed_group_keeps_arrival_order()
{
    sg_plan a = make_plan(64, 1000), b = make_plan(200, 300);
    sg_server *s = nullptr;
    CHECK(sg_server_create(0, 1, &s) == SG_OK);
    char in[4], out;
    uint64_t t[4];
    auto submit = [&](int k, sg_plan *p) { CHECK(sg_submit(s, p, &in[k], nullptr, nullptr, &out, &out, &t[k]) == SG_OK); };
    submit(0, &b);  // holds the only slot while the others arrive
    CHECK(soon([] { return in_flight() == 1; }));
    g_largest = 1500;  // one of a's workspaces (1000 bytes and the error word, rounded up), not two
    submit(1, &a);
    submit(2, &b);
    submit(3, &a);
    for (int k = 0; k < 4; ++k) {
        CHECK(soon([] { return in_flight() == 1; }));
        complete_first();
        sg_status r;
        CHECK(sg_wait(s, t[k], 5000.0, &r, nullptr) == SG_OK && r == SG_OK);
    }
    CHECK(g_groups == 0 && g_started.size() == 4);
    for (int k = 0; k < 4; ++k) CHECK(g_started[k] == &in[k]);
    sg_server_stats st;
    CHECK(sg_server_get_stats(s, &st, 0) == SG_OK);
    CHECK(st.peak_bytes == 1000 && st.bytes_in_use == 0);
    CHECK(sg_server_destroy(s) == SG_OK);
}

// A solve that completes while the worker is still launching is noticed at once, not at
// the worker's next poll a millisecond later.
static void completions_during_a_launch_are_noticed()
{
    sg_plan a = make_plan(64, 1000);
    sg_server *s = nullptr;
    CHECK(sg_server_create(0, 1, &s) == SG_OK);
    CHECK(sg_server_set_group_limit(s, 1) == SG_OK);
    g_at_once = true;
    char in, out;
    const int n = 400;
    uint64_t t[n];
    const double t0 = now_s();
    for (int k = 0; k < n; ++k) CHECK(sg_submit(s, &a, &in, nullptr, nullptr, &out, &out, &t[k]) == SG_OK);
    for (int k = 0; k < n; ++k) {
        sg_status r;
        CHECK(sg_wait(s, t[k], 5000.0, &r, nullptr) == SG_OK && r == SG_OK);
    }
    const double ms = 1e3 * (now_s() - t0);
    printf("%d solves in %.1f ms\n", n, ms);
    CHECK(ms < 0.25 * n);  // a poll each: one millisecond per solve
    CHECK(sg_server_destroy(s) == SG_OK);
}

int main(int argc, char **argv)
{
    const char *s = argc > 1 ? argv[1] : "";
    if (!strcmp(s, "failed_group_keeps_arrival_order")) return failed_group_keeps_arrival_order(), 0;
    if (!strcmp(s, "completions_during_a_launch_are_noticed")) return completions_during_a_launch_are_noticed(), 0;
    fprintf(stderr, "unknown scenario '%s'\n", s);
    return 2;
}

// Host side of the FP32 cross-patch sum (cross32.cu) on a CPU: the CUDA runtime
// calls it makes are replaced by the fakes below, which record every launch.
// Usage: cross_host SCENARIO; exits 0 when the scenario holds.
#include "../paper_2001_02765_gb300/csrc/cross32.cu"

#include <stdio.h>
#include <stdlib.h>

#include <tuple>

struct launch {
    const void *kern;
    unsigned grid;
    void **args;
};
static std::vector<launch> g_launches;
static cudaError_t g_launch_error = cudaSuccess, g_sync_error = cudaSuccess;  // what the fakes report
static int64_t g_live = 0;   // device allocations not yet freed
static int64_t g_sums = -1;  // how many target sums the level-0 charge kernel was told to clear

// the last argument of a kernel, whatever its integer type
template <typename... A>
static int64_t last_arg(void (*)(A...), void **args)
{
    using last = std::tuple_element_t<sizeof...(A) - 1, std::tuple<A...>>;
    return (int64_t)*(const last *)args[sizeof...(A) - 1];
}

#ifndef __CUDA_ARCH__
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n)
{
    ++g_live;
    return (*p = calloc(n, 1)) ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p)
{
    if (p) --g_live;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *kern, void **args)
{
    g_launches.push_back({kern, c->gridDim.x, args});
    if (kern == (const void *)k_p2m) g_sums = last_arg(k_p2m, args);
    return c->gridDim.x >= 1 ? cudaSuccess : cudaErrorInvalidConfiguration;
}
// (a launch by <<<>>>)
cudaError_t __cudaLaunchKernel(cudaKernel_t kern, dim3 grid, dim3, void **args, size_t, cudaStream_t)
{
    g_launches.push_back({(const void *)kern, grid.x, args});
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return g_launch_error; }
cudaError_t cudaDeviceSynchronize() { return g_sync_error; }
}
#endif

// what cross32.cu takes from the rest of the library
void sg_set_last_cuda_error(cudaError_t, const char *) {}
void sg_set_last_error_message(const char *) {}
void sg_timing_begin(const sg_workspace *, int, cudaStream_t) {}
void sg_timing_end(const sg_workspace *, int, cudaStream_t) {}
sg_status sg_plan_upload(sg_plan *plan, void **dst, const void *src, size_t n)
{
    *dst = malloc(n ? n : 1);
    if (n) memcpy(*dst, src, n);
    plan->device_bytes += (int64_t)n;
    return SG_OK;
}

// A plan of the given patches (nx, ny, existing cells or none), all on one level.
struct shape {
    int nx, ny;
    bool any;
};
static sg_status make_plan(sg_plan *plan, sg_workspace *ws, const std::vector<shape> &patches, double z)
{
    memset(plan, 0, sizeof(*plan));
    memset(ws, 0, sizeof(*ws));
    plan->npatches = (int)patches.size();
    plan->pp = new sg_patch_plan[patches.size()]();
    plan->geom.z = z;
    plan->lattice_unit = 1.0;
    std::vector<std::vector<int>> code;
    std::vector<const int *> codes;
    int64_t leaves = 0;
    for (size_t p = 0; p < patches.size(); ++p) {
        plan->pp[p].d.nx = patches[p].nx;
        plan->pp[p].d.ny = patches[p].ny;
        plan->pp[p].d.step = 2;
        code.emplace_back((size_t)patches[p].nx * patches[p].ny, patches[p].any ? SG_CELL_LEAF : SG_CELL_ABSENT);
        if (patches[p].any) leaves += (int64_t)patches[p].nx * patches[p].ny;
    }
    for (const auto &c : code) codes.push_back(c.data());
    plan->ntargets = (int)leaves;
    plan->nblocks = 1;
    return sg_far_setup(plan, codes.data(), 1, &leaves, SG_NT_GMAX);
}

#define CHECK(x)                                                              \
    do {                                                                      \
        if (!(x)) {                                                           \
            fprintf(stderr, "%s:%d: %s does not hold\n", __FILE__, __LINE__, #x); \
            return 1;                                                         \
        }                                                                     \
    } while (0)

// every target's sums are cleared, also where their number exceeds 32 bits
static int clears_every_sum()
{
    for (double z : {0.0, 0.5}) {
        sg_plan plan;
        sg_workspace ws;
        CHECK(make_plan(&plan, &ws, {{8, 8, true}, {8, 8, true}}, z) == SG_OK);
        for (int64_t n : {(int64_t)128, (int64_t)1 << 30, ((int64_t)1 << 31) - 256}) {
            plan.ntargets = (int)n;
            CHECK(sg_far_solve(&plan, &ws, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0) == SG_OK);
            CHECK(g_sums == n * (z != 0.0 ? 3 : 2));
        }
    }
    return 0;
}

// a patch without an existing cell adds no launch (its levels hold no cluster)
static int empty_patch_adds_no_launch()
{
    for (const shape &empty : {shape{256, 256, false}, shape{4, 4, false}}) {
        size_t n[2];
        int nlev[2];
        for (int k = 0; k < 2; ++k) {
            sg_plan plan;
            sg_workspace ws;
            std::vector<shape> patches = {{16, 16, true}, {12, 16, true}};
            if (k == 1) patches.push_back(empty);
            CHECK(make_plan(&plan, &ws, patches, 0.0) == SG_OK);
            g_launches.clear();
            CHECK(sg_far_solve(&plan, &ws, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0) == SG_OK);
            for (const launch &l : g_launches) CHECK(l.grid >= 1);
            n[k] = g_launches.size();
            nlev[k] = plan.far->nlev;
        }
        CHECK(n[0] == n[1] && nlev[0] == nlev[1] && nlev[0] == 3);
    }
    return 0;
}

// tables of the potential that could not be built are not taken for built by the next call
static int unbuilt_tables_are_dropped()
{
    sg_plan plan;
    sg_workspace ws;
    CHECK(make_plan(&plan, &ws, {{16, 16, true}, {12, 16, true}}, 0.0) == SG_OK);
    const int64_t bytes = plan.device_bytes, live = g_live;
    for (int k = 0; k < 2; ++k) {
        (k == 0 ? g_launch_error : g_sync_error) = cudaErrorLaunchFailure;
        CHECK(sg_far_potential_tables(&plan) == SG_ECUDA);
        g_launch_error = g_sync_error = cudaSuccess;
        CHECK(!plan.far->ptab.data && plan.device_bytes == bytes && g_live == live);
    }
    g_launches.clear();
    CHECK(sg_far_potential_tables(&plan) == SG_OK);
    CHECK(g_launches.size() == 1 && plan.far->ptab.data && plan.device_bytes > bytes);
    CHECK(sg_far_potential_tables(&plan) == SG_OK && g_launches.size() == 1);
    return 0;
}

int main(int argc, char **argv)
{
    const char *s = argc > 1 ? argv[1] : "";
    if (!strcmp(s, "clears_every_sum")) return clears_every_sum();
    if (!strcmp(s, "empty_patch_adds_no_launch")) return empty_patch_adds_no_launch();
    if (!strcmp(s, "unbuilt_tables_are_dropped")) return unbuilt_tables_are_dropped();
    fprintf(stderr, "unknown scenario '%s'\n", s);
    return 2;
}

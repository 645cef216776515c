// A device in host memory for tests of the library's host code (csrc/api.cu) where no
// GPU is wanted: device allocations are counted against a total that the test
// sets, a chosen one fails, and the kernels whose results steer the host
// code write what the test says.  Every other kernel launch and CUDA call that
// api.cu makes is a stub that returns 0 (fake_device.py writes them).
#include "../../paper_1107_5719_gb300/csrc/internal.h"

#include <sys/mman.h>
#include <cstdlib>
#include <cstring>
#include <map>

namespace {
std::map<void*, size_t> g_mem;
long long g_total = 284LL << 30, g_live = 0, g_peak = 0, g_large = 1LL << 60, g_large_live = 0, g_large_peak = 0;
int g_sweeps = 5, g_solves = 0, g_graphs = 0, g_marches = 0, g_applies = 0, g_lengths = 0, g_ng = 0,
    g_outside = 0, g_replays = 0, g_chunks = 0, g_mallocs = 0, g_nth = -1;
unsigned long long g_steps = 1ull << 40;
cudaError_t g_last = cudaSuccess;
double g_delta = 0.5;
int g_entries = 64, g_rows = 64;        // of every plane of an operator
}  // namespace

extern "C" {

void fake_memory(long long total) { g_total = total; }
// the n-th allocation from here fails (-1: none; it is -1 again once it has)
void fake_fail(int n) { g_nth = n; }
int fake_failed(void) { return g_nth < 0; }
void fake_solves(int sweeps, double delta) { g_sweeps = sweeps; g_delta = delta; }
void fake_operator(int entries, int rows, unsigned long long steps)
{
    g_entries = entries;
    g_rows = rows;
    g_steps = steps;
}
// the peak of the allocations of at least `bytes` since the last call, which
// sets that size
long long fake_large(long long bytes)
{
    const long long p = g_large_peak;
    g_large = bytes;
    g_large_live = 0;
    for (auto& m : g_mem) g_large_live += (long long)m.second >= g_large ? m.second : 0;
    g_large_peak = g_large_live;
    return p;
}
long long fake_live(void) { return g_live; }
long long fake_peak(int reset)
{
    const long long p = g_peak;
    if (reset) g_peak = g_live;
    return p;
}
// {one-kernel solves, graph launches, marches, applied operators, length marches,
// extrapolations, barrier words outside their allocation, ray-by-ray replays,
// recording marches (one a chunk of planes), device allocations} since the last call
void fake_counts(int* n)
{
    const int c[10] = {g_solves, g_graphs, g_marches, g_applies, g_lengths,
                       g_ng, g_outside, g_replays, g_chunks, g_mallocs};
    std::memcpy(n, c, sizeof c);
    g_solves = g_graphs = g_marches = g_applies = g_lengths = g_ng = g_outside = g_replays = g_chunks = g_mallocs = 0;
}

cudaError_t cudaMalloc(void** p, size_t n)
{
    *p = nullptr;
    ++g_mallocs;
    const bool chosen = g_nth == 0;
    if (g_nth >= 0) --g_nth;
    if (chosen || g_live + (long long)n > g_total) return g_last = cudaErrorMemoryAllocation;
    void* m = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return g_last = cudaErrorMemoryAllocation;
    g_mem[m] = n;
    g_live += (long long)n;
    if (g_live > g_peak) g_peak = g_live;
    if ((long long)n >= g_large) g_large_live += (long long)n;
    if (g_large_live > g_large_peak) g_large_peak = g_large_live;
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (!p) return cudaSuccess;
    auto it = g_mem.find(p);
    if (it == g_mem.end()) return cudaErrorInvalidValue;
    munmap(p, it->second);
    g_live -= (long long)it->second;
    if ((long long)it->second >= g_large) g_large_live -= (long long)it->second;
    g_mem.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return *p = std::calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* fr, size_t* tot)
{
    *fr = (size_t)(g_total - g_live);
    *tot = (size_t)g_total;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int x, size_t n, cudaStream_t)
{
    if (!x && n >= 1 << 24 && (size_t)d % 4096 == 0) {      // without touching the pages
        madvise(d, n / 4096 * 4096, MADV_DONTNEED);
        d = (char*)d + n / 4096 * 4096;
        n %= 4096;
    }
    std::memset(d, x, n);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e)
{
    return e == cudaErrorMemoryAllocation ? "out of memory" : "error";
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return ++g_graphs, cudaSuccess; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                             size_t, cudaGraphNodeParams* p)
{
    static cudaGraph_t body[1];
    p->conditional.phGraph_out = body;
    return cudaSuccess;
}

}  // extern "C"

// Whether [p, p + n) lies in one allocation.
static bool inside(const void* p, long long n)
{
    auto it = g_mem.upper_bound(const_cast<void*>(p));
    if (it == g_mem.begin()) return false;
    --it;
    return n >= 0 && (char*)p + n <= (char*)it->first + it->second;
}

namespace rt3d {

long long os_coef_stride(const Geometry& g, bool split)
{
    return split ? 2LL * ((g.nx + 1) / 2) * g.ny * g.nz : g.N;
}
long long pair_records(const Geometry& g) { return (2LL * g.ny + 1) * 2 * g.nx * g.nz; }
int ng_partial_size() { return 4096; }
int sc_chunk(const Geometry&) { return 1; }
void os_solve_shape(long long, int, bool, OsShape* s)
{
    s->threads = 32;
    s->voxels = s->blocks = 1;
    s->coef = true;
}
cudaError_t launch_plane_order(const Geometry& g, double, const double*, double*, int* order, cudaStream_t)
{
    for (int k = 0; k < g.nz; ++k) order[k] = k;
    return cudaSuccess;
}
cudaError_t launch_op_counts(const Geometry& g, const OpLists&, bool, const int*, int*, int*, int*, int* E,
                             int* rows, cudaStream_t)
{
    for (int k = 0; k < g.nz; ++k) {
        E[k] = g_entries;
        rows[k] = g_rows;
    }
    return cudaSuccess;
}
cudaError_t launch_op_lengths(const Geometry&, const double*, const double*, const double*, const DirInfo*,
                              const int*, const float4*, double, int, bool, int, float2*, int*, int, int*,
                              unsigned long long* steps, cudaStream_t)
{
    *steps = g_steps;
    return ++g_lengths, cudaGetLastError();
}
cudaError_t launch_op_apply64(const Geometry&, const double*, const double*, const OpMap&, double*,
                              unsigned long long*, cudaStream_t)
{
    return ++g_applies, cudaGetLastError();
}
cudaError_t launch_op_apply_df(const Geometry&, const double*, const double*, const OpMap&, double, double*,
                               unsigned long long*, cudaStream_t)
{
    return ++g_applies, cudaGetLastError();
}
cudaError_t launch_fs64(const Geometry&, const double*, const double*, const double*, const double*,
                        const DirInfo*, const StepGeo*, const Bw4d*, const Bw4d*, const double*, double, int,
                        double*, unsigned long long*, cudaStream_t)
{
    return ++g_marches, cudaGetLastError();
}
cudaError_t launch_rec64(const Geometry&, int, int, const double*, const double*, const double*, const DirInfo*,
                         const StepGeo*, const Bw4d*, const Bw4d*, const RecOut&, const int*, int, int, double*,
                         double*, cudaStream_t)
{
    return ++g_chunks, cudaGetLastError();
}
cudaError_t launch_recdf(const ViewDF&, int, int, const RecOut&, const int*, int, int, double*, double*, double*,
                         cudaStream_t)
{
    return ++g_chunks, cudaGetLastError();
}
cudaError_t launch_fs64rep(const Geometry&, const double*, const DirInfo*, const StepGeo*, const Bw4d*, const FsRec&,
                           int, double*, unsigned long long*, cudaStream_t)
{
    return ++g_replays, cudaGetLastError();
}
cudaError_t launch_fsdfrep(const ViewDF&, const Rec32&, int, unsigned long long*, cudaStream_t)
{
    return ++g_replays, cudaGetLastError();
}
cudaError_t launch_fs32rep_batch(const Rep32*, const int*, const long long*, int n, long long, int, int,
                                 unsigned long long*, cudaStream_t)
{
    g_replays += n;
    return cudaGetLastError();
}
cudaError_t launch_fsdf(const ViewDF&, double, int, unsigned long long*, cudaStream_t)
{
    return ++g_marches, cudaGetLastError();
}
cudaError_t launch_os_solve(const OsTask& one, const OsTask* tasks, const int*, int ntask, const OsShape&, bool gs,
                            int, int max_sweeps, double, cudaStream_t)
{
    ++g_solves;
    for (int q = 0; q < (tasks ? ntask : 1); ++q) {
        const OsTask& t = tasks ? tasks[q] : one;
        g_outside += !inside(t.words, 8LL * max_sweeps * (gs ? 2 : 1)) ||
                     (t.nclear && !inside(t.clear, 8LL * t.nclear));
        *t.sweeps = g_sweeps;
        if (t.delta) *t.delta = g_delta;
    }
    return cudaSuccess;
}
cudaError_t launch_ng_apply(long long, const double*, const double*, const double*, double*, cudaStream_t)
{
    return ++g_ng, cudaSuccess;
}
cudaError_t launch_rel_change(long long, const double*, const double*, double* delta, double*, cudaStream_t)
{
    *delta = g_delta;
    return cudaSuccess;
}

}  // namespace rt3d

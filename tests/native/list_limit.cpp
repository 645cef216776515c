// Shared-memory limits of the node-list kernel where two threads launch it: the CUDA
// calls of op.cu are replaced, and between a thread's cudaFuncSetAttribute and its launch
// the other thread's whole call runs.  Prints "nodes other_nodes launches refused" for
// pairs of planes, refused: launches above the limit in force.
#include "../../paper_1107_5719_gb300/csrc/internal.h"

#include <algorithm>
#include <cstdio>
#include <map>

using namespace rt3d;

namespace {
std::map<const void*, int> g_limit;
int g_other = 0, g_launches = 0, g_refused = 0;
size_t g_shm = 0;

void launch(int ny)
{
    Geometry g{};
    g.nx = 100;
    g.ny = ny;
    g.nz = 2;
    g.ndir = 1;
    g.N = 200LL * ny;
    OpLists L{};
    launch_op_lists(g, nullptr, nullptr, nullptr, nullptr, L, nullptr, nullptr);
}
}  // namespace

extern "C" {
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v)
{
    g_limit[f] = v;
    if (const int other = g_other) {
        g_other = 0;
        launch(other);
    }
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t shm, void*) { return g_shm = shm, 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* shm, void*) { return *shm = g_shm, cudaSuccess; }
cudaError_t __cudaGetKernel(const void** k, const void* f) { return *k = f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t shm, cudaStream_t)
{
    ++g_launches;
    const auto it = g_limit.find(f);
    if (shm > (size_t)std::max(48 * 1024, it == g_limit.end() ? 0 : it->second)) ++g_refused;
    return cudaSuccess;
}
}

int main()
{
    for (int ny : {40, 102, 103, 104, 130, 245})
        for (int other : {40, 103, 124, 200}) {
            g_limit.clear();
            g_launches = g_refused = 0;
            g_other = other;
            launch(ny);
            std::printf("%d %d %d %d\n", 100 * ny, 100 * other, g_launches, g_refused);
        }
    return 0;
}

// PinnedDoubles (dp_pinned.h) against a fake of the CUDA runtime's page-locked
// memory: prints nothing and returns 0 when every expectation holds.
#include <cstdio>
#include <cstdlib>

#include "dp_pinned.h"

namespace {
bool g_full = false;       // no page-locked memory left
int g_live = 0;            // buffers handed out
cudaError_t g_last = cudaSuccess;
int fail(int line)
{
    printf("line %d\n", line);
    return 1;
}
}  // namespace

extern "C" cudaError_t cudaMallocHost(void** p, size_t bytes)
{
    if (g_full) return g_last = cudaErrorMemoryAllocation;
    *p = malloc(bytes);
    ++g_live;
    return cudaSuccess;
}
extern "C" cudaError_t cudaFreeHost(void* p)
{
    free(p);
    --g_live;
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}

#define EXPECT(x) \
    if (!(x)) return fail(__LINE__)

int main()
{
    dpk::PinnedDoubles b;
    g_full = true;
    EXPECT(b.reserve(10, 100) == nullptr && g_last == cudaSuccess);   // refused: no pointer, no error left behind
    g_full = false;
    double* p = b.reserve(10, 100);
    EXPECT(p && g_live == 1);
    for (int k = 0; k < 20; ++k) p[k] = k;                            // room for twice as many
    EXPECT(b.reserve(20, 100) == p);
    g_full = true;
    EXPECT(b.reserve(60, 100) == nullptr && g_last == cudaSuccess);   // refused again: the old buffer stays
    EXPECT(b.reserve(20, 100) == p && p[19] == 19.0);
    g_full = false;
    p = b.reserve(60, 100);
    EXPECT(p && g_live == 1);
    for (int k = 0; k < 100; ++k) p[k] = k;
    EXPECT(b.reserve(100, 100) == p);
    b.release();
    EXPECT(g_live == 0);
    return 0;
}

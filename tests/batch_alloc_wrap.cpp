// Linked before the library's objects with --wrap=cudaMalloc: a fake of the call that refuses
// requests of at least `limit` bytes while probe_limit_alloc(limit) is in force (0: none).
#include <stddef.h>

extern "C" int __real_cudaMalloc(void**, size_t);

static size_t g_limit = 0;
static int g_refused = 0;
extern "C" void probe_limit_alloc(long long limit) { g_limit = (size_t)limit; g_refused = 0; }
extern "C" int probe_refused(void) { return g_refused; }

extern "C" int __wrap_cudaMalloc(void** p, size_t bytes) {
    if (!g_limit || bytes < g_limit) return __real_cudaMalloc(p, bytes);
    ++g_refused;
    *p = nullptr;
    return 2;                                              // cudaErrorMemoryAllocation
}

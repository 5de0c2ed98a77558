// Linked before the library's objects with --wrap=cudaGraphInstantiate: a fake of the call that
// fails while probe_fail_instantiate(1) is in force and forwards to the real one otherwise.
typedef struct CUgraphExec_st* cudaGraphExec_t;
typedef struct CUgraph_st* cudaGraph_t;

extern "C" int __real_cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long);

static int g_fail = 0, g_calls = 0;
extern "C" void probe_fail_instantiate(int on) { g_fail = on; }
extern "C" int probe_instantiate_calls(void) { return g_calls; }

extern "C" int __wrap_cudaGraphInstantiate(cudaGraphExec_t* exec, cudaGraph_t graph, unsigned long long flags) {
    ++g_calls;
    return g_fail ? 2 : __real_cudaGraphInstantiate(exec, graph, flags);      // 2: cudaErrorMemoryAllocation
}

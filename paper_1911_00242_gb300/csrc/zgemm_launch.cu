// Instances of the SIMT complex GEMM, one per arithmetic and tile shape that a rule can take
// (zg_built; the callers ask for no other).
#include "zgemm_launch.h"

namespace ccsdk {

namespace {

template <typename T> constexpr int kArith = ZG_FP64;
template <> constexpr int kArith<float> = ZG_FP32;
template <> constexpr int kArith<df> = ZG_DF;

template <typename T>
void launch_one(int shape, const GemmArgs& g, dim3 grid, cudaStream_t st) {
    switch (shape) {
#define X(id, bm, bn, bk, tm, tn, ks) \
    case id:                                                                                  \
        if constexpr (zg_built(kArith<T>, id))                                                \
            zgemm_kb_kernel<bm, bn, bk, tm, tn, T, ks><<<grid, ZG_THREADS, 0, st>>>(g);       \
        break;
        ZG_SHAPES(X)
#undef X
    }
}

template <typename T>
void launch_group(int shape, const GemmArgs* args, const long long* prefix, int n, long long total, int ctas,
                  cudaStream_t st) {
    switch (shape) {
#define X(id, bm, bn, bk, tm, tn, ks)                                                                            \
    case id:                                                                                                     \
        if constexpr (zg_built(kArith<T>, id))                                                                   \
            zgemm_grouped_kernel<bm, bn, bk, tm, tn, T, ks><<<(unsigned)ctas, ZG_THREADS, 0, st>>>(args, prefix, \
                                                                                                   n, total);    \
        break;
        ZG_SHAPES(X)
#undef X
    }
}

}  // namespace

void launch_zgemm(int arith, int shape, const GemmArgs& g, int blocks, cudaStream_t st) {
    const dim3 grid((unsigned)blocks, (unsigned)g.nsplit);
    if (arith == ZG_FP64) launch_one<double>(shape, g, grid, st);
    else if (arith == ZG_FP32) launch_one<float>(shape, g, grid, st);
    else launch_one<df>(shape, g, grid, st);
}

void launch_zgemm_grouped(int arith, int shape, const GemmArgs* args, const long long* prefix, int n,
                          long long total, int ctas, cudaStream_t st) {
    if (arith == ZG_FP32) launch_group<float>(shape, args, prefix, n, total, ctas, st);
    else launch_group<double>(shape, args, prefix, n, total, ctas, st);
}

}  // namespace ccsdk

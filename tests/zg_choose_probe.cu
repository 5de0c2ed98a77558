// Host build of the SIMT GEMM's choice of tile shape and K split (csrc/zgemm_shapes.h).
#include "../paper_1911_00242_gb300/csrc/zgemm_shapes.h"

extern "C" int probe_zg_choose(int arith, int M, int N, int K, long long nchunk, long long nbatch, int* shape) {
    const ccsdk::ZgChoice c = ccsdk::zg_choose(arith, M, N, K, nchunk, nbatch, 1, 152);
    *shape = c.shape;
    return c.nsplit;
}
extern "C" long long probe_zg_least(int arith, int K, long long nchunk) {
    return arith == ccsdk::ZG_FP32 ? ccsdk::zg_fp32_splits(K, nchunk) : 1;
}

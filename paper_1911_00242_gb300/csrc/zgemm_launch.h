// Launchers of the SIMT complex GEMM (zgemm_launch.cu).
#pragma once
#include "zgemm_kb.cuh"
#include "zgemm_shapes.h"

namespace ccsdk {

// One contraction: blocks (tiles x batches) by nsplit CTAs.
void launch_zgemm(int arith, int shape, const GemmArgs& g, int blocks, cudaStream_t st);
// The same step of n problems (grouped iterations run FP64 or FP32).
void launch_zgemm_grouped(int arith, int shape, const GemmArgs* args, const long long* prefix, int n,
                          long long total, int ctas, cudaStream_t st);

}  // namespace ccsdk

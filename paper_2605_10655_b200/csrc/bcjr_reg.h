// Host side of bcjr_reg.cuh: which shapes it covers, and its launches.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "bcjr_common.cuh"

namespace bcjr {

struct RegPlan {
    int grid = 0, parts = 0;          // CTAs, partial codebook gradients (one per cluster)
    size_t smem = 0, hist_floats = 0;
};

// Clusters of the kernel that can be resident at once; 0 if the shape is not covered.
enum RegKind { REG_FWD = 0, REG_BWD = 1, REG_BWD_FIXED = 2 };   // the last: without grad_codebook
int reg_resident(int Lb, int n, RegKind kind, int num_sms);
RegPlan reg_plan(int Lb, int n, int64_t B, bool bwd, int resident, int max_ctas);
cudaError_t reg_forward(const FwdParams &p, const RegPlan &plan, cudaStream_t st);
cudaError_t reg_backward(const BwdParams &p, const RegPlan &plan, bool want_gc, cudaStream_t st);
// Certified Viterbi (bcjr_vitreg.cuh): CTAs resident at once (0: not covered), launch of `grid` of them, floats of history a CTA needs.
int reg_viterbi_resident(int Lb, int n, int num_sms);
size_t reg_viterbi_hist_floats(int Lb, int n);
cudaError_t reg_viterbi(const VitParams &p, int grid, cudaStream_t st);

}  // namespace bcjr

// Host side of bcjr_meet.cuh: which shapes it covers, and its launches.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "bcjr_common.cuh"

namespace bcjr {

// Forms of the kernels for a trellis, see bcjr_meet_launch.cuh
constexpr int MEET_FORMS = 3, MEET_K3 = 2;   // the last one: k = 3
struct MeetPlan {
    bool split = false;               // two launches
    int grid = 0, parts = 0;          // CTAs, partial codebook gradients
    size_t smem = 0, hist_floats = 0, aux_ints = 0;
};

// Sides (two a block) that can be in flight at once; 0 if the shape has no such form.
int meet_fwd_resident(int Lb, int form, int n, int num_sms);
int meet_bwd_resident(int Lb, int form, int n, int num_sms);
MeetPlan meet_fwd_plan(int Lb, int form, int n, int64_t B, int resident);
MeetPlan meet_bwd_plan(int Lb, int form, int n, int64_t B, int resident);
// p.hist, aux: the plan's scratch.  Split form: blocks without a certificate are left flagged in p.lin_flag (p.lin_x >= 0).
cudaError_t meet_forward(const FwdParams &p, int form, const MeetPlan &plan, int *aux, cudaStream_t st);
cudaError_t meet_backward(const BwdParams &p, int form, const MeetPlan &plan, int *aux, bool want_gc, cudaStream_t st);

}  // namespace bcjr

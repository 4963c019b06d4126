// Launches of the two-ended register kernels (bcjr_meet.cuh), forward.
#include "bcjr_meet_launch.cuh"

namespace bcjr {

int meet_fwd_resident(int Lb, int form, int n, int num_sms) { return meet_resident_of<false>(Lb, form, n, num_sms); }
MeetPlan meet_fwd_plan(int Lb, int form, int n, int64_t B, int resident) { return meet_plan_of<false>(Lb, form, n, B, resident); }

cudaError_t meet_forward(const FwdParams &p, int form, const MeetPlan &plan, int *aux, cudaStream_t st)
{
    return dispatch<false>(p.Lb, form, [&](auto c) {
        using C = decltype(c);
        const MeetScratch ms{aux};
        if constexpr (C::SPLIT) {
            const cudaError_t e = launch<C>(meet_fwd_kernel<C, 1>, p, plan, ms, st);
            return e != cudaSuccess ? e : launch<C>(meet_fwd_kernel<C, 2>, p, plan, ms, st);
        } else {
            return launch<C>(meet_fwd_kernel<C, 0>, p, plan, ms, st);
        }
    });
}

}  // namespace bcjr

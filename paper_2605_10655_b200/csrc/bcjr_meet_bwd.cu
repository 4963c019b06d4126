// Launches of the two-ended register kernels (bcjr_meet.cuh), backward.
#include "bcjr_meet_launch.cuh"

namespace bcjr {

int meet_bwd_resident(int Lb, int form, int n, int num_sms) { return meet_resident_of<true>(Lb, form, n, num_sms); }
MeetPlan meet_bwd_plan(int Lb, int form, int n, int64_t B, int resident) { return meet_plan_of<true>(Lb, form, n, B, resident); }

cudaError_t meet_backward(const BwdParams &p, int form, const MeetPlan &plan, int *aux, bool want_gc, cudaStream_t st)
{
    return dispatch<true>(p.Lb, form, [&](auto c) {
        using C = decltype(c);
        const MeetScratch ms{aux};
        if constexpr (C::SPLIT) {
            const cudaError_t e = launch<C>(meet_bwd_kernel<C, false, 1>, p, plan, ms, st);
            if (e != cudaSuccess) return e;
            return want_gc ? launch<C>(meet_bwd_kernel<C, true, 2>, p, plan, ms, st) : launch<C>(meet_bwd_kernel<C, false, 2>, p, plan, ms, st);
        } else {
            return want_gc ? launch<C>(meet_bwd_kernel<C, true, 0>, p, plan, ms, st) : launch<C>(meet_bwd_kernel<C, false, 0>, p, plan, ms, st);
        }
    });
}

}  // namespace bcjr

// Forward call, one CTA per weight block, for the 2^16-state trellis (k = 2, 3), with LINEAR messages.
//
// fwd_solo_kernel carries log2 alpha and log2 beta.  A log-domain step costs, besides the exponential of every
// state's energy, a maximum and a subtraction per state, a logarithm per group and an exponential per group for the
// posterior, and the sweep is bound by exactly those: issue slots and the special-function unit.  With the messages
// themselves in float32,
//     A'(q) = sum_j A((q+jQ)>>k) E(q+jQ),   M'(q) = sum_b M((qK+b) & (Q-1)) E(qK+b),   E(s) = 2^(-lam2 (w-c_s)^2),
// a state costs a subtraction, a square, one exponential and one multiply-add, and a posterior weight is the product
// A M' -- no maximum, no logarithm.  592 blocks of 256 weights, T = 0.1: k = 2 7.34 -> 5.40 ms, k = 3 6.80 -> 5.55 ms
// (special-function unit 72 % busy, FP32 pipe 54 %, before one in four of the alpha sweep's exponentials moved to the
// FP32 pipe: 5.67 -> 5.41 ms at k = 2, 5.78 -> 5.53 at k = 3; the same in the beta sweep loses).
//
// What float32 lacks is range, and it lacks less than one would fear: what has to fit between 2^-126 and 2^127 is not
// the spread of a step's messages but the excess of the paths that carry posterior weight over the best prefix (and
// the best suffix) at that step.  Simulated in float64 on N(0,1) weights and tables, log2(max A max M / Z), maximum
// over the 256 steps of a block: median 6 at T = 0.1, 100 at T = 0.01, 99th percentile 16 and 179.  So a block is run
// in the linear form and its result is CERTIFIED; a block without a certificate is run again in the log domain, from
// the list that lin_list_kernel makes of the flags: up to a few waves of them by fwd_reg_kernel, which spreads a block over
// eight SMs, more by fwd_solo_kernel.
//
// The certificate.  The alpha sweep computes an upper bound of A (up to rounding): an exponential below 2^-126 is flushed to
// zero, which takes less than 2^-126 sum_j A_j from an output, so that much (one sum per butterfly) is added to every
// output, with 2^-126 on top for what subnormal results lose (this also keeps an accepted block's M below 2^111, far enough from
// overflow for the backward call, which multiplies it by zeros).  The beta sweep flushes, so its M is a lower bound.  Let S_t =
// sum_q A_t M_t, normalised by Z_up = sum A_{n+1}.  Then S_1 = Z_lo / Z_up (A_1 is exact) with Z_lo <= Z <= Z_up, and S_t - S_1
// bounds the added weight that passes step t.  If |S_t - 1| <= eps at every step, the added weight at any step is at most
// 2 eps and the weight missing from M at most eps: every posterior is within 3 eps (sum of absolute differences),
// eps = 2e-5, below the log-domain kernel's own rounding of S_t at T = 0.01 (6e-5).  Overflow ends in a NaN or an infinity
// and fails, and so do non-finite inputs, which the log-domain kernel then reports.  Without the added weight six of 16384
// blocks at T = 0.01 passed every test with a wrong result: paths flushed from A early and from M late.
//   * Gauge: every step E is multiplied by 2^-off, off = exponent of the largest input - X, by adding off to the exponent's
//     argument (free: the square becomes a multiply-add).  The beta sweep uses the alpha sweep's offsets in reverse, which
//     makes its messages M_t 2^(O_t) / Z: the posterior is the plain product A M', and no maximum is needed for its gauge.
//     (A larger common factor under the exponential would widen its range, but the argument's rounding at that magnitude
//     costs three digits of S_t.)
//   * X = min(100, 1.33 lam2): at X = 100 A reaches 2^103 and M about 2^110 before the added weight fails a block.  Where the
//     trellis is warm the messages need no such range, and M, which is gamma / A, keeps its small values out of the subnormals
//     (with X = 100 at T = 0.3 the rarest states' grad_codebook was off by 2.8e-3 of its root mean square, now 2e-5).
//
// The table is staged scaled by sqrt(lam2), so that E = 2^-(d d); soft is recovered as w + sum gamma d / sqrt(lam2).
#pragma once
#include "bcjr_solo.cuh"

namespace bcjr {

constexpr int LIN_X_MAX = 100, LIN_STEP_DROP = 120;
constexpr float LIN_DEFECT = 2e-5f;
// what an alpha output can lose to zero, from the sum of its butterfly's inputs
__device__ __forceinline__ float lin_floor(float inputs) { return fmaf(inputs, 1.1756e-38f, 1.1756e-38f); }

__device__ __forceinline__ float pow2i(int e) { return __int_as_float((e + 127) << 23); }     // -126 <= e <= 127
__device__ __forceinline__ int exp2i(float v) { return (int)(__float_as_uint(v) >> 23) - 127; }   // v > 0
// step offset from the largest input message
__device__ __forceinline__ int lin_offset(float vmax, int X) { const int o = exp2i(vmax) - X; return o < -LIN_STEP_DROP ? -LIN_STEP_DROP : o; }
// 2^-a of a pair
__device__ __forceinline__ float2 ex2n2(float2 a) { return make_float2(ex2f(-a.x), ex2f(-a.y)); }
// The same on the FP32 pipe, with a result that does go to zero: ex2_poly2 clamps its argument, and 2^-125 times a
// large message would be a floor under every state.  Here the exponent sum is clamped at zero instead.
__device__ __forceinline__ float2 ex2n_poly2(float2 a)
{
    a.x = fminf(a.x, 250.f); a.y = fminf(a.y, 250.f);            // keeps the exponent arithmetic below from wrapping
    const float2 magic = splat2(12582912.f);
    const float2 t = sub2(magic, a);
    const float2 n = sub2(magic, t);                             // -(nearest integer to -a)
    const float2 f = sub2(n, a);
    float2 p = fma2(splat2(1.3390863e-3f), f, splat2(9.6760318e-3f));
    p = fma2(p, f, splat2(5.5503570e-2f));
    p = fma2(p, f, splat2(2.4022107e-1f));
    p = fma2(p, f, splat2(6.9314718e-1f));
    p = fma2(p, f, splat2(1.0000001f));
    p.x = __int_as_float(__viaddmax_s32(__float_as_int(p.x), __float_as_int(t.x) << 23, 0));
    p.y = __int_as_float(__viaddmax_s32(__float_as_int(p.y), __float_as_int(t.y) << 23, 0));
    return p;
}

// Which blocks can be expected to have a certificate.  A state is what the last Lb / k steps left in it, so those steps' weights share its
// Lb bits.  A weight near the middle of the table is served by half the states, one in its tail by a few, and a window of weights that
// together ask for many more bits than there are is served by paths that were poor prefixes: that excess over the best prefix, times lam2, is
// the range float32 lacks.  The measure: bits a weight asks for, -log2 of the normal tail beyond it (the quadratic is within 0.3 bits up to 7
// sigma, its tangent from there on), summed over the window, maximum over the block.  N(0,1) blocks of 256 weights and 2^16 states: 32 in the
// median, 41 at the 99th percentile; heavy-tailed ones (four degrees of freedom) 40 and 100.  The limits are in the dispatch
// (lin_demand_limit).  A misjudged block costs time only.
__device__ __forceinline__ float lin_demand(const float *__restrict__ w, int t, int n, int window)
{
    float s = 0.f;
    for (int i = t; i < t + window && i < n; ++i) {
        const float a = fabsf(__ldg(w + i)), m = fminf(a, 7.3f);
        s += fmaf(10.2f, a - m, fmaf(m, fmaf(0.63f, m, 1.05f), 1.f));
    }
    return s;
}
// *count (zero before the call): blocks beyond p.demand, a warp per block
static __global__ void __launch_bounds__(256) lin_judge_kernel(FwdParams p, int *count)
{
    const int lane = threadIdx.x & 31;
    int mine = 0;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < p.B; b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        float d = 0.f;
        for (int t = lane; t < p.n; t += 32) d = fmaxf(d, lin_demand(p.W + b * p.n, t, p.n, p.window));
        mine += warp_max(d) > p.demand;
    }
    if (lane == 0 && mine) atomicAdd(count, mine);
}
// calls judged as a whole: true if no block is tried (all are flagged then)
__device__ __forceinline__ bool lin_given_up(const FwdParams &p)
{
    if (!p.unlikely || *p.unlikely <= p.unlikely_max) return false;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < p.B; b += (int64_t)gridDim.x * blockDim.x) p.lin_flag[b] = 1;
    return true;
}

// Backward kernels (see bcjr_lin_bwd.cuh): exponent of a gradient from the bit pattern of its largest |g| (NaN sorts above infinity);
// GRAD_NONE: all zero.  The bounds keep both factors normal numbers.
constexpr int GRAD_LEVEL = 2, GRAD_SPAN = 8, GRAD_ROOM = 2, GRAD_NONE = -1000;
__device__ __forceinline__ uint32_t grad_bits(float g) { return __float_as_uint(fabsf(g)); }
__device__ __forceinline__ int grad_exponent(uint32_t bits)
{
    const int e = (int)(bits >> 23) - 127;
    return bits == 0u ? GRAD_NONE : e < -100 ? -100 : e > 112 ? 112 : e;
}
__device__ __forceinline__ float grad_down(int e) { return e == GRAD_NONE ? 1.f : pow2i(-(e + GRAD_LEVEL)); }
__device__ __forceinline__ float grad_up(int e) { return e == GRAD_NONE ? 1.f : pow2i(e + GRAD_LEVEL); }
// scale of a block in a call: the call's, GRAD_SPAN bits less, twice as many ...; the call's where the block has no gradient
__device__ __forceinline__ int grad_scale(uint32_t bits, uint32_t top_bits)
{
    const int e = grad_exponent(bits), top = grad_exponent(top_bits);
    return e == GRAD_NONE ? top : top - (top - e) / GRAD_SPAN * GRAD_SPAN;
}
// bits[b] of every block, *top (zero before the call) of all: a warp per block
static __global__ void __launch_bounds__(256) grad_bits_kernel(const float *__restrict__ g, int64_t B, int n, uint32_t *__restrict__ bits, uint32_t *__restrict__ top)
{
    const int lane = threadIdx.x & 31;
    uint32_t all = 0;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < B; b += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        uint32_t m = 0;
#pragma unroll 4
        for (int t = lane; t < n; t += 32) m = max(m, grad_bits(__ldg(g + b * n + t)));
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) bits[b] = m;
        all = max(all, m);
    }
    if (lane == 0 && all) atomicMax(top, all);
}

// Indices of the flagged blocks, ascending, behind their number: list[0] = count, list[1 + i].
static __global__ void __launch_bounds__(1024) lin_list_kernel(const uint8_t *__restrict__ flag, int64_t B, int *__restrict__ list)
{
    __shared__ int wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int base = 0;
    for (int64_t b0 = 0; b0 < B; b0 += 4096) {
        const int64_t b = b0 + 4 * tid;
        uint32_t f = 0;
        if (b + 4 <= B) f = *reinterpret_cast<const uint32_t *>(flag + b);
        else for (int i = 0; i < 4; ++i) if (b + i < B) f |= (uint32_t)flag[b + i] << (8 * i);
        const int mine = __popc(f & 0x01010101u);
        int pre = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, pre, o); if (lane >= o) pre += v; }
        if (lane == 31) wsum[warp] = pre;
        __syncthreads();
        int before = 0, total = 0;
        for (int i = 0; i < 32; ++i) { if (i < warp) before += wsum[i]; total += wsum[i]; }
        int at = base + before + pre - mine;
#pragma unroll
        for (int i = 0; i < 4; ++i) if ((f >> (8 * i)) & 1u) list[1 + at++] = (int)(b + i);
        base += total;
        __syncthreads();
    }
    if (tid == 0) list[0] = base;
}

// stage_codebook with the entries scaled
template <typename C>
__device__ __forceinline__ void stage_codebook_scaled(const float *cbk, int x, uint32_t tm_butterfly, bool beta, float scale)
{
    constexpr int K = C::K;
#pragma unroll
    for (int u = 0; u < C::UNITS; ++u) {
        float2 v[8];
#pragma unroll
        for (int hh = 0; hh < C::HPU; ++hh) {
            const int h = u * C::HPU + hh;
#pragma unroll
            for (int o = 0; o < K; ++o) {
                const int slo = beta ? (2 * h) * C::Q + x * K + o : o * C::Q + x * K + 2 * h;
                const int shi = beta ? (2 * h + 1) * C::Q + x * K + o : o * C::Q + x * K + 2 * h + 1;
                v[beta ? C::b_idx(hh, o) : C::a_idx(o, hh)] = make_float2(scale * __ldg(cbk + slo), scale * __ldg(cbk + shi));
            }
        }
        tmem_st16(tm_butterfly + 16u * u, v);
    }
}

template <int KB>
__global__ void __launch_bounds__(SoloCfg<KB>::THREADS, 1) fwd_lin_kernel(FwdParams p)
{
    using C = SoloCfg<KB>;
    constexpr int K = C::K, NB = C::NB, Q = C::Q, BPT = C::BPT, NWARP = C::NWARP, CT = C::CTHREADS, NCH = C::NCH, RD = C::RD;
    constexpr int UNITS = C::UNITS, HPU = C::HPU, NU = BPT * UNITS;
    if (lin_given_up(p)) return;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = p.n, X = p.lin_x;
    const float sl = sqrtf(p.lam2);
    const double isl_d = 1.0 / (double)sl;

    float *msg = smem + C::OFF_MSG;
    float4 *stage4 = reinterpret_cast<float4 *>(smem + C::OFF_RING);
    float *w_s = smem + C::OFF_W, *v_s = w_s + C::MAX_N;          // scaled clamped weight, and the same + 2 delta (step_energy)
    const float c_lo = p.diag->c_lo, c_hi = p.diag->c_hi;
    int *O_s = reinterpret_cast<int *>(smem + C::OFF_O);
    float *wmax = smem + C::OFF_WMAX;
    float *part = smem + C::OFF_PART;
    float *lz = smem + C::OFF_LZ;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_TMEM);
    const uint32_t stage_u32 = smem_u32(stage4) + (uint32_t)tid * 16u;
    float4 *hist4 = reinterpret_cast<float4 *>(p.hist + (size_t)blockIdx.x * n * Q) + tid;

    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tm = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    int push_a[BPT];                                              // destinations of the alpha outputs, as in fwd_solo_kernel
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int x = i * CT + tid;
        const int q2 = x * K, j2 = q2 / NB, x2 = q2 % NB;
        push_a[i] = ((x2 / CT) * K + j2) * CT + (x2 % CT);
    }
    float defect = 0.f, zgap = 0.f;

    for (int64_t blk = blockIdx.x; blk < p.B; blk += gridDim.x) {
        const float *w = p.W + blk * n;
        int outside = 0;
        for (int t = tid; t < n; t += CT) {
            const StepEnergy se = step_energy(__ldg(w + t), c_lo, c_hi, p.lam2);
            w_s[t] = se.wc * sl; v_s[t] = (se.wc + 2.f * se.delta) * sl;
            outside |= se.delta != 0.f;
        }
        const bool recentre = __syncthreads_or(outside) != 0;
        for (int q = tid; q < Q; q += CT) msg[q] = pow2i(X);  // A_1 = 1 = 2^X 2^O_1
        if (tid == 0) O_s[1] = -X;
#pragma unroll 1                                               // unrolled, its addresses cost the sweeps registers
        for (int i = 0; i < BPT; ++i) stage_codebook_scaled<C>(p.cb, i * CT + tid, tm + (uint32_t)(K * K * i), false, sl);
        tmem_wait_st();
        int O = -X, off = 0;
        compute_barrier(CT);
        // ================= alpha sweep
        auto alpha_sweep = [&](auto rc_tag) {
            constexpr bool RC = decltype(rc_tag)::value;
                        for (int t = 1; t <= n; ++t) {
                const int cur = (t - 1) & 1;
                const float *Lin = msg + cur * Q;
                float *Lout = msg + (cur ^ 1) * Q;
                float2 cb[2][8];
                tmem_ld16(tm, cb[0]);
                if (t > 1) off = lin_offset(warp_max(lane < NWARP ? wmax[cur * 32 + lane] : 0.f), X);
                float4 *hrow = hist4 + (size_t)(t - 1) * (BPT * NCH * CT);
                const float2 w2 = splat2(w_s[t - 1]), v2 = splat2(v_s[t - 1]), off2 = splat2((float)off);
                float tmax = 0.f;
#pragma unroll
                for (int i = 0; i < BPT; ++i) {
                    float Aj[K];
#pragma unroll
                    for (int j = 0; j < K; ++j) Aj[j] = Lin[(i * K + j) * CT + tid];
#pragma unroll
                    for (int q = 0; q < NCH; ++q)
                        hrow[(i * NCH + q) * CT] = make_float4(Aj[4 * q], Aj[4 * q + 1], Aj[4 * q + 2], Aj[4 * q + 3]);
                    float in = Aj[0];
#pragma unroll
                    for (int j = 1; j < K; ++j) in += Aj[j];
                    const float2 floor2 = splat2(lin_floor(in));
                    float2 out[K / 2];
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const int g = i * UNITS + u;
                        tmem_wait_ld(cb[g & 1]);
                        if (g + 1 < NU) tmem_ld16(tm + 16u * (g + 1), cb[(g + 1) & 1]);
#pragma unroll
                        for (int hh = 0; hh < HPU; ++hh) {
                            const int h = u * HPU + hh;
                            float2 sum = floor2;
#pragma unroll
                            for (int j = 0; j < K; ++j) {
                                const float2 c2 = cb[g & 1][C::a_idx(j, hh)];
                                const float2 d = sub2(c2, w2);
                                const float2 arg = fma2(d, RC ? sub2(c2, v2) : d, off2);
                                const float2 e = (j & 3) == 3 ? ex2n_poly2(arg) : ex2n2(arg);   // one in four on the FP32 pipe
                                sum = fma2(e, splat2(Aj[j]), sum);
                            }
                            out[h] = sum;
                            tmax = max3f(tmax, sum.x, sum.y);
                        }
                    }
#pragma unroll
                    for (int h = 0; h < K / 2; h += 2)
                        *reinterpret_cast<float4 *>(Lout + push_a[i] + 2 * h) = make_float4(out[h].x, out[h].y, out[h + 1].x, out[h + 1].y);
                }
                tmax = warp_max(tmax);
                if (lane == 0) wmax[(cur ^ 1) * 32 + warp] = tmax;
                O += off;
                if (tid == 0) O_s[t + 1] = O;
                compute_barrier(CT);
            }
        };
        if (recentre) alpha_sweep(std::true_type{}); else alpha_sweep(std::false_type{});
        // ================= Z = 2^O_{n+1} sum_q A_{n+1}(q); A_{n+1} sits in buffer n&1
        {
            const float *Afin = msg + (n & 1) * Q;
            float ssum = 0.f;
            for (int q = tid; q < Q; q += CT) ssum += Afin[q];
            ssum = warp_sum(ssum);
            if (lane == 0) lz[warp] = ssum;
        }
        compute_barrier(CT);
        const float Zs = warp_sum(lane < NWARP ? lz[lane] : 0.f);
        if (!(Zs > 1e-37f && Zs < 1e37f)) {                       // not representable (or not finite): leave it to the log-domain kernel
            if (tid == 0) p.lin_flag[blk] = 1;
            compute_barrier(CT);
            continue;
        }
        const int Ofin = O;
        // ================= beta sweep: messages M_t 2^(O_{t+1} - Ofin) / Zs, so that gamma = A_t M'_{t-1}
        for (int q = tid; q < Q; q += CT) msg[q] = 1.f / Zs;      // M_n = 1 in buffer 0
#pragma unroll 1                                               // unrolled, its addresses cost the sweeps registers
        for (int i = 0; i < BPT; ++i) stage_codebook_scaled<C>(p.cb, i * CT + tid, tm + (uint32_t)(K * K * i), true, sl);
        tmem_wait_st();
        int bad = 0;
        float bdef = 0.f, den1 = 0.f;
        // history stream as in fwd_solo_kernel
        const uint32_t nchunks = (uint32_t)n * BPT;
        const float4 *nsrc = hist4 + (size_t)(n - 1) * (BPT * NCH * CT);
        uint32_t nleft = nchunks;
        int ni = 0;
        auto issue_chunk = [&](uint32_t slot) {
            const uint32_t dst = stage_u32 + slot * (uint32_t)(NCH * CT * 16);
#pragma unroll
            for (int q = 0; q < NCH; ++q)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(q * CT * 16)), "l"(nsrc + q * CT) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
            const bool more = nleft > 1;
            const bool wrap = ni == BPT - 1;
            const ptrdiff_t adv = wrap ? -(ptrdiff_t)((size_t)(2 * BPT - 1) * (NCH * CT)) : (ptrdiff_t)(NCH * CT);
            nsrc += more ? adv : 0;
            ni = wrap ? 0 : ni + 1;
            nleft -= more ? 1u : 0u;
        };
        constexpr bool STATIC_RING = RD == BPT;
        constexpr ptrdiff_t HROW = (ptrdiff_t)BPT * NCH * CT;
        auto issue_static = [&](const float4 *row, int i) {
            const uint32_t dst = stage_u32 + (uint32_t)i * (uint32_t)(NCH * CT * 16);
#pragma unroll
            for (int q = 0; q < NCH; ++q)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(q * CT * 16)), "l"(row + (i * NCH + q) * CT) : "memory");
        };
#pragma unroll
        for (uint32_t c = 0; c + 1 < RD; ++c) {
            if (STATIC_RING) { issue_static(hist4 + (size_t)(n - 1) * HROW, (int)c); asm volatile("cp.async.commit_group;" ::: "memory"); }
            else issue_chunk(c);
        }
        uint32_t slot = 0;
        // warp 0: soft of step t from the partial sums of parity b, kept in v_s until the block has its certificate
        auto finish_step = [&](int t, int b) {
            float a = lane < NWARP ? part[(b * 32 + lane) * 2] : 0.f;
            float c = lane < NWARP ? part[(b * 32 + lane) * 2 + 1] : 0.f;
            a = warp_sum(a); c = warp_sum(c);
            if (lane == 0) {
                const float sw = (float)(((double)w_s[t - 1] + (double)(a / c)) * isl_d);
                v_s[t - 1] = sw;                                     // (step t is done with its entry)
                den1 = c;
                bdef = fmaxf(bdef, fabsf(c - 1.f));
                bad |= !(fabsf(c - 1.f) <= LIN_DEFECT);
            }
        };
        compute_barrier(CT);
        auto beta_sweep = [&](auto rc_tag) {
            constexpr bool RC = decltype(rc_tag)::value;
            for (int t = n; t >= 1; --t) {
                const int cur = (n - t) & 1;
                const float *Min = msg + cur * Q;
                float *Mout = msg + (cur ^ 1) * Q;
                float2 cb[2][8];
                tmem_ld16(tm, cb[0]);
                if (t < n && warp == 0) finish_step(t + 1, cur);
                const float2 w2 = splat2(w_s[t - 1]), v2 = splat2(v_s[t - 1]);
                const float2 off2 = splat2((float)(O_s[t + 1] - O_s[t]));
                float2 num2 = make_float2(0.f, 0.f), den2 = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < BPT; ++i) {
                    if (STATIC_RING) {
                        const float4 *hrow = hist4 + (size_t)(t - 1) * HROW;
                        if (i == 0) issue_static(hrow, BPT - 1);
                        else if (t > 1) issue_static(hrow - HROW, i - 1);
                        asm volatile("cp.async.commit_group;" ::: "memory");
                    } else {
                        issue_chunk(slot == 0 ? RD - 1 : slot - 1);
                    }
                    asm volatile("cp.async.wait_group %0;" ::"n"(RD - 1) : "memory");
                    const uint32_t sl_ = STATIC_RING ? (uint32_t)i : slot;
                    float Ah[K];
#pragma unroll
                    for (int q = 0; q < NCH; ++q) {
                        const float4 l4 = stage4[(sl_ * NCH + q) * CT + tid];
                        Ah[4 * q] = l4.x; Ah[4 * q + 1] = l4.y; Ah[4 * q + 2] = l4.z; Ah[4 * q + 3] = l4.w;
                    }
                    slot = slot + 1 == RD ? 0 : slot + 1;
                    float Mb[K];
#pragma unroll
                    for (int b = 0; b < K; b += 4) {
                        const float4 v = *reinterpret_cast<const float4 *>(Min + (i * CT + tid) * K + b);
                        Mb[b] = v.x; Mb[b + 1] = v.y; Mb[b + 2] = v.z; Mb[b + 3] = v.w;
                    }
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) {
                        const int g = i * UNITS + u;
                        tmem_wait_ld(cb[g & 1]);
                        if (g + 1 < NU) tmem_ld16(tm + 16u * (g + 1), cb[(g + 1) & 1]);
#pragma unroll
                        for (int hh = 0; hh < HPU; ++hh) {
                            const int jh = u * HPU + hh;
                            float2 sum, dsum;
#pragma unroll
                            for (int b = 0; b < K; ++b) {
                                const float2 c2 = cb[g & 1][C::b_idx(hh, b)];
                                const float2 d = sub2(c2, w2);
                                const float2 e = ex2n2(fma2(d, RC ? sub2(c2, v2) : d, off2));
                                const float2 pb = mul2(e, splat2(Mb[b]));
                                sum = b == 0 ? pb : add2(sum, pb);
                                dsum = b == 0 ? mul2(pb, d) : fma2(pb, d, dsum);
                            }
                            Mout[((2 * jh) * (NB / K) + (i * CT + tid) / K) * K + (tid % K)] = sum.x;
                            Mout[((2 * jh + 1) * (NB / K) + (i * CT + tid) / K) * K + (tid % K)] = sum.y;
                            const float2 Ahj = make_float2(Ah[2 * jh], Ah[2 * jh + 1]);
                            num2 = fma2(Ahj, dsum, num2);
                            den2 = fma2(Ahj, sum, den2);
                        }
                    }
                }
                const float nd = warp_sum2_split(num2.x + num2.y, den2.x + den2.y, lane);   // lane 0: numerator, lane 16: denominator
                if ((lane & 15) == 0) part[((cur ^ 1) * 32 + warp) * 2 + (lane >> 4)] = nd;
                compute_barrier(CT);
            }
        };
        if (recentre) beta_sweep(std::true_type{}); else beta_sweep(std::false_type{});
        if (warp == 0) finish_step(1, n & 1);
        if (tid == 0) {
            p.lin_flag[blk] = bad ? 1 : 0;
            lz[0] = bad ? 1.f : 0.f;
            if (!bad) {
                const int ez = exp2i(Zs);
                const float l2z = lg2f(Zs * pow2i(-ez));
                if (p.logZ) {
                    double zshift = 0.0;                             // sum_t lam2 delta_t^2: left out by step_energy
                    if (recentre)
                        for (int t = 0; t < n; ++t) {
                            const double dl = (double)step_energy(__ldg(w + t), c_lo, c_hi, p.lam2).delta;
                            zshift += (double)p.lam2 * dl * dl;
                        }
                    p.logZ[blk] = (float)(((double)(Ofin + ez) + (double)l2z - zshift) * 0.6931471805599453);
                }
                defect = fmaxf(defect, bdef);
                zgap = fmaxf(zgap, fabsf(lg2f(den1)));               // A_1 is constant: the sums of step 1 are the beta side's Z
                if (p.blk_defect) p.blk_defect[blk] = bdef;
            }
        }
        compute_barrier(CT);                                      // part and the messages are free for the next block
        // soft may be W: written where it stands only, and after everything that reads W
        if (lz[0] == 0.f)
            for (int t = tid; t < n; t += CT) {
                p.soft[blk * n + t] = v_s[t];
                if (p.soft_copy) p.soft_copy[blk * n + t] = v_s[t];
            }
    }
    if (tid == 0) {
        diag_max(&p.diag->max_defect, defect);
        diag_max(&p.diag->max_logz_gap, zgap);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

}  // namespace bcjr

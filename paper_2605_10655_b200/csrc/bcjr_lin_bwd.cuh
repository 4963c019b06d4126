// Backward call with linear messages (2^16 states, k = 2): the two kernels of the chunked backward call
// (bcjr_alpha.cuh, bcjr_skew.cuh) with A, M in float32 instead of their logarithms, for the blocks that the forward
// call certified (bcjr_lin.cuh; same gauge, same offsets, same range: what is flushed here is less than what the
// forward call added for its certificate).  The other blocks are skipped here and run from the list: up to a few
// waves of them by bwd_reg_kernel, more by the chunked log-domain kernels.
//
// The alpha sweep carries A and AA = A (At + gs), At the conditional expectation of the increments so far and
// gs_t = g_t (wc_t - soft_t) the part of h_t = g_t (c - soft_t) = (g_t / sl) d + gs_t that is common to the states:
//     A'(q) = sum_j E A_j,    AA'(q) = sum_j E ((g/sl) d A_j + AA_j) + gs_{t+1} A'(q)
// five packed instructions and two exponentials per pair of states, no division.  The beta sweep carries M (already
// divided by Z, see bcjr_lin.cuh) and the conditional expectation Bt -- with y = (g/sl) d + Bt the gradient of a state
// is one product P z, P = E M_b, z = A g + (w - c)/T (A y + AA), where the un-normalised form would need three more
// packed instructions per pair; its price is one reciprocal per group.
//
// Scale of the gradient.  The forward certificate covers A, M and the energies.  What the backward sweeps add to them -- AA, y, z --
// is linear in g: with A at 2^103 a gradient of 2^16 overflows z where the exponential is zero (0 inf in grad_codebook), one of
// 2^-34 loses AA's bits to subnormals.  So a block runs on g 2^-(e + 2), its largest |g| between 2^(e-7) and 2^(e+1): AA stays below
// 2^115, z below 2^126 for weights of twenty units at T = 0.01, and a message of 2^-111 still has a normal AA.  The powers of two are
// exact, so the results are those of any other scale bit for bit.  The accumulators of grad_codebook are at the block's scale; where
// the next block's is another, they are written out first.  e is the exponent of the call's largest |g| for every block within
// eight bits of it (grad_bits_kernel: 3 us for 4 million weights), so that this happens only where blocks differ by more.
//
// 592 blocks of 256 weights, T = 0.1: 11.85 -> 10.1 ms with grad_codebook, 11.2 (bwd_solo_kernel) -> 10.0 without
// (alpha 8.4 k -> 6.1 k, beta 11.6 k clocks per step and block; ncu: alpha XU 67 %, FMA 47 %; beta XU 44 %, FMA 56 %, issue
// 55 % with packed instructions counted once).
#pragma once
#include "bcjr_alpha.cuh"
#include "bcjr_lin.cuh"

namespace bcjr {

// What a step needs besides its messages, formed once per block.  gs is centred on the SCALED table: d / sl is c - wc only up
// to the rounding of c sl and wc sl, and a centring by wc itself would leave that rounding, the same for all states, in
// every r_t; with wc taken back from its scaled value (in double) only the table's own rounding, a half-ulp of c, remains.
__device__ __forceinline__ float lin_gs(float g, float wc_scaled, double isl, float soft) { return (float)((double)g * ((double)wc_scaled * isl - (double)soft)); }

template <int KB_>
struct AlphaLinCfg : AlphaCfg<KB_> {
    using A = AlphaCfg<KB_>;
    static constexpr int OFF_STEP = A::SMEM_FLOATS;             // float4 [MAX_N + 1]: scaled weight, the same + 2 delta, g / sl, gs
    static constexpr size_t SMEM_BYTES = (size_t)(OFF_STEP + 4 * (A::MAX_N + 1)) * 4;
    static_assert(OFF_STEP % 4 == 0, "16-byte step entries");
};

template <int KB>
__global__ void __launch_bounds__(AlphaCfg<KB>::THREADS, 1) bwd_alpha_lin_kernel(BwdParams p)
{
    using C = AlphaLinCfg<KB>;
    constexpr int K = C::K, Q = C::Q, BPT = C::BPT, NWARP = C::NWARP, CT = C::CTHREADS, UNITS = C::UNITS, HPU = C::HPU, NU = BPT * UNITS;
    constexpr ptrdiff_t HSTEP = 2 * Q / 4;                      // float4 per step: (A, AA) of every group
    constexpr int HCH = CT;
    extern __shared__ __align__(16) float smem[];
    const int64_t blk = blockIdx.x;                             // one block per CTA
    if (p.lin_flag[blk]) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = p.n, X = p.lin_x;
    const float sl = sqrtf(p.lam2), isl = 1.f / sl;
    const float c_lo = p.diag->c_lo, c_hi = p.diag->c_hi;

    float *Ls = smem + C::OFF_L, *As = smem + C::OFF_A;
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem + C::OFF_TAB);
    float *wmax = smem + C::OFF_WMAX;
    float *lz = smem + C::OFF_LZ;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_TMEM);

    if (tid < C::NROT * 16) {
        const int r = tid >> 4, e = tid & 15;                            // table row = the rotation itself
        uint32_t v = 0;
        if (e < BPT) v = C::slot((uint32_t)e << 9, r);                   // T_i: butterfly bits above the thread index
        else if (e >= 8 && e < 8 + K) v = C::slot((uint32_t)(e - 8) << (C::QB - KB), r);   // T_j: the input's branch bits
        tab[tid] = v;
    }
    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tm = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    int hpos[BPT];                                                       // see bwd_alpha_kernel
#pragma unroll
    for (int i = 0; i < BPT; ++i) hpos[i] = beta_history_pos<KB>(i * CT + tid);

    const float *w_s = p.W + blk * n, *g_s = p.g + blk * n, *sf_s = p.soft + blk * n;
    float4 *hist4 = reinterpret_cast<float4 *>(p.hist + (size_t)blk * n * 2 * Q);
    int *aux = p.stepO + (size_t)blk * C::AUX_INTS;
    float4 *step = reinterpret_cast<float4 *>(smem + C::OFF_STEP);       // entry t - 1 belongs to step t
    const double isl_d = 1.0 / (double)sl;
    const int e_g = grad_scale(p.g_bits[blk], *p.g_top);
    const float down = grad_down(e_g);
    int outside = 0;
    for (int t = tid; t < n; t += CT) {
        const StepEnergy se = step_energy(__ldg(w_s + t), c_lo, c_hi, p.lam2);
        const float g = __ldg(g_s + t) * down, ws = se.wc * sl;
        step[t] = make_float4(ws, (se.wc + 2.f * se.delta) * sl, g * isl, lin_gs(g, ws, isl_d, __ldg(sf_s + t)));
        outside |= se.delta != 0.f;
    }
    if (tid == 0) { step[n] = make_float4(0.f, 0.f, 0.f, 0.f); aux[1] = -X; }
    const bool recentre = __syncthreads_or(outside) != 0;
    {
        const float a1 = pow2i(X), aa1 = step[0].w * a1;
        for (int q = tid; q < Q; q += CT) { Ls[q] = a1; As[q] = aa1; }
    }
#pragma unroll
    for (int i = 0; i < BPT; ++i) stage_codebook_scaled<C>(p.cb, i * CT + tid, tm + (uint32_t)(K * K * i), false, sl);
    tmem_wait_st();
    int O = -X, off = 0;
    compute_barrier(CT);
    auto alpha_sweep = [&](auto rc_tag) {
        constexpr bool RC = decltype(rc_tag)::value;
        int r = 0;                                                // k (t - 1) mod (Lb - k)
        for (int t = 1; t <= n; ++t) {
            const int cur = (t - 1) & 1;
            float2 cb[2][8];
            tmem_ld16(tm, cb[0]);
            const float4 sp = step[t - 1];
            const float gt = sp.z;
            if (t > 1) off = lin_offset(warp_max(lane < NWARP ? wmax[cur * 32 + lane] : 0.f), X);
            const float2 w2 = splat2(sp.x), v2 = splat2(sp.y), off2 = splat2((float)off), gsn2 = splat2(step[t].w);
            const uint32_t *tb = tab + r * 16;
            const uint32_t st = C::slot((uint32_t)tid, r);
            uint32_t TJ[K];
#pragma unroll
            for (int j = 0; j < K; ++j) TJ[j] = tb[8 + j] ^ st;
            float4 *hrow = hist4 + (size_t)(t - 1) * HSTEP;
            float tmax = 0.f;
#pragma unroll
            for (int i = 0; i < BPT; ++i) {
                const uint32_t ti = tb[i];
                float Lj[K], Aj[K];
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    Lj[j] = Ls[ti ^ TJ[j]];
                    Aj[j] = As[ti ^ TJ[j]];
                }
#pragma unroll
                for (int q = 0; q < K / 4; ++q) {
                    hrow[hpos[i] + q * HCH] = make_float4(Lj[4 * q], Lj[4 * q + 1], Lj[4 * q + 2], Lj[4 * q + 3]);
                    hrow[hpos[i] + (K / 4 + q) * HCH] = make_float4(Aj[4 * q], Aj[4 * q + 1], Aj[4 * q + 2], Aj[4 * q + 3]);
                }
                float2 outL[K / 2], outA[K / 2];
#pragma unroll
                for (int u = 0; u < UNITS; ++u) {
                    const int g = i * UNITS + u;
                    tmem_wait_ld(cb[g & 1]);
                    if (g + 1 < NU) tmem_ld16(tm + 16u * (g + 1), cb[(g + 1) & 1]);
#pragma unroll
                    for (int hh = 0; hh < HPU; ++hh) {
                        const int h = u * HPU + hh;
                        float2 sum, ax;
#pragma unroll
                        for (int j = 0; j < K; ++j) {
                            const float2 c2 = cb[g & 1][C::a_idx(j, hh)];
                            const float2 d = sub2(c2, w2);
                            const float2 e = ex2n2(fma2(d, RC ? sub2(c2, v2) : d, off2));
                            const float2 y = fma2(d, splat2(gt * Lj[j]), splat2(Aj[j]));
                            sum = j == 0 ? mul2(e, splat2(Lj[0])) : fma2(e, splat2(Lj[j]), sum);
                            ax = j == 0 ? mul2(e, y) : fma2(e, y, ax);
                        }
                        outL[h] = sum;
                        outA[h] = fma2(sum, gsn2, ax);
                        tmax = max3f(tmax, sum.x, sum.y);
                    }
                }
                // output [x|l] takes the place of input [l|x]
#pragma unroll
                for (int h = 0; h < K / 2; ++h) {
                    Ls[ti ^ TJ[2 * h]] = outL[h].x; Ls[ti ^ TJ[2 * h + 1]] = outL[h].y;
                    As[ti ^ TJ[2 * h]] = outA[h].x; As[ti ^ TJ[2 * h + 1]] = outA[h].y;
                }
            }
            tmax = warp_max(tmax);
            if (lane == 0) wmax[(cur ^ 1) * 32 + warp] = tmax;
            O += off;
            if (tid == 0) aux[t + 1] = O;
            r += KB; r = r >= C::QB ? r - C::QB : r;
            compute_barrier(CT);
        }
    };
    if (recentre) alpha_sweep(std::true_type{}); else alpha_sweep(std::false_type{});
    {
        float ssum = 0.f;
        for (int q = tid; q < Q; q += CT) ssum += Ls[q];
        ssum = warp_sum(ssum);
        if (lane == 0) lz[warp] = ssum;
        compute_barrier(CT);
    }
    const float Zs = warp_sum(lane < NWARP ? lz[lane] : 0.f);
    if (tid == 0) aux[n + 2] = __float_as_int(1.f / Zs);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

// Beta sweeps of the same blocks on clusters of two CTAs: bwd_skew_kernel<ACC, true> with linear messages.  The slots, their order,
// the two mbarriers per buffer and the history stream are described in bcjr_skew.cuh; what is gone is the gauge exchange
// (the offsets are the alpha sweep's), so "late" carries the last slot's outputs and the posterior sums only.
struct BetaLinCfg : SkewCfg {
    static constexpr int OFF_STEP = SkewCfg::OFF_O;             // float4 [MAX_N]: scaled weight, g, gs, gauge offset
    static constexpr int OFF_PART = OFF_STEP + 4 * MAX_N;       // [2][32][4]
    static constexpr int OFF_MBAR = OFF_PART + 256;
    static constexpr int OFF_TMEM = OFF_MBAR + 8;
    static constexpr int OFF_FLAG = OFF_TMEM + 2;
    static constexpr int OFF_SCALE = OFF_FLAG + 1;              // scale of the accumulators (kept here: the sweep has no register for it)
    static constexpr int OFF_PUSH = OFF_FLAG + 2;
    static constexpr int SMEM_FLOATS = OFF_PUSH + 2 * BPT * THREADS;
    static constexpr size_t SMEM_BYTES = (size_t)SMEM_FLOATS * 4;
    static_assert(OFF_STEP % 4 == 0 && OFF_MBAR % 2 == 0 && SMEM_BYTES <= 232448, "alignment, shared memory of an SM");
};

template <bool ACC>
__global__ void __launch_bounds__(SkewCfg::THREADS, 1) bwd_beta_lin_kernel(BwdParams p)
{
    using C = BetaLinCfg;
    constexpr int K = C::K, BPT = C::BPT, NWARP = C::NWARP, CT = C::THREADS;
    constexpr int CL = C::CL, SLOTS = C::SLOTS, NCH = C::NCH;
    constexpr uint32_t BUF_BYTES = (uint32_t)C::BUF * 4u;
    constexpr int PLANE = C::PLANE;
    constexpr uint32_t TX_EARLY = 3u * CT * 16u, TX_LATE = CT * 16u, TX_PART = SLOTS * 12u;
    constexpr int ORD_B0 = 2, ORD_B1 = 0, ORD_B2 = 3, ORD_B3 = 1;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const uint32_t cid = cluster_id_x(), ncl = cluster_count_x();
    const int n = p.n;
    const float invT = p.invT, sl = sqrtf(p.lam2), isl = 1.f / sl;
    const double isl_d = 1.0 / (double)sl;
    const float c_lo = p.diag->c_lo, c_hi = p.diag->c_hi;

    float *msg = smem + C::OFF_MSG;
    float4 *stage4 = reinterpret_cast<float4 *>(smem + C::OFF_RING);      // [BPT][NCH][CT], thread-private entries
    float4 *step = reinterpret_cast<float4 *>(smem + C::OFF_STEP);         // entry t - 1 belongs to step t
    float *part = smem + C::OFF_PART;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_FLAG);
    Proto pr{1u, abort_flag, p.diag};
    const uint32_t mb_early = smem_u32(smem + C::OFF_MBAR), mb_late = mb_early + 16u;   // [2] each, one per parity
    const uint32_t msg_u32 = smem_u32(msg), stage_u32 = smem_u32(stage4) + (uint32_t)tid * 16u;
    const uint32_t part_u32 = smem_u32(part);
    constexpr ptrdiff_t HSTEP = (ptrdiff_t)CL * BPT * NCH * CT;     // float4 per step

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(mb_early + 8u * s, 1 + NWARP); mbar_init(mb_late + 8u * s, 1 + SLOTS); }
        *abort_flag = 0;
        *reinterpret_cast<int *>(smem + C::OFF_SCALE) = GRAD_NONE;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    uint32_t phase = 0;            // bit b: parity to wait for on early[b]; bit 2 + b: on late[b]
    auto wait_early = [&](int b) { pr.wait(mb_early + 8u * b, (phase >> b) & 1u); phase ^= 1u << b; };
    auto wait_late = [&](int b) { pr.wait(mb_late + 8u * b, (phase >> (2 + b)) & 1u); phase ^= 4u << b; };

    const uint32_t tm_cb = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    const uint32_t tm_acc = tm_cb + 64u;
    const uint32_t peer = rank ^ 1u;
    const uint32_t peer_early = mapa_u32(mb_early, peer), peer_late = mapa_u32(mb_late, peer);
    const uint32_t late_rank0 = mapa_u32(mb_late, 0u);
    // where the outputs go: j = (rank, 0) [+8 KB for (rank, 1)] and j = (!rank, 0) [+4 KB for (!rank, 1)]
    uint32_t *pushtab = reinterpret_cast<uint32_t *>(smem + C::OFF_PUSH) + tid;
#pragma unroll
    for (int i = 0; i < BPT; ++i) {
        const int x = C::x_of((int)rank, tid, i);
        const int bin = x & 3;
        const int xl = ((int)rank << 11) | (x >> 2), xr = ((int)peer << 11) | (x >> 2);     // consumer butterflies of outputs j = (CTA, 0)
        pushtab[(2 * i) * CT] = msg_u32 + (uint32_t)(((bin >> 1) * PLANE + C::slot_of(xl) * CT + C::tid_of(xl)) * 4 + (bin & 1) * 2) * 4u;
        pushtab[(2 * i + 1) * CT] = mapa_u32(msg_u32 + (uint32_t)(((bin >> 1) * PLANE + C::slot_of(xr) * CT + C::tid_of(xr)) * 4 + (bin & 1) * 2) * 4u, peer);
    }
    constexpr uint32_t BL_STEP = CT * 16u, BR_STEP = 256u * 16u;     // j0 = 1: next slot (own CTA) / upper half of the threads (peer)
    const uint32_t part_dst = mapa_u32(part_u32 + (uint32_t)((int)rank * NWARP + warp) * 16u, 0u);
    auto zero_acc = [&]() {                                     // the accumulators (laid out like the beta-paired codebook)
        float2 z[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) z[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int g = 0; g < BPT; ++g) tmem_st16(tm_acc + 16u * g, z);
        tmem_wait_st();
    };
    if (ACC) zero_acc();
#pragma unroll
    for (int i = 0; i < BPT; ++i)                             // codebook -> TMEM, beta pairing: once per launch
        stage_codebook_scaled<C>(p.cb, C::x_of((int)rank, tid, i), tm_cb + (uint32_t)(16 * i), true, sl);
    tmem_wait_st();
    // test hook for the waits' abort path: one warp of CTA 0 withholds an arrival of its first block
    const bool drop_hook = blockIdx.x == 0 && warp == 1 && p.diag->drop_history_load != 0;
    float defect = 0.f;
    int *e_acc = reinterpret_cast<int *>(smem + C::OFF_SCALE);  // scale of the accumulators; the first block sets it
    // this cluster's partial of grad_codebook, added to what earlier launches left
    auto write_acc = [&]() {
        float *gc = p.gc_part + (size_t)cid * C::S;
        const float up = grad_up(*e_acc);
        tmem_wait_st();
#pragma unroll
        for (int i = 0; i < BPT; ++i) {
            const int x = C::x_of((int)rank, tid, i);
            float2 acc[8];
            tmem_ld16(tm_acc + 16u * i, acc);
            tmem_wait_ld(acc);
#pragma unroll
            for (int jh = 0; jh < K / 2; ++jh)
#pragma unroll
                for (int b = 0; b < K; ++b) {
                    gc[(size_t)(2 * jh) * C::Q + (size_t)x * K + b] += up * acc[C::b_idx(jh, b)].x;
                    gc[(size_t)(2 * jh + 1) * C::Q + (size_t)x * K + b] += up * acc[C::b_idx(jh, b)].y;
                }
        }
    };

    for (int64_t blk = cid; blk < p.B; blk += ncl) {
        if (p.lin_flag[blk]) continue;                        // both CTAs alike
        int ib = 0;
        bool dead = false;
        const float *w_s = p.W + blk * n, *g_s = p.g + blk * n, *sf_s = p.soft + blk * n;
        const float4 *hist4 = reinterpret_cast<const float4 *>(p.hist + (size_t)blk * n * 2 * C::Q) + tid;
        const int *aux = p.stepO + (size_t)blk * (C::MAX_N + 4);
        const int e_g = grad_scale(p.g_bits[blk], *p.g_top);
        const bool other = e_g != *e_acc;
        if (ACC && other && *e_acc != GRAD_NONE) { write_acc(); zero_acc(); }
        const float down = grad_down(e_g);
        int outside = 0;
        for (int t = tid; t < n; t += CT) {
            const StepEnergy se = step_energy(__ldg(w_s + t), c_lo, c_hi, p.lam2);
            const float g = __ldg(g_s + t) * down, ws = se.wc * sl;
            step[t] = make_float4(ws, g, lin_gs(g, ws, isl_d, __ldg(sf_s + t)), (float)(aux[t + 2] - aux[t + 1]));
            outside |= se.delta != 0.f;
        }
        const bool recentre = __syncthreads_or(outside) != 0;
        if (other && tid == 0) *e_acc = e_g;
        {
            const float m1 = __int_as_float(aux[n + 2]);         // M_n = 1 / Z, Bt_n = 0
            for (int f = tid; f < C::BUF; f += CT) msg[ib * C::BUF + f] = (f & 1) ? 0.f : m1;
        }
        // history stream: the four butterflies of step t are requested during step t + 1, each into its own staging slot
        const float4 *hsrc = hist4 + (size_t)(n - 1) * HSTEP + (size_t)rank * (BPT * NCH * CT);    // step being requested next
        auto issue_chunk = [&](int slot) {
            const uint32_t dst = stage_u32 + (uint32_t)slot * (uint32_t)(NCH * CT * 16);
#pragma unroll
            for (int q = 0; q < NCH; ++q)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(q * CT * 16)), "l"(hsrc + (slot * NCH + q) * CT) : "memory");
        };
#pragma unroll
        for (int i = 0; i < BPT; ++i) issue_chunk(i);           // the first step's butterflies
        asm volatile("cp.async.commit_group;" ::: "memory");
        cluster_sync();                                          // beta start
        // rank 0, last warp: turn the sums of step t (slots of parity b) into grad_W[t]
        auto finish_step = [&](int t, int b) {
            if (rank == 0 && warp == NWARP - 1) {
                const float *pp = part + (b * 32 + lane) * 4;
                float a0 = lane < SLOTS ? pp[0] : 0.f, a2 = lane < SLOTS ? pp[1] : 0.f, az = lane < SLOTS ? pp[2] : 0.f;
                a0 = warp_sum(a0); a2 = warp_sum(a2); az = warp_sum(az);
                if (lane == 0) {
                    const float i0 = grad_up(*e_acc) / a0;
                    p.gW[blk * n + t - 1] = (__ldg(g_s + t - 1) - az * i0) + (a2 * i0) * (__ldg(w_s + t - 1) - __ldg(sf_s + t - 1)) * invT;
                    defect = fmaxf(defect, fabsf(a0 - 1.f));
                }
            }
        };
        auto beta_sweep = [&](auto rc_tag) {
        constexpr bool RC = decltype(rc_tag)::value;
        for (int t = n; t >= 1 && !dead; --t) {
            const int ob = ib ^ 1;
            float2 cb[8];                                           // one set of table registers (see bcjr_skew.cuh)
            tmem_ld16(tm_cb + 16u * ORD_B0, cb);
            const float4 sp = step[t - 1];
            asm volatile("cp.async.wait_group 0;" ::: "memory");    // this step's history, requested during the previous step
            hsrc -= t > 1 ? HSTEP : 0;                              // next requests: step t - 1 (at t = 1: step 1 again, unread)
            if (t < n) wait_early(ib);
            if (!pr.warp_live()) { tmem_wait_ld(cb); dead = true; break; }
            const float4 *MBin = reinterpret_cast<const float4 *>(msg + ib * C::BUF);
            const uint32_t ob_off = (uint32_t)ob * BUF_BYTES, ob_mbar = 8u * ob;
            if (tid == 0) {
                mbar_expect_tx(mb_early + ob_mbar, TX_EARLY);
                mbar_expect_tx(mb_late + ob_mbar, rank == 0 ? TX_LATE + TX_PART : TX_LATE);
            }
            const float2 w2 = splat2(sp.x), off2 = splat2(sp.w), gd2 = splat2(sp.y * isl), g2 = splat2(sp.y), ni2 = splat2(-invT * isl), gs2 = splat2(sp.z);
            float2 v2 = w2, u2 = w2;                                // scaled weight + 2 delta, + delta
            if (RC) {
                const StepEnergy se = step_energy(__ldg(w_s + t - 1), c_lo, c_hi, p.lam2);
                v2 = splat2((se.wc + 2.f * se.delta) * sl); u2 = splat2((se.wc + se.delta) * sl);
            }
            float2 S0 = make_float2(0.f, 0.f), S2 = S0, ZS = S0;
#pragma unroll
            for (int pos = 0; pos < BPT; ++pos) {
                const int i = pos == 0 ? ORD_B0 : pos == 1 ? ORD_B1 : pos == 2 ? ORD_B2 : ORD_B3;
                const int inext = pos == 0 ? ORD_B1 : pos == 1 ? ORD_B2 : ORD_B3;
                const float4 l4 = stage4[(i * NCH) * CT + tid], a4 = stage4[(i * NCH + 1) * CT + tid];
                issue_chunk(i);                                     // this slot's entry for the next step (a whole step ahead)
                if (pos == BPT - 1) asm volatile("cp.async.commit_group;" ::: "memory");
                float Mb[K], Yb[K];
#pragma unroll
                for (int e = 0; e < K / 2; ++e) {
                    const float4 v = MBin[e * PLANE + i * CT + tid];
                    Mb[2 * e] = v.x; Yb[2 * e] = v.y; Mb[2 * e + 1] = v.z; Yb[2 * e + 1] = v.w;
                }
                float2 acc[8];
                tmem_wait_ld(cb);
                if (ACC) tmem_ld16(tm_acc + 16u * i, acc);
                bool acc_ready = !ACC;
                float2 outM[K / 2], outB[K / 2];
#pragma unroll
                for (int jh = 0; jh < K / 2; ++jh) {
                    const float2 A2 = jh == 0 ? make_float2(l4.x, l4.y) : make_float2(l4.z, l4.w);
                    const float2 AA2 = jh == 0 ? make_float2(a4.x, a4.y) : make_float2(a4.z, a4.w);
                    const float2 fg = mul2(A2, g2), nf = mul2(A2, ni2), nfA = mul2(AA2, ni2);
                    float2 sum, ya, zs;
#pragma unroll
                    for (int b = 0; b < K; ++b) {
                        const float2 c2 = cb[C::b_idx(jh, b)];
                        const float2 d = sub2(c2, w2);
                        const float2 e = ex2n2(fma2(d, RC ? sub2(c2, v2) : d, off2));
                        const float2 y = fma2(gd2, d, splat2(Yb[b]));                                  // h - gs + Bt
                        const float2 z = fma2(RC ? sub2(c2, u2) : d, fma2(nf, y, nfA), fg);            // A (g + (w - c) r / T)
                        const float2 pb = mul2(e, splat2(Mb[b]));
                        if (!acc_ready) { tmem_wait_ld(acc); acc_ready = true; }
                        sum = b == 0 ? pb : add2(sum, pb);
                        ya = b == 0 ? mul2(pb, y) : fma2(pb, y, ya);
                        zs = b == 0 ? mul2(pb, z) : fma2(pb, z, zs);
                        if (ACC) acc[C::b_idx(jh, b)] = fma2(pb, z, acc[C::b_idx(jh, b)]);
                    }
                    outM[jh] = sum;
                    outB[jh] = fma2(ya, rcpf2(make_float2(fmaxf(sum.x, 1e-37f), fmaxf(sum.y, 1e-37f))), gs2);
                    S0 = fma2(A2, sum, S0);
                    S2 = fma2(AA2, sum, fma2(A2, ya, S2));
                    ZS = add2(ZS, zs);
                }
                if (ACC) tmem_st16(tm_acc + 16u * i, acc);
                if (pos == 0) {
                    // everything of the previous step has arrived and every warp of the cluster is done with it: leave to
                    // overwrite the buffer that step read
                    if (t < n) {
                        wait_late(ib);
                        finish_step(t + 1, ib);
                    }
                    if (!pr.warp_live()) { dead = true; break; }
                }
                if (pos + 1 < BPT) tmem_ld16(tm_cb + 16u * inext, cb);
                // outputs j = 2 jh, 2 jh + 1 go to CTA jh: own CTA by plain stores, the peer by st.async
                const uint32_t mbp = (pos == BPT - 1 ? peer_late : peer_early) + ob_mbar;
#pragma unroll
                for (int jh = 0; jh < K / 2; ++jh) {
                    if (jh == (int)rank) {
                        const uint32_t pl = pushtab[(2 * i) * CT] + ob_off;
                        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(pl), "f"(outM[jh].x), "f"(outB[jh].x) : "memory");
                        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(pl + BL_STEP), "f"(outM[jh].y), "f"(outB[jh].y) : "memory");
                    } else {
                        const uint32_t prm = pushtab[(2 * i + 1) * CT] + ob_off;
                        st_async_v2(prm, outM[jh].x, outB[jh].x, mbp);
                        st_async_v2(prm + BR_STEP, outM[jh].y, outB[jh].y, mbp);
                    }
                }
                if (pos == BPT - 2) {                             // "early" also counts the local warps (its arrival count is fixed)
                    __syncwarp();
                    if (lane == 0) mbar_arrive_local(mb_early + ob_mbar);
                }
            }
            if (dead) { tmem_wait_ld(cb); break; }
            if (ACC) tmem_wait_st();
            __syncwarp();
            if (lane == 0 && !(drop_hook && t == n && blk == cid)) {   // this warp has read all its inputs and written its outputs
                mbar_arrive_local(mb_late + ob_mbar);
                mbar_arrive_remote(peer_late + ob_mbar);
            }
            // the posterior sums follow the arrival (see bwd_skew_kernel)
            const float s3 = warp_sum3_split(S0.x + S0.y, S2.x + S2.y, ZS.x + ZS.y, lane);
            if ((lane & 7) == 0 && lane < 24)
                st_async_f32(part_dst + (uint32_t)(ob * 128 + (lane >> 3)) * 4u, s3, late_rank0 + ob_mbar);
            ib = ob;
        }
        };
        if (recentre) beta_sweep(std::true_type{}); else beta_sweep(std::false_type{});
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (!dead) {
            wait_early(ib);
            wait_late(ib);                                       // the sums of step 1
            finish_step(1, ib);
        }
        cluster_sync();                                          // block end
    }
    if (ACC && *e_acc != GRAD_NONE) write_acc();
    if (tid == CT - 32 && rank == 0) diag_max(&p.diag->max_defect, defect);
    asm volatile("cp.async.wait_all;" ::: "memory");           // no copy may be in flight at exit (a warp may have left the loop early)
    tmem_wait_st();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();             // no CTA leaves while a peer may still address its shared memory
    if (*abort_flag) settle_after_abort();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

}  // namespace bcjr

// Vector-emission trellis (16 state bits, 4 bits and V = 2 weights per step) with LINEAR messages: the forward call on
// clusters of two CTAs, the backward call as an alpha kernel on clusters of two and a beta kernel on clusters of four.
// Certificate, gauge and range are those of bcjr_lin.cuh and bcjr_lin_bwd.cuh; ownership, message exchange, table layout and
// the blocks in flight those of bcjr_vec2.cuh and bcjr_vec4.cuh.  Blocks without a certificate are skipped by the backward
// kernels and run from the list by the log-domain kernels, in both directions.
//
// Per pair of states the log-domain forward step costs ten packed FP32 instructions and two exponentials in the alpha sweep,
// thirteen and two (and a second walk over the table) in the beta sweep; here it is five and eight, one walk each, and with the
// offsets known the beta sweep exchanges no gauge.  The backward sweeps: eleven and twenty before, nine and sixteen here.
// 592 blocks of 256 weights, T = 0.1: forward 4.50 -> 3.44 ms (XU 63 %, FMA 55 %, issue 55 % with packed instructions counted
// once), backward 9.90 -> 6.86 (alpha 2.1, beta 4.7 on 132 SMs: FMA 55 %, the rest dependency and shared-memory latency at four
// warps a scheduler); 16 blocks forward 0.67 -> 0.52 (before they were spread over the clusters 1.8).
// Without effect: an exponential in four on the FP32 pipe (forward 3.44 -> 3.62), two branches instead of two groups per register
// pair in the backward alpha sweep (0.98 -> 1.11 ms per 296), four blocks in flight in the beta kernel (7.0 -> 7.7), one set of table
// registers (6.67 -> 6.75).
#pragma once
#include "bcjr_vec2.cuh"
#include "bcjr_lin.cuh"

namespace bcjr {


// Alpha table: a pair of lanes holds two branches j, j + 1 of one group (in bcjr_vec2.cuh: one branch of two groups), so that
// the inputs A_j, A_{j+1} are a register pair as loaded and need no copies.  Group g of the thread at columns 32 g, pair jp = j / 2
// as (c_j.x, c_{j+1}.x), (c_j.y, c_{j+1}.y) at 4 jp.
__device__ __forceinline__ void vec_stage_alpha(uint32_t tm, const float *src, int q0, float scale)
{
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float2 v[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int j = 8 * u + 2 * e;
                const float2 a = __ldg(reinterpret_cast<const float2 *>(src) + (size_t)j * 4096 + q0 + g);
                const float2 b = __ldg(reinterpret_cast<const float2 *>(src) + (size_t)(j + 1) * 4096 + q0 + g);
                v[2 * e] = make_float2(scale * a.x, scale * b.x);
                v[2 * e + 1] = make_float2(scale * a.y, scale * b.y);
            }
            tmem_st16(tm + 32u * g + 16u * u, v);
        }
    tmem_wait_st();
}

// Beta messages of a CTA are kept as [b >> 1][x >> 1][b & 1][x & 1] here: a consumer's float4 is the pairs (M(x,b), M(x+1,b)),
// (M(x,b+1), M(x+1,b+1)), x even.  A producer holds (x', b'), (x', b' + 1), b' even, and lane ^ 8 the same of x' ^ 1: after one
// exchange the lane of even x' has the pair of b', the other that of b' + 1.
__device__ __forceinline__ float2 vec_pair_x(float2 v, int lane)
{
    const bool odd = lane & 8;
    const float got = __shfl_xor_sync(0xffffffffu, odd ? v.x : v.y, 8);
    return odd ? make_float2(got, v.y) : make_float2(v.x, got);
}

// byte offset of that pair in its consumer, which keeps xn values of x
__device__ __forceinline__ uint32_t vec_beta_dst(int q, int xn, int lane)
{
    const int x = (q >> 4) & (xn - 1), b = (q & 15) + ((lane >> 3) & 1);      // q & 15 is even
    return (uint32_t)((b >> 1) * 2 * xn + (x >> 1) * 4 + (b & 1) * 2) * 4u;
}

// soft_v(t) = w_v + (sum gamma d_v) / sqrt(lam2): the table and the weights are staged scaled (see bcjr_lin.cuh)
template <int NBLK_>
__global__ void __launch_bounds__(Vec2Cfg<NBLK_>::THREADS, 1) fwd_vec_lin_kernel(FwdParams p)
{
    using C = Vec2Cfg<NBLK_>;
    constexpr int K = C::K, Q = C::Q, QC = C::QC, CL = C::CL, NWARP = C::NWARP, NBUF = C::NBUF, SLOTS = C::SLOTS, CT = C::THREADS;
    constexpr int NBLK = C::NBLK, OSTR = C::MAX_NT + 4, PP = C::PP;
    constexpr uint32_t TX_ALPHA = QC * 4u + SLOTS * 4u;          // half of the messages + gauge slots
    constexpr uint32_t TX_BETA = QC * 4u, TX_PART = SLOTS * 16u; // half of the messages; posterior sums (rank 0 only)
    if (lin_given_up(p)) return;                                 // (every CTA alike)
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const uint32_t cid = cluster_id_x(), ncl = cluster_count_x();
    const int n = p.n, nt = n / C::V, X = p.lin_x;
    const float sl = sqrtf(p.lam2);
    const double isl_d = 1.0 / (double)sl;
    const VecRange range = vec_range<NBLK>(p.B, cid, ncl);

    float *msg = smem + C::OFF_MSG;
    float *w_s = smem + C::OFF_W;
    float *off_s = smem + C::OFF_O;                              // [NBLK][OSTR]: gauge offset of step t
    float *wmax = smem + C::OFF_WMAX;
    float *part = smem + C::OFF_PART;
    float *lz = smem + C::OFF_LZ;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_FLAG);
    Proto pr{1u, abort_flag, p.diag};
    const uint32_t mbar_full = smem_u32(smem + C::OFF_MBAR);     // [NBUF][NBLK]
    const uint32_t msg_u32 = smem_u32(msg), wmax_u32 = smem_u32(wmax), part_u32 = smem_u32(part), lz_u32 = smem_u32(lz);

    const int q0 = C::alpha_q0((int)rank, tid);                  // alpha sweep: this thread's groups q0 .. q0 + 3
    const int q0b = C::beta_q0((int)rank, warp, lane, 0);        // beta sweep: groups q0b, q0b + 1 and q0b + 256, q0b + 257
    float *hist = p.hist + (size_t)cid * NBLK * nt * Q;          // [NBLK][nt][Q]: row t = A_{t+1}

    // this warp's slots for the gauge maximum (and the sums of Z): lane r sends to CTA r
    const uint32_t wmax_dst = mapa_u32(wmax_u32 + (uint32_t)((int)rank * NWARP + warp) * 4u, (uint32_t)(lane & (CL - 1)));
    const uint32_t wmax_mbar = mapa_u32(mbar_full, (uint32_t)(lane & (CL - 1)));
    const uint32_t part_dst = mapa_u32(part_u32 + (uint32_t)((int)rank * NWARP + warp) * 16u, 0u);
    const int ra = C::alpha_dst_rank(q0);
    const uint32_t push_a = mapa_u32(msg_u32, (uint32_t)ra) + (uint32_t)C::alpha_dst_off(q0) * 4u;
    const uint32_t push_a_mbar = mapa_u32(mbar_full, (uint32_t)ra);
    const int rb = C::beta_dst_rank(q0b);                        // the same for the thread's second pair
    const uint32_t push_b = mapa_u32(msg_u32, (uint32_t)rb) + vec_beta_dst(q0b, 128, lane);
    constexpr uint32_t PUSH_B_PAIR = (uint32_t)(C::beta_dst_off(256) - C::beta_dst_off(0)) * 4u;   // second pair: j + 1
    const uint32_t push_b_mbar = mapa_u32(mbar_full, (uint32_t)rb);
    const uint32_t part_mbar = mapa_u32(mbar_full, 0u);

    if (tid == 0) {
        for (int s = 0; s < NBUF * NBLK; ++s) mbar_init(mbar_full + 8u * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tm = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    uint32_t full_phase = 0;       // bit (b * NBLK + k) = parity to wait for on full[b][k]
    int ib = 0;
    float defect = 0.f, zgap = 0.f;
    auto wait_inputs = [&](int b, int k) {
        const int s = b * NBLK + k;
        pr.wait(mbar_full + 8u * s, (full_phase >> s) & 1u);
        full_phase ^= 1u << s;
    };


    int left = range.count;
    for (int64_t base = range.begin; left > 0; base += range.depth, left -= range.depth) {
        const int nact = left < range.depth ? left : range.depth;      // blocks in flight in this batch
        for (int k = 0; k < nact; ++k) {
            const float *w = p.W + (base + k) * n;
            for (int t = tid; t < n; t += CT) w_s[k * C::MAX_N + t] = __ldg(w + t) * sl;
            for (int q = tid; q < QC; q += CT) msg[(ib * NBLK + k) * QC + q] = pow2i(X);     // A_1 = 1 = 2^X 2^O_1
        }
        vec_stage_alpha(tm, p.cb, q0, sl);
        cluster_sync();
        // ================= alpha sweep: step t maps A_t to A_{t+1}
        for (int t = 1; t <= nt; ++t) {
            const int ob = ib == NBUF - 1 ? 0 : ib + 1;
#pragma unroll
            for (int k = 0; k < NBLK; ++k) {
                if (k < nact) {
                    const int si = ib * NBLK + k, so = ob * NBLK + k;
                    // the first table unit and the step's weights do not depend on the step's inputs: requested before the wait
                    float2 cb[2][8];
                    tmem_ld16(tm, cb[0]);
                    const float *wk = w_s + k * C::MAX_N + 2 * (t - 1);
                    const float2 wx = splat2(wk[0]), wy = splat2(wk[1]);
                    int off = 0;
                    if (t > 1) {
                        wait_inputs(ib, k);
                        off = lin_offset(warp_max(wmax[si * SLOTS + lane]), X);
                    }
                    const float *Lin = msg + si * QC + C::alpha_in(tid);      // [j][x & 127]
                    if (tid == 0) pr.expect_tx(mbar_full + 8u * so, TX_ALPHA);
                    float2 A2[K / 2], in = make_float2(0.f, 0.f);             // inputs 2 jp, 2 jp + 1
#pragma unroll
                    for (int jp = 0; jp < K / 2; ++jp) { A2[jp] = make_float2(Lin[256 * jp], Lin[256 * jp + 128]); in = add2(in, A2[jp]); }
                    const float2 floor2 = make_float2(lin_floor(in.x + in.y), 0.f), off2 = splat2((float)off);
                    float out[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        float2 sum = floor2;
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int c = 2 * g + u;
                            tmem_wait_ld(cb[c & 1]);
                            if (c + 1 < 8) tmem_ld16(tm + 16u * (c + 1), cb[(c + 1) & 1]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 dx = sub2(cb[c & 1][2 * e], wx), dy = sub2(cb[c & 1][2 * e + 1], wy);
                                sum = fma2(ex2n2(fma2(dy, dy, fma2(dx, dx, off2))), A2[4 * u + e], sum);
                            }
                        }
                        out[g] = sum.x + sum.y;
                    }
                    float tmax = fmaxf(fmaxf(out[0], out[1]), fmaxf(out[2], out[3]));
                    pr.async_v4(push_a + (uint32_t)(so * QC) * 4u, out[0], out[1], out[2], out[3], push_a_mbar + 8u * so);
                    if (t < nt) *reinterpret_cast<float4 *>(hist + ((size_t)k * nt + t) * Q + q0) = make_float4(out[0], out[1], out[2], out[3]);
                    tmax = warp_max(tmax);
                    if (lane < CL) pr.async_f32(wmax_dst + (uint32_t)(so * SLOTS) * 4u, tmax, wmax_mbar + 8u * so);
                    if (tid == 0) off_s[k * OSTR + t] = (float)off;
                }
            }
            ib = ob;
        }
        // ================= Z = 2^O_{nt+1} sum_q A_{nt+1}(q), each CTA sums the half it holds
#pragma unroll
        for (int k = 0; k < NBLK; ++k) {
            if (k < nact) {
                wait_inputs(ib, k);
                const float *Afin = msg + (ib * NBLK + k) * QC;
                float ssum = 0.f;
                for (int e = tid; e < QC; e += CT) ssum += Afin[e];
                ssum = warp_sum(ssum);
                if (lane < CL) st_cluster_f32(mapa_u32(lz_u32 + (uint32_t)(k * SLOTS + (int)rank * NWARP + warp) * 4u, (uint32_t)lane), ssum);
            }
        }
        cluster_sync();
        bool bad = false;                                        // warp k: block base + k gets no certificate
#pragma unroll
        for (int k = 0; k < NBLK; ++k) {
            if (k < nact) {
                const float Zs = warp_sum(lz[k * SLOTS + lane]);
                const bool ok = Zs > 1e-37f && Zs < 1e37f;       // else not representable (or not finite)
                if (warp == k) bad = !ok;
                if (ok && warp == k && rank == 0 && p.logZ) {    // (of a block that turns out bad later it is written again)
                    float O = 0.f;                               // whole numbers below 2^24: exact
                    for (int t = 1 + lane; t <= nt; t += 32) O += off_s[k * OSTR + t];
                    const int ez = exp2i(Zs);
                    O = warp_sum(O) + (float)(ez - X);
                    if (lane == 0) p.logZ[base + k] = (float)(((double)O + (double)lg2f(Zs * pow2i(-ez))) * 0.6931471805599453);
                }
                // messages M_t 2^(O_{t+1} - O_{nt+1}) / Zs: the posterior weight is the product A_t M
                for (int q = tid; q < QC; q += CT) msg[(ib * NBLK + k) * QC + q] = 1.f / Zs;
            }
        }
        // ================= beta sweep: step t maps M_t to M_{t-1}
#pragma unroll
        for (int pp = 0; pp < PP; ++pp) vec4_stage_table(tm + 64u * pp, p.cb_beta, q0b + 256 * pp, sl);
        // history of the posterior, requested one turn (block and step) ahead; A_1 is constant
        auto load_history = [&](int t, int k, float2 *L) {
#pragma unroll
            for (int pp = 0; pp < PP; ++pp)
                L[pp] = t > 1 ? __ldcg(reinterpret_cast<const float2 *>(hist + ((size_t)k * nt + t - 1) * Q + q0b + 256 * pp)) : splat2(pow2i(X));
        };
        float2 Ls[PP];
        load_history(nt, 0, Ls);
        float bdef = 0.f, den1 = 1.f;
        cluster_sync();
        // rank 0, warp k: turn the sums of step t of block k (slots of buffer b) into soft[t], which takes the place of the step's weights
        // (every warp has read those) until the block has its certificate
        auto finish_step = [&](int t, int b, int k) {
            if (rank == 0 && warp == k) {
                const float4 s4 = *reinterpret_cast<const float4 *>(part + (size_t)((b * NBLK + k) * SLOTS + lane) * 4);
                const float den = warp_sum(s4.x), n0 = warp_sum(s4.y), n1 = warp_sum(s4.z);
                if (lane == 0) {
                    float *wk = w_s + k * C::MAX_N + 2 * (t - 1);
                    const float s0 = (float)(((double)wk[0] + (double)(n0 / den)) * isl_d), s1 = (float)(((double)wk[1] + (double)(n1 / den)) * isl_d);
                    *reinterpret_cast<float2 *>(wk) = make_float2(s0, s1);
                    bdef = fmaxf(bdef, fabsf(den - 1.f));
                    bad |= !(fabsf(den - 1.f) <= LIN_DEFECT);
                    den1 = den;
                }
            }
        };
        for (int t = nt; t >= 1; --t) {
            const int ob = ib == NBUF - 1 ? 0 : ib + 1;
#pragma unroll
            for (int k = 0; k < NBLK; ++k) {
                if (k < nact) {
                    const int si = ib * NBLK + k, so = ob * NBLK + k;
                    float2 cb[2][8];
                    tmem_ld16(tm, cb[0]);                                     // requested before the wait for the step's inputs
                    const float *wk = w_s + k * C::MAX_N + 2 * (t - 1);
                    const float2 wx = splat2(wk[0]), wy = splat2(wk[1]), off2 = splat2(off_s[k * OSTR + t]);
                    if (t < nt) {
                        wait_inputs(ib, k);
                        finish_step(t + 1, ib, k);
                    }
                    const float *Min = msg + si * QC + C::beta_in(warp, lane);   // [b >> 1][x >> 1][b & 1][x & 1], x = 2 xp
                    if (tid == 0) pr.expect_tx(mbar_full + 8u * so, rank == 0 ? TX_BETA + TX_PART : TX_BETA);
                    float2 Ls_next[PP];
                    if (k + 1 < nact) load_history(t, k + 1, Ls_next); else load_history(t - 1, 0, Ls_next);
                    float2 fd = make_float2(0.f, 0.f), fx = fd, fy = fd;
#pragma unroll
                    for (int pp = 0; pp < PP; ++pp) {
                        float2 sum = make_float2(0.f, 0.f), cx = sum, cy = sum;
#pragma unroll
                        for (int un = 0; un < C::UNITS; ++un) {
                            const int g = pp * C::UNITS + un;
                            tmem_wait_ld(cb[g & 1]);
                            if (g + 1 < PP * C::UNITS) tmem_ld16(tm + 16u * (g + 1), cb[(g + 1) & 1]);
#pragma unroll
                            for (int e = 0; e < 4; e += 2) {
                                const int b = 4 * un + e;
                                const float4 Mv = *reinterpret_cast<const float4 *>(Min + 256 * (b >> 1));   // M(x,b), M(x+1,b), M(x,b+1), M(x+1,b+1)
#pragma unroll
                                for (int bb = 0; bb < 2; ++bb) {
                                    const float2 dx = sub2(cb[g & 1][2 * (e + bb)], wx), dy = sub2(cb[g & 1][2 * (e + bb) + 1], wy);
                                    const float2 ex = ex2n2(fma2(dy, dy, fma2(dx, dx, off2)));
                                    const float2 pb = mul2(ex, bb == 0 ? make_float2(Mv.x, Mv.y) : make_float2(Mv.z, Mv.w));
                                    sum = add2(sum, pb);
                                    cx = fma2(pb, dx, cx);
                                    cy = fma2(pb, dy, cy);
                                }
                            }
                        }
                        const float2 px = vec_pair_x(sum, lane);
                        pr.async_v2(push_b + PUSH_B_PAIR * pp + (uint32_t)(so * QC) * 4u, px.x, px.y, push_b_mbar + 8u * so);
                        fd = fma2(Ls[pp], sum, fd); fx = fma2(Ls[pp], cx, fx); fy = fma2(Ls[pp], cy, fy);
                        Ls[pp] = Ls_next[pp];
                    }
                    const float s3 = warp_sum3_split(fd.x + fd.y, fx.x + fx.y, fy.x + fy.y, lane);   // lanes 0, 8, 16: den, num_0, num_1
                    if ((lane & 7) == 0) pr.async_f32(part_dst + (uint32_t)(so * SLOTS * 4 + (lane >> 3)) * 4u, lane < 24 ? s3 : 0.f, part_mbar + 8u * so);
                }
            }
            ib = ob;
        }
        // ================= the sums of step 1 (A_1 is constant: they are the beta side's Z)
#pragma unroll
        for (int k = 0; k < NBLK; ++k) {
            if (k < nact) {
                wait_inputs(ib, k);
                finish_step(1, ib, k);
            }
        }
        if (rank == 0 && warp < nact) {
            bad = __shfl_sync(0xffffffffu, (int)bad, 0) != 0;
            __syncwarp();
            if (lane == 0) p.lin_flag[base + warp] = bad ? 1 : 0;
            if (!bad) {
                if (lane == 0) {
                    defect = fmaxf(defect, bdef);
                    zgap = fmaxf(zgap, fabsf(lg2f(den1)));
                }
                const float2 *sw = reinterpret_cast<const float2 *>(w_s + warp * C::MAX_N);
                for (int t = lane; t < nt; t += 32) {             // (soft may be W)
                    reinterpret_cast<float2 *>(p.soft + (base + warp) * n)[t] = sw[t];
                    if (p.soft_copy) reinterpret_cast<float2 *>(p.soft_copy + (base + warp) * n)[t] = sw[t];
                }
            }
        }
        cluster_sync();         // nobody still reads this batch's buffers when the next batch starts
    }
    if (rank == 0 && lane == 0 && warp < NBLK) {
        diag_max(&p.diag->max_defect, defect);
        diag_max(&p.diag->max_logz_gap, zgap);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();             // no CTA leaves while a peer may still address its shared memory
    if (*abort_flag) settle_after_abort();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

// --------------------------------------------------------------------------------------
// Backward call.  The alpha sweep carries A and AA = A (At + gs), the beta sweep M and Bt (bcjr_lin_bwd.cuh), with
//     h_t = sum_v g_v (c_v - soft_v) = sum_v (g_v / sl) d_v + gs_t,     gs_t = sum_v g_v (w_v - soft_v).
// Two kernels because they want different clusters: the alpha sweep needs the table alone (two CTAs, all 148 SMs), the beta
// sweep the gradient accumulators next to it (four).  What passes between them is the history, one float4
// (A, A', AA, AA') per pair of adjacent groups and step: 4 MB a block of 256 weights.
// --------------------------------------------------------------------------------------
template <int NBLK_>
struct VecAlphaLinCfg {
    using F = Vec2Cfg<NBLK_>;
    static constexpr int NBUF = F::NBUF, NBLK = NBLK_, QC = F::QC, SLOTS = F::SLOTS;
    static constexpr int MAX_N = 512, MAX_NT = MAX_N / 2, AUX_INTS = MAX_NT + 4;   // aux of a block: 1 / Z, then the offset of every step
    static constexpr int OFF_MSG = 0;                                  // [NBUF][NBLK][2][QC]: A, AA
    static constexpr int OFF_STEP = OFF_MSG + NBUF * NBLK * 2 * QC;    // float4 [NBLK][MAX_NT]: scaled weights, g / sl
    static constexpr int OFF_GS = OFF_STEP + NBLK * MAX_NT * 4;        // [NBLK][MAX_NT + 4]
    static constexpr int OFF_WMAX = OFF_GS + NBLK * (MAX_NT + 4);      // [NBUF][NBLK][SLOTS]
    static constexpr int OFF_LZ = OFF_WMAX + NBUF * NBLK * SLOTS;      // [NBLK][SLOTS]
    static constexpr int OFF_MBAR = OFF_LZ + NBLK * SLOTS;             // uint64 [NBUF][NBLK]
    static constexpr int OFF_TMEM = OFF_MBAR + 2 * NBUF * NBLK + 2;
    static constexpr int OFF_FLAG = OFF_TMEM + 2;
    static constexpr size_t SMEM_BYTES = (size_t)(OFF_FLAG + 4) * 4;
    static_assert(OFF_STEP % 4 == 0 && OFF_MBAR % 2 == 0 && SMEM_BYTES <= 232448, "alignment, shared memory of one CTA");
};

// gs of a step: centred on the scaled weights (lin_gs)
__device__ __forceinline__ float vec_gs(float gx, float gy, float wxs, float wys, double isl, float sx, float sy)
{
    return (float)((double)gx * ((double)wxs * isl - (double)sx) + (double)gy * ((double)wys * isl - (double)sy));
}

// the certified ones of the blocks base .. base + count - 1, as a mask
template <int NBLK>
__device__ __forceinline__ uint32_t vec_live(const uint8_t *flag, int64_t base, int count)
{
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < NBLK; ++k)
        if (k < count && !__ldg(flag + base + k)) m |= 1u << k;
    return m;
}

template <int NBLK_>
__global__ void __launch_bounds__(Vec2Cfg<NBLK_>::THREADS, 1) bwd_vec_alpha_lin_kernel(BwdParams p)
{
    using C = Vec2Cfg<NBLK_>;
    using D = VecAlphaLinCfg<NBLK_>;
    constexpr int K = C::K, Q = C::Q, QC = C::QC, CL = C::CL, NWARP = C::NWARP, NBUF = C::NBUF, SLOTS = C::SLOTS, CT = C::THREADS;
    constexpr int NBLK = C::NBLK, PP = C::PP, MAX_NT = D::MAX_NT, GSTR = D::MAX_NT + 4;
    constexpr uint32_t TX = 2u * QC * 4u + SLOTS * 4u;           // half of both message arrays + gauge slots
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const uint32_t cid = cluster_id_x(), ncl = cluster_count_x();
    const int n = p.n, nt = n / 2, X = p.lin_x;
    const float sl = sqrtf(p.lam2), isl = 1.f / sl;
    const double isl_d = 1.0 / (double)sl;
    const VecRange range = vec_range<NBLK>(p.B, cid, ncl);

    float *msg = smem + D::OFF_MSG;
    float4 *step = reinterpret_cast<float4 *>(smem + D::OFF_STEP);     // entry t - 1 belongs to step t
    float *gs_s = smem + D::OFF_GS;
    float *wmax = smem + D::OFF_WMAX;
    float *lz = smem + D::OFF_LZ;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + D::OFF_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + D::OFF_FLAG);
    Proto pr{1u, abort_flag, p.diag};
    const uint32_t mbar_full = smem_u32(smem + D::OFF_MBAR);     // [NBUF][NBLK]
    const uint32_t msg_u32 = smem_u32(msg), wmax_u32 = smem_u32(wmax), lz_u32 = smem_u32(lz);
    const int q0 = C::alpha_q0((int)rank, tid);                  // this thread's groups q0 .. q0 + 3
    float4 *hist = reinterpret_cast<float4 *>(p.hist) + q0 / 2;  // + (block nt + t - 1) Q / 2

    // this warp's slots for the gauge maximum (and the sums of Z): lane r sends to CTA r
    const uint32_t wmax_dst = mapa_u32(wmax_u32 + (uint32_t)((int)rank * NWARP + warp) * 4u, (uint32_t)(lane & (CL - 1)));
    const uint32_t wmax_mbar = mapa_u32(mbar_full, (uint32_t)(lane & (CL - 1)));
    const int ra = C::alpha_dst_rank(q0);
    const uint32_t push_a = mapa_u32(msg_u32, (uint32_t)ra) + (uint32_t)C::alpha_dst_off(q0) * 4u;
    const uint32_t push_a_mbar = mapa_u32(mbar_full, (uint32_t)ra);

    if (tid == 0) {
        for (int s = 0; s < NBUF * NBLK; ++s) mbar_init(mbar_full + 8u * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tm = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) vec4_stage_table(tm + 64u * pp, p.cb, q0 + 2 * pp, sl);
    uint32_t full_phase = 0;       // bit (b * NBLK + k) = parity to wait for on full[b][k]
    int ib = 0;
    auto wait_inputs = [&](int b, int k) {
        const int s = b * NBLK + k;
        pr.wait(mbar_full + 8u * s, (full_phase >> s) & 1u);
        full_phase ^= 1u << s;
    };

    int left = range.count;
    for (int64_t base = range.begin; left > 0; base += range.depth, left -= range.depth) {
        const uint32_t live = vec_live<NBLK>(p.lin_flag, base, left < range.depth ? left : range.depth);   // both CTAs alike
        if (live == 0) continue;
        for (int k = 0; k < range.depth; ++k) {
            if (!((live >> k) & 1u)) continue;
            const float2 *w = reinterpret_cast<const float2 *>(p.W + (base + k) * n), *g = reinterpret_cast<const float2 *>(p.g + (base + k) * n);
            const float2 *sf = reinterpret_cast<const float2 *>(p.soft + (base + k) * n);
            const float down = grad_down(grad_scale(p.g_bits[base + k], *p.g_top));
            for (int t = tid; t < nt; t += CT) {
                const float2 wt = __ldg(w + t), st = __ldg(sf + t);
                float2 gt = __ldg(g + t);
                gt.x *= down; gt.y *= down;
                step[k * MAX_NT + t] = make_float4(wt.x * sl, wt.y * sl, gt.x * isl, gt.y * isl);
                gs_s[k * GSTR + t] = vec_gs(gt.x, gt.y, wt.x * sl, wt.y * sl, isl_d, st.x, st.y);
            }
            if (tid == 0) gs_s[k * GSTR + nt] = 0.f;
        }
        __syncthreads();
        for (int k = 0; k < range.depth; ++k) {
            if (!((live >> k) & 1u)) continue;
            const float a1 = pow2i(X), aa1 = gs_s[k * GSTR] * a1;             // A_1 = 1 = 2^X 2^O_1
            float *m0 = msg + (size_t)(ib * NBLK + k) * 2 * QC;
            for (int q = tid; q < QC; q += CT) { m0[q] = a1; m0[QC + q] = aa1; }
            float4 *h = hist + (size_t)(base + k) * nt * (Q / 2);
            h[0] = h[1] = make_float4(a1, a1, aa1, aa1);
        }
        cluster_sync();
        for (int t = 1; t <= nt; ++t) {
            const int ob = ib == NBUF - 1 ? 0 : ib + 1;
#pragma unroll
            for (int k = 0; k < NBLK; ++k) {
                if ((live >> k) & 1u) {
                    const int si = ib * NBLK + k, so = ob * NBLK + k;
                    float2 cb[2][8];
                    tmem_ld16(tm, cb[0]);                        // requested before the wait for the step's inputs
                    const float4 sp = step[k * MAX_NT + t - 1];
                    const float2 wx = splat2(sp.x), wy = splat2(sp.y), gx = splat2(sp.z), gy = splat2(sp.w);
                    const float2 gsn = splat2(gs_s[k * GSTR + t]);
                    int off = 0;
                    if (t > 1) {
                        wait_inputs(ib, k);
                        off = lin_offset(warp_max(wmax[si * SLOTS + lane]), X);
                    }
                    const float *Lin = msg + (size_t)si * 2 * QC + C::alpha_in(tid), *Ain = Lin + QC;      // [j][x & 127]
                    if (tid == 0) pr.expect_tx(mbar_full + 8u * so, TX);
                    const float2 off2 = splat2((float)off);
                    float Lj[K], Aj[K];
#pragma unroll
                    for (int j = 0; j < K; ++j) { Lj[j] = Lin[128 * j]; Aj[j] = Ain[128 * j]; }
                    float2 outL[PP], outA[PP];
                    float tmax = 0.f;
#pragma unroll
                    for (int pp = 0; pp < PP; ++pp) {
                        float2 sum = make_float2(0.f, 0.f), ax = sum;
#pragma unroll
                        for (int u = 0; u < C::UNITS; ++u) {
                            const int g = pp * C::UNITS + u;
                            tmem_wait_ld(cb[g & 1]);
                            if (g + 1 < PP * C::UNITS) tmem_ld16(tm + 16u * (g + 1), cb[(g + 1) & 1]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int j = 4 * u + e;
                                const float2 dx = sub2(cb[g & 1][2 * e], wx), dy = sub2(cb[g & 1][2 * e + 1], wy);
                                const float2 ex = ex2n2(fma2(dy, dy, fma2(dx, dx, off2)));
                                const float2 y = fma2(fma2(gx, dx, mul2(gy, dy)), splat2(Lj[j]), splat2(Aj[j]));
                                sum = fma2(ex, splat2(Lj[j]), sum);
                                ax = fma2(ex, y, ax);
                            }
                        }
                        outL[pp] = sum;
                        outA[pp] = fma2(sum, gsn, ax);
                        tmax = max3f(tmax, sum.x, sum.y);
                    }
                    const uint32_t dst = push_a + (uint32_t)(so * 2 * QC) * 4u;
                    pr.async_v4(dst, outL[0].x, outL[0].y, outL[1].x, outL[1].y, push_a_mbar + 8u * so);
                    pr.async_v4(dst + QC * 4u, outA[0].x, outA[0].y, outA[1].x, outA[1].y, push_a_mbar + 8u * so);
                    if (t < nt) {
                        float4 *h = hist + ((size_t)(base + k) * nt + t) * (Q / 2);
                        h[0] = make_float4(outL[0].x, outL[0].y, outA[0].x, outA[0].y);
                        h[1] = make_float4(outL[1].x, outL[1].y, outA[1].x, outA[1].y);
                    }
                    tmax = warp_max(tmax);
                    if (lane < CL) pr.async_f32(wmax_dst + (uint32_t)(so * SLOTS) * 4u, tmax, wmax_mbar + 8u * so);
                    if (tid == 0 && rank == 0) p.stepO[(size_t)(base + k) * D::AUX_INTS + t] = off;
                }
            }
            ib = ob;
        }
#pragma unroll
        for (int k = 0; k < NBLK; ++k) {
            if ((live >> k) & 1u) {
                wait_inputs(ib, k);
                const float *Afin = msg + (size_t)(ib * NBLK + k) * 2 * QC;
                float ssum = 0.f;
                for (int e = tid; e < QC; e += CT) ssum += Afin[e];
                ssum = warp_sum(ssum);
                if (lane < CL) st_cluster_f32(mapa_u32(lz_u32 + (uint32_t)(k * SLOTS + (int)rank * NWARP + warp) * 4u, (uint32_t)lane), ssum);
            }
        }
        cluster_sync();         // and nobody still reads this batch's buffers when the next batch starts
        if (rank == 0 && warp < NBLK && ((live >> warp) & 1u)) {
            const float Zs = warp_sum(lz[warp * SLOTS + lane]);
            if (lane == 0) p.stepO[(size_t)(base + warp) * D::AUX_INTS] = __float_as_int(1.f / Zs);
        }
        cluster_sync();         // nor the sums
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();             // no CTA leaves while a peer may still address its shared memory
    if (*abort_flag) settle_after_abort();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

template <int NBLK_>
struct VecBetaLinCfg {
    using F = Vec4Cfg<NBLK_>;
    static constexpr int Q = F::Q, QC = F::QC, CL = F::CL, THREADS = F::THREADS, NWARP = F::NWARP, SLOTS = F::SLOTS, K = F::K, S = F::S;
    static constexpr int NBUF = 3, NBLK = NBLK_, UNITS = 4;
    static constexpr int MAX_N = 512, MAX_NT = MAX_N / 2;
    static constexpr int OFF_MSG = 0;                                  // [NBUF][NBLK][2][QC]: M, Bt
    static constexpr int OFF_STEP = OFF_MSG + NBUF * NBLK * 2 * QC;    // float4 [NBLK][MAX_NT]: scaled weights, g
    static constexpr int OFF_GS = OFF_STEP + NBLK * MAX_NT * 4;        // float2 [NBLK][MAX_NT]: gs, gauge offset
    static constexpr int OFF_PART = OFF_GS + NBLK * MAX_NT * 2;        // [NBUF][NBLK][64][4]: S0, S2, ZS_0, ZS_1
    static constexpr int OFF_MBAR = OFF_PART + NBUF * NBLK * 64 * 4;   // uint64 [NBUF][NBLK]
    static constexpr int OFF_TMEM = OFF_MBAR + 2 * NBUF * NBLK + 2;
    static constexpr int OFF_FLAG = OFF_TMEM + 2;
    static constexpr size_t SMEM_BYTES = (size_t)(OFF_FLAG + 4) * 4;
    static_assert(OFF_STEP % 4 == 0 && OFF_GS % 4 == 0 && OFF_PART % 4 == 0 && OFF_MBAR % 2 == 0, "alignment");
    static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");
    static_assert(NBLK <= NWARP && NBUF * NBLK <= 32, "one finishing warp per block in flight; phase bits");
};

template <int NBLK_>
__global__ void __launch_bounds__(VecBetaLinCfg<NBLK_>::THREADS, 1) bwd_vec_beta_lin_kernel(BwdParams p)
{
    using C = VecBetaLinCfg<NBLK_>;
    constexpr int K = C::K, Q = C::Q, QC = C::QC, CL = C::CL, NWARP = C::NWARP, NBUF = C::NBUF, SLOTS = C::SLOTS, CT = C::THREADS;
    constexpr int NBLK = C::NBLK, UNITS = C::UNITS, MAX_NT = C::MAX_NT;
    constexpr uint32_t TX_MSG = 2u * QC * 4u, TX_PART = SLOTS * 16u;   // a quarter of both message arrays; the sums (rank 0 only)
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const uint32_t cid = cluster_id_x(), ncl = cluster_count_x();
    const int n = p.n, nt = n / 2;
    const float invT = p.invT, sl = sqrtf(p.lam2), isl = 1.f / sl;
    const double isl_d = 1.0 / (double)sl;
    const VecRange range = vec_range<NBLK>(p.B, cid, ncl);

    float *msg = smem + C::OFF_MSG;
    float4 *step = reinterpret_cast<float4 *>(smem + C::OFF_STEP);     // entry t - 1 belongs to step t
    float2 *gso = reinterpret_cast<float2 *>(smem + C::OFF_GS);
    float *part = smem + C::OFF_PART;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_TMEM);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_FLAG);
    Proto pr{1u, abort_flag, p.diag};
    const uint32_t mbar_full = smem_u32(smem + C::OFF_MBAR);
    const uint32_t msg_u32 = smem_u32(msg), part_u32 = smem_u32(part);
    const int q0b = warp * 256 + (int)rank * 64 + 2 * lane;      // groups q0b, q0b + 1
    const float4 *hist = reinterpret_cast<const float4 *>(p.hist) + q0b / 2;     // + (block nt + t - 1) Q / 2

    const int rb = warp >> 2;                                    // consumer of this thread's outputs (see bwd_vec4_kernel)
    const uint32_t push_b = mapa_u32(msg_u32, (uint32_t)rb) + vec_beta_dst(q0b, 64, lane);
    const uint32_t push_b_mbar = mapa_u32(mbar_full, (uint32_t)rb);
    const uint32_t part_dst = mapa_u32(part_u32 + (uint32_t)((int)rank * NWARP + warp) * 16u, 0u);
    const uint32_t part_mbar = mapa_u32(mbar_full, 0u);

    if (tid == 0) {
        for (int s = 0; s < NBUF * NBLK; ++s) mbar_init(mbar_full + 8u * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc_512(smem_u32(const_cast<uint32_t *>(tmem_slot)));
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tm = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
    const uint32_t tm_acc = tm + 64u;
    auto zero_acc = [&]() {
        float2 z[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) z[e] = make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < UNITS; ++u) tmem_st16(tm_acc + 16u * u, z);
        tmem_wait_st();
    };
    zero_acc();
    vec4_stage_table(tm, p.cb_beta, q0b, sl);
    int e_acc = GRAD_NONE;                                       // scale of the accumulators (see bcjr_lin_bwd.cuh)
    // the accumulators added to this cluster's partial of the table gradient, in the regrouped layout [b][q][V]
    auto write_acc = [&]() {
        float *gc = p.gc_part + (size_t)cid * C::S * 2;
        const float up = grad_up(e_acc);
#pragma unroll
        for (int un = 0; un < UNITS; ++un) {
            float2 acc[8];
            tmem_ld16(tm_acc + 16u * un, acc);
            tmem_wait_ld(acc);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float4 *dst = reinterpret_cast<float4 *>(gc + ((size_t)(4 * un + e) * Q + q0b) * 2);
                const float4 o = *dst;                           // (z0.x, z0.y, z1.x, z1.y)
                *dst = make_float4(o.x + up * acc[2 * e].x, o.y + up * acc[2 * e + 1].x, o.z + up * acc[2 * e].y, o.w + up * acc[2 * e + 1].y);
            }
        }
    };
    uint32_t full_phase = 0;
    int ib = 0;
    float defect = 0.f;
    auto wait_inputs = [&](int b, int k) {
        const int s = b * NBLK + k;
        pr.wait(mbar_full + 8u * s, (full_phase >> s) & 1u);
        full_phase ^= 1u << s;
    };

    int left = range.count;
    for (int64_t base = range.begin; left > 0; base += range.depth, left -= range.depth) {
        uint32_t todo = vec_live<NBLK>(p.lin_flag, base, left < range.depth ? left : range.depth);   // all four CTAs alike
        while (todo) {                                           // blocks with gradients of one scale side by side: as a rule all of them
            int e_g = 0;
            uint32_t live = 0;
            for (int k = 0; k < range.depth; ++k) {
                if (!((todo >> k) & 1u)) continue;
                const int e = grad_scale(p.g_bits[base + k], *p.g_top);
                if (live == 0) e_g = e;
                if (e == e_g) live |= 1u << k;
            }
            todo &= ~live;
            if (e_g != e_acc) {
                if (e_acc != GRAD_NONE) { write_acc(); zero_acc(); }
                e_acc = e_g;
            }
            const float down = grad_down(e_g);
            for (int k = 0; k < range.depth; ++k) {
                if (!((live >> k) & 1u)) continue;
                const float2 *w = reinterpret_cast<const float2 *>(p.W + (base + k) * n), *g = reinterpret_cast<const float2 *>(p.g + (base + k) * n);
                const float2 *sf = reinterpret_cast<const float2 *>(p.soft + (base + k) * n);
                const int *aux = p.stepO + (size_t)(base + k) * VecAlphaLinCfg<1>::AUX_INTS;
                for (int t = tid; t < nt; t += CT) {
                    const float2 wt = __ldg(w + t), st = __ldg(sf + t);
                    float2 gt = __ldg(g + t);
                    gt.x *= down; gt.y *= down;
                    step[k * MAX_NT + t] = make_float4(wt.x * sl, wt.y * sl, gt.x, gt.y);
                    gso[k * MAX_NT + t] = make_float2(vec_gs(gt.x, gt.y, wt.x * sl, wt.y * sl, isl_d, st.x, st.y), (float)aux[t + 1]);
                }
                const float m1 = __int_as_float(aux[0]);             // M_nt = 1 / Z, Bt_nt = 0
                float *m0 = msg + (size_t)(ib * NBLK + k) * 2 * QC;
                for (int q = tid; q < QC; q += CT) { m0[q] = m1; m0[QC + q] = 0.f; }
            }
            // history, requested one turn (block and step) ahead
            const int k0 = __ffs(live) - 1;
            float4 H = __ldcg(hist + ((size_t)(base + k0) * nt + nt - 1) * (Q / 2));
            cluster_sync();
            // rank 0, warp k: turn the sums of step t of block k (slots of buffer b) into grad_W of that step
            auto finish_step = [&](int t, int b, int k) {
                if (rank == 0 && warp == k) {
                    const float *pp = part + (size_t)((b * NBLK + k) * 64) * 4;
                    const float4 s4 = *reinterpret_cast<const float4 *>(pp + lane * 4);
                    const float4 o = *reinterpret_cast<const float4 *>(pp + (lane + 32) * 4);
                    const float v4 = warp_sum4_split(s4.x + o.x, s4.y + o.y, s4.z + o.z, s4.w + o.w, lane);
                    const float a0 = __shfl_sync(0xffffffffu, v4, 0), a2 = __shfl_sync(0xffffffffu, v4, 8);
                    const float z0 = __shfl_sync(0xffffffffu, v4, 16), z1 = __shfl_sync(0xffffffffu, v4, 24);
                    if (lane == 0) {
                        const int64_t at = (base + k) * n + 2 * (t - 1);
                        const float2 wt = __ldg(reinterpret_cast<const float2 *>(p.W + at)), gt = __ldg(reinterpret_cast<const float2 *>(p.g + at));
                        const float2 st = __ldg(reinterpret_cast<const float2 *>(p.soft + at));
                        const float i0 = grad_up(e_acc) / a0;
                        *reinterpret_cast<float2 *>(p.gW + at) = make_float2((gt.x - z0 * i0) + (a2 * i0) * (wt.x - st.x) * invT,
                                                                             (gt.y - z1 * i0) + (a2 * i0) * (wt.y - st.y) * invT);
                        defect = fmaxf(defect, fabsf(a0 - 1.f));
                    }
                }
            };
            for (int t = nt; t >= 1; --t) {
                const int ob = ib == NBUF - 1 ? 0 : ib + 1;
#pragma unroll
                for (int k = 0; k < NBLK; ++k) {
                    if ((live >> k) & 1u) {
                        const int si = ib * NBLK + k, so = ob * NBLK + k;
                        float2 cb[2][8], acc[8];
                        tmem_ld16(tm, cb[0]);
                        const float4 sp = step[k * MAX_NT + t - 1];
                        const float2 so2 = gso[k * MAX_NT + t - 1];
                        const float2 wx = splat2(sp.x), wy = splat2(sp.y), gx = splat2(sp.z * isl), gy = splat2(sp.w * isl), off2 = splat2(so2.y);
                        const float2 A2 = make_float2(H.x, H.y), AA2 = make_float2(H.z, H.w), ni2 = splat2(-invT * isl);
                        const float2 fgx = mul2(A2, splat2(sp.z)), fgy = mul2(A2, splat2(sp.w)), nf = mul2(A2, ni2), nfA = mul2(AA2, ni2);
                        const uint32_t later = live >> (k + 1) << (k + 1);
                        const int tn = later ? t : t > 1 ? t - 1 : 1, kn = later ? __ffs(later) - 1 : k0;
                        H = __ldcg(hist + ((size_t)(base + kn) * nt + tn - 1) * (Q / 2));
                        if (t < nt) {
                            wait_inputs(ib, k);
                            finish_step(t + 1, ib, k);
                        }
                        const float *Min = msg + (size_t)si * 2 * QC + 4 * lane, *Bin = Min + QC;           // [b >> 1][x >> 1][b & 1][x & 1], x = 2 lane
                        if (tid == 0) pr.expect_tx(mbar_full + 8u * so, rank == 0 ? TX_MSG + TX_PART : TX_MSG);
                        float2 sum = make_float2(0.f, 0.f), ya = sum, Z0 = sum, Z1 = sum;
#pragma unroll
                        for (int un = 0; un < UNITS; ++un) {
                            tmem_ld16(tm_acc + 16u * un, acc);
                            if (un + 1 < UNITS) tmem_ld16(tm + 16u * (un + 1), cb[(un + 1) & 1]);
                            if (un == 0) tmem_wait_ld(cb[0]);
                            tmem_wait_ld(acc);
                            if (un + 1 < UNITS) tmem_wait_ld(cb[(un + 1) & 1]);
#pragma unroll
                            for (int e = 0; e < 4; e += 2) {
                                const int b = 4 * un + e;
                                const float4 Mv = *reinterpret_cast<const float4 *>(Min + 128 * (b >> 1));
                                const float4 Bv = *reinterpret_cast<const float4 *>(Bin + 128 * (b >> 1));
#pragma unroll
                                for (int bb = 0; bb < 2; ++bb) {
                                    const int c = 2 * (e + bb);
                                    const float2 dx = sub2(cb[un & 1][c], wx), dy = sub2(cb[un & 1][c + 1], wy);
                                    const float2 ex = ex2n2(fma2(dy, dy, fma2(dx, dx, off2)));
                                    const float2 y = fma2(gx, dx, fma2(gy, dy, bb == 0 ? make_float2(Bv.x, Bv.y) : make_float2(Bv.z, Bv.w)));   // h - gs + Bt
                                    const float2 pb = mul2(ex, bb == 0 ? make_float2(Mv.x, Mv.y) : make_float2(Mv.z, Mv.w));
                                    const float2 r = fma2(nf, y, nfA);                                       // -A r / (T sl)
                                    const float2 zx = fma2(dx, r, fgx), zy = fma2(dy, r, fgy);               // A (g_v + (w_v - c_v) r / T)
                                    sum = add2(sum, pb);
                                    ya = fma2(pb, y, ya);
                                    Z0 = fma2(pb, zx, Z0); Z1 = fma2(pb, zy, Z1);
                                    acc[c] = fma2(pb, zx, acc[c]);
                                    acc[c + 1] = fma2(pb, zy, acc[c + 1]);
                                }
                            }
                            tmem_st16(tm_acc + 16u * un, acc);
                        }
                        const float2 outB = fma2(ya, rcpf2(make_float2(fmaxf(sum.x, 1e-37f), fmaxf(sum.y, 1e-37f))), splat2(so2.x));
                        const uint32_t dst = push_b + (uint32_t)(so * 2 * QC) * 4u;
                        const float2 mx = vec_pair_x(sum, lane), bx = vec_pair_x(outB, lane);
                        pr.async_v2(dst, mx.x, mx.y, push_b_mbar + 8u * so);
                        pr.async_v2(dst + QC * 4u, bx.x, bx.y, push_b_mbar + 8u * so);
                        const float2 S0 = mul2(A2, sum), S2 = fma2(AA2, sum, mul2(A2, ya));
                        const float v4 = warp_sum4_split(S0.x + S0.y, S2.x + S2.y, Z0.x + Z0.y, Z1.x + Z1.y, lane);   // lanes 0, 8, 16, 24
                        if ((lane & 7) == 0)
                            pr.async_f32(part_dst + (uint32_t)(so * 256 + (lane >> 3)) * 4u, v4, part_mbar + 8u * so);
                        tmem_wait_st();
                    }
                }
                ib = ob;
            }
#pragma unroll
            for (int k = 0; k < NBLK; ++k) {
                if ((live >> k) & 1u) {
                    wait_inputs(ib, k);                                          // the sums of step 1
                    finish_step(1, ib, k);
                }
            }
            cluster_sync();         // nobody still reads this batch's buffers when the next batch starts
        }
    }
    if (e_acc != GRAD_NONE) write_acc();
    if (rank == 0 && lane == 0 && warp < NBLK) diag_max(&p.diag->max_defect, defect);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();             // no CTA leaves while a peer may still address its shared memory
    if (*abort_flag) settle_after_abort();
    if (warp == 0) tmem_dealloc_512(tmem_base);
}

}  // namespace bcjr

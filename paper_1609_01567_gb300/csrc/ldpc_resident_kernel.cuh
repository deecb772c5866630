// The resident decode kernel (see ldpc_resident.h).
//
// Algorithm 2 of one frame by one CTA: the check phase and the bit phase of an
// iteration are separated by CTA barriers, every message stays in shared
// memory, and the CTA leaves as soon as its frame's syndrome is zero.
// The arithmetic of a node is that of the pass kernels (ldpc_pass_kernels.cuh),
// operation for operation, so both decodes give the same results bit for bit.
//
// What bounds it: instruction issue (70-80% of the slots at n = 1008 and
// 2048) and, with one CTA an SM, the latencies between two barriers; HBM sees a
// frame's LLRs and decisions once. The pass kernels move a frame's messages
// through HBM or L2 three times a pass, launch at least two kernels a pass up to
// max_iter, and keep a group of 64-128 frames running until its last one stops;
// here a frame costs its own iterations. Measured (pass kernels -> this one,
// early exit unless said): n = 1008, one frame 149-180 -> 17-25 us with the call,
// 1000 frames 576 -> 162 us; n = 2048 (4, 8)-regular, 10,000 frames with channel
// noise and error count 5.74 -> 1.90 ms; n = 8192, 700 frames 916 -> 341 us; n =
// 8192 with a degree-96 check, bfloat16, 256 frames, 10 fixed iterations 271 -> 173
// us; n = 16200 min-sum, 301 frames 1.41 -> 0.83-0.89 ms. These are frames that stop;
// resident_shape weighs frames that do not. Two frames a CTA in packed FP32
// pairs were slower for all but fixed iterations (n = 8192, 700 frames: 916 us):
// both run to the slower one's end.
#pragma once

#include "ldpc_pass_kernels.cuh"
#include "ldpc_resident.h"

namespace ldpc {
namespace resident {

// A check group as a lane sees it: its check's table row, message slots and the
// group's largest degree.
template <int NV, typename M>
struct Group {
    uint32_t v[NV];
    M *r;  // the slot of input 0; input k is 32 k further
    int dm;
    bool zero_neg;  // an input of exactly +0, or NaN, counts as negative (read where D > 16, whatever the group's degree)
    // entry k of the row, held as packed pairs
    __device__ __forceinline__ uint32_t entry(int k) const { return (k & 1) ? v[k / 2] >> 16 : v[k / 2] & 0xFFFFu; }
};

// The sum-product rule of one check per lane, at most D inputs; kAll: every
// check has exactly D. Suffix states are kept at chunk ends only and formed
// again inside a chunk (the same operations on the same values), which bounds
// the registers. Two checks a lane in packed FP32 pairs ran no faster (n = 2048,
// 10,000 frames: 2.15 ms either way) and slower where the registers then halve
// the warps (n = 576, degree 18: 186 us against 108).
template <int D, bool kAll, bool ZN, int NV, typename M>
__device__ __forceinline__ void sp_group(const Group<NV, M> &gr, const unsigned char *app, const ResidentArgs &a,
                                         uint32_t &unsat) {
    constexpr bool kClamp = D <= (kAll ? 2 : 4);  // outputs of three or more inputs never saturate
    constexpr int C = D <= 6 ? D : (D <= 8 ? 4 : 6);
    constexpr int NC = (D + C - 1) / C;
    float t[D];
    uint32_t sb = 0, z = 0, d = 0;  // z, sign bit: parity of the decisions APP > 0, each the sign of 0 - APP
#pragma unroll
    for (int k = 0; k < D; ++k) {
        t[k] = 0.0f;
        if (!kAll && k >= gr.dm) {  // the same for the whole warp
            sb <<= 1;
            continue;
        }
        const uint32_t c = gr.entry(k);
        const bool on = kAll || c != kResidentPad;
        const float av = *reinterpret_cast<const float *>(app + (on ? c : 0u));
        float q = extrinsic(av, MsgIO<M>::load1(gr.r + 32 * k));
        // what is not above zero, NaN included: the sign of its bit in sb
        if ((D > 16 ? gr.zero_neg : ZN) && !(q > 0.0f)) q = __uint_as_float(__float_as_uint(q) | 0x80000000u);
        const float e = exp_neg(fminf(fabsf(q), a.l_max));
        z ^= on ? __float_as_uint(__fsub_rn(0.0f, av)) : 0u;
        sb = __funnelshift_l(on ? __float_as_uint(q) : 0u, sb, 1);
        if (on) t[k] = e;
        if (!kAll) d += on ? 1u : 0u;
    }
    unsat |= z;
    float ea[NC], ed[NC];  // states of the inputs after each chunk
    {
        float ca = 2.0f, cd = 0.0f;
#pragma unroll
        for (int k = D - 1; k >= 0; --k) {
            if (k == D - 1 || k % C == C - 1) {
                ea[k / C] = ca;
                ed[k / C] = cd;
            }
            if (k >= C) pf_merge(ca, cd, t[k]);
        }
    }
    const uint32_t neg = (((kAll ? (uint32_t)D : d) ^ __popc(sb)) & 1u) ? ~sb : sb;
    float pa = 2.0f, pd = 0.0f;
#pragma unroll
    for (int ch = 0; ch < NC; ++ch) {
        float sa[C], sd[C];
        float ca = ea[ch], cd = ed[ch];
#pragma unroll
        for (int i = C - 1; i >= 0; --i) {
            const int k = ch * C + i;
            if (k < D) {
                sa[i] = ca;
                sd[i] = cd;
                if (i > 0) pf_merge(ca, cd, t[k]);
            }
        }
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int k = ch * C + i;
            if (k < D) {
                const float y = pf_out<kClamp>(pa, pd, sa[i], sd[i], a.r_max);
                // padding slots take a value nobody reads
                if (kAll || k < gr.dm) MsgIO<M>::store1(gr.r + 32 * k, with_sign(y, neg << (32 - D + k)));
                if (k + 1 < D) pf_merge(pa, pd, t[k]);
            }
        }
    }
}

// The min-sum family, one check per lane: two sweeps over the slots.
template <int D, bool kAll, int NV, typename M>
__device__ __forceinline__ void ms_group(const Group<NV, M> &gr, const unsigned char *app, const ResidentArgs &a,
                                         uint32_t &unsat) {
    float m1 = a.l_max, m2 = a.l_max;
    int idx = -1, d = kAll ? D : 0;
    uint32_t ones = 0, z = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        if (!kAll && k >= gr.dm) continue;  // the same for the whole warp
        const uint32_t c = gr.entry(k);
        const bool on = kAll || c != kResidentPad;
        const float av = *reinterpret_cast<const float *>(app + (on ? c : 0u));
        const float q = av - MsgIO<M>::load1(gr.r + 32 * k);
        if (!kAll) d += on ? 1 : 0;
        z ^= on ? __float_as_uint(__fsub_rn(0.0f, av)) : 0u;
        ones |= on && q > 0.0f ? 1u << k : 0u;
        const float x = on ? fminf(fabsf(q), a.l_max) : a.l_max;
        const bool lt = x < m1;
        m2 = lt ? m1 : fminf(m2, x);
        m1 = lt ? x : m1;
        idx = lt ? k : idx;
    }
    float alpha = a.ms_alpha, beta = a.ms_beta;
    if (a.ms_table) {
        const float2 ab = __ldg(a.ms_table + d);
        alpha = ab.x;
        beta = ab.y;
    }
    unsat |= z;
    const uint32_t neg = (__popc(ones) & 1u) ? ones : ~ones;
    const float o1 = fminf(fmaxf(fmaf(alpha, m1, -beta), 0.0f), a.l_max);
    const float o2 = fminf(fmaxf(fmaf(alpha, m2, -beta), 0.0f), a.l_max);
#pragma unroll
    for (int k = 0; k < D; ++k)
        if (kAll || k < gr.dm)
            MsgIO<M>::store1(gr.r + 32 * k,
                             __uint_as_float(__float_as_uint(idx == k ? o2 : o1) | ((neg << (31 - k)) & 0x80000000u)));
}

// A check of degree above 32 by one warp: the arithmetic of k_check_wide, whose
// eight warps' partial results (inputs w, w + 8, ...) are lanes w here.
template <int RULE, typename M>
__device__ __forceinline__ void wide_check(const int4 wc, const float *app, M *r, const ResidentArgs &a,
                                           uint32_t &unsat) {
    const int lane = threadIdx.x & 31;
    const int d = wc.y;
    const uint16_t *col = a.list + wc.z;
    r += wc.x;
    float alpha = a.ms_alpha, beta = a.ms_beta;
    if (RULE == 1 && a.ms_table) {
        const float2 ab = __ldg(a.ms_table + d);
        alpha = ab.x;
        beta = ab.y;
    }
    auto input = [&](int k, float &av) {
        av = app[col[k]];
        const float rv = MsgIO<M>::load1(r + k);
        return RULE == 1 ? av - rv : extrinsic(av, rv);
    };
    float hi = RULE == 1 ? a.l_max : 0.0f, lo = hi;
    int idx = -1;
    uint32_t par = 0, z = 0;
    if (lane < 8) {
#pragma unroll 2
        for (int k = lane; k < d; k += 8) {
            float av;
            const float q = input(k, av);
            z ^= av > 0.0f ? 1u : 0u;
            if constexpr (RULE == 1) {
                const float x = fminf(fabsf(q), a.l_max);
                if (x < hi) {
                    lo = hi;
                    hi = x;
                    idx = k;
                } else if (x < lo) {
                    lo = x;
                }
            } else {
                float err;
                hi = two_sum(hi, phi_hat(fabsf(q), a.l_max, a.phi_lmax), err);
                lo += err;
            }
            par ^= q > 0.0f ? 1u : 0u;
        }
    }
    float H = __shfl_sync(kFull, hi, 0), Lw = __shfl_sync(kFull, lo, 0);
    int I = __shfl_sync(kFull, idx, 0);
#pragma unroll
    for (int u = 1; u < 8; ++u) {
        const float h2 = __shfl_sync(kFull, hi, u), l2 = __shfl_sync(kFull, lo, u);
        if constexpr (RULE == 1) {
            const int i2 = __shfl_sync(kFull, idx, u);
            if (h2 < H) {
                Lw = fminf(H, l2);
                H = h2;
                I = i2;
            } else {
                Lw = fminf(Lw, h2);
            }
        } else {
            float err;
            const float s2 = two_sum(H, h2, err);
            Lw = (Lw + l2) + err;
            H = s2;
        }
    }
    const uint32_t par_all = __reduce_xor_sync(kFull, par);
    unsat |= __reduce_xor_sync(kFull, z) << 31;
    for (int k = lane; k < d; k += 32) {
        float av, mm;
        const float q = input(k, av);
        if constexpr (RULE == 1) {
            mm = fminf(fmaxf(fmaf(alpha, I == k ? Lw : H, -beta), 0.0f), a.l_max);
        } else {
            const float own = phi_hat(fabsf(q), a.l_max, a.phi_lmax);
            float err;
            const float s2 = two_sum(H, -own, err);
            mm = phi_hat(s2 + (err + Lw), a.l_max, a.phi_lmax);
        }
        const uint32_t others = par_all ^ (q > 0.0f ? 1u : 0u);
        MsgIO<M>::store1(r + k, others ? mm : -mm);
    }
}

template <int D, bool kAll, int RULE, bool ZN, int NV, typename M>
__device__ __forceinline__ void form(const Group<NV, M> &gr, const unsigned char *app, const ResidentArgs &a,
                                     uint32_t &unsat) {
    if constexpr (RULE == 1)
        ms_group<D, kAll, NV, M>(gr, app, a, unsat);
    else
        sp_group<D, kAll, ZN, NV, M>(gr, app, a, unsat);
}

// Degrees that have a form of their own in the kernel of class DC: groups of 32
// checks of such a degree run without a mask, which takes half the instructions
// (the checks of most codes have two neighbouring degrees).
__host__ __device__ constexpr bool exact_degree(int DC, int d) {
    return DC <= 4   ? d >= 2 && d <= 4
           : DC <= 6 ? d >= 3 && d <= 6
           : DC <= 8 ? d >= 4 && d <= 8
           : DC <= 12 ? d >= 6 && d <= 12
           : DC <= 18 ? d == 8 || d == 12 || d >= 16
                      : d == 8 || d == 16 || d == 24 || d == 32;
}

// Calls f(degree, mask-free) with the form that serves groups of largest degree
// dm, both as compile-time constants.
template <int DC, int D, typename F>
__device__ __forceinline__ void with_form(int dm, bool full, F &&f) {
    if constexpr (D >= 2) {
        if constexpr (exact_degree(DC, D)) {
            if (full && dm == D) {
                f(std::integral_constant<int, D>{}, std::true_type{});
                return;
            }
        }
        with_form<DC, D - 1>(dm, full, f);
    } else if (DC == 4 || dm <= 4) {
        f(std::integral_constant<int, 4>{}, std::false_type{});
    } else {
        f(std::integral_constant<int, DC>{}, std::false_type{});
    }
}

// The same for one group, without the closure (see kStay).
template <int DC, int D, int RULE, bool ZN, int NV, typename M>
__device__ __forceinline__ bool exact_form(const Group<NV, M> &gr, const unsigned char *app, const ResidentArgs &a,
                                           uint32_t &unsat) {
    if constexpr (exact_degree(DC, D)) {
        if (gr.dm == D) {
            form<D, true, RULE, ZN, NV, M>(gr, app, a, unsat);
            return true;
        }
    }
    if constexpr (D > 2) return exact_form<DC, D - 1, RULE, ZN, NV, M>(gr, app, a, unsat);
    return false;
}

// Threads of the largest CTA, and so the registers a thread may take (64 at
// 1024 threads); checks of degree above 12 need more.
template <int DC, int RULE>
__host__ __device__ constexpr int max_threads() { return RULE == 1 || DC <= 12 ? 1024 : 512; }

template <typename M, int DC, int RULE, bool ZN>
__global__ void __launch_bounds__(max_threads<DC, RULE>(), 1) k_resident(const __grid_constant__ ResidentArgs a) {
    constexpr int kRow = resident_row(DC), NV = kRow / 2;
    constexpr bool kAhead = DC <= 12;  // table rows are fetched one group ahead
    // a warp stays in a degree's code while its groups have that degree (n = 2048,
    // 6000 frames, 10 iterations 798 -> 759 us, n = 8192, 700 frames 356 -> 341 us);
    // wider checks are few to a warp and lose by it (n = 1152, degrees 11 and 12,
    // 119 -> 129 us, n = 2304 142 -> 151 us)
    constexpr bool kStay = DC <= 8;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *flag = reinterpret_cast<uint32_t *>(smem);  // [2]: some check is not satisfied
    float *app = reinterpret_cast<float *>(smem + 16);
    const int nv = resident_vars(a.n_vg, a.n_wv);
    float *lam = app + nv;
    M *r = reinterpret_cast<M *>(lam + (a.lam_shared ? nv : 0));
    const unsigned char *rb = reinterpret_cast<const unsigned char *>(r);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
    const int4 *wide_vars = a.wide + a.n_wc;
    const int frame = a.f0 + (int)blockIdx.x;
    const float *llr = a.llr + (size_t)frame * a.n;

    uint32_t cw = 0, cv[NV];        // the warp's next check group: word and table rows
    uint4 vv = make_uint4(0u, 0u, 0u, 0u);  // its next variable group: entries 0-3
    auto fetch_check = [&](int g) {
        if (g >= a.n_cg) return;
        cw = __ldg(a.cg + g);
        const uint2 *x = reinterpret_cast<const uint2 *>(a.crow + (size_t)(g * 32 + lane) * kRow);
        if constexpr (kRow % 8 == 0) {
#pragma unroll
            for (int i = 0; i < kRow / 8; ++i) {
                const uint4 y = __ldg(reinterpret_cast<const uint4 *>(x) + i);
                cv[4 * i] = y.x;
                cv[4 * i + 1] = y.y;
                cv[4 * i + 2] = y.z;
                cv[4 * i + 3] = y.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kRow / 4; ++i) {
                const uint2 y = __ldg(x + i);
                cv[2 * i] = y.x;
                cv[2 * i + 1] = y.y;
            }
        }
    };
    auto take = [&](Group<NV, M> &gr) {
#pragma unroll
        for (int k = 0; k < NV; ++k) gr.v[k] = cv[k];
        gr.r = r + (int)(cw & 0xFFFFu) * 32 + lane;
    };
    auto fetch_var = [&](int g) {
        if (g < a.n_v1) vv = __ldg(a.v4 + g * 32 + lane);
    };
    if constexpr (kAhead) fetch_check(warp);

    if (tid < 2) flag[tid] = 0u;
    for (int j = tid; j < a.n; j += blockDim.x) {
        const int v = a.place[j];
        const float x = __ldg(llr + j);
        app[v] = x;
        if (a.lam_shared) lam[v] = x;
    }
    {
        const uint32_t zero = std::is_same_v<M, int8_t> ? 0x80808080u : 0u;  // the stored form of 0
        uint32_t *rw = reinterpret_cast<uint32_t *>(r);
        const int words = a.slots * (int)sizeof(M) / 4;  // slots is a multiple of 32
        for (int i = tid; i < words; i += blockDim.x) rw[i] = zero;
        if (tid == 0) MsgIO<M>::store1(r + a.slots, -0.0f);
    }
    __syncthreads();

    bool stopped = false;
    int t = 0;
    for (; t <= a.max_iter; ++t) {
        // check phase: new messages, and the syndrome of the decision after pass t - 1
        uint32_t unsat = 0u;  // sign bit: a check of this lane is not satisfied
        for (int g = warps - 1 - warp; g < a.n_wc; g += warps) wide_check<RULE, M>(a.wide[g], app, r, a, unsat);
        if constexpr (kStay) {
            for (int g = warp; g < a.n_cg;) {
                const uint32_t kind = cw >> 16;  // degree and mask of this group, and of those that follow it here
                with_form<DC, DC>((int)kind & 63, (cw & kResidentFull) != 0u, [&](auto dc, auto all) {
                    Group<NV, M> gr;
                    gr.dm = (int)kind & 63;
                    gr.zero_neg = false;
                    do {
                        take(gr);
                        g += warps;
                        fetch_check(g);
                        form<decltype(dc)::value, decltype(all)::value, RULE, ZN, NV, M>(gr, smem + 16, a, unsat);
                    } while (g < a.n_cg && cw >> 16 == kind);
                });
            }
        } else {
            for (int g = warp; g < a.n_cg; g += warps) {
                if constexpr (!kAhead) fetch_check(g);
                Group<NV, M> gr;
                take(gr);
                gr.dm = (int)(cw >> 16) & 63;
                // by the group's own degree: the general form of a wide class serves narrow groups too
                gr.zero_neg = gr.dm > 16 ? a.zero_neg_wide == 2 || (ZN && a.zero_neg_wide == 1) : ZN;
                const bool full = cw & kResidentFull;
                if constexpr (kAhead) fetch_check(g + warps);
                if (full && exact_form<DC, DC, RULE, ZN, NV, M>(gr, smem + 16, a, unsat)) continue;
                if (gr.dm <= 4)
                    form<4, false, RULE, ZN, NV, M>(gr, smem + 16, a, unsat);
                else if (gr.dm <= 8)
                    form<8, false, RULE, ZN, NV, M>(gr, smem + 16, a, unsat);
                else
                    form<DC, false, RULE, ZN, NV, M>(gr, smem + 16, a, unsat);
            }
        }
        fetch_var(warp);
        if (a.early && t > 0 && __any_sync(kFull, (int)unsat < 0) && lane == 0) flag[t & 1] = 1u;
        __syncthreads();
        if (a.early && t > 0) {
            if (flag[t & 1] == 0u) {
                stopped = true;
                break;
            }
            if (tid == 0) flag[(t + 1) & 1] = 0u;
        }
        // bit phase
        auto add2 = [&](float &acc, uint32_t x, uint32_t y) {
            const float m0 = MsgIO<M>::load1(reinterpret_cast<const M *>(rb + x));
            const float m1 = MsgIO<M>::load1(reinterpret_cast<const M *>(rb + y));
            acc = __fadd_rn(__fadd_rn(acc, m0), m1);
        };
        auto lambda = [&](int v) {  // channel LLR of an internal index
            if (a.lam_shared) return lam[v];
            const uint32_t j = a.var[v];
            return j != kResidentPad ? __ldg(llr + j) : 0.0f;
        };
        int vg = warp;
        auto sum_edges = [&](auto kc, int end) {  // groups of variables with up to K edges, below `end`
            constexpr int K = decltype(kc)::value;
            for (; vg < end; vg += warps) {
                const uint4 e = vv;
                fetch_var(vg + warps);
                const int v = vg * 32 + lane;
                float acc = lambda(v);
                add2(acc, e.x, e.y);
                if constexpr (K > 2) add2(acc, e.z, e.w);
                if constexpr (K > 4) {
                    const uint4 x = __ldg(a.v8 + v);
                    add2(acc, x.x, x.y);
                    add2(acc, x.z, x.w);
                }
                if constexpr (K > 8) {
                    const uint4 x = __ldg(a.v16 + 2 * v), y = __ldg(a.v16 + 2 * v + 1);
                    add2(acc, x.x, x.y);
                    add2(acc, x.z, x.w);
                    add2(acc, y.x, y.y);
                    add2(acc, y.z, y.w);
                }
                app[v] = acc;
            }
        };
        sum_edges(std::integral_constant<int, 16>{}, a.n_v16);  // groups are in falling order of degree
        sum_edges(std::integral_constant<int, 8>{}, a.n_v8);
        sum_edges(std::integral_constant<int, 4>{}, a.n_v3);
        sum_edges(std::integral_constant<int, 2>{}, a.n_v1);  // those without a check keep what they have
        // variables of degree above kWideVarDegree: eight partial sums (lane u
        // over edges u, u + 8, ...) added to lambda in order
        for (int g = warps - 1 - warp; g < a.n_wv; g += warps) {
            const int4 wv = wide_vars[g];
            float acc = 0.0f;
            if (lane < 8)
                for (int k = lane; k < wv.y; k += 8) acc = __fadd_rn(acc, MsgIO<M>::load1(r + a.list[wv.x + k]));
            float s = lambda(wv.z);
#pragma unroll
            for (int u = 0; u < 8; ++u) s = __fadd_rn(s, __shfl_sync(kFull, acc, u));
            if (lane == 0) app[wv.z] = s;
        }
        if constexpr (kAhead) fetch_check(warp);
        __syncthreads();
    }

    if (!stopped) {  // syndrome of the last decision
        uint32_t *fin = flag + (t & 1);
        if (tid == 0) *fin = 0u;
        __syncthreads();
        bool unsat = false;
        for (int g = warp; g < a.n_cg; g += warps) {
            const uint16_t *row = a.crow + (size_t)(g * 32 + lane) * kRow;
            const int dm = (int)(a.cg[g] >> 16) & 63;
            bool z = false;
#pragma unroll 4
            for (int k = 0; k < dm; ++k) {
                const uint32_t c = row[k];
                if (c != kResidentPad) z ^= app[c / 4] > 0.0f;
            }
            unsat |= z;
        }
        for (int g = warp; g < a.n_wc; g += warps) {
            const int4 wc = a.wide[g];
            uint32_t z = 0;
            for (int k = lane; k < wc.y; k += 32) z ^= app[a.list[wc.z + k]] > 0.0f ? 1u : 0u;
            unsat |= __reduce_xor_sync(kFull, z) != 0u;
        }
        if (__any_sync(kFull, unsat) && lane == 0) *fin = 1u;
        __syncthreads();
    }
    if (tid == 0) {
        a.iters[frame] = stopped ? t - 1 : a.max_iter;
        a.ok[frame] = stopped || flag[t & 1] == 0u ? 1 : 0;
    }
    // four variables a thread, bytes of their decisions as one word where the rows allow it
    const bool vec = (a.n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.bits) & 3) == 0 &&
                     (reinterpret_cast<uintptr_t>(a.post) & 15) == 0;
    const size_t row0 = (size_t)frame * a.n;
    for (int q = tid; q < (a.n + 3) / 4; q += blockDim.x) {
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = 4 * q + i < a.n ? app[a.place[4 * q + i]] : 0.0f;
        const size_t o = row0 + 4 * q;
        if (vec) {
            uint32_t word = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) word |= (x[i] > 0.0f ? 1u : 0u) << (8 * i);
            *reinterpret_cast<uint32_t *>(a.bits + o) = word;
            if (a.post) *reinterpret_cast<float4 *>(a.post + o) = make_float4(x[0], x[1], x[2], x[3]);
        } else {
            for (int i = 0; i < 4 && 4 * q + i < a.n; ++i) {
                a.bits[o + i] = x[i] > 0.0f ? 1 : 0;
                if (a.post) a.post[o + i] = x[i];
            }
        }
    }
}

template <typename M, int DC, int RULE, bool ZN>
cudaError_t launch_frames(const ResidentArgs &a, int32_t frames, const ResidentShape &sh, cudaStream_t s) {
    static std::atomic<bool> ready[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (!ready[dev & 63].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(k_resident<M, DC, RULE, ZN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kResidentSmem);
        if (e != cudaSuccess) return e;
        ready[dev & 63].store(true, std::memory_order_release);
    }
    const unsigned threads = (unsigned)std::min(sh.threads, max_threads<DC, RULE>());
    // the launch's own status: cudaGetLastError would also report what an earlier,
    // refused call left (a decode that was refused inside a capture)
    void *args[] = {const_cast<ResidentArgs *>(&a)};
    return cudaLaunchKernel(reinterpret_cast<const void *>(k_resident<M, DC, RULE, ZN>), dim3((unsigned)frames),
                            dim3(threads), args, sh.smem, s);
}

template <typename M, int DC, int RULE>
cudaError_t launch(const ResidentArgs &a, const ResidentShape &sh, cudaStream_t s, int64_t *launched) {
    if constexpr (RULE == 1) {
        *launched += 1;
        return launch_frames<M, DC, 1, false>(a, a.F, sh, s);
    } else {
        const int32_t plain = std::min(a.F, a.zero_neg_from);
        cudaError_t e = plain > 0 ? launch_frames<M, DC, 0, false>(a, plain, sh, s) : cudaSuccess;
        *launched += plain > 0 ? 1 : 0;
        if (e == cudaSuccess && plain < a.F) {
            ResidentArgs b = a;
            b.f0 = plain;
            e = launch_frames<M, DC, 0, true>(b, a.F - plain, sh, s);
            *launched += 1;
        }
        return e;
    }
}

}  // namespace resident

template <typename M, int RULE>
cudaError_t launch_resident_m(const ResidentArgs &a, int32_t dclass, const ResidentShape &sh, cudaStream_t s,
                              int64_t *launched) {
    switch (dclass) {
    case 4: return resident::launch<M, 4, RULE>(a, sh, s, launched);
    case 6:
        if constexpr (RULE == 0) return resident::launch<M, 6, RULE>(a, sh, s, launched);
        [[fallthrough]];
    case 8: return resident::launch<M, 8, RULE>(a, sh, s, launched);
    case 12: return resident::launch<M, 12, RULE>(a, sh, s, launched);
    case 18: return resident::launch<M, 18, RULE>(a, sh, s, launched);
    default: return resident::launch<M, 32, RULE>(a, sh, s, launched);
    }
}

}  // namespace ldpc

#define LDPC_INSTANTIATE_RESIDENT(M, RULE)                                                                  \
    namespace ldpc {                                                                                        \
    template cudaError_t launch_resident_m<M, RULE>(const ResidentArgs &, int32_t, const ResidentShape &,   \
                                                    cudaStream_t, int64_t *);                               \
    }

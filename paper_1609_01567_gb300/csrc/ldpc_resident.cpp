// Plan and dispatch of the resident decode (ldpc_resident.h).
#include <algorithm>
#include <climits>
#include <cmath>
#include <initializer_list>
#include <new>

#include "ldpc_internal.h"
#include "ldpc_resident.h"

namespace ldpc {

// Nodes `ids` sorted by falling degree, cut into groups of 32; no group holds
// degrees on both sides of a border (degrees up to `b` and above it).
static std::vector<std::vector<int32_t>> degree_groups(std::vector<int32_t> ids, const std::vector<int32_t> &ptr,
                                                       std::initializer_list<int32_t> borders) {
    auto deg = [&](int32_t i) { return ptr[i + 1] - ptr[i]; };
    int32_t top = 0;
    for (int32_t id : ids) top = std::max(top, deg(id));
    std::vector<int32_t> at((size_t)top + 2, 0), sorted(ids.size());  // counting sort: creating a code waits for this
    for (int32_t id : ids) at[top - deg(id) + 1] += 1;
    for (int32_t d = 0; d <= top; ++d) at[d + 1] += at[d];
    for (int32_t id : ids) sorted[at[top - deg(id)]++] = id;
    ids.swap(sorted);
    std::vector<std::vector<int32_t>> groups;
    for (int32_t id : ids) {
        bool cut = groups.empty() || groups.back().size() == 32;
        for (int32_t b : borders) cut = cut || (deg(groups.back()[0]) > b && deg(id) <= b);
        if (cut) {
            groups.emplace_back();
            groups.back().reserve(32);
        }
        groups.back().push_back(id);
    }
    return groups;
}

static cudaError_t make_plan(const ldpc_code *c, ResidentPlan *p) {
    *p = ResidentPlan{};
    // 16-bit indexes
    if (c->m == 0 || c->n == 0 || c->E == 0 || c->n >= kResidentPad || c->E >= kResidentPad) return cudaSuccess;
    std::vector<int32_t> checks, wide_checks, vars, wide_vars;
    for (int32_t i = 0; i < c->m; ++i) {
        const int32_t d = c->row_ptr[i + 1] - c->row_ptr[i];
        if (d > kMaxRegisterDegree) wide_checks.push_back(i);
        else if (d > 0) checks.push_back(i);
    }
    for (int32_t j = 0; j < c->n; ++j)
        (c->col_ptr[j + 1] - c->col_ptr[j] > kWideVarDegree ? wide_vars : vars).push_back(j);
    // variables without a check keep their channel value as it is: their own groups
    const auto vg = degree_groups(vars, c->col_ptr, {0});
    // outputs of checks of up to four inputs can saturate, and the sign of an
    // input of exactly zero changes above 16 (see zero_sign)
    const auto cg = degree_groups(checks, c->row_ptr, {4, 16});
    auto degree = [](const std::vector<int32_t> &ptr, int32_t i) { return ptr[i + 1] - ptr[i]; };
    std::vector<uint16_t> place((size_t)c->n), var((vg.size() * 32 + wide_vars.size() + 3) / 4 * 4, kResidentPad);
    if (var.size() * 4 >= kResidentPad) return cudaSuccess;  // 16-bit byte offsets
    auto put = [&](size_t v, int32_t j) {
        place[j] = (uint16_t)v;
        var[v] = (uint16_t)j;
    };
    for (size_t g = 0; g < vg.size(); ++g)
        for (size_t l = 0; l < vg[g].size(); ++l) put(g * 32 + l, vg[g][l]);
    for (size_t i = 0; i < wide_vars.size(); ++i) put(vg.size() * 32 + i, wide_vars[i]);

    const int32_t top = cg.empty() ? 1 : degree(c->row_ptr, cg[0][0]);
    p->dclass = top <= 4 ? 4 : (top <= 6 ? 6 : (top <= 8 ? 8 : (top <= 12 ? 12 : (top <= 18 ? 18 : 32))));
    const int32_t row = resident_row(p->dclass);
    std::vector<uint32_t> words;
    std::vector<uint16_t> crow(cg.size() * 32 * row, kResidentPad), list;
    std::vector<int32_t> slot_of((size_t)c->E);  // message slot of each check-order entry
    int64_t slots = 0;
    for (size_t g = 0; g < cg.size(); ++g) {
        const int32_t d0 = degree(c->row_ptr, cg[g][0]);
        const bool full = cg[g].size() == 32 && degree(c->row_ptr, cg[g][31]) == d0;
        words.push_back((uint32_t)(slots / 32) | (uint32_t)d0 << 16 | (full ? kResidentFull : 0u));
        for (size_t l = 0; l < cg[g].size(); ++l)
            for (int32_t k = 0, b = c->row_ptr[cg[g][l]]; b + k < c->row_ptr[cg[g][l] + 1]; ++k) {
                crow[(g * 32 + l) * row + k] = (uint16_t)(4 * place[c->col_idx[b + k]]);
                slot_of[b + k] = (int32_t)slots + 32 * k + (int32_t)l;
            }
        slots += 32 * d0;
    }
    std::vector<int4> wide;
    for (int32_t i : wide_checks) {
        const int32_t b = c->row_ptr[i], d = degree(c->row_ptr, i);
        wide.push_back(make_int4((int)slots, d, (int)list.size(), 0));
        for (int32_t k = 0; k < d; ++k) {
            slot_of[b + k] = (int32_t)slots++;
            list.push_back(place[c->col_idx[b + k]]);
        }
    }
    slots = (slots + 31) / 32 * 32;
    p->slots = (int32_t)slots;
    // 16-bit slots, and one frame's smallest messages must fit
    if (slots >= kResidentPad || (size_t)c->n * 4 + (size_t)slots + 64 > (size_t)kResidentSmem) return cudaSuccess;
    std::vector<uint32_t> v4, v8, v16;
    v4.reserve(vg.size() * 128);
    for (const auto &g : vg) {
        const int32_t d0 = degree(c->col_ptr, g[0]);
        p->n_v1 += d0 > 0 ? 1 : 0;
        p->n_v3 += d0 > 2 ? 1 : 0;
        p->n_v8 += d0 > 4 ? 1 : 0;
        p->n_v16 += d0 > 8 ? 1 : 0;
        for (size_t l = 0; l < 32; ++l)
            for (int32_t k = 0; k < (d0 > 8 ? 16 : (d0 > 4 ? 8 : 4)); ++k) {
                const bool real = l < g.size() && k < degree(c->col_ptr, g[l]);
                (k < 4 ? v4 : (k < 8 ? v8 : v16))
                    .push_back((uint32_t)(real ? slot_of[c->edge_slot[c->col_ptr[g[l]] + k]] : slots));
            }
    }
    for (size_t i = 0; i < wide_vars.size(); ++i) {
        const int32_t e = c->col_ptr[wide_vars[i]], d = degree(c->col_ptr, wide_vars[i]);
        wide.push_back(make_int4((int)list.size(), d, (int)(vg.size() * 32 + i), 0));
        for (int32_t k = 0; k < d; ++k) list.push_back((uint16_t)slot_of[c->edge_slot[e + k]]);
    }
    p->n_cg = (int32_t)cg.size();
    p->n_vg = (int32_t)vg.size();
    p->n_wc = (int32_t)wide_checks.size();
    p->n_wv = (int32_t)wide_vars.size();
    std::vector<unsigned char> tab;
    int at = 0;
    auto add = [&](const void *src, size_t bytes) {
        const auto *b = static_cast<const unsigned char *>(src);
        p->off[at++] = tab.size();
        if (bytes) tab.insert(tab.end(), b, b + bytes);
        tab.resize((tab.size() + 15) / 16 * 16);
    };
    add(crow.data(), crow.size() * 2);
    add(words.data(), words.size() * 4);
    add(place.data(), place.size() * 2);
    add(var.data(), var.size() * 2);
    add(wide.data(), wide.size() * sizeof(int4));
    add(list.data(), list.size() * 2);
    for (int bytes = 1; bytes <= 4; bytes *= 2) {  // of a message
        for (auto *v : {&v4, &v8, &v16}) {
            add(v->data(), v->size() * 4);
            for (auto &x : *v) x *= 2;
        }
    }
    cudaError_t e = cudaMalloc(&p->tab, tab.size());
    if (e == cudaSuccess) e = cudaMemcpy(p->tab, tab.data(), tab.size(), cudaMemcpyHostToDevice);
    p->ok = e == cudaSuccess;
    return e;
}

cudaError_t resident_plan_create(const ldpc_code *c, ResidentPlan *p) {
    try {
        return make_plan(c, p);
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

constexpr int32_t kPassChunk = 8192;  // frames of a chunk of the pass kernels

// The sum-product kernels count an input of exactly +0, or NaN, as a positive one,
// all but the register kernel (k_check_reg). The resident decode counts it as the
// kernel does that serves the check in a decode with passes: frames from
// `from` on (chunks of up to 32 frames) for degrees up to 16, `wide` above.
static void zero_sign(const ldpc_code *c, int32_t F, ResidentArgs *a) {
    const int32_t last = F > kPassChunk ? F % kPassChunk : F;
    a->zero_neg_from = last > 0 && last <= 32 ? F - last : INT_MAX;
    const bool staged = c->bin_off[5] - c->bin_off[4] >= kWideBinAnyKernel;
    a->zero_neg_wide = staged ? 0 : (c->bin_max_degree[4] > 18 ? 2 : 1);  // 2: all frames, 1: from zero_neg_from
}

void resident_plan_free(ResidentPlan *p) {
    cudaFree(p->tab);
    *p = ResidentPlan{};
}

// One iteration of F frames, in us, here and by the pass kernels: estimates for
// the choice between the two, fitted to 1515 timed pairs of 35 codes of 576 to
// 16,200 bits (rates 1/3 to 5/6, check degrees 3 to 22 and one of 96, 1 to 5000
// frames, all message formats, 10 fixed iterations). 9% and 12% root-mean-square off.
// By the widest check's class: degree 8, 12, 18, 32.
static int degree_class(const ResidentPlan &p) { return p.dclass <= 8 ? 0 : (p.dclass <= 12 ? 1 : (p.dclass <= 18 ? 2 : 3)); }

// An SM takes a time per message slot (instruction issue) for each of its
// frames, and latency (barriers) once where several CTAs cover each other's,
// else for each.
static double resident_us(const ldpc_code *c, const ResidentShape &sh, int32_t per_sm, int32_t F,
                          const ldpc_decode_opts_t &o) {
    constexpr double kSlotNs[2][4] = {{0.249, 0.298, 0.426, 0.485}, {0.235, 0.257, 0.287, 0.352}};
    constexpr double kLatency = 1.17;
    const ResidentPlan &p = c->resident;
    const int32_t sms = std::max(1, c->sm_count), rounds = F / sms + (F % sms != 0);
    double work = kSlotNs[o.check_rule == LDPC_RULE_SUM_PRODUCT ? 0 : 1][degree_class(p)] * 1e-3 * p.slots;
    if (!sh.lam_shared) work *= 1.23;
    if (msg_bytes(o.msg_dtype) == 1) work *= 1.08;
    return per_sm <= 1 ? rounds * (work + kLatency) : rounds * work + kLatency;
}

// Launches (one check kernel a degree bin), a time per slot and padded frame,
// and the messages and posteriors that L2 does not hold at 6.4 TB/s.
static double passes_us(const ldpc_code *c, int32_t F, const ldpc_decode_opts_t &o) {
    constexpr double kFramePs[2][4] = {{1.20, 1.96, 2.50, 5.86}, {1.73, 2.12, 2.67, 3.27}};
    constexpr double kL2 = 47e6;
    const ResidentPlan &p = c->resident;
    int bins = 0;
    for (int b = 0; b < kNumCheckBins; ++b) bins += c->bin_off[b + 1] > c->bin_off[b] ? 1 : 0;
    const int dc = degree_class(p);
    const double ps = kFramePs[o.check_rule == LDPC_RULE_SUM_PRODUCT ? 0 : 1][dc];
    auto chunk = [&](int64_t frames) {
        // up to 64 frames of narrow checks take the time of 32
        const double Fp = (double)(frames <= 32 || (frames <= 64 && dc < 3) ? 32 : (frames <= 64 ? 64 : (frames + 127) / 128 * 128));
        const double bytes = ((double)p.slots * msg_bytes(o.msg_dtype) + 4.0 * c->n) * Fp;
        return 7.2 + 3.2 * (bins - 1) + 5e-5 * p.slots + ps * 1e-6 * p.slots * Fp +
               std::max(0.0, bytes - kL2) / 6.4e6;
    };
    double us = (F / kPassChunk) * chunk(kPassChunk);
    if (F % kPassChunk) us += chunk(F % kPassChunk);
    return us;
}

ResidentShape resident_shape(const ldpc_code *c, int32_t F, int32_t max_iter, const ldpc_decode_opts_t &o,
                             bool wherever_it_fits) {
    ResidentShape sh;
    const ResidentPlan &p = c->resident;
    if (!p.ok || F <= 0 || o.frames_per_lane || o.check_schedule || o.tile_frames || o.streams || o.r_out || o.profile ||
        o.check_rule == LDPC_RULE_SP_TABLE)
        return sh;
    const size_t nv = (size_t)resident_vars(p.n_vg, p.n_wv);
    auto bytes = [&](bool lam) {
        return 16 + nv * 4 * (lam ? 2 : 1) + (size_t)(p.slots + 4) * msg_bytes(o.msg_dtype);
    };
    sh.lam_shared = bytes(true) <= (size_t)kResidentSmem;
    sh.smem = bytes(sh.lam_shared);
    if (sh.smem > (size_t)kResidentSmem) return ResidentShape{};
    const int32_t sms = std::max(1, c->sm_count);
    const int32_t per_sm = (int32_t)((size_t)228 * 1024 / (sh.smem + 1024));
    // Fixed iterations: the faster one (10 iterations, passes / here: n = 6000 rate
    // 1/2, 304 frames, half 196 / 147 us; n = 5000 rate 5/6, 1000 frames 1735 / 795;
    // n = 8000 rate 1/2, int8, 1600 frames 911 / 1079; n = 9000 rate 3/4, 32 frames
    // 130 / 165). Early exit stops every frame on its own here, while the passes keep
    // a group of 64-128 frames running until its last one stops and launch up to
    // max_iter: calls whose frames stop early gain, the more the larger max_iter is
    // (n = 10000, 620 frames, bfloat16, max_iter 50, 0.4 dB above the code's
    // threshold 763 / 433 us), and calls whose frames use all their iterations lose an
    // iteration's ratio (the same 1.5 dB below it 2370 / 2700). A call does not know which it
    // has, so an iteration may cost up to 1.2 times as much here at max_iter 20 and
    // 1.4 from 33 on, near where the sums of both losses over the timed codes are
    // least. streams = 1 keeps the passes. Against the passes, in 35 codes: fixed
    // iterations at most 1.19 times their time (0.70 in the geometric mean of 2015
    // calls), frames that never stop 1.45 (0.66 of 2821), that stop 1.17 (0.43 of 6851).
    if (!wherever_it_fits) {
        const double limit = o.early_exit ? std::min(1.4, 1.05 + 0.015 * std::max(0, max_iter - 10)) : 1.05;
        if (resident_us(c, sh, per_sm, F, o) > limit * passes_us(c, F, o)) return ResidentShape{};
    }
    // Warps of a CTA. 64 registers a thread let 32 warps run on an SM (16 where
    // checks of degree above 12 take 128). With many frames to each SM, few warps
    // a CTA and many CTAs: one CTA's barriers are covered by the others (n = 576,
    // 3 / 8 warps: 522 / 813 us; n = 1008, 4 / 16 warps 608 / 770 us, 10,000
    // frames, 10 iterations). With few, the slowest frame decides and takes 16
    // warps (n = 1008, 1000 frames, 4 / 8 / 16 warps: 150 / 135 / 133 us; n =
    // 4096, 355 frames, 8 / 16 warps 433 / 312 us), or 32 where no SM has a second
    // frame (n = 5000, 32 frames, bfloat16, 50 iterations 16 / 32 warps 313 / 255 us).
    // Short codes of wide checks would leave one CTA an SM by their registers: few
    // warps there from the second frame of an SM on (n = 576 rate 5/6, 1000 frames, 10
    // iterations 151 us with nine warps, 70 with four; codes with fewer than
    // eight frames an SM keep 16: n = 6000 rate 3/4, int8, 400 frames 329 / 486 us).
    const int32_t work = std::max({p.n_cg, (p.n_vg + 1) / 2, 1});  // warps with something to do
    const double per = (double)F / sms;                            // frames to an SM
    const int32_t fit = p.dclass <= 12 || o.check_rule != LDPC_RULE_SUM_PRODUCT ? 32 : 16;
    int32_t warps = per_sm <= 1 || F <= sms ? 32 : 16;
    if (per >= (o.early_exit ? 32 : 8)) {
        warps = std::max((fit + per_sm - 1) / per_sm, std::min(4, p.n_cg));
    } else if (per >= 8 && per_sm >= 4) {
        warps = 8;
    } else if (fit < 32 && !o.early_exit && per_sm >= 8 && F > sms) {
        const int32_t at_once = std::min(per_sm, (F + sms - 1) / sms);
        warps = std::max((fit + at_once - 1) / at_once, std::min(4, p.n_cg));
    }
    sh.threads = 32 * std::min(warps, work);
    return sh;
}

cudaError_t launch_resident(const ldpc_code *c, const ResidentShape &sh, const float *llr, int32_t F, int32_t max_iter,
                            const ldpc_decode_opts_t &o, float l_max, uint8_t *bits, int32_t *iters, uint8_t *ok,
                            float *post, cudaStream_t s, int64_t *launched) {
    NvtxRange nvtx_decode("ldpc decode (one SM a frame)");
    const ResidentPlan &p = c->resident;
    ResidentArgs a{};
    a.crow = reinterpret_cast<const uint16_t *>(p.tab + p.off[0]);
    a.cg = reinterpret_cast<const uint32_t *>(p.tab + p.off[1]);
    a.place = reinterpret_cast<const uint16_t *>(p.tab + p.off[2]);
    a.var = reinterpret_cast<const uint16_t *>(p.tab + p.off[3]);
    a.wide = reinterpret_cast<const int4 *>(p.tab + p.off[4]);
    a.list = reinterpret_cast<const uint16_t *>(p.tab + p.off[5]);
    const int mb = msg_bytes(o.msg_dtype), vt = 6 + 3 * (mb == 4 ? 2 : mb - 1);
    a.v4 = reinterpret_cast<const uint4 *>(p.tab + p.off[vt]);
    a.v8 = reinterpret_cast<const uint4 *>(p.tab + p.off[vt + 1]);
    a.v16 = reinterpret_cast<const uint4 *>(p.tab + p.off[vt + 2]);
    a.n_cg = p.n_cg;
    a.n_vg = p.n_vg;
    a.n_v1 = p.n_v1;
    a.n_v3 = p.n_v3;
    a.n_v8 = p.n_v8;
    a.n_v16 = p.n_v16;
    a.n_wc = p.n_wc;
    a.n_wv = p.n_wv;
    a.n = c->n;
    a.F = F;
    a.slots = p.slots;
    a.max_iter = max_iter;
    a.early = o.early_exit ? 1 : 0;
    a.lam_shared = sh.lam_shared ? 1 : 0;
    zero_sign(c, F, &a);
    a.l_max = l_max;
    a.phi_lmax = (float)std::log1p(2.0 / std::expm1((double)l_max));
    a.r_max = (float)std::exp((double)l_max);
    a.ms_alpha = o.rule_alpha > 0.0f ? o.rule_alpha : 1.0f;
    a.ms_beta = o.rule_beta;
    a.ms_table = o.check_rule == LDPC_RULE_MIN_SUM_ADAPTIVE ? c->d.ms_table : nullptr;
    a.llr = llr;
    a.bits = bits;
    a.iters = iters;
    a.ok = ok;
    a.post = post;
    return with_msg_type(o.msg_dtype, [&](auto tag) {
        using M = typename decltype(tag)::type;
        return o.check_rule == LDPC_RULE_SUM_PRODUCT ? launch_resident_m<M, 0>(a, p.dclass, sh, s, launched)
                                                     : launch_resident_m<M, 1>(a, p.dclass, sh, s, launched);
    });
}

}  // namespace ldpc

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
    std::stable_sort(ids.begin(), ids.end(), [&](int32_t a, int32_t b) { return deg(a) > deg(b); });
    std::vector<std::vector<int32_t>> groups;
    for (int32_t id : ids) {
        bool cut = groups.empty() || groups.back().size() == 32;
        for (int32_t b : borders) cut = cut || (deg(groups.back()[0]) > b && deg(id) <= b);
        if (cut) groups.emplace_back();
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
    const auto vg = degree_groups(vars, c->col_ptr, {});
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
    for (const auto &g : vg) {
        const int32_t d0 = degree(c->col_ptr, g[0]);
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

// The sum-product kernels count an input of exactly +0 as a positive one, all
// but the register kernel (k_check_reg). The resident decode counts it as the
// kernel does that serves the check in a decode with passes: frames from
// `from` on (chunks of up to 32 frames) for degrees up to 16, `wide` above.
static void zero_sign(const ldpc_code *c, int32_t F, ResidentArgs *a) {
    constexpr int32_t chunk = 8192;  // frames of a chunk of the pass kernels
    const int32_t last = F > chunk ? F % chunk : F;
    a->zero_neg_from = last > 0 && last <= 32 ? F - last : INT_MAX;
    const bool staged = c->bin_off[5] - c->bin_off[4] >= kWideBinAnyKernel;
    a->zero_neg_wide = staged ? 0 : (c->bin_max_degree[4] > 18 ? 2 : 1);  // 2: all frames, 1: from zero_neg_from
}

void resident_plan_free(ResidentPlan *p) {
    cudaFree(p->tab);
    *p = ResidentPlan{};
}

ResidentShape resident_shape(const ldpc_code *c, int32_t F, int32_t max_iter, const ldpc_decode_opts_t &o) {
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
    // Fixed iterations take a frame and pass of the same time either way, and
    // the pass kernels are the faster ones for long codes in narrow formats,
    // where only one or two frames fit on an SM and there are more frames than
    // that: n = 16200 int8, 1000 frames, 10 iterations 821 us against 1072; n =
    // 8192 int8 717 / 833; n = 10000 bfloat16, 160 frames 225 / 263; FP32, one
    // frame an SM, 160 frames 249 / 339, 304 frames 353 / 347. Shorter codes and
    // FP32: n = 4096 bfloat16, 10,000 frames 2459 / 2227, n = 2048 FP32, 6000
    // frames 1154 / 822, n = 576, 10,000 frames 543 / 522. Early exit stops every
    // frame on its own and is faster here throughout (n = 16200 int8, 1000 frames
    // 2694 / 2376, one frame n = 1008 149 / 17).
    // `ahead` is that ratio for full waves of CTAs; a last wave that is not full
    // takes as long.
    const bool narrow = msg_bytes(o.msg_dtype) < 4;
    const int64_t cap = (int64_t)per_sm * sms;
    // A few frames of a long code leave most SMs idle here, while the passes spread
    // one frame over all of them (n = 16200, 4 frames, 10 iterations 138 / 172 us,
    // n = 7152, 5 frames, 50 iterations 408 / 439; n = 6376, 11 frames 184 / 166, n
    // = 16200, 109 frames 750 / 571). So few iterations that a long code's frames
    // mostly use them all count as fixed.
    const bool fixed = !o.early_exit || (max_iter <= 12 && p.slots > 32000);
    if (fixed && F <= 64 && p.slots > 26000) return ResidentShape{};
    if (fixed && per_sm <= 2 && F > cap) {
        const double ahead = (narrow ? 0.7 : 0.9) + 0.1 * per_sm +
                             (o.check_rule == LDPC_RULE_SUM_PRODUCT ? 0.0 : (narrow ? 0.1 : 0.3));
        if (ahead * (double)F < (double)((F + cap - 1) / cap * cap)) return ResidentShape{};
    }
    // Warps of a CTA. 64 registers a thread let 32 warps run on an SM (16 where
    // checks of degree above 12 take 128). With many frames to each SM, few warps
    // a CTA and many CTAs: one CTA's barriers are covered by the others (n = 576,
    // 3 / 8 warps: 522 / 813 us; n = 1008, 4 / 16 warps 608 / 770 us, 10,000
    // frames, 10 iterations). With few, the slowest frame decides and takes 16
    // warps (n = 1008, 1000 frames, 4 / 8 / 16 warps: 150 / 135 / 133 us; n =
    // 4096, 355 frames, 8 / 16 warps 433 / 312 us).
    const int32_t work = std::max({p.n_cg, (p.n_vg + 1) / 2, 1});  // warps with something to do
    const double per = (double)F / sms;                            // frames to an SM
    int32_t warps = per_sm <= 1 ? 32 : 16;
    if (per >= (o.early_exit ? 32 : 8)) {
        const int32_t fit = p.dclass <= 12 || o.check_rule != LDPC_RULE_SUM_PRODUCT ? 32 : 16;
        warps = std::max((fit + per_sm - 1) / per_sm, std::min(4, p.n_cg));
    } else if (per >= 8 && per_sm >= 4) {
        warps = 8;
    }
    sh.threads = 32 * std::min(warps, work);
    return sh;
}

cudaError_t launch_resident(const ldpc_code *c, const ResidentShape &sh, const float *llr, int32_t F, int32_t max_iter,
                            const ldpc_decode_opts_t &o, float l_max, uint8_t *bits, int32_t *iters, uint8_t *ok,
                            float *post, cudaStream_t s, int64_t *launched) {
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

// The resident decode: every iteration of a frame inside one CTA, its
// messages, posteriors and channel LLRs in that CTA's shared memory. This
// header holds the plan (the code's tables in the order the kernel walks
// them), the kernel's arguments and the launcher.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "ldpc.h"

struct ldpc_code;

namespace ldpc {

// Tables of one code. Checks and variables are sorted by degree and walked in
// groups of 32, one node per lane of a warp. Input k of the check in lane l of a
// group with base b has its message in slot b + 32 k + l, so a warp's message
// accesses are consecutive words. Variables are renumbered in their sorted
// order, so a warp's posteriors and channel LLRs are consecutive too. The
// tables hold a lane's entries next to each other, so a node's row is read by
// one or a few vector loads, as byte offsets into the CTA's arrays (16 bits for
// variables, 32 for messages, a table per message size): a shared-memory access
// then takes no address arithmetic but the row's unpacking. A missing entry of a check is
// kResidentPad; a missing edge of a variable is the slot past the last one,
// whose message is always -0 (+0 in int8, which has no other zero, so that a sum
// with at least one message is the same). The checks of degree above 32 and the variables
// of degree above kWideVarDegree follow, each worked on by a warp.
constexpr uint16_t kResidentPad = 0xFFFF;

struct ResidentPlan {
    bool ok = false;
    int32_t slots = 0;   // message slots (padding included, the -0 slot not)
    int32_t dclass = 0;  // inputs the check rows have room for: 4, 6 or 8 (rows of 8), 12, 18 (20) or 32
    int32_t n_cg = 0, n_vg = 0, n_v1 = 0, n_v3 = 0, n_v8 = 0, n_v16 = 0;  // groups; of them with variables of degree above 0, 2, 4, 8
    int32_t n_wc = 0, n_wv = 0;
    size_t off[15] = {0};          // byte offsets in tab of the tables below, in order
    unsigned char *tab = nullptr;  // device
};

// check group word: base / 32 (low 16 bits), largest degree (bits 16-21), bit 22: all 32 lanes have that degree
constexpr uint32_t kResidentFull = 1u << 22;

constexpr int kResidentSmem = 227 * 1024;  // shared memory a CTA may take

// entries of a check's table row
__host__ __device__ constexpr int resident_row(int dclass) { return dclass <= 4 ? 4 : (dclass <= 8 ? 8 : (dclass <= 12 ? 12 : (dclass <= 18 ? 20 : 32))); }

// internal variable indexes (a multiple of 4)
__host__ __device__ constexpr int resident_vars(int n_vg, int n_wv) { return (n_vg * 32 + n_wv + 3) / 4 * 4; }

struct ResidentArgs {
    const uint16_t *crow;        // [n_cg * 32][resident_row], variables as byte offsets (4 x internal index)
    const uint32_t *cg;          // [n_cg]
    // messages of a variable's edges as byte offsets: entries 0-3 of every variable, 4-7 of the first n_v8
    // groups, 8-15 of the first n_v16
    const uint4 *v4, *v8, *v16;
    const uint16_t *place;       // [n] internal index of a variable
    const uint16_t *var;         // [n_vg * 32 + n_wv] variable of an internal index
    const int4 *wide;            // n_wc checks (first slot, degree, first entry in list), n_wv variables (first entry, degree, internal index)
    const uint16_t *list;        // entries of the wide nodes
    int32_t n_cg, n_vg, n_v1, n_v3, n_v8, n_v16, n_wc, n_wv;
    int32_t n, F, f0, slots;  // frames f0 + blockIdx.x
    int32_t max_iter, early;
    int32_t lam_shared;  // channel LLRs kept in shared memory (else re-read from llr)
    // an input of exactly +0, or NaN, counts as negative: frames from zero_neg_from on; in checks of degree above 16
    // never (0), as the others (1) or always (2)
    int32_t zero_neg_from, zero_neg_wide;
    float l_max, phi_lmax, r_max, ms_alpha, ms_beta;
    const float2 *ms_table;
    const float *llr;
    uint8_t *bits;
    int32_t *iters;
    uint8_t *ok;
    float *post;
};

// Builds the plan's host tables and uploads them (device >= 0 selected).
cudaError_t resident_plan_create(const ldpc_code *c, ResidentPlan *p);
void resident_plan_free(ResidentPlan *p);

// Threads and shared memory of a decode of F frames, a CTA each; threads = 0
// when the resident decode does not serve it, or the pass kernels are the better
// choice (not asked for wherever_it_fits: a tuner that times both).
struct ResidentShape {
    int32_t threads = 0;
    bool lam_shared = true;
    size_t smem = 0;
};
ResidentShape resident_shape(const ldpc_code *c, int32_t F, int32_t max_iter, const ldpc_decode_opts_t &o,
                             bool wherever_it_fits = false);

// Adds the kernels it launches to `launched`.
cudaError_t launch_resident(const ldpc_code *c, const ResidentShape &sh, const float *llr, int32_t F, int32_t max_iter,
                            const ldpc_decode_opts_t &o, float l_max, uint8_t *bits, int32_t *iters, uint8_t *ok,
                            float *post, cudaStream_t s, int64_t *launched);

template <typename M, int RULE>
cudaError_t launch_resident_m(const ResidentArgs &a, int32_t dclass, const ResidentShape &sh, cudaStream_t s,
                              int64_t *launched);

}  // namespace ldpc

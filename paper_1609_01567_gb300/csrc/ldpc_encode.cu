// Systematic encoder of IRA codes (H = [H1 | H2], H2 the dual-diagonal
// staircase in columns k .. n-1): c = [u | p] with p_i = s_i xor p_(i-1),
// s = H1 u. The BER simulator (Section IV) needs codewords; the paper sends
// the all-zero word or encodes on the host. Here the whole chain (information
// bits, encoder, channel, decoder, error count) stays on the device.
//
// Frames travel bit-sliced: word g of a row holds one bit of frames
// 32g .. 32g + 31, so one XOR combines 32 frames.
//
// A code whose word fits in shared memory takes one kernel (k_encode_ira). The
// general path, for longer words, a few long ones and codes with a few very heavy
// checks:
//   1. pack      u [F][k] bytes      -> U [k][G] words
//   2. checks    s_i = xor over the H1 neighbours of check i of U[j], and
//                its running xor within a chunk of checks
//   3. carries   exclusive xor-scan of the chunk totals
//   4. write     c [F][n] bytes: the information bytes, then bit f of
//                p_i = (running xor) xor (carry of the chunk)
//
// The dense systematic encoder serves any code (lifted codes without a
// staircase included): the host reduces H over GF(2) once, and the device
// forms each parity bit as the xor of the information bits its reduced row
// holds.
#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

#include "ldpc_internal.h"

namespace ldpc {
namespace {

__global__ void k_pack_info(const uint8_t *__restrict__ info, int32_t F, int32_t k, int32_t G,
                            uint32_t *__restrict__ U) {
    const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= k) return;
    for (int32_t g = blockIdx.y; g < G; g += gridDim.y) {
        uint32_t w = 0;
        const int32_t nb = min(32, F - 32 * g);
        for (int32_t b = 0; b < nb; ++b) w |= (uint32_t)(info[(size_t)(32 * g + b) * k + j] & 1u) << b;
        U[(size_t)j * G + g] = w;
    }
}

// Checks are scanned in chunks of kChunk: one thread per (chunk, word
// column) forms s_i and its running xor inside the chunk, then one warp per
// word column turns the chunk totals into carries, and the write kernel
// applies the carry of each chunk.
constexpr int kChunk = 64;

__global__ void k_chunk_prefix(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col_idx, int32_t m,
                               int32_t k, int32_t G, const uint32_t *__restrict__ U, uint32_t *__restrict__ Pl,
                               uint32_t *__restrict__ T) {
    const int32_t nC = (m + kChunk - 1) / kChunk;
    const int64_t total = (int64_t)nC * G;
    for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < total;
         id += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = (int32_t)(id / G);
        const int32_t g = (int32_t)(id - (int64_t)c * G);
        const int32_t i1 = min(m, (c + 1) * kChunk);
        uint32_t run = 0;
        for (int32_t i = c * kChunk; i < i1; ++i) {
            uint32_t s = 0;
            for (int32_t e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
                const int32_t j = col_idx[e];
                if (j < k) s ^= U[(size_t)j * G + g];
            }
            run ^= s;
            Pl[(size_t)i * G + g] = run;
        }
        T[(size_t)c * G + g] = run;
    }
}

// Exclusive xor-scan of the chunk totals T[c][g] over c, in place: one warp
// per word column g.
__global__ void k_chunk_carry(uint32_t *__restrict__ T, int32_t nC, int32_t G) {
    const int lane = threadIdx.x & 31;
    const int32_t per = (nC + 31) / 32;
    const int32_t c0 = min(nC, lane * per), c1 = min(nC, c0 + per);
    for (int32_t g = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); g < G; g += gridDim.x * (blockDim.x / 32)) {
        uint32_t x = 0;
        for (int32_t c = c0; c < c1; ++c) x ^= T[(size_t)c * G + g];
        uint32_t inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc ^= y;
        }
        uint32_t run = inc ^ x;  // xor of the chunks before this lane's range
        for (int32_t c = c0; c < c1; ++c) {
            const uint32_t t = T[(size_t)c * G + g];
            T[(size_t)c * G + g] = run;
            run ^= t;
        }
    }
}

__global__ void k_write_codeword(const uint8_t *__restrict__ info, const uint32_t *__restrict__ Pl,
                                 const uint32_t *__restrict__ carry, int32_t F, int32_t n, int32_t k, int32_t G,
                                 uint8_t *__restrict__ cw) {
    const int64_t total = (int64_t)F * n;
    for (int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; id < total;
         id += (int64_t)gridDim.x * blockDim.x) {
        const int32_t f = (int32_t)(id / n);
        const int32_t j = (int32_t)(id - (int64_t)f * n);
        uint8_t v;
        if (j < k)
            v = info[(size_t)f * k + j] & 1u;
        else {
            const int32_t i = j - k, g = f >> 5;
            v = (uint8_t)(((Pl[(size_t)i * G + g] ^ carry[(size_t)(i / kChunk) * G + g]) >> (f & 31)) & 1u);
        }
        cw[id] = v;
    }
}

// ---------------------------------------------------------------------------
// IRA codes whose word fits in shared memory: one kernel, one CTA per eight
// frames. A byte of shared memory holds one bit position of the CTA's eight
// frames. The information bytes are read once, written to the codeword and
// packed on the way (byte lane b of (w & 0x01..01) << f over f). Each warp
// forms s_i of a contiguous range of checks, lane = check, from a table with
// the lanes' entries next to each other, with a running xor by shuffles; after
// one barrier for the warps' totals it writes its range as bytes of the eight
// rows, W bytes a store. Bound by the bytes read and written once and by the
// latency of the table rows between them: n = 64800, 1024 frames 259 -> 36-39 us
// against the four kernels of the general path, whose write kernel divides a
// 64-bit index for every codeword byte (100 MB at the copy rate: 15 us). Rows
// read through row_ptr and col_idx instead of the padded table: 54 us, every
// load of a warp touching six lines.
// ---------------------------------------------------------------------------

template <int W>
struct Wide;
template <>
struct Wide<1> {
    using T = uint8_t;
};
template <>
struct Wide<4> {
    using T = uint32_t;
};
template <>
struct Wide<16> {
    using T = uint4;
};
__device__ __forceinline__ uint32_t ones_of(uint8_t x) { return x & 1u; }
__device__ __forceinline__ uint32_t ones_of(uint32_t x) { return x & 0x01010101u; }
__device__ __forceinline__ uint4 ones_of(uint4 x) {
    return make_uint4(x.x & 0x01010101u, x.y & 0x01010101u, x.z & 0x01010101u, x.w & 0x01010101u);
}
__device__ __forceinline__ void add_frame(uint32_t &acc, uint32_t x, int f) { acc |= x << f; }
__device__ __forceinline__ void add_frame(uint4 &acc, uint4 x, int f) {
    acc.x |= x.x << f;
    acc.y |= x.y << f;
    acc.z |= x.z << f;
    acc.w |= x.w << f;
}
__device__ __forceinline__ uint32_t frame_of(uint32_t x, int f) { return (x >> f) & 0x01010101u; }
__device__ __forceinline__ uint4 frame_of(uint4 x, int f) {
    return make_uint4(frame_of(x.x, f), frame_of(x.y, f), frame_of(x.z, f), frame_of(x.w, f));
}
__device__ __forceinline__ uint32_t flip(uint32_t x, uint32_t c) { return x ^ c; }
__device__ __forceinline__ uint4 flip(uint4 x, uint32_t c) { return make_uint4(x.x ^ c, x.y ^ c, x.z ^ c, x.w ^ c); }

constexpr int kWordFrames = 8;
constexpr int kWarpTotals = 32 * sizeof(uint32_t);

// WI: bytes per access of the information part, WP: of the parity part.
template <int WI, int WP>
__global__ void __launch_bounds__(1024) k_encode_ira(const uint8_t *__restrict__ info,
                                                     const int2 *__restrict__ groups,
                                                     const uint32_t *__restrict__ rows, int32_t F, int32_t m,
                                                     int32_t k, uint8_t *__restrict__ cw) {
    extern __shared__ __align__(16) uint8_t es[];
    uint32_t *total = reinterpret_cast<uint32_t *>(es);  // [32] xor of a warp's range
    uint8_t *U = es + kWarpTotals;                       // [k] bits of the information positions, then a zero
    uint8_t *P = U + ((k + 16) & ~15);                   // [m] running xor within a warp's range
    const int32_t n = k + m;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
    const int64_t f0 = (int64_t)blockIdx.x * kWordFrames;
    const int nf = (int)min((int64_t)kWordFrames, F - f0);
    {
        using T = typename Wide<WI>::T;
        using A = std::conditional_t<WI == 16, uint4, uint32_t>;
        for (int32_t q = tid; q < k / WI; q += blockDim.x) {
            A x[kWordFrames];
#pragma unroll
            for (int f = 0; f < kWordFrames; ++f)
                x[f] = f < nf ? ones_of(reinterpret_cast<const T *>(info + (f0 + f) * k)[q]) : A{};
            A acc{};
#pragma unroll
            for (int f = 0; f < kWordFrames; ++f) {
                add_frame(acc, x[f], f);
                if (f < nf) {
                    if constexpr (WI == 1) cw[(f0 + f) * n + q] = (uint8_t)x[f];
                    else reinterpret_cast<T *>(cw + (f0 + f) * n)[q] = x[f];
                }
            }
            if constexpr (WI == 1) U[q] = (uint8_t)acc;
            else reinterpret_cast<T *>(U)[q] = acc;
        }
    }
    if (tid == 0) U[k] = 0;
    __syncthreads();
    const int32_t per = ((m + warps - 1) / warps + 127) / 128 * 128;
    const int32_t lo = min(m, warp * per), hi = min(m, lo + per);
    uint32_t run = 0;
    for (int32_t i0 = lo; i0 < hi; i0 += 128) {
        // four groups of 32 checks, byte c of w for group c, so that the shuffles of
        // the running xor serve four groups
        uint32_t w = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int32_t g = i0 / 32 + c;
            if (32 * g >= hi) continue;
            const int2 gd = groups[g];  // first entry, entries per lane
            const uint32_t *p = rows + gd.x + lane;
            uint32_t x = 0;
            for (int32_t e = 0; e < gd.y; e += 8) {
                uint32_t j[8];
#pragma unroll
                for (int v = 0; v < 8; ++v) j[v] = e + v < gd.y ? __ldg(p + 32 * (e + v)) : (uint32_t)k;
#pragma unroll
                for (int v = 0; v < 8; ++v) x ^= U[j[v]];
            }
            w |= x << (8 * c);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w ^= y;
        }
        uint32_t t = __shfl_sync(0xffffffffu, w, 31);  // the groups' totals, then the xor of those before
        t ^= t << 8;
        t ^= t << 16;
        w ^= (t << 8) ^ (run * 0x01010101u);
        run ^= t >> 24;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (i0 + 32 * c + lane < hi) P[i0 + 32 * c + lane] = (uint8_t)(w >> (8 * c));
    }
    if (lane == 0) total[warp] = run;
    __syncthreads();
    // xor of the totals of the warps before this one, in every byte
    const uint32_t before = lane < warp ? total[lane] : 0u;
    const uint32_t carry = __reduce_xor_sync(0xffffffffu, before) * 0x01010101u;
    for (int32_t q = lo / WP + lane; q < (hi + WP - 1) / WP; q += 32) {
        using T = typename Wide<WP>::T;
        using A = std::conditional_t<WP == 16, uint4, uint32_t>;
        const A x = flip(A(reinterpret_cast<const T *>(P)[q]), carry);
#pragma unroll
        for (int f = 0; f < kWordFrames; ++f) {
            if (f >= nf) break;
            uint8_t *dst = cw + (f0 + f) * n + k;
            if constexpr (WP == 1) dst[q] = (uint8_t)frame_of(x, f);
            else reinterpret_cast<T *>(dst)[q] = frame_of(x, f);
        }
    }
}

constexpr int kEncodeSmem = 224 * 1024;  // a word's bits; the warps' totals come on top

// Bytes an access of the one-kernel form takes in the information or parity part:
// every row start and the part's length are multiples of them.
int ira_width(const uint8_t *info, const uint8_t *cw, int32_t m, int32_t k, bool par) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(cw) | (uintptr_t)(k + m) | (uintptr_t)k |
                        (par ? (uintptr_t)m : reinterpret_cast<uintptr_t>(info));
    return a % 16 == 0 ? 16 : (a % 4 == 0 ? 4 : 1);
}

// Few long words leave most SMs idle in the one-kernel form, whose CTA then takes a
// time per bit, the more the narrower its accesses are; the general path spreads
// them over the GPU. n = 200,001, general / one kernel: 8 frames 100 / 146 us, 100
// frames 142 / 150, 300 frames 244 / 152; n = 130,001, 8 frames 96 / 97; n =
// 229,000 (four bytes an access) 109 / 119; n = 200,000 (16 bytes) 100 / 86.
bool ira_one_kernel(int width, int32_t F, int32_t n) {
    const double ns = width == 16 ? 0.43 : (width == 4 ? 0.52 : 0.53 + 0.0275 * std::min(F, kWordFrames));
    return ns * 1e-3 * n < 90.0 + 0.45 * F;
}

cudaError_t launch_encode_ira(const uint8_t *info, const int2 *groups, const uint32_t *rows, int32_t F, int32_t m,
                              int32_t k, uint8_t *cw, cudaStream_t s) {
    const size_t smem = kWarpTotals + (size_t)((k + 16) & ~15) + ((m + 15) & ~15);
    const int32_t n = k + m;
    const int wi = ira_width(info, cw, m, k, false), wp = ira_width(info, cw, m, k, true);
    const int32_t threads = n <= 2048 ? 128 : (n <= 8192 ? 256 : (n <= 16384 ? 512 : 1024));
    auto go = [&](auto kernel) {
        // all of the kernel's shared memory is dynamic, so that `smem` is what the
        // 48 KB limit of a launch without the opt-in applies to
        cudaError_t e = cudaSuccess;
        if (smem > 48 * 1024)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEncodeSmem + kWarpTotals);
        if (e != cudaSuccess) return e;
        kernel<<<(unsigned)((F + kWordFrames - 1) / kWordFrames), threads, smem, s>>>(info, groups, rows, F, m, k,
                                                                                      cw);
        return cudaGetLastError();
    };
    auto pick = [&](auto wi) {
        constexpr int WI = decltype(wi)::value;
        if (wp == 16) return go(k_encode_ira<WI, 16>);
        if (wp == 4) return go(k_encode_ira<WI, 4>);
        return go(k_encode_ira<WI, 1>);
    };
    if (wi == 16) return pick(std::integral_constant<int, 16>{});
    if (wi == 4) return pick(std::integral_constant<int, 4>{});
    return pick(std::integral_constant<int, 1>{});
}

// ---------------------------------------------------------------------------
// Dense systematic encoder (any code): parity row i of the reduced H sets the
// bit of its pivot column to the xor of the information bits it holds, a
// product over GF(2). Bit-sliced: word g of a row holds 32 frames, Gp words a
// row (a multiple of 32, one per lane).
// ---------------------------------------------------------------------------

// U [k][Gp] from info [F][k]; also clears P [r][Gp]. A CTA packs 4 x 32
// columns of eight words: lane q takes four bytes of each of a word's 32
// frames, from the one or two aligned words that hold them (rows of k bytes
// start anywhere), and the tile leaves as 32-byte runs.
template <bool kEnds>
__global__ void __launch_bounds__(256) k_dense_pack(const uint8_t *__restrict__ info, int32_t F, int32_t k, int32_t Gp,
                                                    uint32_t *__restrict__ U, uint32_t *__restrict__ P,
                                                    int64_t p_words) {
    __shared__ uint32_t tile[128][9];
    for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 256 + threadIdx.x; i < p_words;
         i += (int64_t)gridDim.x * gridDim.y * 256)
        P[i] = 0u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t j = blockIdx.x * 128 + 4 * lane;
    const int32_t g = blockIdx.y * 8 + warp;
    const int need = min(4, k - j);  // columns of this lane; more bytes than that go nowhere
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    // kEnds: info's first or last byte is unaligned, so that the word that holds it
    // reaches past the buffer: put together from its bytes inside. (For all calls:
    // n = 8192, 1000 frames 40.7 us instead of 38.9; byte loads of all columns at the
    // ends: up to 4 us longer.)
    uintptr_t first = 0, last = 0;
    uint32_t head = 0, tail = 0;
    if constexpr (kEnds) {
        const uintptr_t lo = reinterpret_cast<uintptr_t>(info), hi = lo + (size_t)F * k;
        first = lo & 3 ? lo & ~(uintptr_t)3 : 0;
        last = hi & 3 ? hi & ~(uintptr_t)3 : 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uintptr_t h = first + i, t = last + i;
            if (first && h >= lo && h < hi) head |= (uint32_t)*reinterpret_cast<const uint8_t *>(h) << (8 * i);
            if (last && t >= lo && t < hi) tail |= (uint32_t)*reinterpret_cast<const uint8_t *>(t) << (8 * i);
        }
    }
    auto word = [&](uintptr_t a) {
        if (!kEnds) return *reinterpret_cast<const uint32_t *>(a);
        uint32_t x = a == first ? head : tail;
        if (a != first && a != last) x = *reinterpret_cast<const uint32_t *>(a);
        return x;
    };
#pragma unroll
    for (int b = 0; b < 4; ++b) {  // eight frames: byte i of acc has column j + i
        uint32_t acc = 0;
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            const int64_t fr = 32 * (int64_t)g + 8 * b + f;
            uint32_t x = 0;
            if (fr < F && need > 0) {
                const uintptr_t at = reinterpret_cast<uintptr_t>(info + fr * k + j);
                const uintptr_t w32 = at & ~(uintptr_t)3;
                const int off = (int)(at & 3);
                x = __funnelshift_r(word(w32), off + need > 4 ? word(w32 + 4) : 0u, 8 * off);
            }
            acc |= (x & 0x01010101u) << f;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] |= ((acc >> (8 * i)) & 0xFFu) << (8 * b);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) tile[4 * lane + i][warp] = w[i];
    __syncthreads();
    for (int i = threadIdx.x; i < 128 * 8; i += 256) {
        const int32_t c = blockIdx.x * 128 + i / 8;
        if (c < k) U[(size_t)c * Gp + blockIdx.y * 8 + i % 8] = tile[i / 8][i % 8];
    }
}

// P ^= R U over GF(2) by tables (the method of four Russians, Arlazarov,
// Dinic, Kronrod and Faradzhev 1970): for each four information bits a table
// of the 16 xors of their words, built once per CTA and read by its kDenseRows
// parity rows, so a row takes one shared-memory word a lane for four bits
// instead of two xors on average. A half-warp's lanes are the 32 words of a
// group, two each, so a table access of a warp reads two conflict-free rows of
// 128 bytes for two parity rows at once; a CTA takes a slice of the
// information bits and adds its part to P by atomic xor. Bound by shared-memory
// rows and the address arithmetic around them: n = 8192 with 4093 dense rows,
// 1000 frames: the whole call 264 -> 39 us against a thread walking the set
// bits of a row, one dependent load each; a parity row a warp access (one word a
// lane): 50 us, and with two CTAs an SM instead of four: 63 us.
constexpr int kDenseRows = 128;
constexpr int32_t kDenseFrames = 65536;  // frames a launch of each kernel (bounds the grids and the scratch)

__global__ void __launch_bounds__(256) k_dense_parity(const uint32_t *__restrict__ R, int32_t r, int32_t k, int32_t kw,
                                                      int32_t slice, const uint32_t *__restrict__ U, int32_t Gp,
                                                      uint32_t *__restrict__ P) {
    __shared__ __align__(16) uint32_t tab[2][8][16][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kPer = kDenseRows / 8;  // rows per warp
    const int32_t row0 = blockIdx.x * kDenseRows + warp * kPer;
    const int32_t w0 = blockIdx.y * slice, w1 = min(kw, w0 + slice);
    const uint32_t *Ug = U + blockIdx.z * 32 + lane;
    const int half = lane >> 4, pair = lane & 15;  // parity row 2 i + half, words 2 pair and 2 pair + 1
    const unsigned char *tb = reinterpret_cast<const unsigned char *>(tab);
    uint2 acc[kPer / 2];
#pragma unroll
    for (int i = 0; i < kPer / 2; ++i) acc[i] = make_uint2(0u, 0u);
    const bool mine = lane < kPer && row0 + lane < r;
    const uint32_t *Rl = R + (size_t)(mine ? row0 + lane : 0) * kw;
    uint32_t u[4], rw = 0;
    auto fetch = [&](int32_t w) {  // this warp's four information words, and its rows' 32 coefficients
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int32_t j = 32 * w + 4 * warp + b;
            u[b] = w < w1 && j < k ? Ug[(size_t)j * Gp] : 0u;
        }
        rw = w < w1 && mine ? Rl[w] : 0u;
    };
    fetch(w0);
    for (int32_t w = w0; w < w1; ++w) {
        uint32_t(*t)[16][32] = tab[(w - w0) & 1];
        uint32_t x = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {  // Gray code: one xor per entry
            const int code = i ^ (i >> 1);
            if (i) {
                const int b = (i & 1) ? 0 : ((i & 2) ? 1 : ((i & 4) ? 2 : 3));
                x ^= u[b];
            }
            t[warp][code][lane] = x;
        }
        const uint32_t coef = rw;
        fetch(w + 1);
        __syncthreads();  // one barrier a step: the tables alternate
        const uint32_t at = (uint32_t)pair * 8u + (((w - w0) & 1) ? (uint32_t)sizeof(tab[0]) : 0u);
#pragma unroll
        for (int i = 0; i < kPer / 2; ++i) {
            const uint32_t c = __shfl_sync(0xffffffffu, coef, 2 * i + half);
            uint2 y = make_uint2(0u, 0u);
#pragma unroll
            for (int q = 0; q < 8; ++q) {  // byte offset of the entry of bits 4 q .. 4 q + 3: 128 times their value
                const uint32_t e = (q < 2 ? c << (7 - 4 * q) : c >> (4 * q - 7)) & 0x780u;
                const uint2 x = *reinterpret_cast<const uint2 *>(tb + q * (int)sizeof(tab[0][0]) + (e | at));
                y.x ^= x.x;
                y.y ^= x.y;
            }
            acc[i].x ^= y.x;
            acc[i].y ^= y.y;
        }
    }
#pragma unroll
    for (int i = 0; i < kPer / 2; ++i) {
        const int32_t row = row0 + 2 * i + half;
        if (row >= r) continue;
        uint32_t *dst = P + (size_t)row * Gp + blockIdx.z * 32 + 2 * pair;
        atomicXor(dst, acc[i].x);
        atomicXor(dst + 1, acc[i].y);
    }
}

// c[f][j] from the words of its row: information row colmap[j] of U, or parity
// row -1 - colmap[j] of P. A thread holds four columns of one word (32
// frames): byte b of the four words makes eight frames' four bytes.
template <bool V4>
__global__ void __launch_bounds__(256) k_dense_write(const uint32_t *__restrict__ U, const uint32_t *__restrict__ P,
                                                     const int32_t *__restrict__ colmap, int32_t F, int32_t n,
                                                     int32_t Gp, uint8_t *__restrict__ cw) {
    const int32_t j = (blockIdx.x * 256 + threadIdx.x) * 4;
    const int32_t g = blockIdx.y;
    if (j >= n) return;
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int32_t cm = j + i < n ? colmap[j + i] : 0;
        w[i] = j + i < n ? (cm >= 0 ? U[(size_t)cm * Gp + g] : P[(size_t)(-1 - cm) * Gp + g]) : 0u;
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const uint32_t s = (uint32_t)(b | (4 + b) << 4);
        const uint32_t x = __byte_perm(__byte_perm(w[0], w[1], s), __byte_perm(w[2], w[3], s), 0x5410u);
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            const int64_t fr = 32 * (int64_t)g + 8 * b + f;
            if (fr >= F) return;
            const uint32_t y = frame_of(x, f);
            uint8_t *dst = cw + fr * n + j;
            if (V4) {
                *reinterpret_cast<uint32_t *>(dst) = y;
            } else {
                for (int i = 0; i < 4; ++i)
                    if (j + i < n) dst[i] = (uint8_t)(y >> (8 * i));
            }
        }
    }
}

unsigned grid_of(int64_t threads, int per_block, int sm_count) {
    int64_t b = (threads + per_block - 1) / per_block;
    const int64_t cap = (int64_t)std::max(sm_count, 1) * 16;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

}  // namespace
}  // namespace ldpc

namespace ldpc {

// The information columns of the checks in groups of 32, entry e of a group's
// lane l at first + 32 e + l (k, a zero bit, where a check has fewer). Not made
// for a code whose padded table would be four times its edges (a few very
// heavy checks among light ones): the general path serves it.
cudaError_t encoder_rows_create(ldpc_code *c) {
    if (c->ira_k < 0 || c->m == 0 || (size_t)c->n + 48 > (size_t)kEncodeSmem) return cudaSuccess;
    const uint32_t k = (uint32_t)c->ira_k;
    try {
        std::vector<int2> groups;
        std::vector<uint32_t> rows;
        rows.reserve((size_t)c->E);
        for (int32_t i0 = 0; i0 < c->m; i0 += 32) {
            const int32_t i1 = std::min(c->m, i0 + 32);
            int32_t in[32] = {0}, width = 0;  // information columns of a check
            for (int32_t i = i0; i < i1; ++i) {
                for (int32_t e = c->row_ptr[i]; e < c->row_ptr[i + 1]; ++e) in[i - i0] += (uint32_t)c->col_idx[e] < k;
                width = std::max(width, in[i - i0]);
            }
            const size_t first = rows.size();
            groups.push_back(make_int2((int)first, width));
            rows.resize(first + 32 * (size_t)width, k);
            for (int32_t i = i0; i < i1; ++i) {
                uint32_t *to = rows.data() + first + (i - i0);
                for (int32_t e = c->row_ptr[i]; e < c->row_ptr[i + 1]; ++e) {
                    if ((uint32_t)c->col_idx[e] >= k) continue;
                    *to = (uint32_t)c->col_idx[e];
                    to += 32;
                }
            }
            if (rows.size() > 4 * (size_t)c->E + 4096) return cudaSuccess;
        }
        cudaError_t e = cudaMalloc(&c->ira_groups, sizeof(int2) * groups.size());
        if (e == cudaSuccess) e = cudaMalloc(&c->ira_rows, sizeof(uint32_t) * std::max<size_t>(rows.size(), 1));
        if (e == cudaSuccess)
            e = cudaMemcpy(c->ira_groups, groups.data(), sizeof(int2) * groups.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && !rows.empty())
            e = cudaMemcpy(c->ira_rows, rows.data(), sizeof(uint32_t) * rows.size(), cudaMemcpyHostToDevice);
        return e;
    } catch (const std::bad_alloc &) {
        return cudaErrorMemoryAllocation;
    }
}

}  // namespace ldpc

using namespace ldpc;

extern "C" int ldpc_encode_ira(ldpc_code_t *c, const uint8_t *info, int32_t n_frames, uint8_t *codeword,
                               void *stream) {
    if (!c) return set_error(LDPC_EINVAL, "ldpc_encode_ira: code is NULL");
    if (c->device < 0) return set_error(LDPC_ENODEV, "ldpc_encode_ira: host-only code");
    if (c->ira_k < 0)
        return set_error(LDPC_EINVAL, "ldpc_encode_ira: H has no staircase parity part in its last m columns");
    if (n_frames < 0) return set_error(LDPC_EINVAL, "ldpc_encode_ira: n_frames < 0");
    const int32_t k = c->ira_k, m = c->m, n = c->n;
    if (n_frames == 0 || n == 0) return LDPC_OK;
    if (!codeword || (k > 0 && !info)) return set_error(LDPC_EINVAL, "ldpc_encode_ira: NULL buffer");
    cudaStream_t s = (cudaStream_t)stream;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(c->device);
    if (c->ira_groups &&
        ira_one_kernel(std::min(ira_width(info, codeword, m, k, false), ira_width(info, codeword, m, k, true)), n_frames,
                       n)) {
        const cudaError_t e = launch_encode_ira(info, c->ira_groups, c->ira_rows, n_frames, m, k, codeword, s);
        if (prev >= 0) cudaSetDevice(prev);
        return e == cudaSuccess ? LDPC_OK : cuda_error(e, "ldpc_encode_ira");
    }
    const int32_t G = (n_frames + 31) / 32;
    // stream-ordered scratch: U [k][G], Pl [m][G] and T [chunks][G] words
    const int32_t nC = (m + kChunk - 1) / kChunk;
    uint32_t *U = nullptr;
    const size_t words = ((size_t)k + (size_t)m + (size_t)nC) * G;
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&U), sizeof(uint32_t) * std::max<size_t>(words, 1), s);
    if (e == cudaSuccess) {
        uint32_t *Pl = U + (size_t)k * G;
        uint32_t *T = Pl + (size_t)m * G;
        if (k > 0) {
            dim3 grid((unsigned)((k + 255) / 256), (unsigned)std::min(G, 65535));
            k_pack_info<<<grid, 256, 0, s>>>(info, n_frames, k, G, U);
        }
        if (m > 0) {
            k_chunk_prefix<<<grid_of((int64_t)nC * G, 128, c->sm_count), 128, 0, s>>>(c->d.row_ptr, c->d.col_idx, m,
                                                                                      k, G, U, Pl, T);
            k_chunk_carry<<<(unsigned)std::min((G + 7) / 8, 65535), 256, 0, s>>>(T, nC, G);
        }
        k_write_codeword<<<grid_of((int64_t)n_frames * n, 256, c->sm_count), 256, 0, s>>>(info, Pl, T, n_frames, n, k,
                                                                                          G, codeword);
        e = cudaGetLastError();
        cudaError_t e2 = cudaFreeAsync(U, s);
        if (e == cudaSuccess) e = e2;
    }
    if (prev >= 0) cudaSetDevice(prev);
    if (e != cudaSuccess) return cuda_error(e, "ldpc_encode_ira");
    return LDPC_OK;
}

namespace {

// Reduced row echelon form of H over GF(2) (dense rows of 64-bit words),
// pivots taken column by column from the last column down, so that a code in
// IRA form keeps its staircase columns as the parity positions. Fills the
// column map (information index, or -1 - pivot row) and the parity rows over
// the information bits; returns the rank.
int32_t reduce_parity_check(const ldpc_code *c, std::vector<int32_t> &colmap, std::vector<uint32_t> &R, int32_t *k_out) {
    const int32_t m = c->m, n = c->n;
    const size_t nw = ((size_t)n + 63) / 64;
    std::vector<uint64_t> A((size_t)m * nw, 0);
    for (int32_t i = 0; i < m; ++i)
        for (int32_t e = c->row_ptr[i]; e < c->row_ptr[i + 1]; ++e) {
            const int32_t j = c->col_idx[e];
            A[(size_t)i * nw + j / 64] ^= 1ull << (j % 64);
        }
    std::vector<int32_t> pivot_col;
    int32_t rank = 0;
    for (int32_t j = n - 1; j >= 0 && rank < m; --j) {
        const size_t w = (size_t)j / 64;
        const uint64_t bit = 1ull << (j % 64);
        int32_t p = -1;
        for (int32_t i = rank; i < m && p < 0; ++i)
            if (A[(size_t)i * nw + w] & bit) p = i;
        if (p < 0) continue;
        uint64_t *pr = &A[(size_t)p * nw], *rr = &A[(size_t)rank * nw];
        if (p != rank) std::swap_ranges(pr, pr + nw, rr);
        for (int32_t i = 0; i < m; ++i) {
            uint64_t *ri = &A[(size_t)i * nw];
            if (i == rank || !(ri[w] & bit)) continue;
            for (size_t t = 0; t < nw; ++t) ri[t] ^= rr[t];
        }
        pivot_col.push_back(j);
        ++rank;
    }
    colmap.assign((size_t)n, 0);
    std::vector<char> is_pivot((size_t)n, 0);
    for (int32_t i = 0; i < rank; ++i) {
        colmap[pivot_col[i]] = -1 - i;
        is_pivot[pivot_col[i]] = 1;
    }
    std::vector<int32_t> info_col;
    for (int32_t j = 0; j < n; ++j)
        if (!is_pivot[j]) {
            colmap[j] = (int32_t)info_col.size();
            info_col.push_back(j);
        }
    const int32_t k = (int32_t)info_col.size();
    const size_t kw = ((size_t)k + 31) / 32;
    R.assign((size_t)rank * std::max<size_t>(kw, 1), 0u);
    for (int32_t i = 0; i < rank; ++i) {
        const uint64_t *ri = &A[(size_t)i * nw];
        for (int32_t t = 0; t < k; ++t) {
            const int32_t j = info_col[t];
            if ((ri[j / 64] >> (j % 64)) & 1ull) R[(size_t)i * kw + t / 32] |= 1u << (t % 32);
        }
    }
    *k_out = k;
    return rank;
}

}  // namespace

// The handle's memory pool of ldpc_encode's scratch: kept between calls up to
// kEncoderPoolBytes (a pool without a threshold gives its memory back to the
// driver at every synchronisation: a call followed by one took 461 us, 264 of
// them its kernels), given back with the handle. Allocation and release are
// ordered by the caller's stream, so calls on several streams and threads have
// their own scratch.
constexpr uint64_t kEncoderPoolBytes = uint64_t(64) << 20;

static cudaError_t encoder_pool(int device, cudaMemPool_t *pool) {
    cudaMemPoolProps p = {};
    p.allocType = cudaMemAllocationTypePinned;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = device;
    cudaError_t e = cudaMemPoolCreate(pool, &p);
    uint64_t keep = kEncoderPoolBytes;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(*pool, cudaMemPoolAttrReleaseThreshold, &keep);
    return e;
}

extern "C" int ldpc_code_build_encoder(ldpc_code_t *c, int32_t *k_out) {
    if (!c) return set_error(LDPC_EINVAL, "ldpc_code_build_encoder: code is NULL");
    if ((int64_t)c->m * c->n > ((int64_t)1 << 26))
        return set_error(LDPC_EINVAL, "ldpc_code_build_encoder: m * n = %lld exceeds 2^26 (dense elimination)",
                         (long long)c->m * c->n);
    std::lock_guard<std::mutex> lock(c->mu);
    if (c->enc_k < 0) {
        std::vector<int32_t> colmap;
        std::vector<uint32_t> R;
        int32_t k = 0;
        const int32_t r = reduce_parity_check(c, colmap, R, &k);
        if (c->device >= 0) {
            int prev = -1;
            cudaGetDevice(&prev);
            cudaSetDevice(c->device);
            uint32_t *dR = nullptr;
            int32_t *dmap = nullptr;
            cudaError_t e = cudaMalloc(&dR, sizeof(uint32_t) * std::max<size_t>(R.size(), 1));
            if (e == cudaSuccess) e = cudaMalloc(&dmap, sizeof(int32_t) * std::max<size_t>(colmap.size(), 1));
            if (e == cudaSuccess) e = encoder_pool(c->device, &c->enc_pool);
            if (e == cudaSuccess && !R.empty())
                e = cudaMemcpy(dR, R.data(), sizeof(uint32_t) * R.size(), cudaMemcpyHostToDevice);
            if (e == cudaSuccess && !colmap.empty())
                e = cudaMemcpy(dmap, colmap.data(), sizeof(int32_t) * colmap.size(), cudaMemcpyHostToDevice);
            if (prev >= 0) cudaSetDevice(prev);
            if (e != cudaSuccess) {
                cudaFree(dR);
                cudaFree(dmap);
                if (c->enc_pool) cudaMemPoolDestroy(c->enc_pool);
                c->enc_pool = nullptr;
                return cuda_error(e, "ldpc_code_build_encoder");
            }
            c->enc_R = dR;
            c->enc_colmap = dmap;
        }
        c->enc_r = r;
        c->enc_k = k;
    }
    if (k_out) *k_out = c->enc_k;
    return LDPC_OK;
}

extern "C" int ldpc_encode(ldpc_code_t *c, const uint8_t *info, int32_t n_frames, uint8_t *codeword, void *stream) {
    if (!c) return set_error(LDPC_EINVAL, "ldpc_encode: code is NULL");
    if (c->device < 0) return set_error(LDPC_ENODEV, "ldpc_encode: host-only code");
    if (c->enc_k < 0) return set_error(LDPC_EINVAL, "ldpc_encode: no encoder (call ldpc_code_build_encoder first)");
    if (n_frames < 0) return set_error(LDPC_EINVAL, "ldpc_encode: n_frames < 0");
    const int32_t k = c->enc_k, r = c->enc_r, n = c->n;
    if (n_frames == 0 || n == 0) return LDPC_OK;
    if (!codeword || (k > 0 && !info)) return set_error(LDPC_EINVAL, "ldpc_encode: NULL buffer");
    cudaStream_t s = (cudaStream_t)stream;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(c->device);
    const int32_t kw = (k + 31) / 32;
    const int32_t most = std::min(n_frames, kDenseFrames);
    const int32_t Gp = (most + 1023) / 1024 * 32;  // words a row, 32 to a lane group
    uint32_t *U = nullptr;  // stream-ordered scratch: U [k][Gp], then P [r][Gp]
    const size_t words = ((size_t)k + (size_t)r) * Gp;
    cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&U),
                                            sizeof(uint32_t) * std::max<size_t>(words, 1), c->enc_pool, s);
    if (e == cudaSuccess) {
        uint32_t *P = U + (size_t)k * Gp;
        // slices of the information bits until the grid covers the SMs four times
        const int32_t blocks = (r + kDenseRows - 1) / kDenseRows;
        const int32_t cover = 4 * std::max(c->sm_count, 1), all = std::max(blocks * (Gp / 32), 1);
        const int32_t want = std::max(1, std::min(kw, (cover + all - 1) / all));
        const int32_t slice = std::max(1, (kw + want - 1) / want);
        for (int64_t f0 = 0; f0 < n_frames; f0 += kDenseFrames) {  // 64 bits: the last step may pass 2^31
            const int32_t F = (int32_t)std::min<int64_t>(kDenseFrames, n_frames - f0);
            const uint8_t *in = info + (size_t)f0 * k;
            uint8_t *out = codeword + (size_t)f0 * n;
            const dim3 pack((unsigned)std::max((k + 127) / 128, 1), (unsigned)(Gp / 8));
            const bool ends = ((reinterpret_cast<uintptr_t>(in) | (uintptr_t)((int64_t)F * k)) & 3) != 0;
            (ends ? k_dense_pack<true> : k_dense_pack<false>)<<<pack, 256, 0, s>>>(in, F, k, Gp, U, P, (int64_t)r * Gp);
            if (r > 0 && k > 0) {
                const dim3 grid((unsigned)blocks, (unsigned)((kw + slice - 1) / slice), (unsigned)(Gp / 32));
                k_dense_parity<<<grid, 256, 0, s>>>(c->enc_R, r, k, kw, slice, U, Gp, P);
            }
            const dim3 wr((unsigned)((n + 1023) / 1024), (unsigned)((F + 31) / 32));
            const bool out4 = n % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 4 == 0;
            (out4 ? k_dense_write<true> : k_dense_write<false>)<<<wr, 256, 0, s>>>(U, P, c->enc_colmap, F, n, Gp, out);
        }
        e = cudaGetLastError();
        cudaError_t e2 = cudaFreeAsync(U, s);
        if (e == cudaSuccess) e = e2;
    }
    if (prev >= 0) cudaSetDevice(prev);
    if (e != cudaSuccess) return cuda_error(e, "ldpc_encode");
    return LDPC_OK;
}

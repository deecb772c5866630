// Error counting of the BER simulator (Section IV): Hamming distance between
// decoded words and the transmitted ones (or the all-zero word, which is
// enough by linearity), accumulated on the device.
#include <algorithm>
#include <type_traits>

#include "ldpc_internal.h"

namespace ldpc {

// Differing bytes of W-byte words.
__device__ __forceinline__ unsigned int differ(uint32_t a, uint32_t b) { return __popc(__vsetne4(a, b)); }

// TPF threads compare a frame, W bytes a load (ref null: the zero word). The
// sums stay in registers over a thread group's frames and meet in one set of
// atomics per CTA: an atomic per frame on four shared counters serialises in
// L2, and byte loads keep too few bytes in flight (10,000 frames of 2048 bits
// 24 -> 8 us, 256 frames of 64800 bits against a reference 52 -> 12 us with the
// call).
template <int TPF, int W>
__global__ void __launch_bounds__(256) k_count_errors(const uint8_t *__restrict__ bits, const uint8_t *__restrict__ ref,
                                                      int32_t F, int32_t n, const int32_t *__restrict__ iters,
                                                      const uint8_t *__restrict__ ok,
                                                      unsigned long long *__restrict__ counts) {
    __shared__ unsigned int partial[8];
    __shared__ unsigned long long sums[4];
    constexpr int kPer = 256 / TPF;  // frames at once
    const int t = threadIdx.x % TPF;
    unsigned long long sum[4] = {0, 0, 0, 0};  // of the group's first thread
    if (threadIdx.x < 4) sums[threadIdx.x] = 0ull;
    for (int64_t f0 = (int64_t)blockIdx.x * kPer; f0 < F; f0 += (int64_t)gridDim.x * kPer) {
        const int64_t f = f0 + threadIdx.x / TPF;
        unsigned int errs = 0;
        if (f < F) {
            const uint8_t *b = bits + (size_t)f * n;
            const uint8_t *r = ref ? ref + (size_t)f * n : nullptr;
#pragma unroll 4
            for (int j = t; j < n / W; j += TPF) {
                if constexpr (W == 16) {
                    const uint4 x = reinterpret_cast<const uint4 *>(b)[j];
                    const uint4 y = r ? reinterpret_cast<const uint4 *>(r)[j] : make_uint4(0, 0, 0, 0);
                    errs += differ(x.x, y.x) + differ(x.y, y.y) + differ(x.z, y.z) + differ(x.w, y.w);
                } else if constexpr (W == 4) {
                    errs += differ(reinterpret_cast<const uint32_t *>(b)[j], r ? reinterpret_cast<const uint32_t *>(r)[j] : 0u);
                } else {
                    errs += b[j] != (r ? r[j] : 0) ? 1u : 0u;
                }
            }
        }
        errs = __reduce_add_sync(0xffffffffu, errs);
        if constexpr (TPF == 256) {
            __syncthreads();
            if ((threadIdx.x & 31) == 0) partial[threadIdx.x >> 5] = errs;
            __syncthreads();
            if (t == 0) {
                errs = 0;
                for (int w = 0; w < 8; ++w) errs += partial[w];
            }
        }
        if (t == 0 && f < F) {
            sum[0] += errs;
            sum[1] += errs ? 1u : 0u;
            if (iters) sum[2] += (unsigned long long)iters[f];
            if (ok && !ok[f]) sum[3] += 1u;
        }
    }
    __syncthreads();
    if (t == 0)
        for (int i = 0; i < 4; ++i)
            if (sum[i]) atomicAdd(&sums[i], sum[i]);
    __syncthreads();
    if (threadIdx.x < 4 && sums[threadIdx.x]) atomicAdd(counts + threadIdx.x, sums[threadIdx.x]);
}

template <int TPF, int W>
cudaError_t launch_count(const uint8_t *bits, const uint8_t *ref, int32_t F, int32_t n, const int32_t *iters,
                         const uint8_t *ok, unsigned long long *counts, cudaStream_t s) {
    // byte loads need all the warps an SM holds to keep enough of them in flight
    // (n = 64801, 1000 frames against a reference: 254 us with four CTAs an SM)
    const int64_t most = 152 * (W == 1 ? 16 : 4);
    const unsigned blocks = (unsigned)std::min<int64_t>(((int64_t)F + 256 / TPF - 1) / (256 / TPF), most);
    k_count_errors<TPF, W><<<blocks, 256, 0, s>>>(bits, ref, F, n, iters, ok, counts);
    return cudaGetLastError();
}

}  // namespace ldpc

using namespace ldpc;

extern "C" int ldpc_count_errors(const uint8_t *bits, const uint8_t *ref, int32_t n_frames, int32_t n,
                                 const int32_t *iters, const uint8_t *syndrome_ok, int64_t *counts, void *stream) {
    if (n_frames < 0 || n < 0) return set_error(LDPC_EINVAL, "ldpc_count_errors: negative size");
    if (!counts) return set_error(LDPC_EINVAL, "ldpc_count_errors: counts is NULL");
    if (n_frames == 0) return LDPC_OK;
    if (n > 0 && !bits) return set_error(LDPC_EINVAL, "ldpc_count_errors: bits is NULL");
    // a warp per frame, a CTA where a warp alone would walk a long word: above 4096
    // bits (eight 16-byte or 32 four-byte loads a lane; n = 3004, 10,000 frames a warp
    // 11 us, a CTA 19), byte by byte above 2048 (n = 4095, 1000 frames 16.7 / 12.5 us)
    auto *c = reinterpret_cast<unsigned long long *>(counts);
    const cudaStream_t st = (cudaStream_t)stream;
    const uintptr_t a = reinterpret_cast<uintptr_t>(bits) | reinterpret_cast<uintptr_t>(ref) | (uintptr_t)n;
    auto go = [&](auto width) {
        constexpr int W = decltype(width)::value;
        return n <= (W == 1 ? 2048 : 4096) ? launch_count<32, W>(bits, ref, n_frames, n, iters, syndrome_ok, c, st)
                                            : launch_count<256, W>(bits, ref, n_frames, n, iters, syndrome_ok, c, st);
    };
    const cudaError_t e = a % 16 == 0  ? go(std::integral_constant<int, 16>{})
                          : a % 4 == 0 ? go(std::integral_constant<int, 4>{})
                                       : go(std::integral_constant<int, 1>{});
    if (e != cudaSuccess) return cuda_error(e, "ldpc_count_errors: launch");
    return LDPC_OK;
}

// 2:4 prune + compress (prune24_compress) and its inverse.
//
// Vector path: a thread takes pieces of 16 input bytes (four groups of four
// codes): one 16-byte load, a branch-free selection for the four groups at
// once (select_groups4), an 8-byte store of the kept codes and a 2-byte
// store of the four metadata nibbles.  Rows whose length or alignment does
// not allow it fall back to one metadata byte per iteration.
// Bandwidth-bound: 1 byte read, 0.625 bytes written per element; no
// allocation, one launch.  The inverse moves the same bytes the other way.
#include <algorithm>

#include "common.cuh"
#include "prune_select.cuh"

namespace gb300 {
namespace {

constexpr int kThreads = 256;

// Vector path: K % 16 == 0, a 16-aligned with lda % 16 == 0, vals 8-aligned,
// meta 2-aligned.  blockIdx.y walks rows.  A thread takes U pieces of
// 16 codes (four groups) spaced kThreads apart, so each load instruction of
// a warp reads 512 contiguous bytes; all loads are issued before any
// selection.  Per piece: 8 bytes of kept codes and 16 bits of metadata.
// Contiguous rows (lda == K) come as one long row, so every block but the
// last has all its pieces whatever K is: a block per row of K = 8192 has
// work for half of its loads, one of K = 1024 for a sixteenth.  Measured
// (GB300, inputs rotated beyond L2) with both changes, the four-group
// selection and the one long row: 23.3 -> 17.3 us at 8192 x 8192 (6.3 TB/s),
// 75.8 -> 62.4 us at 16384 x 16384, 18.5 -> 6.5 us at 16384 x 1024.
// U = kPieces while that leaves every SM a few blocks, else 1: with less
// work the spread over the SMs counts for more than the loads in flight.
constexpr int kPieces = 4;

int pieces_per_thread(int64_t total)
{
    return total < static_cast<int64_t>(sm_count()) * 8 * kThreads ? 1 : kPieces;
}

template <int U>
__global__ void __launch_bounds__(kThreads) prune24_vec_kernel(const uint8_t* __restrict__ a,
                                                               int64_t M, int64_t K, int64_t lda,
                                                               uint8_t* __restrict__ vals,
                                                               uint8_t* __restrict__ meta)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int pieces = static_cast<int>(K / 16);
    const int64_t ldv = K / 2, ldm = K / 8;
    const int p_first = blockIdx.x * (kThreads * U) + threadIdx.x;
    for (int64_t r = blockIdx.y; r < M; r += gridDim.y) {
        const uint4* src = reinterpret_cast<const uint4*>(a + r * lda);
        uint4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p_first + u * kThreads;
            if (p < pieces)
                x[u] = __ldg(src + p);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = p_first + u * kThreads;
            if (p >= pieces)
                continue;
            uint2 v;
            const uint32_t nib = select_groups4(x[u].x, x[u].y, x[u].z, x[u].w, &v.x, &v.y);
            *reinterpret_cast<uint2*>(vals + r * ldv + static_cast<int64_t>(p) * 8) = v;
            *reinterpret_cast<uint16_t*>(meta + r * ldm + static_cast<int64_t>(p) * 2) = static_cast<uint16_t>(nib);
        }
    }
}

// Scalar path (any K % 4 == 0 and any alignment): one metadata byte (two
// groups, or one at an odd tail) per iteration so that no two threads write
// the same byte.
__global__ void __launch_bounds__(kThreads) prune24_kernel(const uint8_t* __restrict__ a,
                                                           int64_t M, int64_t K, int64_t lda,
                                                           uint8_t* __restrict__ vals,
                                                           uint8_t* __restrict__ meta)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t ldv = K / 2, ldm = (K + 7) / 8;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
    const int64_t tid = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x;
    for (int64_t i = tid; i < M * ldm; i += stride) {
        const int64_t r = i / ldm, b = i - r * ldm;
        uint8_t out = 0;
        for (int h = 0; h < 2; ++h) {
            const int64_t g = 2 * b + h;
            if (4 * g >= K)
                break;
            const uint8_t* p = a + r * lda + 4 * g;
            const uint32_t w = p[0] | (p[1] << 8) | (p[2] << 16) | (static_cast<uint32_t>(p[3]) << 24);
            const uint32_t sel = select_group(w);
            vals[r * ldv + 2 * g] = static_cast<uint8_t>(sel & 0xFFu);
            vals[r * ldv + 2 * g + 1] = static_cast<uint8_t>((sel >> 8) & 0xFFu);
            out |= static_cast<uint8_t>(((sel >> 16) & 0xFu) << (4 * h));
        }
        meta[r * ldm + b] = out;
    }
}

// One group expanded: the two kept codes of v's low half at the bytes the
// nibble names (any nibble, equal indices included, as the scalar path).
__device__ __forceinline__ uint32_t expand_group(uint32_t v, uint32_t nib)
{
    return ((v & 0xFFu) << ((nib << 3) & 24u)) | (((v >> 8) & 0xFFu) << ((nib << 1) & 24u));
}

// Vector path of the inverse: K % 16 == 0, out 16-aligned, vals 8-aligned,
// meta 2-aligned.  All three arrays are contiguous, so the matrix is one run
// of pieces (8 kept codes and 16 metadata bits -> 16 codes); a thread takes
// U of them (pieces_per_thread) spaced kThreads apart, all loads before any
// store.  Bound by HBM: 18.0 us at 8192 x 8192 (6.1 TB/s), 64.3 us at 16384 x
// 16384, against 56.1 and 212 us for the scalar path below (single-byte
// loads and stores, a 64-bit division per group).
template <int U>
__global__ void __launch_bounds__(kThreads) decompress24_vec_kernel(const uint2* __restrict__ vals,
                                                                    const uint16_t* __restrict__ meta,
                                                                    int64_t pieces, uint4* __restrict__ out)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t step = static_cast<int64_t>(gridDim.x) * (kThreads * U);
    for (int64_t p0 = static_cast<int64_t>(blockIdx.x) * (kThreads * U) + threadIdx.x; p0 < pieces;
         p0 += step) {
        uint2 v[U];
        uint32_t n[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t p = p0 + u * kThreads;
            if (p < pieces) {
                v[u] = __ldg(vals + p);
                n[u] = __ldg(meta + p);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t p = p0 + u * kThreads;
            if (p < pieces)
                out[p] = make_uint4(expand_group(v[u].x, n[u]), expand_group(v[u].x >> 16, n[u] >> 4),
                                    expand_group(v[u].y, n[u] >> 8), expand_group(v[u].y >> 16, n[u] >> 12));
        }
    }
}

// Scalar path (any K % 4 == 0 and any alignment): one group per iteration.
__global__ void __launch_bounds__(kThreads) decompress24_kernel(const uint8_t* __restrict__ vals,
                                                                const uint8_t* __restrict__ meta,
                                                                int64_t M, int64_t K,
                                                                uint8_t* __restrict__ out)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t ldv = K / 2, ldm = (K + 7) / 8, groups = K / 4;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; i < M * groups;
         i += stride) {
        const int64_t r = i / groups, g = i - r * groups;
        const uint32_t nib = (meta[r * ldm + g / 2] >> (4 * (g % 2))) & 0xFu;
        const uint32_t i0 = nib & 3u, i1 = nib >> 2;
        uint32_t w = 0;
        w |= static_cast<uint32_t>(vals[r * ldv + 2 * g]) << (8 * i0);
        w |= static_cast<uint32_t>(vals[r * ldv + 2 * g + 1]) << (8 * i1);
        uint8_t* o = out + r * K + 4 * g;
        o[0] = w & 0xFFu;
        o[1] = (w >> 8) & 0xFFu;
        o[2] = (w >> 16) & 0xFFu;
        o[3] = (w >> 24) & 0xFFu;
    }
}

int grid_for(int64_t items)
{
    const int64_t blocks = (items + kThreads - 1) / kThreads;
    const int64_t cap = static_cast<int64_t>(sm_count()) * 16;
    return static_cast<int>(blocks < cap ? (blocks > 0 ? blocks : 1) : cap);
}

}  // namespace
}  // namespace gb300

extern "C" int prune24_compress(const uint8_t* a, int64_t M, int64_t K, int64_t lda,
                                uint8_t* a_vals, uint8_t* a_meta, fp8_stream_t stream)
{
    using namespace gb300;
    if (M < 0 || K < 0)
        return FP8_ERR_INVALID;
    if (K % 4 != 0)
        return FP8_ERR_SHAPE;
    if (M == 0 || K == 0)
        return FP8_OK;
    if (!a || !a_vals || !a_meta)
        return FP8_ERR_INVALID;
    if (lda < K)
        return FP8_ERR_SHAPE;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const bool vec = (K % 16 == 0) && aligned16(a) && (lda % 16 == 0) &&
                     (reinterpret_cast<uintptr_t>(a_vals) % 8 == 0) &&
                     (reinterpret_cast<uintptr_t>(a_meta) % 2 == 0);
    if (vec) {
        // contiguous rows as one (the piece index of a row is 32 bits)
        if (lda == K && M * (K / 16) < INT32_MAX - kThreads * kPieces) {
            K *= M;
            lda = K;
            M = 1;
        }
        const int64_t pieces = K / 16;
        const int u = pieces_per_thread(M * pieces);
        const unsigned gx = static_cast<unsigned>((pieces + kThreads * u - 1) / (kThreads * u));
        const unsigned gy = static_cast<unsigned>(M < 65535 ? M : 65535);
        if (u == 1)
            launch_dependent(prune24_vec_kernel<1>, dim3(gx, gy), kThreads, st, a, M, K, lda, a_vals, a_meta);
        else
            launch_dependent(prune24_vec_kernel<kPieces>, dim3(gx, gy), kThreads, st, a, M, K, lda, a_vals, a_meta);
    } else {
        launch_dependent(prune24_kernel, grid_for(M * ((K + 7) / 8)), kThreads, st, a, M, K, lda, a_vals, a_meta);
    }
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

extern "C" int prune24_decompress(const uint8_t* a_vals, const uint8_t* a_meta, int64_t M,
                                  int64_t K, uint8_t* out, fp8_stream_t stream)
{
    using namespace gb300;
    if (M < 0 || K < 0)
        return FP8_ERR_INVALID;
    if (K % 4 != 0)
        return FP8_ERR_SHAPE;
    if (M == 0 || K == 0)
        return FP8_OK;
    if (!a_vals || !a_meta || !out)
        return FP8_ERR_INVALID;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (K % 16 == 0 && aligned16(out) && reinterpret_cast<uintptr_t>(a_vals) % 8 == 0 &&
        reinterpret_cast<uintptr_t>(a_meta) % 2 == 0) {
        const int64_t pieces = M * (K / 16);
        const int u = pieces_per_thread(pieces);
        const int64_t blocks = std::min<int64_t>((pieces + kThreads * u - 1) / (kThreads * u), INT32_MAX);
        const auto* v8 = reinterpret_cast<const uint2*>(a_vals);
        const auto* m2 = reinterpret_cast<const uint16_t*>(a_meta);
        auto* o16 = reinterpret_cast<uint4*>(out);
        if (u == 1)
            launch_dependent(decompress24_vec_kernel<1>, static_cast<unsigned>(blocks), kThreads, st, v8, m2, pieces, o16);
        else
            launch_dependent(decompress24_vec_kernel<kPieces>, static_cast<unsigned>(blocks), kThreads, st, v8, m2, pieces, o16);
    } else {
        launch_dependent(decompress24_kernel, grid_for(M * (K / 4)), kThreads, st, a_vals, a_meta, M, K, out);
    }
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

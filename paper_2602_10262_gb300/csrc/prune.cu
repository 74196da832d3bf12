// 2:4 prune + compress (prune24_compress) and its inverse.
//
// Vector path: a thread takes pieces of 16 input bytes (four groups of four
// codes): one 16-byte load, a branch-free selection for the four groups at
// once (select_groups4), an 8-byte store of the kept codes and a 2-byte
// store of the four metadata nibbles.  Rows whose length or alignment does
// not allow it take the same pieces with narrower accesses.
// Bandwidth-bound: 1 byte read, 0.625 bytes written per element; no
// allocation, one launch.  Loads are ordinary ones (of whole pieces, at L2):
// these kernels may start before their input is written (launch_dependent),
// which the read-only path does not allow.  The inverse moves the same bytes
// the other way.
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
// Contiguous rows (lda == K, K % 8 == 0) come as one long row, so every block
// but the last has all its pieces whatever K is: a block per row of K = 8192 has
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
                x[u] = __ldcg(src + p);
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

// Any K % 4 == 0 and any alignment: a row is pieces of up to four groups (G),
// and a thread takes U pieces of the whole matrix (kThreads apart, the row by
// one 32-bit division), each with the widest loads and stores its arrays
// allow.  16384 x 4100 (rows of half metadata bytes): 28.6
// us, and 46.2 to expand it again; one metadata byte, or one group, per
// thread with single-byte accesses and a 64-bit division took 46.8 and 54.9.
struct PieceShape {
    int64_t total;             // pieces of the matrix
    int64_t per_row;
    int64_t groups;            // of a row
    int64_t ldv, ldm;          // kept-code and metadata bytes of a row
};

__device__ __forceinline__ void piece_row(const PieceShape& s, int64_t i, int64_t* r, int64_t* p)
{
    if (s.total <= 0xFFFFFFFFll) {
        const uint32_t n = static_cast<uint32_t>(s.per_row);
        const uint32_t q = static_cast<uint32_t>(i) / n;
        *r = q;
        *p = static_cast<uint32_t>(i) - q * n;
    } else {
        *r = i / s.per_row;
        *p = i - *r * s.per_row;
    }
}

// n bytes (a multiple of 2, at most 4 * W) between memory of alignment
// `align` (16, 8, 4, 2 or 1) and words.
template <int W>
__device__ __forceinline__ void load_words(const uint8_t* p, int n, int align, uint32_t (&w)[W])
{
#pragma unroll
    for (int i = 0; i < W; ++i)
        w[i] = 0;
    if (W == 4 && align >= 16 && n == 16) {
        const uint4 v = __ldca(reinterpret_cast<const uint4*>(p));
        w[0] = v.x, w[W > 1 ? 1 : 0] = v.y, w[W > 2 ? 2 : 0] = v.z, w[W > 3 ? 3 : 0] = v.w;
    } else if (W >= 2 && align >= 8 && n == 4 * W) {
#pragma unroll
        for (int i = 0; i + 1 < W; i += 2) {
            const uint2 v = __ldca(reinterpret_cast<const uint2*>(p + 4 * i));
            w[i] = v.x, w[i + 1] = v.y;
        }
    } else if (align >= 4) {
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (4 * i + 4 <= n)
                w[i] = __ldca(reinterpret_cast<const uint32_t*>(p + 4 * i));
            else if (4 * i + 2 <= n)
                w[i] = __ldca(reinterpret_cast<const uint16_t*>(p + 4 * i));
    } else if (align >= 2) {
#pragma unroll
        for (int i = 0; i < 2 * W; ++i)
            if (2 * i + 2 <= n)
                w[i / 2] |= static_cast<uint32_t>(__ldca(reinterpret_cast<const uint16_t*>(p + 2 * i))) << (16 * (i & 1));
    } else {
#pragma unroll
        for (int i = 0; i < 4 * W; ++i)
            if (i < n)
                w[i / 4] |= static_cast<uint32_t>(__ldca(p + i)) << (8 * (i & 3));
    }
}

template <int W>
__device__ __forceinline__ void store_words(uint8_t* p, int n, int align, const uint32_t (&w)[W])
{
    if (W >= 2 && align >= 8 && n == 4 * W) {
#pragma unroll
        for (int i = 0; i + 1 < W; i += 2)
            *reinterpret_cast<uint2*>(p + 4 * i) = make_uint2(w[i], w[i + 1]);
    } else if (align >= 4) {
#pragma unroll
        for (int i = 0; i < W; ++i)
            if (4 * i + 4 <= n)
                *reinterpret_cast<uint32_t*>(p + 4 * i) = w[i];
            else if (4 * i + 2 <= n)
                *reinterpret_cast<uint16_t*>(p + 4 * i) = static_cast<uint16_t>(w[i]);
    } else if (align >= 2) {
#pragma unroll
        for (int i = 0; i < 2 * W; ++i)
            if (2 * i + 2 <= n)
                *reinterpret_cast<uint16_t*>(p + 2 * i) = static_cast<uint16_t>(w[i / 2] >> (16 * (i & 1)));
    } else {
#pragma unroll
        for (int i = 0; i < 4 * W; ++i)
            if (i < n)
                p[i] = static_cast<uint8_t>(w[i / 4] >> (8 * (i & 3)));
    }
}

// Pieces of two groups (G = 2) where a or the kept codes start on any byte and
// there is too little work to fill the SMs: sixteen single-byte loads, or eight
// stores, one after the other are then all the time there is (320 x 4100: 3.7
// us with four groups a thread, 2.6 with two).  Not for short rows of half
// metadata bytes, which lose more to their last piece (4096 x 132: 1.9, 2.2).
template <int U, int G>
__global__ void __launch_bounds__(kThreads) prune24_any_kernel(const uint8_t* __restrict__ a, PieceShape s,
                                                               int64_t lda, int a_align, uint8_t* __restrict__ vals,
                                                               int v_align, uint8_t* __restrict__ meta, int m_align)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t step = static_cast<int64_t>(gridDim.x) * (kThreads * U);
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kThreads * U) + threadIdx.x; i0 < s.total; i0 += step) {
        uint32_t w[U][G];
        int64_t r[U], p[U];
        int n[U];                          // groups of the piece
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * kThreads;
            n[u] = 0;
            if (i < s.total) {
                piece_row(s, i, &r[u], &p[u]);
                n[u] = static_cast<int>(min(static_cast<int64_t>(G), s.groups - G * p[u]));
                load_words<G>(a + r[u] * lda + 4 * G * p[u], 4 * n[u], a_align, w[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (n[u] == 0)
                continue;
            uint32_t v01, v23;
            const uint32_t nib = select_groups4(w[u][0], w[u][1], G == 4 ? w[u][G - 2] : 0u, G == 4 ? w[u][G - 1] : 0u,
                                                &v01, &v23) & ((1u << (4 * n[u])) - 1u);
            uint32_t v[G / 2];
            v[0] = v01;
            if constexpr (G == 4)
                v[1] = v23;
            store_words<G / 2>(vals + r[u] * s.ldv + 2 * G * p[u], 2 * n[u], v_align, v);
            uint8_t* md = meta + r[u] * s.ldm + G / 2 * p[u];
            if (m_align >= 2 && n[u] > 2) {
                *reinterpret_cast<uint16_t*>(md) = static_cast<uint16_t>(nib);
            } else {
                md[0] = static_cast<uint8_t>(nib);
                if (n[u] > 2)
                    md[1] = static_cast<uint8_t>(nib >> 8);
            }
        }
    }
}

// One group expanded: the two kept codes of v's low half at the bytes the
// nibble names (any nibble: equal or descending indices combine with OR).
__device__ __forceinline__ uint32_t expand_group(uint32_t v, uint32_t nib)
{
    return ((v & 0xFFu) << ((nib << 3) & 24u)) | (((v >> 8) & 0xFFu) << ((nib << 1) & 24u));
}

// Vector path of the inverse: K % 16 == 0, out 16-aligned, vals 8-aligned,
// meta 2-aligned.  All three arrays are contiguous, so the matrix is one run
// of pieces (8 kept codes and 16 metadata bits -> 16 codes); a thread takes
// U of them (pieces_per_thread) spaced kThreads apart, all loads before any
// store.  Bound by HBM: 18.0 us at 8192 x 8192 (6.1 TB/s), 64.3 us at 16384 x
// 16384, against 56.1 and 212 us with single-byte loads and stores and a
// 64-bit division per group.
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
                v[u] = __ldcg(vals + p);
                n[u] = __ldcg(meta + p);
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

// The inverse for any K % 4 == 0 and any alignment of its inputs, out on a
// 4-byte boundary, by the same pieces.
template <int U>
__global__ void __launch_bounds__(kThreads) decompress24_any_kernel(const uint8_t* __restrict__ vals, int v_align,
                                                                    const uint8_t* __restrict__ meta, int m_align,
                                                                    PieceShape s, uint8_t* __restrict__ out,
                                                                    int64_t ldo, int o_align)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t step = static_cast<int64_t>(gridDim.x) * (kThreads * U);
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kThreads * U) + threadIdx.x; i0 < s.total; i0 += step) {
        uint32_t v[U][2], m[U];
        int64_t r[U], p[U];
        int n[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * kThreads;
            n[u] = 0;
            if (i < s.total) {
                piece_row(s, i, &r[u], &p[u]);
                n[u] = static_cast<int>(min(static_cast<int64_t>(4), s.groups - 4 * p[u]));
                load_words<2>(vals + r[u] * s.ldv + 8 * p[u], 2 * n[u], v_align, v[u]);
                const uint8_t* md = meta + r[u] * s.ldm + 2 * p[u];
                if (m_align >= 2 && n[u] > 2) {
                    m[u] = __ldca(reinterpret_cast<const uint16_t*>(md));
                } else {
                    m[u] = __ldca(md);
                    if (n[u] > 2)
                        m[u] |= static_cast<uint32_t>(__ldca(md + 1)) << 8;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (n[u] == 0)
                continue;
            const uint32_t w[4] = {expand_group(v[u][0], m[u]), expand_group(v[u][0] >> 16, m[u] >> 4),
                                   expand_group(v[u][1], m[u] >> 8), expand_group(v[u][1] >> 16, m[u] >> 12)};
            store_words<4>(out + r[u] * ldo + 16 * p[u], 4 * n[u], o_align, w);
        }
    }
}

// The inverse with out off a 4-byte boundary: one group a thread and step, as
// the 16 single bytes that a thread of the kernel above would store one by one,
// 16 apart from its neighbour's, write every sector 16 times (16384 x 4100 from
// an odd byte: 180 us, 51.6 this way; 16384 x 14336 586 and 156).  Kept codes and output have no gaps
// between rows, so a group's place in them is its index alone; ROWS: metadata
// rows end in half a byte, and only they need the row (a thread's next group
// is step_rows rows and step_groups groups on: one division a thread).
template <int U, bool ROWS>
__global__ void __launch_bounds__(kThreads) decompress24_group_kernel(const uint8_t* __restrict__ vals, int v_align,
                                                                      const uint8_t* __restrict__ meta, PieceShape s,
                                                                      int step_rows, int step_groups,
                                                                      uint8_t* __restrict__ out, int o_align)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t step = static_cast<int64_t>(gridDim.x) * (kThreads * U);
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kThreads * U) + threadIdx.x; i0 < s.total; i0 += step) {
        uint32_t v[U][1], m[U];
        int64_t r = 0, p = i0;
        if (ROWS)
            piece_row(s, i0, &r, &p);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * kThreads;
            if (ROWS && u > 0) {
                r += step_rows;
                p += step_groups;
                if (p >= s.per_row) {
                    p -= s.per_row;
                    ++r;
                }
            } else if (!ROWS) {
                p = i;
            }
            if (i < s.total) {
                load_words<1>(vals + 2 * i, 2, v_align, v[u]);
                m[u] = __ldca(meta + r * s.ldm + (p >> 1)) >> (4 * (p & 1));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * kThreads;
            if (i < s.total) {
                const uint32_t w[1] = {expand_group(v[u][0], m[u])};
                store_words<1>(out + 4 * i, 4, o_align, w);
            }
        }
    }
}

// The largest of 16, 8, 4, 2, 1 that divides a base address and a row stride.
int bytes_align(const void* p, int64_t ld)
{
    const uint64_t v = reinterpret_cast<uintptr_t>(p) | static_cast<uint64_t>(ld) | 16;
    return static_cast<int>(v & (~v + 1));
}

PieceShape piece_shape(int64_t M, int64_t K, int groups = 4)
{
    const int64_t per_row = (K + 4 * groups - 1) / (4 * groups);
    return {M * per_row, per_row, K / 4, K / 2, (K + 7) / 8};
}

unsigned piece_grid(int64_t total, int u)
{
    return static_cast<unsigned>(std::min<int64_t>((total + kThreads * u - 1) / (kThreads * u), INT32_MAX));
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
    // contiguous rows of whole metadata bytes are one row (the vector path's
    // piece index is 32 bits)
    if (lda == K && K % 8 == 0 && M * (K / 8) < INT32_MAX) {
        K *= M;
        lda = K;
        M = 1;
    }
    const int64_t row_a = M == 1 ? 0 : lda;       // one row: its start alone decides the alignment
    const bool vec = (K % 16 == 0) && aligned16(a) && (row_a % 16 == 0) && K / 16 < INT32_MAX - kThreads * kPieces &&
                     (reinterpret_cast<uintptr_t>(a_vals) % 8 == 0) &&
                     (reinterpret_cast<uintptr_t>(a_meta) % 2 == 0);
    if (vec) {
        const int64_t pieces = K / 16;
        const int u = pieces_per_thread(M * pieces);
        const unsigned gx = static_cast<unsigned>((pieces + kThreads * u - 1) / (kThreads * u));
        const unsigned gy = static_cast<unsigned>(M < 65535 ? M : 65535);
        if (u == 1)
            launch_dependent(prune24_vec_kernel<1>, dim3(gx, gy), kThreads, st, a, M, K, lda, a_vals, a_meta);
        else
            launch_dependent(prune24_vec_kernel<kPieces>, dim3(gx, gy), kThreads, st, a, M, K, lda, a_vals, a_meta);
    } else {
        PieceShape s = piece_shape(M, K);
        const int u = pieces_per_thread(s.total);
        const int aa = bytes_align(a, row_a), va = bytes_align(a_vals, M == 1 ? 0 : s.ldv),
                  ma = bytes_align(a_meta, M == 1 ? 0 : s.ldm);
        const bool halves = u == 1 && std::min(aa, va) == 1 && (K % 8 == 0 || K >= 1024);
        if (halves)
            s = piece_shape(M, K, 2);
        launch_dependent(halves    ? prune24_any_kernel<1, 2>
                         : u == 1 ? prune24_any_kernel<1, 4>
                                  : prune24_any_kernel<kPieces, 4>,
                         piece_grid(s.total, u), kThreads, st, a, s, lda, aa, a_vals, va, a_meta, ma);
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
    if (K % 8 == 0) {                             // rows of whole metadata bytes: one row
        K *= M;
        M = 1;
    }
    if (K % 16 == 0 && aligned16(out) && reinterpret_cast<uintptr_t>(a_vals) % 8 == 0 &&
        reinterpret_cast<uintptr_t>(a_meta) % 2 == 0) {
        const int64_t pieces = M * (K / 16);
        const int u = pieces_per_thread(pieces);
        const int64_t blocks = std::min<int64_t>((pieces + kThreads * u - 1) / (kThreads * u), INT32_MAX);
        const auto* v8 = reinterpret_cast<const uint2*>(a_vals);
        const auto* m2 = reinterpret_cast<const uint16_t*>(a_meta);
        auto* o16 = reinterpret_cast<uint4*>(out);
        if (u == 1)
            launch_dependent(decompress24_vec_kernel<1>, static_cast<unsigned>(blocks), kThreads, st, v8, m2, pieces,
                             o16);
        else
            launch_dependent(decompress24_vec_kernel<kPieces>, static_cast<unsigned>(blocks), kThreads, st, v8, m2,
                             pieces, o16);
    } else {
        const int oa = bytes_align(out, M == 1 ? 0 : K);
        const PieceShape s = piece_shape(M, K, oa < 4 ? 1 : 4);
        const int u = pieces_per_thread(oa < 4 ? s.total / 2 : s.total);
        const int va = bytes_align(a_vals, M == 1 ? 0 : s.ldv), ma = bytes_align(a_meta, M == 1 ? 0 : s.ldm);
        if (oa < 4) {
            const bool rows = K % 8 != 0 && M > 1;
            launch_dependent(rows ? (u == 1 ? decompress24_group_kernel<1, true>
                                            : decompress24_group_kernel<kPieces, true>)
                                  : (u == 1 ? decompress24_group_kernel<1, false>
                                            : decompress24_group_kernel<kPieces, false>),
                             piece_grid(s.total, u), kThreads, st, a_vals, va, a_meta, s,
                             static_cast<int>(kThreads / s.per_row), static_cast<int>(kThreads % s.per_row), out, oa);
        } else {
            launch_dependent(u == 1 ? decompress24_any_kernel<1> : decompress24_any_kernel<kPieces>,
                             piece_grid(s.total, u), kThreads, st, a_vals, va, a_meta, ma, s, out, K, oa);
        }
    }
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

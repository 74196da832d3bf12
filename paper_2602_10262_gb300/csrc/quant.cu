// Scale selection + FP8 quantisation (fp8_quantize_e4m3, fp8_quantize_e5m2).
//
// Per row (scale_mode 1): a group of TPR threads holds a whole row in
// registers: it is loaded once, its amax is a max reduction on the fp32 bit
// patterns of |x| (monotone for non-negative floats; Inf and NaN compare
// above every finite value, which is how non-finite input is detected), and
// the codes come from the registers.  Rows of more than kRowMaxCols columns
// are read twice instead, the second time from L2.  HBM traffic: 4 bytes
// read + 1 byte written per element.
//
// fp8_quantize_e4m3_rows_grouped runs the per-row path for up to 32
// independent matrices in one launch (job table in the kernel parameters).
//
// Per tensor (scale_mode 0): up to a quarter million elements are held in the
// registers of one cluster, which exchanges its maxima through distributed
// shared memory: one launch.  Beyond that an amax kernel folds into the
// dequant_scale[0] slot with atomicMax, an encode kernel reads it (the tensor
// backwards, its end being what is left in L2), and a one-thread kernel turns
// the slot into d = amax / 448.
//
// Most of these kernels start before the one that writes their input has
// ended (programmatic serialization): their loads are ordinary or L2 ones,
// never the read-only path, whose data may not change while a kernel runs.
// The kernels that read long rows twice are launched plainly and do use it
// (1024 x 32768: 48 us, 57 with ordinary loads; held in registers 30).
//
// The scale is s = T / amax with an IEEE-rounded division (__fdiv_rn), T the
// format's largest finite value (448 for E4M3, 57344 for E5M2), and each code
// is cvt.rn.satfinite of the IEEE product x * s (__fmul_rn) to that format.
// Every kernel is a template on the format (FMT 0: E4M3, 1: E5M2).
#include <algorithm>

#include <cuda_fp8.h>

#include "common.cuh"
#include "prune_select.cuh"
#include "ptx.cuh"

namespace gb300 {
namespace {

constexpr int kThreads = 256;
constexpr uint32_t kInfBits = 0x7F800000u;

__device__ __forceinline__ uint32_t abs_bits(float v)
{
    return __float_as_uint(v) & 0x7FFFFFFFu;
}

// Largest finite value of the format: the target of amax.
template <int FMT>
__device__ __forceinline__ float fmt_max()
{
    return FMT == 1 ? 57344.0f : 448.0f;
}

// Two fp32 values -> two codes (a in the low byte), round to nearest even,
// saturating to the largest finite value.
template <int FMT>
__device__ __forceinline__ uint32_t enc2(float a, float b)
{
    return static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE,
                                                          FMT == 1 ? __NV_E5M2 : __NV_E4M3));
}

template <int FMT>
__device__ __forceinline__ uint32_t enc4(float4 v, float s)
{
    return enc2<FMT>(__fmul_rn(v.x, s), __fmul_rn(v.y, s)) |
           (enc2<FMT>(__fmul_rn(v.z, s), __fmul_rn(v.w, s)) << 16);
}

__device__ __forceinline__ uint32_t block_max_u32(uint32_t v, uint32_t* red)
{
    v = __reduce_max_sync(0xFFFFFFFFu, v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
        red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < (blockDim.x >> 5) ? red[lane] : 0u;
        w = __reduce_max_sync(0xFFFFFFFFu, w);
        if (lane == 0)
            red[0] = w;
    }
    __syncthreads();
    uint32_t r = red[0];
    __syncthreads();
    return r;
}

// scale and dequant factor from the amax bit pattern
template <int FMT>
__device__ __forceinline__ void scale_from_amax(uint32_t amax_bits, float& s, float& d)
{
    const float amax = __uint_as_float(amax_bits);
    if (amax_bits == 0u) {
        s = 1.0f;
        d = 1.0f;
    } else {
        s = __fdiv_rn(fmt_max<FMT>(), amax);
        d = __fdiv_rn(amax, fmt_max<FMT>());
    }
}

// ---------------------------------------------------------------- rows in registers
//
// TPR threads (a warp, or a whole number of warps of one block) take a row,
// each holding U vectors of W = vector_of(A) consecutive elements: vector u of
// thread t starts at column (u * TPR + t) * W.  A is the alignment of x's
// rows in elements: 8, vectors of eight by one 32-byte load; 4, by two 16-byte
// ones (guarded scalar loads past the last whole vector in both); 1, where x
// or q allows neither, single elements, which keeps a warp's scalar loads and
// byte stores side by side: 4096 x 14336 at odd offsets 49.9 us (four
// consecutive elements a thread 94.6, the row read twice 86.2; 43.5 aligned).
// Two 16-byte loads a vector, not vectors of four: half as many addresses and
// guards, and the registers that they took left one block an SM (the same size
// at 16-byte offsets 64.3 -> 45.6 us).
//
// What bounds it: HBM, once enough bytes are in flight.  Rows are loaded
// once instead of twice (the second pass over L2 cost issue slots and load
// latency with nothing else to do), short rows share a block (one warp each
// up to 1024 columns) and the few long rows of a decode step get up to 1024
// threads each, since there the row's own latency is all there is.
// quant_row_kernel lets the GEMM that follows it start its setup at entry
// (quantise + GEMM at 16 x 12288 x 4096: 14.6 us, 15.6 when it signals
// after its loads, 15.8 without); launched with programmatic serialization
// itself, a 16 x 4096 call takes 1.41 us of its stream instead of 1.84.
// Measured (GB300, inputs rotated beyond L2), against one block of 256
// threads per row that read it twice: 16384 x 4096 58.0 -> 49.2 us (6.8
// TB/s), 16384 x 14336 183 -> 165 us (7.1 TB/s), 16384 x 512 28.5 -> 8.5 us,
// 16 x 14336 3.4 -> 2.5 us.  Fused with 2:4 compression: 14336 x 4096 64.7
// -> 50.2 us (6.6 TB/s), 16384 x 16384 250 -> 216 us (the
// four-group selection takes less than half of the instructions).  1024 x 32768 47.7
// -> 29.8 us.
constexpr int kRowBlock = 256;            // threads of a block where TPR is smaller
constexpr int kRowMaxCols = 32768;        // longest row held in registers

template <int TPR>
constexpr int row_block()
{
    return TPR > kRowBlock ? TPR : kRowBlock;
}

// 8 consecutive floats at p, the first `left` of them inside the row (0 for
// the others).  vec: p is aligned for whole-vector loads.
__device__ __forceinline__ void load_vec8(const float* p, int64_t left, bool vec, float (&v)[8])
{
    if (vec && left >= 8) {
        asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
                       "=f"(v[7])
                     : "l"(p));
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = i < left ? __ldca(p + i) : 0.0f;
    }
}

// As load_vec8 for rows that are only 16-byte aligned (left is 0 or >= 8).
__device__ __forceinline__ void load_two_vec4(const float* p, int64_t left, float (&v)[8])
{
    const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float4 a = left > 0 ? __ldca(reinterpret_cast<const float4*>(p)) : z;
    const float4 b = left > 0 ? __ldca(reinterpret_cast<const float4*>(p) + 1) : z;
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// 8 elements at p, the first `left` inside the row.  xa: alignment of the
// rows in elements (8, 4 or 1).
__device__ __forceinline__ void load_8(const float* p, int64_t left, int xa, float (&v)[8])
{
    if (xa == 8 || left < 8)
        load_vec8(p, left, xa == 8, v);
    else if (xa == 4)
        load_two_vec4(p, left, v);
    else
        load_vec8(p, left, false, v);
}

// Max over the tpr threads of a row group (tpr a power of two, the same for
// the whole block).  red: one entry per warp of the block, not in use by an
// earlier call since the last barrier; there is one barrier here if tpr > 32.
__device__ __forceinline__ uint32_t row_max(uint32_t m, int tpr, uint32_t* red)
{
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (tpr > 32) {
        const int warps = tpr / 32;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane == 0)
            red[warp] = m;
        __syncthreads();
        const int first = warp & ~(warps - 1);
        m = __reduce_max_sync(0xFFFFFFFFu, lane < warps ? red[first + lane] : 0u);
    }
    return m;
}

template <int U, int W>
__device__ __forceinline__ uint32_t held_amax(const float (&v)[U][W])
{
    uint32_t m = 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < W; ++i)
            m = max(m, abs_bits(v[u][i]));
    return m;
}

template <int FMT>
__device__ __forceinline__ uint32_t enc4(const float* v, float s)
{
    return enc4<FMT>(make_float4(v[0], v[1], v[2], v[3]), s);
}

// The codes of 8 elements to qr, the first `left` inside the row (qa: the
// row's store alignment, 8, 4 or 1).
template <int FMT>
__device__ __forceinline__ void store_codes8(uint8_t* qr, int64_t left, int qa, const float (&v)[8], float s)
{
    if (left <= 0)
        return;
    const uint32_t w[2] = {enc4<FMT>(v, s), enc4<FMT>(v + 4, s)};
    if (left >= 8 && qa >= 8) {
        *reinterpret_cast<uint2*>(qr) = make_uint2(w[0], w[1]);
    } else if (left >= 8 && qa >= 4) {
        reinterpret_cast<uint32_t*>(qr)[0] = w[0];
        reinterpret_cast<uint32_t*>(qr)[1] = w[1];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < left)
                qr[i] = static_cast<uint8_t>(w[i / 4] >> (8 * (i % 4)));
    }
}

template <int FMT>
__device__ __forceinline__ uint8_t enc1(float v, float s)
{
    return static_cast<uint8_t>(enc2<FMT>(__fmul_rn(v, s), 0.0f) & 0xFFu);
}

__host__ __device__ constexpr int vector_of(int a)
{
    return a == 1 ? 1 : 8;
}

// One row by its tpr threads (t: index within them; ok: the row exists).
// A, qa: alignment of the rows of x and q in elements (8, 4 or 1).
template <int FMT, int U, int A>
__device__ __forceinline__ void quantize_held_row(const float* xr, int cols, uint8_t* qr, float* d_out, int qa,
                                                  int* err, int tpr, uint32_t* red, int t, bool ok)
{
    constexpr int W = vector_of(A);
    float v[U][W];
    const int n = ok ? cols : 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int c = (u * tpr + t) * W;
        if constexpr (W == 8)
            load_8(xr + c, n - c, A, v[u]);
        else
            v[u][0] = c < n ? __ldca(xr + c) : 0.0f;
    }
    const uint32_t m = row_max(held_amax(v), tpr, red);
    float s, dq;
    scale_from_amax<FMT>(m, s, dq);
    if (t == 0 && ok) {
        if (m >= kInfBits)
            report_device_error(err, FP8_ERR_NONFINITE);
        *d_out = dq;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int c = (u * tpr + t) * W;
        if constexpr (W == 8)
            store_codes8<FMT>(qr + c, n - c, qa, v[u], s);
        else if (c < n)
            qr[c] = enc1<FMT>(v[u][0], s);
    }
}

template <int FMT, int TPR, int U, int A>
__global__ void __launch_bounds__(row_block<TPR>()) quant_row_kernel(const float* __restrict__ x, int64_t rows,
                                                                     int64_t cols, int64_t ldx,
                                                                     uint8_t* __restrict__ q, int64_t ldq,
                                                                     float* __restrict__ d, int qa, int early,
                                                                     int* err)
{
    grid_launch_dependents();
    __shared__ uint32_t red[2][32];
    constexpr int kRows = row_block<TPR>() / TPR;         // rows per block
    const int t = threadIdx.x % TPR;
    if (early) {
        // the row into L2 while the previous kernel still runs (L2 is
        // coherent: what that kernel writes is what the loads below return)
        const int64_t r = static_cast<int64_t>(blockIdx.x) * kRows + threadIdx.x / TPR;
        if (r < rows) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t c = static_cast<int64_t>(u * TPR + t) * vector_of(A);
                if (c < cols)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(x + r * ldx + c));
            }
        }
    }
    grid_dependency_wait();
    int flip = 0;
    for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRows; r0 < rows;
         r0 += static_cast<int64_t>(gridDim.x) * kRows, flip ^= 1) {
        const int64_t r = r0 + threadIdx.x / TPR;
        quantize_held_row<FMT, U, A>(x + r * ldx, static_cast<int>(cols), q + r * ldq, d + r, qa, err, TPR, red[flip], t, r < rows);
    }
}

// Per-row E4M3 quantisation and 2:4 compression of the codes in one pass
// (fp8_quantize_e4m3_prune24): as quant_row_kernel with W = 8, and a
// thread's vectors two at a time are four 2:4 groups, whose kept codes and
// index nibbles come from their codes exactly as prune24_compress's do
// (select_groups4): 4 bytes of kept codes and one metadata byte per vector,
// next to the neighbouring lanes'.  Needs cols % 128 == 0, x 16-aligned with
// ldx % 4 == 0, q 4-aligned with ldq % 4 == 0, a_vals 2-aligned (checked by
// the host).  It lets the next kernel's blocks in once its row is read, not
// at entry: what follows a weight load is mostly another one, whose waiting
// blocks cost this one's loads their slots (128 x 4096: 1.9 against 2.4 us).
// wide: x rows are 32-aligned; out8: q rows are 8-aligned and
// vals rows 4-aligned.
template <int TPR, int U>
__global__ void __launch_bounds__(row_block<TPR>()) quant_row_prune_kernel(const float* __restrict__ x, int64_t rows,
                                                                           int64_t cols, int64_t ldx,
                                                                           uint8_t* __restrict__ q, int64_t ldq,
                                                                           float* __restrict__ d,
                                                                           uint8_t* __restrict__ vals,
                                                                           uint8_t* __restrict__ meta, int wide,
                                                                           int out8, int* err)
{
    grid_dependency_wait();
    __shared__ uint32_t red[2][32];
    constexpr int kRows = row_block<TPR>() / TPR;
    const int t = threadIdx.x % TPR;
    const int64_t ldv = cols / 2, ldm = cols / 8;
    int flip = 0;
    for (int64_t r0 = static_cast<int64_t>(blockIdx.x) * kRows; r0 < rows;
         r0 += static_cast<int64_t>(gridDim.x) * kRows, flip ^= 1) {
        const int64_t r = r0 + threadIdx.x / TPR;
        const int64_t n = r < rows ? cols : 0;
        const float* xr = x + r * ldx;
        float v[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t c = static_cast<int64_t>(u * TPR + t) * 8;
            if (wide)
                load_vec8(xr + c, n - c, true, v[u]);
            else
                load_two_vec4(xr + c, n - c, v[u]);
        }
        const uint32_t m = row_max(held_amax(v), TPR, red[flip]);
        grid_launch_dependents();
        float s, dq;
        scale_from_amax<0>(m, s, dq);
        if (t == 0 && r < rows) {
            if (m >= kInfBits)
                report_device_error(err, FP8_ERR_NONFINITE);
            d[r] = dq;
        }
        uint8_t* qr = q + r * ldq;
        uint8_t* vr = vals + r * ldv;
        uint8_t* mr = meta + r * ldm;
        const auto put = [&](int64_t c, uint32_t w0, uint32_t w1, uint32_t kept, uint32_t nibs) {
            if (c >= n)
                return;
            if (out8) {
                *reinterpret_cast<uint2*>(qr + c) = make_uint2(w0, w1);
                *reinterpret_cast<uint32_t*>(vr + c / 2) = kept;
            } else {
                reinterpret_cast<uint32_t*>(qr + c)[0] = w0;
                reinterpret_cast<uint32_t*>(qr + c)[1] = w1;
                reinterpret_cast<uint16_t*>(vr + c / 2)[0] = static_cast<uint16_t>(kept);
                reinterpret_cast<uint16_t*>(vr + c / 2)[1] = static_cast<uint16_t>(kept >> 16);
            }
            mr[c / 8] = static_cast<uint8_t>(nibs);
        };
#pragma unroll
        for (int u = 0; u < U; u += 2) {
            const bool two = u + 1 < U;
            const int u1 = two ? u + 1 : u;
            const uint32_t w0 = enc4<0>(v[u], s), w1 = enc4<0>(v[u] + 4, s);
            const uint32_t w2 = two ? enc4<0>(v[u1], s) : 0u, w3 = two ? enc4<0>(v[u1] + 4, s) : 0u;
            uint32_t v01, v23;
            const uint32_t nibs = select_groups4(w0, w1, w2, w3, &v01, &v23);
            put(static_cast<int64_t>(u * TPR + t) * 8, w0, w1, v01, nibs);
            if (two)
                put(static_cast<int64_t>(u1 * TPR + t) * 8, w2, w3, v23, nibs >> 8);
        }
    }
}

// ---------------------------------------------------------------- rows read twice

// One row by a whole block of kThreads: amax, scale, codes.  vec: the row
// allows 16-byte loads and 4-byte stores (x 16-aligned, q 4-aligned).
template <int FMT>
__device__ __forceinline__ void quantize_row(const float* __restrict__ xr, int64_t cols,
                                             uint8_t* __restrict__ qr, float* __restrict__ d_out,
                                             int vec, int* err, uint32_t* red)
{
    const int64_t nvec = vec ? cols / 4 : 0;
    uint32_t m = 0;
    for (int64_t i = threadIdx.x; i < nvec; i += kThreads) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(xr) + i);
        m = max(m, max(max(abs_bits(v.x), abs_bits(v.y)), max(abs_bits(v.z), abs_bits(v.w))));
    }
    for (int64_t c = nvec * 4 + threadIdx.x; c < cols; c += kThreads)
        m = max(m, abs_bits(xr[c]));
    m = block_max_u32(m, red);
    if (m >= kInfBits && threadIdx.x == 0)
        report_device_error(err, FP8_ERR_NONFINITE);
    float s, dq;
    scale_from_amax<FMT>(m, s, dq);
    if (threadIdx.x == 0)
        *d_out = dq;
    for (int64_t i = threadIdx.x; i < nvec; i += kThreads) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(xr) + i);
        reinterpret_cast<uint32_t*>(qr)[i] = enc4<FMT>(v, s);
    }
    for (int64_t c = nvec * 4 + threadIdx.x; c < cols; c += kThreads)
        qr[c] = enc1<FMT>(xr[c], s);
}

template <int FMT>
__global__ void __launch_bounds__(kThreads) quant_long_row_kernel(const float* __restrict__ x,
                                                                  int64_t rows, int64_t cols,
                                                                  int64_t ldx, uint8_t* __restrict__ q,
                                                                  int64_t ldq, float* __restrict__ d,
                                                                  int vec, int* err)
{
    grid_launch_dependents();
    __shared__ uint32_t red[kThreads / 32];
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x)
        quantize_row<FMT>(x + r * ldx, cols, q + r * ldq, d + r, vec, err, red);
}

// Rows of more than kRowMaxCols columns, quantised and compressed: the
// encode pass re-reads the row and takes one 2:4 group per lane and step
// (lanes 2i and 2i + 1 join their nibbles into one metadata byte).
__global__ void __launch_bounds__(kThreads) quant_long_row_prune_kernel(const float* __restrict__ x, int64_t rows,
                                                                        int64_t cols, int64_t ldx,
                                                                        uint8_t* __restrict__ q, int64_t ldq,
                                                                        float* __restrict__ d,
                                                                        uint8_t* __restrict__ vals,
                                                                        uint8_t* __restrict__ meta, int* err)
{
    grid_launch_dependents();
    __shared__ uint32_t red[kThreads / 32];
    const int64_t n4 = cols / 4;
    const int64_t ldv = cols / 2, ldm = cols / 8;
    const int lane = threadIdx.x & 31;
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const float4* xr = reinterpret_cast<const float4*>(x + r * ldx);
        uint32_t m = 0;
        for (int64_t i = threadIdx.x; i < n4; i += kThreads) {
            const float4 v = __ldg(xr + i);
            m = max(m, max(max(abs_bits(v.x), abs_bits(v.y)), max(abs_bits(v.z), abs_bits(v.w))));
        }
        m = block_max_u32(m, red);
        if (m >= kInfBits && threadIdx.x == 0)
            report_device_error(err, FP8_ERR_NONFINITE);
        float s, dq;
        scale_from_amax<0>(m, s, dq);
        if (threadIdx.x == 0)
            d[r] = dq;
        uint8_t* qr = q + r * ldq;
        uint8_t* vr = vals + r * ldv;
        uint8_t* mr = meta + r * ldm;
        for (int64_t i = threadIdx.x; i < n4; i += kThreads) {
            const uint32_t w = enc4<0>(__ldg(xr + i), s);
            reinterpret_cast<uint32_t*>(qr)[i] = w;
            const uint32_t sel = select_group(w);
            reinterpret_cast<uint16_t*>(vr)[i] = static_cast<uint16_t>(sel & 0xFFFFu);
            const uint32_t nib = sel >> 16;
            const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, nib, 1);
            if ((lane & 1) == 0)
                mr[i >> 1] = static_cast<uint8_t>(nib | (next << 4));
        }
    }
}

// Many independent per-row quantisations in one launch: the job table is
// passed by value.  A block of TB threads takes one unit at a time: as many
// consecutive rows of one job as it has groups of that job's tpr threads.
// Units of job j follow those of job j - 1.
// Few rows (no more than two per SM) take a block of 512 each, for their own
// latency.  Of many, a row takes the fewest threads (a warp up to the block)
// that hold it in U vectors of eight each, so a launch may mix short rows and
// long ones, in blocks of 256 up to 8192 columns, so that several are resident
// on an SM.
// One block of 512 a row whatever its length took as long for rows of 64 as
// of 4096 columns: 32 jobs of 1024 rows of 64 columns 163 -> 10.6 us (85 with
// a block of 256 a row that read it twice), of 1024 columns 162 -> 26.0 (97),
// of 4096 166 -> 96 (116); 32 x 256 rows of 64 and 14336 columns in turn 79.2
// -> 45.2 (48.2).
struct RowJobs {
    fp8_quant_job job[FP8_QUANT_GROUPED_MAX];
    int64_t start[FP8_QUANT_GROUPED_MAX + 1];     // first unit of each job (read twice: first row)
    int xa[FP8_QUANT_GROUPED_MAX];        // alignment of the rows of x and of the codes, in elements: 8, 4 or 1
    int qa[FP8_QUANT_GROUPED_MAX];
    int shift[FP8_QUANT_GROUPED_MAX];     // log2 of the threads per row
    int n;
};

__device__ __forceinline__ int job_of(const RowJobs& jobs, int64_t g)
{
    int lo = 0, hi = jobs.n;                      // start[lo] <= g < start[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (jobs.start[mid] <= g)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

template <int TB, int U, int A, bool FEW>
__global__ void __launch_bounds__(TB, (!FEW && U * vector_of(A) == 16 ? 1536 : 1024) / TB)
    quant_rows_grouped_kernel(const __grid_constant__ RowJobs jobs, int* err)
{
    grid_launch_dependents();
    grid_dependency_wait();
    __shared__ uint32_t red[2][32];
    const int64_t total = jobs.start[jobs.n];
    int flip = 0;
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        const int j = job_of(jobs, g);
        const fp8_quant_job& J = jobs.job[j];
        constexpr int kShift = TB == 512 ? 9 : 8;
        const int shift = FEW ? kShift : jobs.shift[j], tpr = 1 << shift;
        const int t = FEW ? threadIdx.x : threadIdx.x & (tpr - 1);
        const int64_t unit = g - jobs.start[j];
        const int64_t r = FEW ? unit : (unit << (kShift - shift)) + (threadIdx.x >> shift);
        const float* xr = J.x + r * J.ldx;
        uint8_t* qr = J.q + r * J.ldq;
        quantize_held_row<0, U, A>(xr, static_cast<int>(J.cols), qr, J.dequant_scale + r, jobs.qa[j], err, tpr,
                                   red[flip], t, FEW || r < J.rows);
        if (tpr > 32)                             // (the buffers alternate from barrier to barrier)
            flip ^= 1;
    }
}

__global__ void __launch_bounds__(kThreads) quant_long_rows_grouped_kernel(const __grid_constant__ RowJobs jobs,
                                                                           int* err)
{
    grid_launch_dependents();
    __shared__ uint32_t red[kThreads / 32];
    const int64_t total = jobs.start[jobs.n];
    for (int64_t g = blockIdx.x; g < total; g += gridDim.x) {
        const int j = job_of(jobs, g);
        const fp8_quant_job& J = jobs.job[j];
        const int64_t r = g - jobs.start[j];
        quantize_row<0>(J.x + r * J.ldx, J.cols, J.q + r * J.ldq, J.dequant_scale + r, jobs.xa[j] >= 4 && jobs.qa[j] >= 4,
                        err, red);
    }
}

// ---------------------------------------------------------------- one scale per tensor
//
// A matrix is cut into vectors of 8 consecutive elements of a row, ceil(cols
// / 8) per row; a contiguous matrix comes as one long row.

// Whole tensor in one cluster: thread t of CTA c holds vectors (u * kCtas + c)
// * kClusterThreads + t.  What bounds it is latency: one launch, one load
// round trip, one cluster exchange, against a memset and three kernels
// before (256 x 256: 2.8 us of its stream, 9.0 before; and 3 launches less to
// issue).  262144 elements is what its registers hold: 512 x 512 takes 4.5
// us, 520 x 512 the long way 5.7.
constexpr int kCtas = 8, kClusterThreads = 512, kClusterMaxU = 8;
constexpr int64_t kClusterVecs = static_cast<int64_t>(kCtas) * kClusterThreads;      // per vector a thread

template <int FMT, int U>
__global__ void __launch_bounds__(kClusterThreads) quant_cluster_kernel(const float* __restrict__ x, int rows,
                                                                        int cols, int64_t ldx,
                                                                        uint8_t* __restrict__ q, int64_t ldq,
                                                                        float* __restrict__ d, int xa, int qa,
                                                                        int* err)
{
    grid_launch_dependents();
    grid_dependency_wait();
    __shared__ uint32_t red[32];
    __shared__ uint32_t cta_max;
    const uint32_t rank = cluster_ctarank();
    const int per_row = (cols + 7) / 8;
    float v[U][8];
    int r[U], c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int i = (u * kCtas + static_cast<int>(rank)) * kClusterThreads + static_cast<int>(threadIdx.x);
        r[u] = i / per_row;
        c[u] = (i - r[u] * per_row) * 8;
        load_8(x + r[u] * ldx + c[u], r[u] < rows ? cols - c[u] : 0, xa, v[u]);
    }
    uint32_t m = row_max(held_amax(v), kClusterThreads, red);
    if (threadIdx.x == 0)
        cta_max = m;
    cluster_sync();
    m = 0;
    const uint32_t slot = smem_u32(&cta_max);
#pragma unroll
    for (int k = 0; k < kCtas; ++k)
        m = max(m, ld_shared_cluster_u32(cluster_map(slot, static_cast<uint32_t>(k))));
    float s, dq;
    scale_from_amax<FMT>(m, s, dq);
    if (rank == 0 && threadIdx.x == 0) {
        if (m >= kInfBits)
            report_device_error(err, FP8_ERR_NONFINITE);
        *d = dq;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        store_codes8<FMT>(q + r[u] * ldq + c[u], r[u] < rows ? cols - c[u] : 0, qa, v[u], s);
    cluster_sync();                        // no CTA leaves while a peer may read its maximum
}

// Larger tensors.  A warp's 32 lanes take `1 << shift` vectors of 32 >> shift
// rows at a time (shift 5 but for rows of fewer than 32 vectors), one item;
// kItems items in flight.  Bound by HBM twice over (each pass reads x; what
// the first leaves in L2 spares the second a little: the second pass going
// backwards, and loads marked evict-first besides, which gave 2 to 4 % more
// and are not used).  3001 x 4100 28.7 -> 20.2 us, 8192 x 8192 110 -> 93 us
// against one element index division per 16 bytes and a memset.
constexpr int kItems = 4;

struct Items {
    int64_t rows, cols;
    int64_t segs;                          // items per row (groups)
    int64_t total;
    int shift;
};

// Row and column of this lane's vector of an item; row >= rows: none.
__device__ __forceinline__ void item_vec(const Items& it, int64_t item, int64_t* r, int64_t* c)
{
    int64_t g, seg;
    if (it.total <= 0xFFFFFFFFll) {
        const uint32_t n = static_cast<uint32_t>(it.segs);
        g = static_cast<uint32_t>(item) / n;
        seg = static_cast<uint32_t>(item) - static_cast<uint32_t>(g) * n;
    } else {
        g = item / it.segs;
        seg = item - g * it.segs;
    }
    const int lane = threadIdx.x & 31;
    *r = (g << (5 - it.shift)) + (lane >> it.shift);
    *c = ((seg << it.shift) + (lane & ((1 << it.shift) - 1))) * 8;
}

__global__ void quant_zero_kernel(uint32_t* slot)
{
    grid_launch_dependents();
    grid_dependency_wait();
    *slot = 0u;
}

__global__ void __launch_bounds__(kThreads) quant_amax_kernel(const float* __restrict__ x, Items it, int64_t ldx,
                                                              int xa, uint32_t* __restrict__ slot)
{
    grid_launch_dependents();
    grid_dependency_wait();
    __shared__ uint32_t red[kThreads / 32];
    uint32_t m = 0;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (kThreads / 32);
    for (int64_t i0 = (static_cast<int64_t>(blockIdx.x) * (kThreads / 32) + (threadIdx.x >> 5)) * kItems;
         i0 < it.total; i0 += warps * kItems) {
        float v[kItems][8];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            int64_t r, c;
            item_vec(it, i0 + k, &r, &c);
            load_8(x + r * ldx + c, i0 + k < it.total && r < it.rows ? it.cols - c : 0, xa, v[k]);
        }
        m = max(m, held_amax(v));
    }
    m = block_max_u32(m, red);
    if (threadIdx.x == 0 && m != 0u)
        atomicMax(slot, m);
}

template <int FMT>
__global__ void __launch_bounds__(kThreads) quant_encode_kernel(const float* __restrict__ x, Items it, int64_t ldx,
                                                                int xa, uint8_t* __restrict__ q, int64_t ldq, int qa,
                                                                const uint32_t* __restrict__ slot)
{
    grid_launch_dependents();
    grid_dependency_wait();
    float s, dq;
    scale_from_amax<FMT>(__ldcg(slot), s, dq);
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (kThreads / 32);
    for (int64_t i0 = (static_cast<int64_t>(blockIdx.x) * (kThreads / 32) + (threadIdx.x >> 5)) * kItems;
         i0 < it.total; i0 += warps * kItems) {
        float v[kItems][8];
        int64_t r[kItems], c[kItems], left[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const int64_t item = it.total - 1 - (i0 + k);          // the end first: it is in L2
            item_vec(it, item < 0 ? 0 : item, &r[k], &c[k]);
            left[k] = item >= 0 && r[k] < it.rows ? it.cols - c[k] : 0;
            load_8(x + r[k] * ldx + c[k], left[k], xa, v[k]);
        }
#pragma unroll
        for (int k = 0; k < kItems; ++k)
            store_codes8<FMT>(q + r[k] * ldq + c[k], left[k], qa, v[k], s);
    }
}

template <int FMT>
__global__ void quant_finalize_kernel(uint32_t* slot, int* err)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const uint32_t m = *slot;
    if (m >= kInfBits)
        report_device_error(err, FP8_ERR_NONFINITE);
    float s, dq;
    scale_from_amax<FMT>(m, s, dq);
    *reinterpret_cast<float*>(slot) = dq;
}

// Alignment of matrix rows of `esz`-byte elements: the largest of 8, 4 and
// 1 elements that every row starts on a multiple of.
int row_align(const void* p, int64_t ld, int esz)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    if (a % (8 * esz) == 0 && ld % 8 == 0)
        return 8;
    return a % (4 * esz) == 0 && ld % 4 == 0 ? 4 : 1;
}

int row_grid(int64_t rows, int rows_per_block)
{
    const int64_t blocks = (rows + rows_per_block - 1) / rows_per_block;
    return static_cast<int>(std::min<int64_t>(blocks, 65535LL * 8));
}

// Calls f.template operator()<TPR, U8>() with the threads per row and
// 8-element vectors per thread for rows of `cols` columns.  Few rows (no
// more than two per SM): as many threads as the row has work for.  Many:
// warps up to 1024 columns, then blocks of 128 to 512 threads with two to
// four vectors each, in steps of a vector where half a vector more would
// leave lanes idle (4100 columns: 16.5 us for 4096 rows with three vectors
// a thread, 20.8 with four).
template <typename F>
void with_row_shape(int64_t rows, int64_t cols, F f)
{
    if (rows <= 2 * sm_count()) {
        if (cols <= 1024)
            f.template operator()<128, 1>();
        else if (cols <= 4096)
            f.template operator()<512, 1>();
        else if (cols <= 16384)
            f.template operator()<1024, 2>();
        else
            f.template operator()<1024, 4>();
    } else if (cols <= 256) {
        f.template operator()<32, 1>();
    } else if (cols <= 512) {
        f.template operator()<32, 2>();
    } else if (cols <= 1024) {
        f.template operator()<32, 4>();
    } else if (cols <= 2048) {
        f.template operator()<128, 2>();
    } else if (cols <= 4096) {
        f.template operator()<256, 2>();
    } else if (cols <= 6144) {
        f.template operator()<256, 3>();
    } else if (cols <= 8192) {
        f.template operator()<256, 4>();
    } else if (cols <= 12288) {
        f.template operator()<512, 3>();
    } else if (cols <= 16384) {
        f.template operator()<512, 4>();
    } else {
        f.template operator()<1024, 4>();
    }
}

// The items of a matrix (flat: contiguous, one long row).
Items items_of(int64_t rows, int64_t cols, bool flat)
{
    Items it;
    it.rows = flat ? 1 : rows;
    it.cols = flat ? rows * cols : cols;
    const int64_t vecs = (it.cols + 7) / 8;
    it.shift = 5;
    while (it.shift > 0 && (int64_t{1} << (it.shift - 1)) >= vecs)
        --it.shift;
    it.segs = (vecs + (int64_t{1} << it.shift) - 1) >> it.shift;
    it.total = it.segs * ((it.rows + (32 >> it.shift) - 1) >> (5 - it.shift));
    return it;
}

int item_grid(const Items& it)
{
    const int64_t per_block = kThreads / 32 * kItems;
    return static_cast<int>(std::min<int64_t>((it.total + per_block - 1) / per_block, sm_count() * 8));
}

template <int FMT>
struct RowLaunch {
    const float* x;
    int64_t rows, cols, ldx;
    uint8_t* q;
    int64_t ldq;
    float* d;
    int* err;
    cudaStream_t st;

    template <int TPR, int U>
    void operator()() const
    {
        const int xa = row_align(x, ldx, 4), qa = row_align(q, ldq, 1);
        const int grid = row_grid(rows, row_block<TPR>() / TPR);
        const auto launch = [&](auto* kernel) {
            launch_dependent(kernel, grid, row_block<TPR>(), st, x, rows, cols, ldx, q, ldq, d, qa,
                             rows <= 2 * sm_count(), err);
        };
        if (xa == 8 && qa >= 4)
            launch(quant_row_kernel<FMT, TPR, U, 8>);
        else if (xa == 4 && qa >= 4)
            launch(quant_row_kernel<FMT, TPR, U, 4>);
        else
            launch(quant_row_kernel<FMT, TPR, 8 * U, 1>);
    }
};

struct RowPruneLaunch {
    const float* x;
    int64_t rows, cols, ldx;
    uint8_t* q;
    int64_t ldq;
    float* d;
    uint8_t *vals, *meta;
    int* err;
    cudaStream_t st;

    template <int TPR, int U>
    void operator()() const
    {
        const int out8 = row_align(q, ldq, 1) == 8 && reinterpret_cast<uintptr_t>(vals) % 4 == 0;
        launch_dependent(quant_row_prune_kernel<TPR, U>, row_grid(rows, row_block<TPR>() / TPR), row_block<TPR>(), st,
                         x, rows, cols, ldx, q, ldq, d, vals, meta, row_align(x, ldx, 4) == 8, out8, err);
    }
};

template <int FMT>
int quantize(const float* x, int64_t rows, int64_t cols, int64_t ldx, int scale_mode, uint8_t* q,
             int64_t ldq, float* dequant_scale, cudaStream_t st)
{
    if (rows < 0 || cols < 0 || (scale_mode != 0 && scale_mode != 1))
        return FP8_ERR_INVALID;
    if (rows == 0 || cols == 0)
        return FP8_OK;
    if (!x || !q || !dequant_scale)
        return FP8_ERR_INVALID;
    if (ldx < cols || ldq < cols)
        return FP8_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(x) & 3u) || (reinterpret_cast<uintptr_t>(dequant_scale) & 3u))
        return FP8_ERR_ALIGN;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    int* err = device_error_word();
    const int vec = aligned16(x) && (ldx % 4 == 0) &&
                    (reinterpret_cast<uintptr_t>(q) % 4 == 0) && (ldq % 4 == 0);
    if (scale_mode == 1) {
        if (cols <= kRowMaxCols)
            with_row_shape(rows, cols, RowLaunch<FMT>{x, rows, cols, ldx, q, ldq, dequant_scale, err, st});
        else
            quant_long_row_kernel<FMT><<<row_grid(rows, 1), kThreads, 0, st>>>(x, rows, cols, ldx, q, ldq,
                                                                               dequant_scale, vec, err);
        GB_CUDA_OK(cudaGetLastError());
        return FP8_OK;
    }
    const int xa = row_align(x, ldx, 4), qa = row_align(q, ldq, 1);
    const int64_t vecs = rows <= kClusterVecs * kClusterMaxU && cols <= 8 * kClusterVecs * kClusterMaxU
                             ? rows * ((cols + 7) / 8)
                             : INT64_MAX;
    if (vecs <= kClusterVecs * kClusterMaxU) {
        const auto launch = [&](auto* kernel) {
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            attr[1].id = cudaLaunchAttributeClusterDimension;
            attr[1].val.clusterDim.x = kCtas;
            attr[1].val.clusterDim.y = 1;
            attr[1].val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kCtas);
            cfg.blockDim = dim3(kClusterThreads);
            cfg.stream = st;
            cfg.attrs = attr;
            cfg.numAttrs = 2;
            return cudaLaunchKernelEx(&cfg, kernel, x, static_cast<int>(rows), static_cast<int>(cols), ldx, q, ldq,
                                      dequant_scale, xa, qa, err);
        };
        GB_CUDA_OK(vecs <= kClusterVecs       ? launch(quant_cluster_kernel<FMT, 1>)
                   : vecs <= 2 * kClusterVecs ? launch(quant_cluster_kernel<FMT, 2>)
                   : vecs <= 4 * kClusterVecs ? launch(quant_cluster_kernel<FMT, 4>)
                                              : launch(quant_cluster_kernel<FMT, kClusterMaxU>));
        return FP8_OK;
    }
    uint32_t* slot = reinterpret_cast<uint32_t*>(dequant_scale);
    launch_dependent(quant_zero_kernel, 1, 1, st, slot);
    GB_CUDA_OK(cudaGetLastError());
    // (a flat matrix is as aligned as its start, whatever its columns)
    const bool x_flat = ldx == cols, flat = x_flat && ldq == cols;
    const Items xi = items_of(rows, cols, x_flat), qi = items_of(rows, cols, flat);
    launch_dependent(quant_amax_kernel, item_grid(xi), kThreads, st, x, xi, ldx, x_flat ? row_align(x, 0, 4) : xa,
                     slot);
    GB_CUDA_OK(cudaGetLastError());
    launch_dependent(quant_encode_kernel<FMT>, item_grid(qi), kThreads, st, x, qi, ldx,
                     flat ? row_align(x, 0, 4) : xa, q, ldq, flat ? row_align(q, 0, 1) : qa, slot);
    GB_CUDA_OK(cudaGetLastError());
    launch_dependent(quant_finalize_kernel<FMT>, 1, 1, st, slot, err);
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

// ---------------------------------------------------------------- block-scaled (MX)

// Byte offset of the scale of row r, 32-element block b, in the tiled layout
// (include/gb300fp8.h): 512-byte chunks per 128 rows x 128 columns, chunk
// (r / 128, b / 4) at (r / 128) * kb + b / 4, and within a chunk row r % 32
// at 16-byte row r % 32, 4-byte word (r % 128) / 32, byte b % 4.
__device__ __forceinline__ int64_t mx_tiled_offset(int64_t r, int64_t b, int64_t kb)
{
    return 512 * ((r >> 7) * kb + (b >> 2)) + 16 * (r & 31) + 4 * ((r & 127) >> 5) + (b & 3);
}

// Scale code of a block and its encoding scale 2^-e from the block's amax bits
// (see quant_mx_kernel; 0 and 1 where amax is 0 or not finite).
template <int FMT>
__device__ __forceinline__ uint32_t mx_block_scale(uint32_t m, float& s)
{
    constexpr int kEmax = FMT == 1 ? 15 : 8;
    s = 1.0f;
    if (m == 0u || m >= kInfBits)
        return 0u;
    const int E = static_cast<int>(m >> 23);      // biased exponent of amax
    const int e = E == 0 ? -127 : max(E - 127 - kEmax, -127);
    s = __uint_as_float(static_cast<uint32_t>(127 - e) << 23);         // normal
    return static_cast<uint32_t>(e + 127);
}

// One warp quantises a 256-column window of one row at a time: lane l holds
// columns 8l .. 8l + 7, so a 32-element block is four lanes, and its amax is
// their local maxima and two shuffles.  For a non-zero block, e = floor(log2
// amax) - emax (emax 8 for E4M3, 15 for E5M2) read from amax's exponent field
// (a subnormal amax gives the floor -127), so amax * 2^-e lies in [2^emax,
// 2^(emax+1)); the scale code is e + 127 and the codes are the format's
// round-to-nearest-even, saturating encoding of the IEEE product x * 2^-e
// (exact unless it falls below 2^-126).  An all-zero block gets scale code 0
// and the codes of its (signed) zeros.  The four codes of a 128-column
// k-block are joined over its 16 lanes and leave as one word.
// The windows of the matrix are one list, the row by one 32-bit division, a
// warp takes one at a time; with the tiled scale layout the list goes on over
// the padding rows of the last 128, whose scales are 1 (a memset before it
// kept the launch from overlapping the kernel before).  What bounds it beside
// HBM is instructions: 128-column windows of four columns a lane spent twice
// as many on the same data (4096 x 4096 19.5 us, 15.0 now; 4096 x 14336 54.8,
// 46.5; 16384 x 8192 112, 103; 16 x 4096 3.6, 2.0).  Two, four or eight
// windows a warp at once, loads first, were slower (16.7, 17.6 and 23.9 us at
// 4096 x 4096): enough warps have a load in flight.
// WIDE = false, where the rows of x or q start on any element: lane l holds
// columns l, l + 32, ..., one of each block, so that loads and byte stores lie
// side by side and a block's amax is one warp reduction; lane k takes the
// scale of block k (16384 x 4096 at odd offsets with tiled scales: 72.5 us,
// eight consecutive elements a lane 92.1, four 74.3; each lane taking all
// eight scales 94.8).
template <int FMT, int TILED, bool WIDE>
__global__ void __launch_bounds__(kThreads) quant_mx_kernel(const float* __restrict__ x, int64_t rows,
                                                            int64_t cols, int64_t ldx, int xa,
                                                            uint8_t* __restrict__ q, int64_t ldq, int qa,
                                                            uint8_t* __restrict__ sc, int* err)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int64_t kb = (cols + 127) / 128;
    const int64_t segs = (cols + 255) / 256;
    const int64_t total = (TILED ? (rows + 127) / 128 * 128 : rows) * segs;
    const int64_t step = static_cast<int64_t>(gridDim.x) * (kThreads / 32);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * (kThreads / 32) + (threadIdx.x >> 5); i < total; i += step) {
        int64_t r, seg;
        if (total <= 0xFFFFFFFFll) {
            const uint32_t n = static_cast<uint32_t>(segs), g = static_cast<uint32_t>(i) / n;
            r = g;
            seg = static_cast<uint32_t>(i) - g * n;
        } else {
            r = i / segs;
            seg = i - r * segs;
        }
        uint32_t word;                            // the four scale codes of this half warp's k-block
        if constexpr (WIDE) {
            const int64_t c = seg * 256 + 8 * lane;
            const bool in = c < cols && r < rows; // cols % 32 == 0: a lane's eight columns are all in or out
            float v[8];
            load_8(x + r * ldx + c, in ? 8 : 0, xa, v);
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                m = max(m, abs_bits(v[k]));
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
            if (m >= kInfBits && (lane & 3) == 0)
                report_device_error(err, FP8_ERR_NONFINITE);
            float s;
            const uint32_t code = mx_block_scale<FMT>(m, s);
            store_codes8<FMT>(q + r * ldq + c, in ? 8 : 0, qa, v, s);
            // blocks past cols and padding rows: scale 1
            word = (in ? code : 127u) << (8 * ((lane >> 2) & 3));
            word |= __shfl_xor_sync(0xFFFFFFFFu, word, 4);
            word |= __shfl_xor_sync(0xFFFFFFFFu, word, 8);
        } else {
            // blocks of this window inside the matrix
            const int nb = r < rows ? static_cast<int>(min(cols - seg * 256, static_cast<int64_t>(256))) / 32 : 0;
            const float* xw = x + r * ldx + seg * 256 + lane;
            uint8_t* qw = q + r * ldq + seg * 256 + lane;
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = k < nb ? __ldca(xw + 32 * k) : 0.0f;
            // block k's amax to lane k, which takes its scale
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t mk = __reduce_max_sync(0xFFFFFFFFu, abs_bits(v[k]));
                m = lane == k ? mk : m;
            }
            if (m >= kInfBits)
                report_device_error(err, FP8_ERR_NONFINITE);
            float s;
            const uint32_t code = mx_block_scale<FMT>(m, s);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float sk = __shfl_sync(0xFFFFFFFFu, s, k);
                if (k < nb)
                    qw[32 * k] = enc1<FMT>(v[k], sk);
            }
            // (blocks past cols and padding rows: scale 1)
            word = (lane < nb ? code : 127u) << (8 * (lane & 3));
            word |= __shfl_xor_sync(0xFFFFFFFFu, word, 1);
            word |= __shfl_xor_sync(0xFFFFFFFFu, word, 2);
            word = __shfl_sync(0xFFFFFFFFu, word, lane >> 4 << 2);       // blocks 0 .. 3, 4 .. 7
        }
        const int64_t k = 2 * seg + (lane >> 4);              // k-block of this half warp
        if ((lane & 15) != 0 || k >= kb)
            continue;
        if (TILED) {
            *reinterpret_cast<uint32_t*>(sc + mx_tiled_offset(r, 4 * k, kb)) = word;
        } else {
            uint8_t* sr = sc + r * (cols / 32) + 4 * k;
            const int nb = static_cast<int>(min(static_cast<int64_t>(4), cols / 32 - 4 * k));
            if (nb == 4 && (reinterpret_cast<uintptr_t>(sr) & 3u) == 0) {
                *reinterpret_cast<uint32_t*>(sr) = word;
            } else {
                for (int j = 0; j < nb; ++j)
                    sr[j] = static_cast<uint8_t>(word >> (8 * j));
            }
        }
    }
}

// Row-major scales [rows, cols / 32] -> the tiled layout (one 4-byte word,
// four blocks of one row, per thread; padding rows and blocks get 127).
__global__ void __launch_bounds__(kThreads) mx_scales_tile_kernel(const uint8_t* __restrict__ src, int64_t rows,
                                                                  int64_t cols, uint8_t* __restrict__ dst)
{
    grid_launch_dependents();
    grid_dependency_wait();
    const int64_t kb = (cols + 127) / 128;
    const int64_t nbr = cols / 32;
    const int64_t total = (rows + 127) / 128 * 128 * kb;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; i < total; i += stride) {
        const int64_t r = i / kb, k = i - r * kb;
        uint32_t word = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t b = 4 * k + j;
            const uint32_t v = (r < rows && b < nbr) ? __ldca(src + r * nbr + b) : 127u;
            word |= v << (8 * j);
        }
        *reinterpret_cast<uint32_t*>(dst + mx_tiled_offset(r, 4 * k, kb)) = word;
    }
}

int grid_for_items(int64_t items)
{
    const int64_t blocks = (items + kThreads - 1) / kThreads;
    const int64_t cap = static_cast<int64_t>(sm_count()) * 8;
    return static_cast<int>(blocks < cap ? (blocks > 0 ? blocks : 1) : cap);
}

template <int FMT>
int quantize_mx(const float* x, int64_t rows, int64_t cols, int64_t ldx, uint8_t* q, int64_t ldq,
                uint8_t* scales, int layout, cudaStream_t st)
{
    if (rows < 0 || cols < 0 || (layout != 0 && layout != 1))
        return FP8_ERR_INVALID;
    if (cols % 32 != 0)
        return FP8_ERR_SHAPE;
    if (rows == 0 || cols == 0)
        return FP8_OK;
    if (!x || !q || !scales)
        return FP8_ERR_INVALID;
    if (ldx < cols || ldq < cols)
        return FP8_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(x) & 3u) || (layout == 1 && !aligned16(scales)))
        return FP8_ERR_ALIGN;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    const int xa = row_align(x, ldx, 4), qa = row_align(q, ldq, 1);
    // a few blocks per SM, each walking windows (short-lived blocks cost more
    // in launch and tail than they save)
    const int64_t windows = (layout == 1 ? (rows + 127) / 128 * 128 : rows) * ((cols + 255) / 256);
    const int64_t per_block = kThreads / 32;
    const int grid = static_cast<int>(std::min<int64_t>((windows + per_block - 1) / per_block, sm_count() * 16));
    int* err = device_error_word();
    const auto launch = [&](auto* wide, auto* single) {
        launch_dependent(xa >= 4 && qa >= 4 ? wide : single, grid, kThreads, st, x, rows, cols, ldx, xa, q, ldq, qa,
                         scales, err);
    };
    if (layout == 1)
        launch(quant_mx_kernel<FMT, 1, true>, quant_mx_kernel<FMT, 1, false>);
    else
        launch(quant_mx_kernel<FMT, 0, true>, quant_mx_kernel<FMT, 0, false>);
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

}  // namespace
}  // namespace gb300

extern "C" size_t fp8_mx_scale_tiled_bytes(int64_t rows, int64_t cols)
{
    if (rows <= 0 || cols <= 0)
        return 0;
    return static_cast<size_t>((rows + 127) / 128) * static_cast<size_t>((cols + 127) / 128) * 512;
}

extern "C" int fp8_quantize_mx(const float* x, int64_t rows, int64_t cols, int64_t ldx, int format,
                               uint8_t* q, int64_t ldq, uint8_t* scales, int scale_layout,
                               fp8_stream_t stream)
{
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (format == FP8_E4M3)
        return gb300::quantize_mx<0>(x, rows, cols, ldx, q, ldq, scales, scale_layout, st);
    if (format == FP8_E5M2)
        return gb300::quantize_mx<1>(x, rows, cols, ldx, q, ldq, scales, scale_layout, st);
    return FP8_ERR_INVALID;
}

extern "C" int fp8_mx_scales_to_tiled(const uint8_t* scales, int64_t rows, int64_t cols, uint8_t* tiled,
                                      fp8_stream_t stream)
{
    using namespace gb300;
    if (rows < 0 || cols < 0)
        return FP8_ERR_INVALID;
    if (cols % 32 != 0)
        return FP8_ERR_SHAPE;
    if (rows == 0 || cols == 0)
        return FP8_OK;
    if (!scales || !tiled)
        return FP8_ERR_INVALID;
    if (!aligned16(tiled))
        return FP8_ERR_ALIGN;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    const int64_t words = (rows + 127) / 128 * 128 * ((cols + 127) / 128);
    launch_dependent(mx_scales_tile_kernel, grid_for_items(words), kThreads, reinterpret_cast<cudaStream_t>(stream),
                     scales, rows, cols, tiled);
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

extern "C" int fp8_quantize_e4m3(const float* x, int64_t rows, int64_t cols, int64_t ldx,
                                 int scale_mode, uint8_t* q, int64_t ldq, float* dequant_scale,
                                 fp8_stream_t stream)
{
    return gb300::quantize<0>(x, rows, cols, ldx, scale_mode, q, ldq, dequant_scale,
                              reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int fp8_quantize_e4m3_prune24(const float* x, int64_t rows, int64_t cols, int64_t ldx, uint8_t* q,
                                         int64_t ldq, float* dequant_scale, uint8_t* a_vals, uint8_t* a_meta,
                                         fp8_stream_t stream)
{
    using namespace gb300;
    if (rows < 0 || cols < 0)
        return FP8_ERR_INVALID;
    if (rows == 0 || cols == 0)
        return FP8_OK;
    if (!x || !q || !dequant_scale || !a_vals || !a_meta)
        return FP8_ERR_INVALID;
    if (cols % 128 != 0 || ldx < cols || ldq < cols)
        return FP8_ERR_SHAPE;
    if (!aligned16(x) || ldx % 4 != 0 || reinterpret_cast<uintptr_t>(q) % 4 != 0 || ldq % 4 != 0 ||
        reinterpret_cast<uintptr_t>(a_vals) % 2 != 0 || reinterpret_cast<uintptr_t>(dequant_scale) % 4 != 0)
        return FP8_ERR_ALIGN;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int* err = device_error_word();
    if (cols <= kRowMaxCols)
        with_row_shape(rows, cols, RowPruneLaunch{x, rows, cols, ldx, q, ldq, dequant_scale, a_vals, a_meta, err, st});
    else
        quant_long_row_prune_kernel<<<row_grid(rows, 1), kThreads, 0, st>>>(x, rows, cols, ldx, q, ldq, dequant_scale,
                                                                            a_vals, a_meta, err);
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

extern "C" int fp8_quantize_e5m2(const float* x, int64_t rows, int64_t cols, int64_t ldx,
                                 int scale_mode, uint8_t* q, int64_t ldq, float* dequant_scale,
                                 fp8_stream_t stream)
{
    return gb300::quantize<1>(x, rows, cols, ldx, scale_mode, q, ldq, dequant_scale,
                              reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int fp8_quantize_e4m3_rows_grouped(const fp8_quant_job* jobs, int num_jobs,
                                              fp8_stream_t stream)
{
    using namespace gb300;
    if (num_jobs < 0 || (num_jobs > 0 && !jobs))
        return FP8_ERR_INVALID;
    if (num_jobs > FP8_QUANT_GROUPED_MAX)
        return FP8_ERR_SHAPE;
    RowJobs rj;
    memset(&rj, 0, sizeof(rj));
    int64_t rows = 0, max_cols = 0;
    int a = 8;                                    // the least alignment of any job's rows
    for (int i = 0; i < num_jobs; ++i) {
        const fp8_quant_job& J = jobs[i];
        if (J.rows < 0 || J.cols < 0)
            return FP8_ERR_INVALID;
        if (J.rows == 0 || J.cols == 0)
            continue;
        if (!J.x || !J.q || !J.dequant_scale)
            return FP8_ERR_INVALID;
        if (J.ldx < J.cols || J.ldq < J.cols)
            return FP8_ERR_SHAPE;
        if ((reinterpret_cast<uintptr_t>(J.x) & 3u) ||
            (reinterpret_cast<uintptr_t>(J.dequant_scale) & 3u))
            return FP8_ERR_ALIGN;
        const int k = rj.n++;
        rj.job[k] = J;
        rj.xa[k] = row_align(J.x, J.ldx, 4);
        rj.qa[k] = row_align(J.q, J.ldq, 1);
        a = std::min(a, rj.qa[k] >= 4 ? rj.xa[k] : 1);
        max_cols = std::max(max_cols, J.cols);
        rows += J.rows;
    }
    if (rows == 0)
        return FP8_OK;
    if (!device_supported())
        return FP8_ERR_UNSUPPORTED;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int* err = device_error_word();
    // threads a block and vectors a thread (see quant_rows_grouped_kernel)
    const bool few = rows <= 2 * sm_count();
    const bool held = max_cols <= 4 * 8 * 512;
    const int tb = few || max_cols > 4 * 8 * 256 ? 512 : 256;
    const int u = max_cols > 2 * 8 * tb ? 4 : (few && max_cols <= 8 * tb ? 1 : 2);
    int64_t units = 0;
    for (int i = 0; i < rj.n; ++i) {
        int shift = few ? 9 : 5;
        while ((1 << shift) < tb && (int64_t{8} * u << shift) < rj.job[i].cols)
            ++shift;
        const int per_unit = held ? tb >> shift : 1;
        rj.shift[i] = shift;
        rj.start[i] = units;
        units += (rj.job[i].rows + per_unit - 1) / per_unit;
    }
    rj.start[rj.n] = units;
    const int grid = row_grid(units, 1);
    const auto launch = [&](auto* a8, auto* a4, auto* a1) {
        launch_dependent(a == 8 ? a8 : a == 4 ? a4 : a1, grid, tb, st, rj, err);
    };
    if (!held)
        quant_long_rows_grouped_kernel<<<grid, kThreads, 0, st>>>(rj, err);
    else if (few && u == 1)
        launch(quant_rows_grouped_kernel<512, 1, 8, true>, quant_rows_grouped_kernel<512, 1, 4, true>,
               quant_rows_grouped_kernel<512, 8, 1, true>);
    else if (few && u == 2)
        launch(quant_rows_grouped_kernel<512, 2, 8, true>, quant_rows_grouped_kernel<512, 2, 4, true>,
               quant_rows_grouped_kernel<512, 16, 1, true>);
    else if (few)
        launch(quant_rows_grouped_kernel<512, 4, 8, true>, quant_rows_grouped_kernel<512, 4, 4, true>,
               quant_rows_grouped_kernel<512, 32, 1, true>);
    else if (u == 2)
        launch(quant_rows_grouped_kernel<256, 2, 8, false>, quant_rows_grouped_kernel<256, 2, 4, false>,
               quant_rows_grouped_kernel<256, 16, 1, false>);
    else if (tb == 256)
        launch(quant_rows_grouped_kernel<256, 4, 8, false>, quant_rows_grouped_kernel<256, 4, 4, false>,
               quant_rows_grouped_kernel<256, 32, 1, false>);
    else
        launch(quant_rows_grouped_kernel<512, 4, 8, false>, quant_rows_grouped_kernel<512, 4, 4, false>,
               quant_rows_grouped_kernel<512, 32, 1, false>);
    GB_CUDA_OK(cudaGetLastError());
    return FP8_OK;
}

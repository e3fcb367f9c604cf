// Packers and quantisers: tensor scale, NVFP4 and LUT3 round-to-nearest,
// LUT3 -> NVFP4 autocast, canonical export, and the activation quantiser of the
// prefill path.  (App. A.3 "Quantization formats", Sec. 2.3, App. C.2 storage.)
//
// Quantiser arithmetic is fp32 with explicit round-to-nearest intrinsics so the
// compiler cannot contract or reorder it:
//   rc6 = 1/(6 s);  t = extreme * rc6;  d = E4M3(t);  r = 1/(s * dec(d));  y = x * r
#include <atomic>

#include "dq_common.cuh"
#include "dq_quant.cuh"

namespace dq {

// ------------------------------------------------------------------ header

struct Codebook8 { unsigned short h[8]; };
static_assert(kHeaderBytes == 256 * 4, "one word per thread of pack_header_kernel");

__global__ void __launch_bounds__(256) pack_header_kernel(PackedHeader *hdr, Codebook8 cb)
{
    reinterpret_cast<uint32_t *>(hdr)[threadIdx.x] = 0u;                     // the whole kilobyte
    __syncthreads();
    if (threadIdx.x != 0) return;
    hdr->s = 1.0f;
    int zero_idx = 0;
    unsigned int amap = 0;
    for (int j = 0; j < 8; ++j) {
        float g = __half2float(__ushort_as_half(cb.h[j]));
        hdr->lut_levels[j] = g;
        hdr->lut_f16[j] = cb.h[j];
        if (g == 0.0f) zero_idx = j;
        amap |= (f32x2_to_e2m1x2(g, 0.0f) & 0xFu) << (4 * j);
    }
    for (int j = 0; j < 7; ++j)
        hdr->lut_thresholds[j] = __fmul_rn(__fadd_rn(hdr->lut_levels[j], hdr->lut_levels[j + 1]), 0.5f);
    hdr->lut_thresholds[7] = __int_as_float(0x7f800000);
    hdr->lut_zero_idx = zero_idx;
    hdr->autocast_map = amap;
    // LUT2A16 grid (App. A.3 "LUT formats"), rounded to fp16
    const float grid2[4] = {-3.6517f, 0.0f, 2.5227f, 6.0f};
    for (int j = 0; j < 4; ++j) {
        const __half h = __float2half_rn(grid2[j]);
        hdr->lut2_f16[j] = __half_as_ushort(h);
        hdr->lut2_levels[j] = __half2float(h);
        if (hdr->lut2_levels[j] == 0.0f) hdr->lut2_zero_idx = j;
    }
    for (int j = 0; j < 3; ++j)
        hdr->lut2_thresholds[j] = __fmul_rn(__fadd_rn(hdr->lut2_levels[j], hdr->lut2_levels[j + 1]), 0.5f);
    hdr->lut2_thresholds[3] = __int_as_float(0x7f800000);
    for (int q = 0; q < 4; ++q) { hdr->lut_prmt[q] = 0u; hdr->lut2_prmt[q] = 0u; }
    for (int j = 0; j < 8; ++j) {
        hdr->lut_prmt[j >> 2] |= (hdr->lut_f16[j] & 0xFFu) << (8 * (j & 3));
        hdr->lut_prmt[2 + (j >> 2)] |= ((hdr->lut_f16[j] >> 8) & 0xFFu) << (8 * (j & 3));
    }
    for (int j = 0; j < 4; ++j) {
        hdr->lut2_prmt[0] |= (hdr->lut2_f16[j] & 0xFFu) << (8 * j);
        hdr->lut2_prmt[2] |= ((hdr->lut2_f16[j] >> 8) & 0xFFu) << (8 * j);
    }
}

cudaError_t launch_pack_header(PackedHeader *hdr, const uint16_t *codebook_f16_host, cudaStream_t stream)
{
    Codebook8 cb;
    for (int j = 0; j < 8; ++j) cb.h[j] = codebook_f16_host[j];
    pack_header_kernel<<<1, 256, 0, stream>>>(hdr, cb);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ absmax

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t min_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// Largest magnitude of W: one streaming read, four 16-byte loads in flight per thread.  grid.y walks rows, grid.x the
// 16-byte pieces of a row; a matrix without gaps between its rows is one long row.  HBM-bound: 17408 x 5120 bf16
// (178 MB) in 29 us, 6.1 TB/s.
template <bool FP32IN>
__global__ void __launch_bounds__(256) absmax_kernel(const uint4 *__restrict__ W, int64_t rows, int64_t len, int64_t ld, PackedHeader *hdr)
{
    uint32_t m[4] = {0u, 0u, 0u, 0u};                       // fp32 bits, or two bf16 magnitudes; a NaN is passed over
    auto take = [&](uint32_t &acc, const uint4 &v) {
        if (FP32IN) {
            const float a = fmaxf(fabsf(__uint_as_float(v.x)), fabsf(__uint_as_float(v.y)));
            const float b = fmaxf(fabsf(__uint_as_float(v.z)), fabsf(__uint_as_float(v.w)));
            acc = __float_as_uint(fmaxf(__uint_as_float(acc), fmaxf(a, b)));
        } else {
            acc = max_bf16x2(max_bf16x2(acc, max_bf16x2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu)),
                             max_bf16x2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu));
        }
    };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const uint4 *p = W + r * ld;
        int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i + 3 * stride < len; i += 4 * stride) {
            const uint4 v0 = __ldg(p + i), v1 = __ldg(p + i + stride), v2 = __ldg(p + i + 2 * stride), v3 = __ldg(p + i + 3 * stride);
            take(m[0], v0);
            take(m[1], v1);
            take(m[2], v2);
            take(m[3], v3);
        }
        for (; i < len; i += stride) take(m[0], __ldg(p + i));
    }
    uint32_t a;                                             // magnitudes order like unsigned integers
    if (FP32IN) {
        a = max(max(m[0], m[1]), max(m[2], m[3]));
    } else {
        const uint32_t q = max_bf16x2(max_bf16x2(m[0], m[1]), max_bf16x2(m[2], m[3]));
        a = max(q >> 16, q & 0xFFFFu) << 16;
    }
    a = __reduce_max_sync(0xffffffffu, a);
    __shared__ uint32_t red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) a = max(a, red[i]);
        atomicMax(&hdr->amax_bits, a);
    }
}

cudaError_t launch_absmax(const void *W, int w_dtype, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr,
                          cudaStream_t stream)
{
    const int64_t per16 = (w_dtype == DQ_DT_FP32) ? 4 : 8;
    int64_t rows = N, len = K / per16;
    if (ldw == K) { len *= rows; rows = 1; }
    const int64_t want = (len + 1023) / 1024, slots = 148 * 8;
    const unsigned gx = (unsigned)(want < slots ? want : slots);
    int64_t gy = slots / gx;
    if (gy > rows) gy = rows;
    const dim3 grid(gx, (unsigned)(gy < 1 ? 1 : gy));
    const uint4 *p = reinterpret_cast<const uint4 *>(W);
    if (w_dtype == DQ_DT_FP32) absmax_kernel<true><<<grid, 256, 0, stream>>>(p, rows, len, ldw / per16, hdr);
    else absmax_kernel<false><<<grid, 256, 0, stream>>>(p, rows, len, ldw / per16, hdr);
    return cudaGetLastError();
}

// -------------------------------------------------------------------- pack

// tensor scale from the largest magnitude (App. A.3): s = max|W| / (6 * 448), 1 for an all-zero tensor
__device__ __forceinline__ float tensor_scale(const PackedHeader *hdr)
{
    const float amax = __uint_as_float(hdr->amax_bits);
    return (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, 2688.0f);
}

// four floats -> two bytes of E2M1 codes (element 0 in the low nibble of byte 0), at the low end
__device__ __forceinline__ uint32_t f32x4_to_e2m1x4(const float (&f)[4])
{
    uint32_t r;
    asm("{\n\t.reg .b8 b0, b1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
        "mov.b32 %0, {b0, b1, b0, b1};\n\t}"
        : "=r"(r) : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]));
    return r;
}
// Transpose of 16-bit pieces between the four threads of a quad.  Thread t comes with v[j] = its pieces of blocks 2j (low
// half) and 2j + 1 (high half) and leaves with the sixteen bytes of blocks 2t and 2t + 1, pieces in thread order.
__device__ __forceinline__ uint4 quad_transpose(const uint32_t (&v)[4], int t)
{
    const bool hi2 = (t & 2) != 0, hi1 = (t & 1) != 0;
    const uint32_t a0 = hi2 ? v[2] : v[0], a1 = hi2 ? v[3] : v[1];
    const uint32_t b0 = __shfl_xor_sync(0xffffffffu, hi2 ? v[0] : v[2], 2), b1 = __shfl_xor_sync(0xffffffffu, hi2 ? v[1] : v[3], 2);
    const uint32_t k0 = hi1 ? a1 : a0, k1 = hi1 ? b1 : b0;              // from thread t and from thread t ^ 2
    const uint32_t g0 = __shfl_xor_sync(0xffffffffu, hi1 ? a0 : a1, 1), g1 = __shfl_xor_sync(0xffffffffu, hi1 ? b0 : b1, 1);
    const uint32_t p0 = hi1 ? g0 : k0, p1 = hi1 ? k0 : g0;              // from threads (t & 2), (t & 2) + 1
    const uint32_t q0 = hi1 ? g1 : k1, q1 = hi1 ? k1 : g1;              // from the other two
    const uint32_t u0 = hi2 ? q0 : p0, u1 = hi2 ? q1 : p1, u2 = hi2 ? p0 : q0, u3 = hi2 ? p1 : q1;
    return make_uint4(__byte_perm(u0, u1, 0x5410), __byte_perm(u2, u3, 0x5410), __byte_perm(u0, u1, 0x7632),
                      __byte_perm(u2, u3, 0x7632));
}

// Number of thresholds below y (the index of the nearest level, a value on a threshold taking the lower level).  The line is cut into
// kBins bins, the outermost open-ended, none of which holds more than one threshold (pack_bins_fit); a bin's entry, found through
// y's place on the line, says how many thresholds lie below the bin and where its own is, and one multiply-add that saturates at 0 and
// 1 compares with that: y * 2^60 - T * 2^60 is rounded once, so it is positive exactly where y > T, and then at least 1.  A NaN
// counts none: the saturated place of a NaN is 0, and so is the comparison.  Entries are 8 bytes, one copy per lane: no bank conflicts.
// Nearly all of it is multiply-adds, whose pipe has room beside the logic, shifts and converts of the rest.
constexpr int kBins = 64;
constexpr float kBinSpan = 32.0f;                          // places from -16 to 16
constexpr float kCmpScale = 1152921504606846976.0f;        // 2^60; thresholds are multiples of 2^-25 and at most 65504
// By how much a bin may reach beyond its edges: the place is rounded to 1/256 of a bin, so it begins up to 1/512 of one early (9.92e-4), and
// places and edges are rounded in fp32 (about 2^-24 of the span); a quarter more
constexpr float kBinReach = kBinSpan / (512.0f * (kBins - 1)), kBinSlack = 1.25f * kBinReach;
static_assert(kBinSlack > kBinReach + kBinSpan / 4194304.0f && kBinSlack < kBinSpan / (4.0f * (kBins - 1)), "room for the rounding, well inside a bin");
__host__ __device__ inline float bin_edge(int b) { return ((float)b / (float)(kBins - 1) - 0.5f) * kBinSpan; }
// thresholds (ascending) below bin b, and the one inside it or +inf; false where it holds more
__host__ __device__ inline bool bin_entry(const float *T, int n, int b, int &below, float &own)
{
    below = 0;
    own = INFINITY;
    int inside = 0;
    for (int l = 0; l < n; ++l) {
        if (b > 0 && T[l] < bin_edge(b) - kBinSlack) ++below;
        else if (b == kBins - 1 || T[l] <= bin_edge(b + 1) + kBinSlack) { if (inside++ == 0) own = T[l]; }
    }
    return inside <= 1;
}
__device__ __forceinline__ float ffma_sat(float a, float b, float c)
{
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// appends the level of y, or of -y for per_bin = -1 / kBinSpan, to a number in base 16
__device__ __forceinline__ float push_level(float acc, float y, float per_bin, const float2 *bins, uint32_t lane8)
{
    const float place = ffma_sat(y, per_bin, 0.5f);
    const uint32_t at = (__float_as_uint(__fmaf_rn(place, (float)(256 * (kBins - 1)), 8388608.0f)) & (uint32_t)(256 * (kBins - 1))) | lane8;
    const float2 e = *reinterpret_cast<const float2 *>(reinterpret_cast<const uint8_t *>(bins) + at);
    return __fadd_rn(__fmaf_rn(acc, 16.0f, e.x), ffma_sat(y, per_bin * (kBinSpan * kCmpScale), e.y));
}
// The same by comparing with every threshold, for codebooks with two of them in a bin: T - y is negative exactly where y > T.
template <int N>
__device__ __forceinline__ float push_level_all(float acc, float y, float sign, const float (&T)[N])
{
    uint32_t n = 0;
#pragma unroll
    for (int l = 0; l < N; ++l) n += __float_as_uint(__fmaf_rn(y, -sign, T[l])) >> 31;
    return __fmaf_rn(acc, 16.0f, (float)n);
}

// Transpose of 32-bit words between the four threads of a quad: thread t comes with v[q] and leaves with word t of threads 0..3
__device__ __forceinline__ void quad_transpose_words(uint32_t (&v)[4], int t)
{
    const bool hi2 = (t & 2) != 0, hi1 = (t & 1) != 0;
    const uint32_t a0 = hi2 ? v[2] : v[0], a1 = hi2 ? v[3] : v[1];
    const uint32_t b0 = __shfl_xor_sync(0xffffffffu, hi2 ? v[0] : v[2], 2), b1 = __shfl_xor_sync(0xffffffffu, hi2 ? v[1] : v[3], 2);
    const uint32_t k0 = hi1 ? a1 : a0, k1 = hi1 ? b1 : b0;              // of threads t and t ^ 2
    const uint32_t g0 = __shfl_xor_sync(0xffffffffu, hi1 ? a0 : a1, 1), g1 = __shfl_xor_sync(0xffffffffu, hi1 ? b0 : b1, 1);
    const uint32_t p0 = hi1 ? g0 : k0, p1 = hi1 ? k0 : g0, q0 = hi1 ? g1 : k1, q1 = hi1 ? k1 : g1;
    v[0] = hi2 ? q0 : p0;
    v[1] = hi2 ? q1 : p1;
    v[2] = hi2 ? p0 : q0;
    v[3] = hi2 ? p1 : q1;
}

// CTAs per SM: what the registers of bf16, and the copy buffers of fp32, leave room for
constexpr int pack_ctas(bool fp32) { return fp32 ? 2 : 4; }
__host__ __device__ constexpr int pack_stage_bytes(bool fp32) { return 8 * 128 * (fp32 ? 4 : 2); }      // one word group of a warp: 8 rows x 128 weights
__device__ __forceinline__ void copy16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Round-to-nearest packing of the master weights (App. A.3): NVFP4 (NV) and / or one LUT format (BITS = 3 or 2) in one
// read of W.  A warp takes atoms of 8 rows x 512 weights, 128 weights (eight blocks) of every row at a time; lane (g, t) takes blocks
// 2t and 2t + 1 of row g whole: extremes, scale and reciprocal (a table of the 127 scales per CTA), which serve both encodings, are its
// own, and its E2M1 codes are 16 bytes of the output as they are.  The index words of the LUT layout hold quarters of eight blocks:
// one transpose inside the quad brings them about.  Index words and scales leave as whole 512- and 256-byte rows of the atom.
// The next word group is on its way to shared memory meanwhile (loaded straight into registers, a lane's 64 or 128 contiguous bytes touch
// 16 or 32 lines per instruction); its 16-byte pieces are placed so that the lanes' reads hit different banks.
// Bound by instruction issue.  17408 x 5120 bf16 to NVFP4 and LUT3: 73 us, 3.4 TB/s; with a quarter of every block per lane, its extremes reduced
// and its scale made in all four lanes of the quad, and seven subtractions and seven logic operations and shifts per weight, 116 us.
template <bool FP32IN, bool NV, int BITS, bool BINNED>
__global__ void __launch_bounds__(256, pack_ctas(FP32IN)) pack_kernel(const void *__restrict__ W, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr,
                                                                      uint8_t *__restrict__ codes, uint8_t *__restrict__ sf, uint8_t *__restrict__ lut)
{
    constexpr bool LUT = BITS > 0;
    constexpr int B = LUT ? BITS : 2;                      // dummy where there is no LUT format
    constexpr int NT = (1 << B) - 1;
    __shared__ float2 bins[LUT && BINNED ? kBins * 32 : 1];
    __shared__ float rtab[128];                            // 1 / (s * d) by the byte of d; 0 for a scale that rounded to zero
    extern __shared__ __align__(128) uint8_t stages[];     // [warp][2]
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const float s = tensor_scale(hdr);
    const float rc6 = __frcp_rn(__fmul_rn(6.0f, s));
    if (blockIdx.x == 0 && threadIdx.x == 0) { hdr->s = s; hdr->rc6 = rc6; }
    if (threadIdx.x < 128) rtab[threadIdx.x] = (threadIdx.x == 0) ? 0.0f : __frcp_rn(__fmul_rn(s, e4m3_to_f32(threadIdx.x)));
    float T[NT];
    if (LUT) {
#pragma unroll
        for (int l = 0; l < NT; ++l) T[l] = (BITS == 3) ? hdr->lut_thresholds[l] : hdr->lut2_thresholds[l & 3];
    }
    if (LUT && BINNED) {
        for (int b = threadIdx.x >> 5; b < kBins; b += 8) {
            int below;
            float own;
            bin_entry(T, NT, b, below, own);
            bins[b * 32 + lane] = make_float2((float)below, __fmul_rn(own, -kCmpScale));
        }
    }
    __syncthreads();
    const uint32_t atoms_k = (uint32_t)(2 * lut_slices(K));               // atoms along a row, a short last slice padded
    const uint32_t katoms = NV && !LUT ? (uint32_t)((K + 511) / 512) : atoms_k;
    // tasks of this warp: atoms first, first + step, .. in row-major order, as (rows of eight, atom of the row) without a division each
    const uint32_t step = gridDim.x * 8u, step_row = step / katoms, step_atom = step - step_row * katoms;
    const uint32_t first = blockIdx.x * 8u + (threadIdx.x >> 5), rowgrps = (uint32_t)(N / 8);
    struct Task { uint32_t row, atom; int groups; };                      // groups: word groups inside K, 0 for padding
    const int kgroups = (int)(K / 128);
    auto count = [&](Task &q) { q.groups = max(0, min(4, kgroups - 4 * (int)q.atom)); };
    auto next = [&](Task &q) {
        q.row += step_row;
        q.atom += step_atom;
        if (q.atom >= katoms) { q.atom -= katoms; ++q.row; }
        count(q);
    };
    Task task = {first / katoms, first % katoms, 0};
    count(task);

    // copies: the word groups of this warp's tasks in turn, one ahead of the one in work.  Piece c of a row (16 bytes) goes to place
    // c ^ swizzle: the four lanes of a quad and the rows g, g + 1 that read together then find theirs in eight different places of 128 bytes.
    constexpr int kElem = FP32IN ? 4 : 2, kRow = 128 * kElem / 16, kPieces = kElem;      // pieces of a row, of a block
    constexpr uint32_t kStage = (uint32_t)pack_stage_bytes(FP32IN);
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(stages) + (threadIdx.x >> 5) * 2u * kStage;
    auto swizzle = [](int row, int c) { return FP32IN ? (c >> 3) | ((row & 1) << 2) : (c >> 3) | ((row & 1) << 1); };
    // an instruction copies 32 pieces: two rows of bf16 or one of fp32
    constexpr int kRowsPer = 32 / kRow;
    const int prow = lane / kRow, pc = lane % kRow;
    const int64_t row_bytes = ldw * kElem, lane_src = prow * row_bytes + pc * 16;
    Task ptask = task;
    while (ptask.row < rowgrps && ptask.groups == 0) next(ptask);
    auto source = [&]() { return reinterpret_cast<const uint8_t *>(W) + (int64_t)ptask.row * (8 * row_bytes) + (int64_t)ptask.atom * (512 * kElem) + lane_src; };
    const uint8_t *psrc = source();
    uint32_t pstage = 0;
    auto copy_next = [&]() {
        if (ptask.row < rowgrps) {
            const uint8_t *q = psrc;
#pragma unroll
            for (int i = 0; i < kRow / 4; ++i, q += kRowsPer * row_bytes) {
                const int row = i * kRowsPer + (kRowsPer > 1 ? prow : 0);
                copy16(ring + pstage + (uint32_t)(row * kRow + (pc ^ swizzle(row, pc))) * 16u, q);
            }
            psrc += 128 * kElem;
            if (--ptask.groups == 0) {
                do next(ptask); while (ptask.row < rowgrps && ptask.groups == 0);
                psrc = source();
            }
        }
        pstage ^= kStage;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy_next();
    uint32_t cstage = 0;
    for (; task.row < rowgrps; next(task)) {
        const int64_t rowgrp = task.row;
        const uint32_t atom = task.atom;
        const int64_t r = rowgrp * 8 + g;
        const int nwi = task.groups;
        uint4 *out_codes = nullptr;
        uint32_t *out_sf = nullptr;
        if (NV) {
            out_codes = reinterpret_cast<uint4 *>(codes + r * (K / 2) + (int64_t)atom * 256 + t * 16);
            out_sf = reinterpret_cast<uint32_t *>(sf + sf_swizzled_offset(r, (int64_t)atom * 32 + 4 * (t >> 1), K));
        }
        uint32_t words[4][B];
        uint2 my_scales = make_uint2(0u, 0u);              // LUT scale bytes of word group t
#pragma unroll
        for (int wi = 0; wi < 4; ++wi) {
#pragma unroll
            for (int p = 0; p < B; ++p) words[wi][p] = 0u;
            if (wi >= nwi) continue;                       // whole warps
            __syncwarp();                                  // everybody has read the stage that is filled next
            copy_next();
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
            uint4 raw[2][kPieces];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < kPieces; ++i) {
                    const int c = (2 * t + j) * kPieces + i;
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(raw[j][i].x), "=r"(raw[j][i].y), "=r"(raw[j][i].z), "=r"(raw[j][i].w)
                                 : "r"(ring + cstage + (uint32_t)(g * kRow + (c ^ swizzle(g, c))) * 16u) : "memory");
                }
            cstage ^= kStage;
            float rs[2], sign[2];
            uint32_t sc = 0;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float mx, mn;                              // largest value and largest of the negated values
                if (FP32IN) {
#pragma unroll
                    for (int i = 0; i < kPieces; ++i) {
                        const float x0 = __uint_as_float(raw[j][i].x), x1 = __uint_as_float(raw[j][i].y), x2 = __uint_as_float(raw[j][i].z), x3 = __uint_as_float(raw[j][i].w);
                        const float px = fmaxf(fmaxf(x0, x1), fmaxf(x2, x3)), pn = fmaxf(fmaxf(-x0, -x1), fmaxf(-x2, -x3));
                        mx = i ? fmaxf(mx, px) : px;       // NaN only where all of the block is
                        mn = i ? fmaxf(mn, pn) : pn;
                    }
                } else {
                    const uint4 u = raw[j][0], v = raw[j][1];
                    const uint32_t hi = max_bf16x2(max_bf16x2(max_bf16x2(u.x, u.y), max_bf16x2(u.z, u.w)), max_bf16x2(max_bf16x2(v.x, v.y), max_bf16x2(v.z, v.w)));
                    const uint32_t lo = min_bf16x2(min_bf16x2(min_bf16x2(u.x, u.y), min_bf16x2(u.z, u.w)), min_bf16x2(min_bf16x2(v.x, v.y), min_bf16x2(v.z, v.w)));
                    mx = fmaxf(__uint_as_float(hi << 16), __uint_as_float(hi & 0xFFFF0000u));
                    mn = -fminf(__uint_as_float(lo << 16), __uint_as_float(lo & 0xFFFF0000u));
                }
                // the LUT scale takes the sign of the block's extreme; where both signs reach the magnitude, plus.  It goes with the reciprocal, but
                // where there are E2M1 codes too, with the levels' constants: codes have the plain reciprocal (taken back from the codes, it would
                // leave one on those of a NaN, which come without)
                const uint32_t d8 = f32_to_e4m3(__fmul_rn(fmaxf(mx, mn), rc6)) & 0x7Fu;
                const bool neg = LUT && mn > mx;
                const float rr = rtab[d8];
                rs[j] = neg && !NV ? -rr : rr;
                sign[j] = (BINNED ? 1.0f / kBinSpan : 1.0f) * (neg && NV ? -1.0f : 1.0f);
                sc |= (neg && d8 ? d8 | 0x80u : d8) << (8 * j);
            }
            const bool zeros = NV && __any_sync(0xffffffffu, !((sc & 0x7Fu) && (sc & 0x7F00u)));
            const uint32_t s4 = __shfl_xor_sync(0xffffffffu, sc, 1);
            const uint32_t sc4 = (t & 1) ? (sc << 16) | s4 : (s4 << 16) | sc;     // blocks 4 (t / 2) .. + 3
            if (LUT) {
                const uint32_t so = __shfl_xor_sync(0xffffffffu, sc4, 2);
                if (t == wi) my_scales = (t & 2) ? make_uint2(so, sc4) : make_uint2(sc4, so);
            }
            uint32_t cw[4], sel[4];                        // E2M1 codes; levels, quarter q of both blocks
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float acc[2];
                uint32_t c2[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float y[4];
                    if (FP32IN) {
                        const uint4 v = raw[j][FP32IN ? q : 0];
                        y[0] = __uint_as_float(v.x); y[1] = __uint_as_float(v.y); y[2] = __uint_as_float(v.z); y[3] = __uint_as_float(v.w);
                    } else {
                        const uint4 v = raw[j][q >> 1];
                        const uint32_t w0 = (q & 1) ? v.z : v.x, w1 = (q & 1) ? v.w : v.y;
                        y[0] = __uint_as_float(w0 << 16); y[1] = __uint_as_float(w0 & 0xFFFF0000u);
                        y[2] = __uint_as_float(w1 << 16); y[3] = __uint_as_float(w1 & 0xFFFF0000u);
                    }
                    acc[j] = 0.0f;
#pragma unroll
                    for (int n4 = 3; n4 >= 0; --n4) {
                        y[n4] = __fmul_rn(y[n4], rs[j]);
                        if (LUT) acc[j] = BINNED ? push_level(acc[j], y[n4], sign[j], bins, (uint32_t)lane * 8u) : push_level_all(acc[j], y[n4], sign[j], T);
                    }
                    if (NV) c2[j] = f32x4_to_e2m1x4(y);
                }
                if (NV) {
                    if (q & 1) { cw[q >> 1] = __byte_perm(cw[q >> 1], c2[0], 0x5410); cw[2 + (q >> 1)] = __byte_perm(cw[2 + (q >> 1)], c2[1], 0x5410); }
                    else { cw[q >> 1] = c2[0]; cw[2 + (q >> 1)] = c2[1]; }
                }
                // the sixteen bits of each half sit at the low end of the significand
                if (LUT) sel[q] = __byte_perm(__float_as_uint(__fadd_rn(acc[0], 8388608.0f)), __float_as_uint(__fadd_rn(acc[1], 8388608.0f)), 0x5410);
            }
            if (LUT) {
                quad_transpose_words(sel, t);
                if (BITS == 3) {
#pragma unroll
                    for (int p = 0; p < B; ++p) words[wi][p] = sel[p] | (((sel[3] >> p) & 0x11111111u) << 3);
                } else {
#pragma unroll
                    for (int p = 0; p < 2; ++p) words[wi][p] = sel[2 * p] | (sel[2 * p + 1] << 2);
                }
            }
            if (NV) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    // under a zero scale: zeros without a sign
                    if (zeros && rs[j] == 0.0f) cw[2 * j] = cw[2 * j + 1] = 0u;
                }
                out_codes[wi * 4] = make_uint4(cw[0], cw[1], cw[2], cw[3]);
                if ((t & 1) == 0) out_sf[wi * 256] = sc4 & 0x7F7F7F7Fu;           // two k atoms of 512 bytes per word group
            }
        }
        if (LUT) {
            uint8_t *out = lut + lut_atom_offset(rowgrp * 8, atom, K, B);
#pragma unroll
            for (int p = 0; p < B; ++p)
                *reinterpret_cast<uint4 *>(out + p * 512 + lane * 16) = make_uint4(words[0][p], words[1][p], words[2][p], words[3][p]);
            *reinterpret_cast<uint2 *>(out + lut_plane_bytes(B) + lane * 8) = my_scales;
        }
    }
}

// Has no bin of the LUT3 codebook more than one threshold?  (Thresholds 0.52 apart never share one; the default codebook's are 1.2 apart.)
static bool pack_bins_fit(const uint16_t *codebook_f16)
{
    float T[7];
    for (int l = 0; l < 7; ++l) {
        const float a = __half2float(__ushort_as_half(codebook_f16[l])), b = __half2float(__ushort_as_half(codebook_f16[l + 1]));
        T[l] = (a + b) * 0.5f;
    }
    int below;
    float own;
    for (int b = 0; b < kBins; ++b)
        if (!bin_entry(T, 7, b, below, own)) return false;
    return true;
}

template <bool FP32IN, bool NV, int BITS, bool BINNED>
static cudaError_t launch_pack_one(const void *W, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr, uint8_t *codes, uint8_t *sf, uint8_t *lut,
                                   cudaStream_t stream)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    const DeviceInfo *di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    auto kernel = pack_kernel<FP32IN, NV, BITS, BINNED>;
    const int smem = 8 * 2 * pack_stage_bytes(FP32IN);
    if (!attr_set[di->device].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set[di->device].store(true, std::memory_order_release);
    }
    const int64_t atoms_k = BITS ? 2 * lut_slices(K) : (K + 511) / 512, need = (N / 8 * atoms_k + 7) / 8;
    const int64_t slots = (int64_t)di->sms * pack_ctas(FP32IN);                  // all resident: a CTA makes its tables once
    kernel<<<(unsigned)(need < slots ? need : slots), 256, smem, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
    return cudaGetLastError();
}
template <bool FP32IN>
static cudaError_t launch_pack_typed(const void *W, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr, uint8_t *codes, uint8_t *sf,
                                     uint8_t *lut, int bits, bool binned, cudaStream_t stream)
{
    if (codes && bits == 3 && binned) return launch_pack_one<FP32IN, true, 3, true>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    if (codes && bits == 3) return launch_pack_one<FP32IN, true, 3, false>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    if (codes && bits == 2) return launch_pack_one<FP32IN, true, 2, true>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    if (codes) return launch_pack_one<FP32IN, true, 0, false>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    if (bits == 3 && binned) return launch_pack_one<FP32IN, false, 3, true>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    if (bits == 3) return launch_pack_one<FP32IN, false, 3, false>(W, N, K, ldw, hdr, codes, sf, lut, stream);
    return launch_pack_one<FP32IN, false, 2, true>(W, N, K, ldw, hdr, codes, sf, lut, stream);
}

// codes / sf: NVFP4 output or nullptr; lut with bits = 3 or 2: LUT output, bits = 0: none
cudaError_t launch_pack(const void *W, int w_dtype, int64_t N, int64_t K, int64_t ldw, const uint16_t *codebook_f16_host, PackedHeader *hdr,
                        uint8_t *codes, uint8_t *sf_swizzled, uint8_t *lut_dev, int bits, cudaStream_t stream)
{
    const bool binned = bits == 3 && pack_bins_fit(codebook_f16_host);
    if (w_dtype == DQ_DT_FP32) return launch_pack_typed<true>(W, N, K, ldw, hdr, codes, sf_swizzled, lut_dev, bits, binned, stream);
    return launch_pack_typed<false>(W, N, K, ldw, hdr, codes, sf_swizzled, lut_dev, bits, binned, stream);
}

// ---------------------------------------------------------------- autocast

// NVFP4 view of the LUT3 codes (Sec. 2.3): level -> nearest E2M1 value, element signs
// flipped under a negative block scale, block scale |d|, same tensor scale.
// A warp takes an atom (8 rows x 512 weights): 16-byte loads of index words, a byte permute looks up the E2M1 codes of four
// weights, and a transpose inside the quad leaves every lane 16 bytes of codes to store.  Signs and zero scales are masks made
// by the permute's sign replication: under a negative scale the looked-up table is exchanged for the one with the signs of
// non-zero codes flipped, under a zero scale the codes are cleared.
// byte permute with the selector as it is: the intrinsic clears the top bits of its nibbles first
__device__ __forceinline__ uint32_t prmt_raw(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t prmt_sign(uint32_t a, uint32_t sel) { return prmt_raw(a, a, sel); }      // nibbles 8-11: sign of byte 0-3
__device__ __forceinline__ void autocast_atom(const PackedHeader *hdr, const uint8_t *lut, int64_t rowgrp, uint32_t atom, int64_t K,
                                              uint8_t *codes, uint8_t *sf)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t r = rowgrp * 8 + g;
    const uint8_t *src = lut + lut_atom_offset(rowgrp * 8, atom, K, 3);
    uint4 w[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) w[p] = __ldg(reinterpret_cast<const uint4 *>(src + p * 512 + lane * 16));
    const uint2 s8 = __ldg(reinterpret_cast<const uint2 *>(src + lut_plane_bytes(3) + lane * 8));
    // E2M1 codes of the levels as bytes, and what a negative block scale flips: the sign bits of non-zero codes
    const uint32_t amap = hdr->autocast_map;
    uint32_t pos[2], flip[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t m = amap >> (16 * i);
        pos[i] = (m & 0xFu) | ((m & 0xF0u) << 4) | ((m & 0xF00u) << 8) | ((m & 0xF000u) << 12);
        flip[i] = ((pos[i] | (pos[i] >> 1) | (pos[i] >> 2)) & 0x01010101u) << 3;
    }
    const int nwi = min(4, (int)(K / 128) - 4 * (int)atom);
    uint4 *out = reinterpret_cast<uint4 *>(codes + r * (K / 2) + (int64_t)atom * 256 + t * 16);
    uint32_t *out_sf = reinterpret_cast<uint32_t *>(sf + sf_swizzled_offset(r, (int64_t)atom * 32 + 4 * (t & 1), K));
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
        if (wi >= nwi) break;                              // whole warps
        uint32_t wd[3], sel[4];
#pragma unroll
        for (int p = 0; p < 3; ++p) wd[p] = wi == 0 ? w[p].x : wi == 1 ? w[p].y : wi == 2 ? w[p].z : w[p].w;
        lut_selectors<3>(wd, sel);
        // the row's scales of this word group sit in lane wi of the quad
        const uint32_t sc[2] = {__shfl_sync(0xffffffffu, s8.x, (lane & ~3) | wi), __shfl_sync(0xffffffffu, s8.y, (lane & ~3) | wi)};
        uint32_t v[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            // top bit of every byte: the block's scale byte is not zero
            const uint32_t live = (((sc[i] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | sc[i]) & 0x80808080u;
#pragma unroll
            for (int k = 0; k < 2; ++k) {                  // blocks 4 i + 2 k and the next
                const int a = 2 * i + k;
                const uint32_t m0 = prmt_sign(sc[i], 0x8888u + 0x1111u * (2 * k)), m1 = prmt_sign(sc[i], 0x8888u + 0x1111u * (2 * k + 1));
                const uint32_t x0 = prmt_raw(pos[0] ^ (m0 & flip[0]), pos[1] ^ (m0 & flip[1]), sel[a]);
                const uint32_t x1 = prmt_raw(pos[0] ^ (m1 & flip[0]), pos[1] ^ (m1 & flip[1]), sel[a] >> 16);
                // codes 0, 2 of both blocks and codes 1, 3 of both blocks
                const uint32_t e = __byte_perm(x0, x1, 0x6420), o = __byte_perm(x0, x1, 0x7531);
                v[a] = (e | (o << 4)) & prmt_sign(live, k ? 0xBBAAu : 0x9988u);
            }
        }
        out[wi * 4] = quad_transpose(v, t);
        if (t < 2) out_sf[wi * 256] = (t ? sc[1] : sc[0]) & 0x7F7F7F7Fu;      // two k atoms of 512 bytes per word group
    }
}

__global__ void __launch_bounds__(128) autocast_kernel(const PackedHeader *__restrict__ hdr, const uint8_t *__restrict__ lut, int64_t N,
                                                       int64_t K, uint8_t *__restrict__ codes, uint8_t *__restrict__ sf)
{
    const uint32_t natoms = (uint32_t)((K + 511) / 512);
    const int64_t task = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int64_t rowgrp = task / natoms;
    if (rowgrp < N / 8) autocast_atom(hdr, lut, rowgrp, (uint32_t)(task - rowgrp * natoms), K, codes, sf);
}

cudaError_t launch_autocast(const PackedHeader *hdr, const uint8_t *lut_dev, int64_t N,
                            int64_t K, uint8_t *codes, uint8_t *sf_swizzled, cudaStream_t stream)
{
    const int64_t warps = N / 8 * ((K + 511) / 512);
    autocast_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, stream>>>(hdr, lut_dev, N, K, codes, sf_swizzled);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ export

// Codes are row-major on both sides: 16-byte copies, four in flight per thread.  Scales: a warp takes 32 rows of each quarter
// of a 128-row band and four 64-wide k atoms, reads the atoms' 16-byte groups (scales of rows r, r+32, r+64, r+96)
// and writes 16 scales of each of its rows at once.
__global__ void __launch_bounds__(256) export_nvfp4_kernel(const PackedHeader *__restrict__ hdr, const uint4 *__restrict__ codes,
                                                           const uint8_t *__restrict__ sf, int64_t N, int64_t K, uint4 *__restrict__ codes_out,
                                                           uint8_t *__restrict__ scales_out, float *s_out, int code_blocks)
{
    if (blockIdx.x == 0 && threadIdx.x == 0 && s_out) *s_out = hdr->s;
    if ((int)blockIdx.x < code_blocks) {
        const int64_t n16 = N * (K / 2) / 16, base = (int64_t)blockIdx.x * 1024 + threadIdx.x;
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) if (base + u * 256 < n16) v[u] = __ldg(codes + base + u * 256);
#pragma unroll
        for (int u = 0; u < 4; ++u) if (base + u * 256 < n16) codes_out[base + u * 256] = v[u];
        return;
    }
    const int64_t katoms = K / 64, groups = (katoms + 3) / 4;
    const int64_t task = ((int64_t)blockIdx.x - code_blocks) * 8 + (threadIdx.x >> 5);
    const int64_t band = task / groups, kg = task - band * groups;
    if (band * 128 >= N) return;
    const int lane = threadIdx.x & 31;
    const int nk = (int)min((int64_t)4, katoms - kg * 4);           // K % 128 == 0: two or four
    uint4 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
        v[c] = (c < nk) ? __ldg(reinterpret_cast<const uint4 *>(sf + (band * katoms + kg * 4 + c) * 512 + lane * 16)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t r = band * 128 + q * 32 + lane;
        if (r >= N) continue;
        uint32_t o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c] = q == 0 ? v[c].x : q == 1 ? v[c].y : q == 2 ? v[c].z : v[c].w;
        uint8_t *dst = scales_out + r * (K / 16) + kg * 16;          // 8-byte aligned (K / 16 is a multiple of 8)
        *reinterpret_cast<uint2 *>(dst) = make_uint2(o[0], o[1]);
        if (nk == 4) *reinterpret_cast<uint2 *>(dst + 8) = make_uint2(o[2], o[3]);
    }
}

// codes_out and scales_out need 8-byte alignment only: the general form for pointers that are not 16-byte aligned
__global__ void export_nvfp4_narrow_kernel(const PackedHeader *hdr, const uint8_t *codes, const uint8_t *sf, int64_t N,
                                           int64_t K, uint8_t *codes_out, uint8_t *scales_out, float *s_out)
{
    const int64_t nb = K / 16;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && s_out) *s_out = hdr->s;
    if (i >= N * nb) return;
    const int64_t r = i / nb, b = i % nb;
    *reinterpret_cast<uint2 *>(codes_out + r * (K / 2) + b * 8) =
        *reinterpret_cast<const uint2 *>(codes + r * (K / 2) + b * 8);
    scales_out[r * nb + b] = sf[sf_swizzled_offset(r, b, K)];
}

cudaError_t launch_export_nvfp4(const PackedHeader *hdr, const uint8_t *codes, const uint8_t *sf_swizzled, int64_t N,
                                int64_t K, uint8_t *codes_out, uint8_t *scales_out, float *s_out,
                                cudaStream_t stream)
{
    if (reinterpret_cast<uintptr_t>(codes_out) % 16 || reinterpret_cast<uintptr_t>(scales_out) % 8) {
        const int64_t total = N * (K / 16);
        export_nvfp4_narrow_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(hdr, codes, sf_swizzled, N, K, codes_out,
                                                                                        scales_out, s_out);
        return cudaGetLastError();
    }
    const int64_t code_blocks = (N * (K / 2) / 16 + 1023) / 1024;
    const int64_t warps = (N + 127) / 128 * ((K / 64 + 3) / 4);
    export_nvfp4_kernel<<<(unsigned)(code_blocks + (warps + 7) / 8), 256, 0, stream>>>(
        hdr, reinterpret_cast<const uint4 *>(codes), sf_swizzled, N, K, reinterpret_cast<uint4 *>(codes_out), scales_out, s_out,
        (int)code_blocks);
    return cudaGetLastError();
}

// LSB-first bit-planes (App. C.2) from the device layout.  A warp takes an atom; lane (g, t) holds weights 4t .. 4t+3 of every
// block of row g, i.e. bits 4t .. 4t+3 of each half of a canonical word.  Per plane and word group it has eight such nibbles, a pair for each
// of four words: a multiplication brings the four bits of a half together (bit 4i times 2^(12 - 3j) lands on 12 + i where j = i,
// and no two products meet anywhere else), and the pairs go into one word, so that one transpose inside the quad hands lane t
// all nibbles of its word group; spread by two byte transposes they are the four words.  Bound by instruction issue
// beside HBM: 17408 x 5120 LUT3 21 us a call (one word per nibble pair exchanged, 24.9).
template <int BITS>
__global__ void __launch_bounds__(128) export_lut_kernel(const PackedHeader *__restrict__ hdr, const uint8_t *__restrict__ lut, int64_t N,
                                                         int64_t K, uint32_t *__restrict__ planes_out, uint8_t *__restrict__ scales_out, float *s_out)
{
    if (blockIdx.x == 0 && threadIdx.x == 0 && s_out) *s_out = hdr->s;
    const uint32_t natoms = (uint32_t)((K + 511) / 512);
    const uint32_t task = blockIdx.x * 4u + (threadIdx.x >> 5), rowgrp = task / natoms;
    if (rowgrp >= N / 8) return;
    const uint32_t atom = task - rowgrp * natoms;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t r = (int64_t)rowgrp * 8 + g;
    const uint8_t *src = lut + lut_atom_offset((int64_t)rowgrp * 8, atom, K, BITS);
    uint4 w[BITS];
#pragma unroll
    for (int p = 0; p < BITS; ++p) w[p] = __ldg(reinterpret_cast<const uint4 *>(src + p * 512 + lane * 16));
    const uint2 s8 = __ldg(reinterpret_cast<const uint2 *>(src + lut_plane_bytes(BITS) + lane * 8));
    const bool mine = (int)(K / 128) - 4 * (int)atom > t;   // word group t of the atom lies inside the row
    uint32_t v[BITS][4];                                    // [plane][word group]
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
        uint32_t wd[BITS], sel[4];
#pragma unroll
        for (int p = 0; p < BITS; ++p) wd[p] = wi == 0 ? w[p].x : wi == 1 ? w[p].y : wi == 2 ? w[p].z : w[p].w;
        lut_selectors<BITS>(wd, sel);
#pragma unroll
        for (int p = 0; p < BITS; ++p) {
            uint32_t m[4];                                  // nibbles of word a: top of bytes 1 (low half) and 3 (high half)
#pragma unroll
            for (int a = 0; a < 4; ++a) m[a] = ((sel[a] >> p) & 0x11111111u) * 0x1248u;
            const uint32_t lo = __byte_perm(m[0], m[1], 0x7531), hi = __byte_perm(m[2], m[3], 0x7531);
            v[p][wi] = ((lo >> 4) & 0x0F0F0F0Fu) | (hi & 0xF0F0F0F0u);     // bytes: words 0|2 low, 0|2 high, 1|3 low, 1|3 high
        }
    }
#pragma unroll
    for (int p = 0; p < BITS; ++p) {
        quad_transpose_words(v[p], t);                      // word group t: the four lanes' nibbles
        const uint32_t e0 = __byte_perm(v[p][0], v[p][1], 0x5140), e1 = __byte_perm(v[p][2], v[p][3], 0x5140);     // lanes 0, 1 (2, 3): low, low, high, high of words 0|2
        const uint32_t f0 = __byte_perm(v[p][0], v[p][1], 0x7362), f1 = __byte_perm(v[p][2], v[p][3], 0x7362);     // of words 1|3
        uint32_t o[4];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const uint32_t x = a ? f0 : e0, y = a ? f1 : e1;
            // bytes (lane 0, lane 1) of a half: low nibbles are word a's, high nibbles word a + 2's
            const uint32_t l01 = (x & 0x000F000Fu) | ((x >> 4) & 0x00F000F0u), h01 = ((x >> 4) & 0x000F000Fu) | ((x >> 8) & 0x00F000F0u);
            const uint32_t l23 = (y & 0x000F000Fu) | ((y >> 4) & 0x00F000F0u), h23 = ((y >> 4) & 0x000F000Fu) | ((y >> 8) & 0x00F000F0u);
            o[a] = l01 | (l23 << 8);
            o[a + 2] = h01 | (h23 << 8);
        }
        if (mine) {
            uint32_t *dst = planes_out + (r * BITS + p) * (K / 32) + (int64_t)atom * 16 + t * 4;
            if ((reinterpret_cast<uintptr_t>(planes_out) & 15) == 0) {
                *reinterpret_cast<uint4 *>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int a = 0; a < 4; ++a) dst[a] = o[a];
            }
        }
    }
    if (mine) {
        uint8_t *dst = scales_out + r * (K / 16) + (int64_t)atom * 32 + t * 8;
        if ((reinterpret_cast<uintptr_t>(scales_out) & 7) == 0) {
            *reinterpret_cast<uint2 *>(dst) = s8;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = (uint8_t)((i < 4 ? s8.x : s8.y) >> (8 * (i & 3)));
        }
    }
}

cudaError_t launch_export_lut(int bits, const PackedHeader *hdr, const uint8_t *lut_dev, int64_t N,
                              int64_t K, uint32_t *planes_out, uint8_t *scales_out, float *s_out,
                              cudaStream_t stream)
{
    const int64_t warps = N / 8 * ((K + 511) / 512);
    const unsigned blocks = (unsigned)((warps + 3) / 4);
    if (bits == 3) export_lut_kernel<3><<<blocks, 128, 0, stream>>>(hdr, lut_dev, N, K, planes_out, scales_out, s_out);
    else export_lut_kernel<2><<<blocks, 128, 0, stream>>>(hdr, lut_dev, N, K, planes_out, scales_out, s_out);
    return cudaGetLastError();
}

// Last launch of every pack / import: does nothing.  The decode kernel is launched so that its set-up may
// overlap the kernel before it in the stream; with this launch in between, that kernel is never one that
// writes the packed buffer.
__global__ void pack_done_kernel() {}
cudaError_t launch_pack_done(cudaStream_t stream)
{
    pack_done_kernel<<<1, 32, 0, stream>>>();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ import

// Canonical codes / scales (the layouts of the export) -> device layouts.  Inverse of the export kernels.
__global__ void import_nvfp4_kernel(const uint8_t *codes_in, const uint8_t *scales_in, int64_t N, int64_t K,
                                    uint8_t *codes, uint8_t *sf)
{
    const int64_t nb = K / 16;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * nb) return;
    const int64_t r = i / nb, b = i % nb;
    *reinterpret_cast<uint2 *>(codes + r * (K / 2) + b * 8) =
        *reinterpret_cast<const uint2 *>(codes_in + r * (K / 2) + b * 8);
    sf[sf_swizzled_offset(r, b, K)] = scales_in[r * nb + b];
}

// one thread per word group, as in the packer
template <int BITS>
__global__ void import_lut_kernel(const uint32_t *planes_in, const uint8_t *scales_in, int64_t N, int64_t K,
                                  uint8_t *lut)
{
    const int64_t nq = K / 128, nw = K / 32;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t quad = i >> 2;
    const int t = (int)(i & 3);
    if (quad >= N * nq) return;
    const int64_t r = quad / nq, q = quad % nq;
    uint32_t wd[BITS];
#pragma unroll
    for (int p = 0; p < BITS; ++p) wd[p] = 0u;
#pragma unroll
    for (int bb = 0; bb < 8; ++bb) {
        // weights 16 bb + 4 t .. + 3 of the 128: bits 16 (bb % 2) + 4 t .. of canonical word 4 q + bb / 2
        uint32_t c[BITS];
#pragma unroll
        for (int p = 0; p < BITS; ++p) c[p] = planes_in[(r * BITS + p) * nw + q * 4 + (bb >> 1)] >> (16 * (bb & 1) + 4 * t);
#pragma unroll
        for (int n4 = 0; n4 < 4; ++n4)
#pragma unroll
            for (int b = 0; b < BITS; ++b) {
                int word, pos;
                lut_locate<BITS>(bb, n4, b, word, pos);
                wd[word] |= ((c[b] >> n4) & 1u) << pos;
            }
    }
#pragma unroll
    for (int p = 0; p < BITS; ++p) *reinterpret_cast<uint32_t *>(lut + lut_word_offset(r, q, t, p, K, BITS)) = wd[p];
    if (t == 0) {
#pragma unroll
        for (int bb = 0; bb < 8; ++bb) lut[lut_scale_offset(r, q * 8 + bb, K, BITS)] = scales_in[r * (K / 16) + q * 8 + bb];
    }
}

__global__ void set_scale_kernel(PackedHeader *hdr, float s)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    hdr->s = s;
    hdr->rc6 = __frcp_rn(__fmul_rn(6.0f, s));
    hdr->amax_bits = __float_as_uint(__fmul_rn(s, 2688.0f));
}

cudaError_t launch_set_scale(PackedHeader *hdr, float s, cudaStream_t stream)
{
    set_scale_kernel<<<1, 32, 0, stream>>>(hdr, s);
    return cudaGetLastError();
}

cudaError_t launch_import_nvfp4(const uint8_t *codes_in, const uint8_t *scales_in, int64_t N, int64_t K, uint8_t *codes,
                                uint8_t *sf_swizzled, cudaStream_t stream)
{
    const int64_t total = N * (K / 16);
    import_nvfp4_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(codes_in, scales_in, N, K, codes,
                                                                             sf_swizzled);
    return cudaGetLastError();
}

cudaError_t launch_import_lut(int bits, const uint32_t *planes_in, const uint8_t *scales_in, int64_t N, int64_t K,
                              uint8_t *lut_dev, cudaStream_t stream)
{
    const int64_t total = N * (K / 128) * 4;
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (bits == 3) import_lut_kernel<3><<<blocks, 256, 0, stream>>>(planes_in, scales_in, N, K, lut_dev);
    else import_lut_kernel<2><<<blocks, 256, 0, stream>>>(planes_in, scales_in, N, K, lut_dev);
    return cudaGetLastError();
}

// ------------------------------------------------------ measurement kernel

// Read-only streaming sum with 128-bit loads: the practical ceiling of a kernel that only reads (the decode
// kernels' roofline is quoted against the copy bandwidth; this number shows what a pure reader reaches).
__global__ void __launch_bounds__(512) stream_read_kernel(const uint4 *__restrict__ src, size_t n16, unsigned long long *out)
{
    uint32_t acc = 0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n16; i += 4 * stride) {          // four independent loads in flight per thread
        const uint4 a = __ldg(src + i), b = __ldg(src + i + stride), c = __ldg(src + i + 2 * stride), d = __ldg(src + i + 3 * stride);
        acc += (a.x ^ a.y ^ a.z ^ a.w) + (b.x ^ b.y ^ b.z ^ b.w) + (c.x ^ c.y ^ c.z ^ c.w) + (d.x ^ d.y ^ d.z ^ d.w);
    }
    for (; i < n16; i += stride) {
        const uint4 a = __ldg(src + i);
        acc += a.x ^ a.y ^ a.z ^ a.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc == 0x9E3779B9u) atomicAdd(out, 1ull);     // keeps the loads alive; almost never taken
}

cudaError_t launch_stream_read(const void *src_dev, size_t bytes, void *out_dev, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    stream_read_kernel<<<sms * 4, 512, 0, stream>>>(reinterpret_cast<const uint4 *>(src_dev), bytes / 16,
                                                    reinterpret_cast<unsigned long long *>(out_dev));
    return cudaGetLastError();
}

// --------------------------------------------------- activation quantiser

// bf16 -> NVFP4 with a static tensor scale (App. A.3 "NVFP4").  One thread per
// 16-block: 32 B in, 8 B of codes out; four neighbouring lanes (one 64-wide k
// atom) merge their scale bytes into one 32-bit store of the MMA scale layout.
// Block (bx, by): 64 blocks of one row per 64 threads, four rows; no division, 32-bit index arithmetic.
template <bool SWIZZLED>
__device__ __forceinline__ void quant_act_block(const __nv_bfloat16 *A, int M, int nb, int64_t lda, float s, uint8_t *codes, uint8_t *sf,
                                                int bx, int by, int tx, int ty)
{
    const int b = by * 64 + tx;
    const int r = bx * 4 + ty;
    const bool live = (b < nb) && (r < M);
    const float rc6 = __frcp_rn(__fmul_rn(6.0f, s));
    uint32_t d8 = 0;
    if (live) {
        const uint4 *p = reinterpret_cast<const uint4 *>(A + (int64_t)r * lda + b * 16);
        const uint4 v0 = __ldg(p), v1 = __ldg(p + 1);
        const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        uint2 c;
        d8 = quant_block_nvfp4_bf16(w, s, rc6, c);
        *reinterpret_cast<uint2 *>(codes + ((int64_t)r * nb + b) * 8) = c;
    }
    // K % 64 == 0, so lanes 4q..4q+3 always hold the four blocks of one k atom of one row
    uint32_t w = d8 << (8 * (tx & 3));
    w |= __shfl_xor_sync(0xffffffffu, w, 1);
    w |= __shfl_xor_sync(0xffffffffu, w, 2);
    if (live && (tx & 3) == 0) {
        if (SWIZZLED) {
            // atom (r / 128, b / 4) of 512 bytes; row rr of the atom at (rr % 32) * 16 + (rr / 32) * 4
            const int rr = r & 127;
            const size_t off = ((size_t)(r >> 7) * (size_t)(nb >> 2) + (size_t)(b >> 2)) * 512 + (size_t)((rr & 31) * 16 + (rr >> 5) * 4);
            *reinterpret_cast<uint32_t *>(sf + off) = w;
        } else {
            *reinterpret_cast<uint32_t *>(sf + (int64_t)r * nb + b) = w;
        }
    }
}

template <bool SWIZZLED>
__global__ void __launch_bounds__(256) quant_act_kernel(const __nv_bfloat16 *A, int M, int nb, int64_t lda,
                                                        float s, uint8_t *codes, uint8_t *sf)
{
    // launched with programmatic stream serialization (hides the launch latency behind the previous
    // kernel); that kernel may produce A or still read the workspace, so wait for it before anything else
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    quant_act_block<SWIZZLED>(A, M, nb, lda, s, codes, sf, (int)blockIdx.x, (int)blockIdx.y, (int)threadIdx.x, (int)threadIdx.y);
}

// The activation quantiser and the cast of a LUT3 matrix to NVFP4 in one launch: the first `cast_blocks` blocks take eight atoms
// each, the others a block of the quantiser.  Both are bound by instruction issue, and nothing orders them.  5120 x 17408 and 1000
// rows of activations: 31.6 us, one after the other 36.
__global__ void __launch_bounds__(256) quant_act_cast_kernel(const __nv_bfloat16 *A, int M, int nb, int64_t lda, float s, uint8_t *codes,
                                                             uint8_t *sf, const PackedHeader *hdr, const uint8_t *lut, int64_t N, int64_t K,
                                                             uint8_t *w_codes, uint8_t *w_sf, int64_t cast_blocks, int quant_x)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int64_t)blockIdx.x < cast_blocks) {
        const uint32_t natoms = (uint32_t)((K + 511) / 512);
        const int64_t task = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
        const int64_t rowgrp = task / natoms;
        if (rowgrp < N / 8) autocast_atom(hdr, lut, rowgrp, (uint32_t)(task - rowgrp * natoms), K, w_codes, w_sf);
        return;
    }
    const uint32_t q = (uint32_t)((int64_t)blockIdx.x - cast_blocks), by = q / (uint32_t)quant_x;
    quant_act_block<true>(A, M, nb, lda, s, codes, sf, (int)(q - by * (uint32_t)quant_x), (int)by, (int)(threadIdx.x & 63), (int)(threadIdx.x >> 6));
}

static cudaLaunchConfig_t overlapped(cudaLaunchAttribute (&attr)[1], dim3 grid, dim3 block, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

cudaError_t launch_quant_act(const void *A_bf16, int64_t M, int64_t K, int64_t lda, float act_scale, uint8_t *codes,
                             uint8_t *sf, int swizzled, cudaStream_t stream)
{
    const int nb = (int)(K / 16);
    const int m = (int)M;
    const __nv_bfloat16 *A = reinterpret_cast<const __nv_bfloat16 *>(A_bf16);
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = overlapped(attr, dim3((unsigned)((m + 3) / 4), (unsigned)((nb + 63) / 64)), dim3(64, 4), stream);
    if (swizzled) return cudaLaunchKernelEx(&cfg, quant_act_kernel<true>, A, m, nb, lda, act_scale, codes, sf);
    return cudaLaunchKernelEx(&cfg, quant_act_kernel<false>, A, m, nb, lda, act_scale, codes, sf);
}

cudaError_t launch_quant_act_cast(const void *A_bf16, int64_t M, int64_t K, int64_t lda, float act_scale, uint8_t *codes, uint8_t *sf,
                                  const PackedHeader *hdr, const uint8_t *lut_dev, int64_t N, uint8_t *w_codes, uint8_t *w_sf,
                                  cudaStream_t stream)
{
    const int nb = (int)(K / 16), m = (int)M;
    const int64_t cast_blocks = (N / 8 * ((K + 511) / 512) + 7) / 8;
    const int quant_x = (m + 3) / 4;
    const int64_t blocks = cast_blocks + (int64_t)quant_x * ((nb + 63) / 64);
    if (blocks > 0x7FFFFFFFll) {                             // beyond one grid: one after the other
        const cudaError_t e = launch_quant_act(A_bf16, M, K, lda, act_scale, codes, sf, 1, stream);
        return e != cudaSuccess ? e : launch_autocast(hdr, lut_dev, N, K, w_codes, w_sf, stream);
    }
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = overlapped(attr, dim3((unsigned)blocks), dim3(256), stream);
    return cudaLaunchKernelEx(&cfg, quant_act_cast_kernel, reinterpret_cast<const __nv_bfloat16 *>(A_bf16), m, nb, lda, act_scale, codes,
                              sf, hdr, lut_dev, N, K, w_codes, w_sf, cast_blocks, quant_x);
}

}  // namespace dq

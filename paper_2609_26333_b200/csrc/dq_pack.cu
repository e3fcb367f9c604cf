// Packers and quantisers: tensor scale, NVFP4 and LUT3 round-to-nearest,
// LUT3 -> NVFP4 autocast, canonical export, and the activation quantiser of the
// prefill path.  (App. A.3 "Quantization formats", Sec. 2.3, App. C.2 storage.)
//
// Quantiser arithmetic is fp32 with explicit round-to-nearest intrinsics so the
// compiler cannot contract or reorder it:
//   rc6 = 1/(6 s);  t = extreme * rc6;  d = E4M3(t);  r = 1/(s * dec(d));  y = x * r
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

// four floats -> two bytes of E2M1 codes (element 0 in the low nibble of byte 0)
__device__ __forceinline__ uint32_t f32x4_to_e2m1x4(float f0, float f1, float f2, float f3)
{
    uint32_t r;
    asm("{\n\t.reg .b8 b0, b1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
        "mov.b32 %0, {b0, b1, b0, b1};\n\t}"
        : "=r"(r) : "f"(f0), "f"(f1), "f"(f2), "f"(f3));
    return r & 0xFFFFu;
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

// Number of thresholds below y (the index of the nearest level, a value on a threshold taking the lower level), as index
// bits in the sign bits of the results: T - y is negative exactly where y > T, and with increasing thresholds the bits of the count
// are parities of those signs.
template <int BITS>
__device__ __forceinline__ void level_bits(float y, const float (&T)[(1 << BITS) - 1], uint32_t (&bit)[BITS])
{
    uint32_t d[(1 << BITS) - 1];
#pragma unroll
    for (int l = 0; l < (1 << BITS) - 1; ++l) d[l] = __float_as_uint(__fsub_rn(T[l], y));
    if (BITS == 3) {
        bit[BITS - 1] = d[3];
        bit[1] = d[1] ^ d[3] ^ d[BITS == 3 ? 5 : 0];
        bit[0] = (d[0] ^ d[1] ^ d[2]) ^ (d[3] ^ d[BITS == 3 ? 4 : 0] ^ d[BITS == 3 ? 5 : 0]) ^ d[BITS == 3 ? 6 : 0];
    } else {
        bit[1] = d[1];
        bit[0] = d[0] ^ d[1] ^ d[2];
    }
}
// appends a nibble [index bits, BITS of them][garbage bit] at the low end of acc (LUT2: [0][bits][garbage])
template <int BITS>
__device__ __forceinline__ uint32_t push_level(uint32_t acc, const uint32_t (&bit)[BITS])
{
    if (BITS == 2) acc <<= 1;
#pragma unroll
    for (int b = BITS - 1; b > 0; --b) acc = __funnelshift_l(bit[b], acc, 1);
    return __funnelshift_l(bit[0], acc, 2);
}

// Round-to-nearest packing of the master weights (App. A.3): NVFP4 (NV) and / or one LUT format (BITS = 3 or 2) in one
// read of W.  A warp takes an atom of 8 rows x 512 weights; lane (g, t) = (row, quarter of a 16-block) takes weights
// 4t .. 4t+3 of every block of its row, which is what its index words of the LUT layout store, 128 weights at a time.
// Both encodings share the block's largest magnitude, its E4M3 scale and the reciprocal (a table of the 127 scales per CTA);
// index words and scales leave as whole 512- and 256-byte rows of the atom, E2M1 codes after a transpose inside
// the quad as 16 bytes per lane.
// Bound by instruction issue (the thresholds: 7 subtractions, 4 logic ops and 3 shifts per weight).  17408 x 5120 bf16 to
// NVFP4 and LUT3: 116 us, 2.3 TB/s; a pass per format with compares and one bit placed at a time took about 250.
template <bool FP32IN, bool NV, int BITS>
__global__ void __launch_bounds__(128) pack_kernel(const void *__restrict__ W, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr,
                                                   uint8_t *__restrict__ codes, uint8_t *__restrict__ sf, uint8_t *__restrict__ lut)
{
    constexpr bool LUT = BITS > 0;
    constexpr int B = LUT ? BITS : 2;                      // dummy where there is no LUT format
    __shared__ float rtab[128];                            // 1 / (s * d) by the byte of d; 0 for a scale that rounded to zero
    const float s = tensor_scale(hdr);
    const float rc6 = __frcp_rn(__fmul_rn(6.0f, s));
    if (blockIdx.x == 0 && threadIdx.x == 0) { hdr->s = s; hdr->rc6 = rc6; }
    rtab[threadIdx.x] = (threadIdx.x == 0) ? 0.0f : __frcp_rn(__fmul_rn(s, e4m3_to_f32(threadIdx.x)));
    __syncthreads();
    const uint32_t atoms_k = (uint32_t)(2 * lut_slices(K));               // atoms along a row, a short last slice padded
    const uint32_t katoms = NV && !LUT ? (uint32_t)((K + 511) / 512) : atoms_k;
    const int64_t task = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int64_t rowgrp = task / katoms;
    if (rowgrp >= N / 8) return;
    const uint32_t atom = (uint32_t)(task - rowgrp * katoms);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t r = rowgrp * 8 + g;
    const int nwi = max(0, min(4, (int)(K / 128) - 4 * (int)atom));
    float T[(1 << B) - 1];
    if (LUT) {
#pragma unroll
        for (int l = 0; l < (1 << B) - 1; ++l) T[l] = (BITS == 3) ? hdr->lut_thresholds[l] : hdr->lut2_thresholds[l & 3];
    }
    uint4 *out_codes = nullptr;
    uint32_t *out_sf = nullptr;
    if (NV) {
        out_codes = reinterpret_cast<uint4 *>(codes + r * (K / 2) + (int64_t)atom * 256 + t * 16);
        out_sf = reinterpret_cast<uint32_t *>(sf + sf_swizzled_offset(r, (int64_t)atom * 32 + 4 * (t & 1), K));
    }
    const int64_t src = r * ldw + (int64_t)atom * 512 + t * 4;
    uint32_t words[4][B];
    uint2 my_scales = make_uint2(0u, 0u);                  // LUT scale bytes of word group t
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
#pragma unroll
        for (int p = 0; p < B; ++p) words[wi][p] = 0u;
        if (wi >= nwi) continue;                           // whole warps
        uint4 raw[8];                                      // bf16: two words of it are used
#pragma unroll
        for (int bb = 0; bb < 8; ++bb) {
            if (FP32IN) {
                raw[bb] = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const float *>(W) + src + wi * 128 + bb * 16));
            } else {
                const uint2 v = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const __nv_bfloat16 *>(W) + src + wi * 128 + bb * 16));
                raw[bb] = make_uint4(v.x, v.y, 0u, 0u);
            }
        }
        uint32_t nv_pieces[4] = {0u, 0u, 0u, 0u};
        uint32_t nv_sc[2] = {0u, 0u}, lut_sc[2] = {0u, 0u};
        uint32_t sel[4];
#pragma unroll
        for (int a = 3; a >= 0; --a) {
            uint32_t acc = 0u;
#pragma unroll
            for (int h = 1; h >= 0; --h) {                 // selector nibbles from the top: second block first
                const int bb = 2 * a + h;
                // largest and most negative value of the block across the quad
                float mx, mn;
                float x[4];
                if (FP32IN) {
                    x[0] = __uint_as_float(raw[bb].x); x[1] = __uint_as_float(raw[bb].y);
                    x[2] = __uint_as_float(raw[bb].z); x[3] = __uint_as_float(raw[bb].w);
                    mx = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
                    mn = fmaxf(fmaxf(-x[0], -x[1]), fmaxf(-x[2], -x[3]));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                    mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                    mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
                } else {
                    x[0] = __uint_as_float(raw[bb].x << 16); x[1] = __uint_as_float(raw[bb].x & 0xFFFF0000u);
                    x[2] = __uint_as_float(raw[bb].y << 16); x[3] = __uint_as_float(raw[bb].y & 0xFFFF0000u);
                    const uint32_t pm = max_bf16x2(raw[bb].x, raw[bb].y);
                    const uint32_t nm = max_bf16x2(raw[bb].x ^ 0x80008000u, raw[bb].y ^ 0x80008000u);
                    uint32_t e = max_bf16x2(__byte_perm(pm, nm, 0x5410), __byte_perm(pm, nm, 0x7632));    // (max, -min)
                    e = max_bf16x2(e, __shfl_xor_sync(0xffffffffu, e, 1));
                    e = max_bf16x2(e, __shfl_xor_sync(0xffffffffu, e, 2));
                    mx = __uint_as_float(e << 16);
                    mn = __uint_as_float(e & 0xFFFF0000u);
                }
                const uint32_t d8 = f32_to_e4m3(__fmul_rn(fmaxf(mx, mn), rc6)) & 0x7Fu;
                const float rr = rtab[d8];
                if (NV) {
                    const uint32_t c = f32x4_to_e2m1x4(__fmul_rn(x[0], rr), __fmul_rn(x[1], rr), __fmul_rn(x[2], rr), __fmul_rn(x[3], rr));
                    nv_pieces[a] |= (d8 ? c : 0u) << (16 * h);
                    nv_sc[bb >> 2] |= d8 << (8 * (bb & 3));
                }
                if (LUT) {
                    // the scale takes the sign of the block's extreme; where both signs reach the magnitude, plus
                    const bool neg = mn > mx;
                    lut_sc[bb >> 2] |= (d8 ? (d8 | (neg ? 0x80u : 0u)) : 0u) << (8 * (bb & 3));
                    const float rs = neg ? -rr : rr;
#pragma unroll
                    for (int n4 = 3; n4 >= 0; --n4) {
                        uint32_t bit[B];
                        level_bits<B>(__fmul_rn(x[n4], rs), T, bit);
                        acc = push_level<B>(acc, bit);
                    }
                }
            }
            sel[a] = acc >> 1;
        }
        if (LUT) {
            if (BITS == 3) {
#pragma unroll
                for (int p = 0; p < B; ++p)
                    words[wi][p] = (sel[p] & 0x77777777u) | (((sel[3] >> p) & 0x11111111u) << 3);
            } else {
#pragma unroll
                for (int p = 0; p < 2; ++p)
                    words[wi][p] = (sel[2 * p] & 0x33333333u) | ((sel[2 * p + 1] & 0x33333333u) << 2);
            }
            if (t == wi) my_scales = make_uint2(lut_sc[0], lut_sc[1]);
        }
        if (NV) {
            out_codes[wi * 4] = quad_transpose(nv_pieces, t);
            if (t < 2) out_sf[wi * 256] = t ? nv_sc[1] : nv_sc[0];              // two k atoms of 512 bytes per word group
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

template <bool FP32IN>
static void launch_pack_typed(const void *W, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr, uint8_t *codes, uint8_t *sf,
                              uint8_t *lut, int bits, cudaStream_t stream)
{
    const int64_t atoms_k = bits ? 2 * lut_slices(K) : (K + 511) / 512;
    const unsigned blocks = (unsigned)((N / 8 * atoms_k + 3) / 4);
    if (codes && bits == 3) pack_kernel<FP32IN, true, 3><<<blocks, 128, 0, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
    else if (codes && bits == 2) pack_kernel<FP32IN, true, 2><<<blocks, 128, 0, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
    else if (codes) pack_kernel<FP32IN, true, 0><<<blocks, 128, 0, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
    else if (bits == 3) pack_kernel<FP32IN, false, 3><<<blocks, 128, 0, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
    else pack_kernel<FP32IN, false, 2><<<blocks, 128, 0, stream>>>(W, N, K, ldw, hdr, codes, sf, lut);
}

// codes / sf: NVFP4 output or nullptr; lut with bits = 3 or 2: LUT output, bits = 0: none
cudaError_t launch_pack(const void *W, int w_dtype, int64_t N, int64_t K, int64_t ldw, PackedHeader *hdr, uint8_t *codes,
                        uint8_t *sf_swizzled, uint8_t *lut_dev, int bits, cudaStream_t stream)
{
    if (w_dtype == DQ_DT_FP32) launch_pack_typed<true>(W, N, K, ldw, hdr, codes, sf_swizzled, lut_dev, bits, stream);
    else launch_pack_typed<false>(W, N, K, ldw, hdr, codes, sf_swizzled, lut_dev, bits, stream);
    return cudaGetLastError();
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
// block of row g, i.e. bits 4t .. 4t+3 of each half of a canonical word.  It gathers its bits of the sixteen words of the atom
// per plane; two exchanges inside the quad OR them together so that lane t ends up with the four words of word group t.
template <int BITS>
__global__ void __launch_bounds__(128) export_lut_kernel(const PackedHeader *__restrict__ hdr, const uint8_t *__restrict__ lut, int64_t N,
                                                         int64_t K, uint32_t *__restrict__ planes_out, uint8_t *__restrict__ scales_out, float *s_out)
{
    if (blockIdx.x == 0 && threadIdx.x == 0 && s_out) *s_out = hdr->s;
    const uint32_t natoms = (uint32_t)((K + 511) / 512);
    const int64_t task = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int64_t rowgrp = task / natoms;
    if (rowgrp >= N / 8) return;
    const uint32_t atom = (uint32_t)(task - rowgrp * natoms);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t r = rowgrp * 8 + g;
    const uint8_t *src = lut + lut_atom_offset(rowgrp * 8, atom, K, BITS);
    uint4 w[BITS];
#pragma unroll
    for (int p = 0; p < BITS; ++p) w[p] = __ldg(reinterpret_cast<const uint4 *>(src + p * 512 + lane * 16));
    const uint2 s8 = __ldg(reinterpret_cast<const uint2 *>(src + lut_plane_bytes(BITS) + lane * 8));
    const bool mine = (int)(K / 128) - 4 * (int)atom > t;   // word group t of the atom lies inside the row
    uint32_t sel[4][4];                                     // [word group][selector]
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
        uint32_t wd[BITS];
#pragma unroll
        for (int p = 0; p < BITS; ++p) wd[p] = wi == 0 ? w[p].x : wi == 1 ? w[p].y : wi == 2 ? w[p].z : w[p].w;
        lut_selectors<BITS>(wd, sel[wi]);
    }
    const bool hi2 = (t & 2) != 0, hi1 = (t & 1) != 0;
#pragma unroll
    for (int p = 0; p < BITS; ++p) {
        uint32_t o[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            uint32_t z[4];
#pragma unroll
            for (int wi = 0; wi < 4; ++wi) {                // bit p of the eight nibbles -> bits 0-3 of both halves, then to 4t
                uint32_t x = (sel[wi][a] >> p) & 0x11111111u;
                x = (x | (x >> 3)) & 0x03030303u;
                x = (x | (x >> 6)) & 0x000F000Fu;
                z[wi] = x << (4 * t);
            }
            const uint32_t a0 = (hi2 ? z[2] : z[0]) | __shfl_xor_sync(0xffffffffu, hi2 ? z[0] : z[2], 2);
            const uint32_t a1 = (hi2 ? z[3] : z[1]) | __shfl_xor_sync(0xffffffffu, hi2 ? z[1] : z[3], 2);
            o[a] = (hi1 ? a1 : a0) | __shfl_xor_sync(0xffffffffu, hi1 ? a0 : a1, 1);
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

// Weight-only decode of batches on the 5th-generation tensor cores, for all three encodings (LUT3, LUT2: App. C.2 "Kernel
// specification"; NVFP4A16: Sec. 2.3 / Table 1):
//   Y[b][n] = bf16( s * sum_k d_blk(n,k) * level(n,k) * X[b][k] ),   up to 64 batch columns in one pass over the weights.
//
// Arithmetic.  A weight is dequantised with its block scale to fp16: E2M1 * E4M3 is exact (3 + 4 bits of significand); an
// fp16 codebook level times E4M3 has up to 15 bits and is kept as a pair hi = rn(G d), lo = G d - hi, both fp16 and exact for
// codebooks whose levels are multiples of 2^-15 (every d is a multiple of 2^-9, fp16 reaches down to 2^-24) and at most 146.2 in
// magnitude (d goes to 448, fp16 to 65504); the launcher asks for it.  Activations: per batch column and slice of 512 weights one power of two brings the largest
// magnitude into [2^14, 2^15); fp16 then holds every element within 2^28 of it exactly.  So products are exact; a group (128
// weights of a LUT format, a slice of NVFP4) is summed in fp32 by the tensor cores, groups are added in fp32 by FMA with the inverse
// power of two.
//
// Work split.  A CTA (one per SM, 16 warps) takes tiles of 256 rows as two halves of 128, the tensor-memory lanes.  Where there
// are too few tiles for the chip a cluster of up to 8 CTAs shares a tile, each taking a range of slices; at the end
// they exchange partial sums through distributed shared memory, every CTA adding a share of the columns in rank order.
//   warps 0-3, 4-7 : dequantise half 0 / half 1: ring stage -> registers -> tcgen05.st into the A operand in tensor memory
//                    (lane (g, t) of the device layout holds what tcgen05.st.16x256b wants from it), 64 columns a step: 64
//                    weights of hi and lo, or 128 NVFP4 weights; two A buffers per half.  They also read finished slices back.
//   warps 8-11     : activations of the next slice: global -> fp16 in shared memory, one column at a time per warp
//   warp 12        : tcgen05.mma (M = 128, N = 16 / 32 / 48 / 64, K = 16, A in tensor memory, B in shared memory)
//   warp 13        : weights of the next slices, bulk / TMA copies into a ring per half
// Two accumulators per half alternate, so reading one back overlaps the MMAs of the next.
//
// What bounds it: look-ups and stores of the dequantising warps, which add up on a scheduler (32 PRMT, 16 HFMA2 and a store of 16
// registers: 89 to 97 cycles a warp in every store shape) on top of the loop's hand-overs.  34816x5120 LUT3 batch 40 takes 70.0 us;
// without staging 63.8, without read-back 67.9, without MMAs (N / 2 cycles each) 65.1, without all three 57.0, of these without
// look-ups 39.2, without stores too 31.7.  It is not latency: sixteen dequantising warps take 73.6, waits that spin 72.4.
#include <atomic>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dq_common.cuh"
#include "dq_tcgen05.cuh"

namespace dq {

namespace {

using namespace tc;

constexpr int kSlice = 512;                        // weights along K per accumulator
constexpr int kThreads = 512;
constexpr uint32_t kSmemMax = 227 * 1024;
constexpr uint32_t kXinvOff = 512;                 // [4][4][64] floats: inverse activation scales of the last slices' 128-weight groups,
constexpr uint32_t kXinvGroup = 68;                // a group's 64 padded: the four stores of a column go to different banks
constexpr uint32_t kRingOff = 5120;

// FMT: 0 = NVFP4, 2 = LUT2, 3 = LUT3; NC: batch columns of the pass, padded
template <int FMT, int NC>
struct Cfg {
    static constexpr bool kLut = FMT != 0;
    static constexpr uint32_t kAtom = kLut ? (uint32_t)lut_atom_bytes(kLut ? FMT : 3) : 0u;
    // one ring stage, 128 rows: LUT 512 weights along K; NVFP4 256, codes and then scale atoms
    static constexpr uint32_t kStageBytes = kLut ? 16u * kAtom : 2u * 8192u + 2048u;
    static constexpr uint32_t kXStride = (uint32_t)NC * 16u + 16u;             // 8 weights of all columns; 16 B of padding: no bank conflicts
    static constexpr uint32_t kXBytes = (kSlice / 8) * kXStride;
    static constexpr uint32_t kXTotal = 2u * kXBytes;
    static constexpr int kFit = (int)((kSmemMax - 1024u - kRingOff - kXTotal) / (2u * kStageBytes));
    static constexpr int S = kFit < 1 ? 1 : kFit > 4 ? 4 : (kLut && kFit > 2) ? 2 : kFit;
    static constexpr uint32_t kXOff = kRingOff + 2u * S * kStageBytes;
    static constexpr uint32_t kSmem = kXOff + kXTotal + 1024u;
    static_assert(kFit >= 1 && kSmem <= kSmemMax, "shared memory");
    static_assert((uint32_t)(NC / 4 + 8) * 256u * 16u <= kXOff + kXTotal - kRingOff, "partial sums of a cluster must fit the ring and X area");
    static constexpr int kStepK = kLut ? 64 : 128;                             // weights per 64 columns of A
    // Steps summed by the tensor cores before the accumulator is read back.  They drop bits below the accumulator's last place at
    // every addition where FMA rounds; products of a 7-bit weight and an 8-bit activation lose next to nothing over a slice, the
    // pairs of LUT weights do: with 64 additions per group 7e-4 of the bf16 outputs differ from the rounded exact sum, with 16
    // (128 weights) as few as with the mma.sync kernels, 2e-4.
    static constexpr int kGroupSteps = kLut ? 128 / kStepK : kSlice / kStepK;
    static constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(NC >> 3) << 17) | ((128u >> 4) << 24);    // fp16 x fp16 -> fp32, K-major
};

// barriers, 8 bytes each, from byte 64 of shared memory
enum : uint32_t {
    kWFull = 64,                 // [half][S <= 4]
    kWEmpty = kWFull + 64,       // [half][4]
    kAFull = kWEmpty + 64,       // [half][2]
    kAEmpty = kAFull + 32,
    kDFull = kAEmpty + 32,       // [buffer 2][half 2]
    kDEmpty = kDFull + 32,       // [buffer 2][half 2]
    kXFull = kDEmpty + 32,       // [2]
    kXEmpty = kXFull + 16,
    kBarEnd = kXEmpty + 16,
};
static_assert(kBarEnd <= kXinvOff && kXinvOff + 16u * 4u * kXinvGroup <= kRingOff, "barriers, scales");

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t hfms2(uint32_t a, uint32_t b, uint32_t c)        // a * b - c
{
    uint32_t r;
    asm("{\n\t.reg .b32 n;\n\tneg.f16x2 n, %3;\n\tfma.rn.f16x2 %0, %1, %2, n;\n\t}" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// the low / high half on both halves: written so that the multiply takes it as an operand modifier
__device__ __forceinline__ uint32_t both_lo(uint32_t v)
{
    uint32_t r;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tmov.b32 %0, {l, l};\n\t}" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t both_hi(uint32_t v)
{
    uint32_t r;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tmov.b32 %0, {h, h};\n\t}" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t two)
{
    uint32_t r;
    asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %1;\n\tcvt.rn.f16x2.e4m3x2 %0, lo;\n\t}" : "=r"(r) : "r"(two));
    return r;
}
// magnitude of the larger magnitude, per half; the sign is of no use
__device__ __forceinline__ uint32_t max_abs_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// A bf16 pair as fp16: +-1 in the place of an infinity, NaN stays, anything else is zero
__device__ __forceinline__ uint32_t inf_to_one(uint32_t w)
{
    uint32_t r = 0;
#pragma unroll
    for (int s = 0; s < 32; s += 16) {
        const uint32_t h = (w >> s) & 0xFFFFu, mag = h & 0x7FFFu;
        r |= (mag == 0x7F80u ? (h & 0x8000u) | 0x3C00u : mag > 0x7F80u ? 0x7FFFu : 0u) << s;
    }
    return r;
}
// Infinite activations of a LUT format.  Both parts of a weight meet the same activation, and a part that is zero would make a NaN of an
// infinite one: a warp's columns of the slice (every fourth from c0) that hold an infinity are staged again with +-1 for it and
// zeros beside it, and the inverse scale of their 128-weight groups is infinite.  A function of its own: inside the loop of the
// activation warps its code costs every call of more than 32 columns 1 % (5120x17408 LUT3 batch 40: 44.5 us so, 45.0 inside).
__device__ __noinline__ void stage_infinite(const __nv_bfloat16 *X, int64_t ldx, int c0, int cols, int live, uint32_t xb, uint32_t stride,
                                            float *xinv)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int c = c0; c < cols; c += 4) {
        const uint4 *xp = reinterpret_cast<const uint4 *>(X + (int64_t)c * ldx);
        uint4 x[2];
        uint32_t inf = 0;                                    // groups with an infinity
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint4 v = lane + 32 * i < live ? __ldg(xp + lane + 32 * i) : make_uint4(0u, 0u, 0u, 0u);
            x[i] = make_uint4(inf_to_one(v.x), inf_to_one(v.y), inf_to_one(v.z), inf_to_one(v.w));
            // 1 has bit 12 set and bit 14 clear, NaN has both
            const uint32_t ones = (x[i].x & ~(x[i].x >> 2)) | (x[i].y & ~(x[i].y >> 2)) | (x[i].z & ~(x[i].z >> 2)) | (x[i].w & ~(x[i].w >> 2));
            const uint32_t any = __ballot_sync(0xffffffffu, (ones & 0x10001000u) != 0u);
            inf |= ((any & 0xFFFFu ? 1u : 0u) | (any >> 16 ? 2u : 0u)) << (2 * i);
        }
        if (inf == 0) continue;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         ::"r"(xb + (uint32_t)c * 16u + (uint32_t)(lane + 32 * i) * stride), "r"(x[i].x), "r"(x[i].y), "r"(x[i].z), "r"(x[i].w) : "memory");
        if (lane < 4) xinv[lane * kXinvGroup + c] = (inf >> lane) & 1u ? __uint_as_float(0x7F800000u) : 1.0f;
    }
}
// four code bytes -> four fp16 pairs (low nibble first)
__device__ __forceinline__ void e2m1x8_to_f16(uint32_t w, uint32_t (&p)[4])
{
    asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\tmov.b32 {b0, b1, b2, b3}, %4;\n\t"
        "cvt.rn.f16x2.e2m1x2 %0, b0;\n\tcvt.rn.f16x2.e2m1x2 %1, b1;\n\t"
        "cvt.rn.f16x2.e2m1x2 %2, b2;\n\tcvt.rn.f16x2.e2m1x2 %3, b3;\n\t}"
        : "=r"(p[0]), "=r"(p[1]), "=r"(p[2]), "=r"(p[3]) : "r"(w));
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds_v2(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void tmem_st_x4(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_x8(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
          "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
          "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
                   "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr) : "memory");
}
// K-major, unswizzled operand: 8-row groups of 16-byte rows; `kstep` bytes between the two 8-element halves of K,
// `nstep` bytes between 8-row groups of N
__device__ __forceinline__ uint64_t make_desc_plain(uint32_t saddr, uint32_t kstep, uint32_t nstep)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((kstep >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((nstep >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// D (tensor memory, fp32) (+)= A (tensor memory, fp16, 128 x 16) * B (shared memory, fp16, 16 x N)
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate ? 1u : 0u) : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t rank, float4 v)
{
    asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.v4.f32 [a], {%2, %3, %4, %5};\n\t}"
                 ::"r"(addr), "r"(rank), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// Wait with the kernel's own budget (a test shortens it); warp-uniform.  The time hint parks the warp in hardware until the phase
// completes: polling from the six warps that mostly wait would take issue slots from the eight that dequantise.
__device__ __forceinline__ bool try_park(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag, long long budget)
{
    if (__all_sync(0xffffffffu, try_park(bar, parity))) return true;
    const long long t0 = clock64();
    while (true) {
        if (__all_sync(0xffffffffu, try_park(bar, parity))) return true;
        const bool over = clock64() - t0 > budget;
        if (__any_sync(0xffffffffu, over || *abort_flag != 0)) { *abort_flag = 1; return false; }
    }
}

// the same for one thread
__device__ __forceinline__ bool wait_one(uint32_t bar, uint32_t parity, volatile int *abort_flag, long long budget)
{
    if (try_park(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (try_park(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) { *abort_flag = 1; return false; }
    }
}

struct Codebook { uint32_t tl0, tl1, th0, th1; };    // low bytes of levels 0-3 / 4-7, high bytes of levels 0-3 / 4-7

struct TcDecodeArgs {
    const uint8_t *weights;              // LUT atoms (NVFP4 codes come through the tensor map)
    const uint8_t *sf;                   // NVFP4 scale atoms
    const PackedHeader *hdr;
    const __nv_bfloat16 *X;
    __nv_bfloat16 *Y;
    int64_t ldx, ldy;
    int b0, cols, N, K;
    int csize;                           // CTAs that share a tile
    long long wait_cycles;
    int drop_first_copy;                 // test hook: the first ring stage of CTA 0 is never requested
    StatusWord *status;
};

template <int FMT, int NC>
__global__ void __launch_bounds__(kThreads, 1)
decode_tc_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ TcDecodeArgs P)
{
    using C = Cfg<FMT, NC>;
    constexpr bool kLut = C::kLut;
    constexpr int BITS = kLut ? FMT : 3;
    constexpr int S = C::S;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t win0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (win0 - smem_u32(smem_raw));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem);
    volatile uint32_t *tmem_ptr = reinterpret_cast<volatile uint32_t *>(smem + 8);
    float *xinv_s = reinterpret_cast<float *>(smem + kXinvOff);

    // roles by number; the dequantising warps, which always have something to issue, are the youngest of their schedulers
    const int warp = (int)(threadIdx.x >> 5) ^ 8, lane = threadIdx.x & 31;
    const int csize = P.csize;
    const uint32_t rank = csize > 1 ? cluster_ctarank() : 0u;
    const int first_tile = (int)blockIdx.x / csize, tile_stride = (int)gridDim.x / csize;
    const int ntiles = (P.N + 255) >> 8;
    const int nslices = (P.K + kSlice - 1) / kSlice;
    const int s0 = (int)((long long)nslices * rank / csize), s1 = (int)((long long)nslices * (rank + 1) / csize);
    const long long budget = P.wait_cycles;
    // halves of a tile with rows in them, 128-weight groups of a slice inside K
    auto halves = [&](int tile) { return P.N - tile * 256 > 128 ? 2 : 1; };
    auto groups = [&](int sl) { return min(kSlice, P.K - sl * kSlice) >> 7; };

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int h = 0; h < 2; ++h) {
            for (int i = 0; i < S; ++i) {
                mbar_init(win0 + kWFull + (h * 4 + i) * 8, 1);
                mbar_init(win0 + kWEmpty + (h * 4 + i) * 8, 4);
            }
            for (int i = 0; i < 2; ++i) {
                mbar_init(win0 + kAFull + (h * 2 + i) * 8, 4);
                mbar_init(win0 + kAEmpty + (h * 2 + i) * 8, 1);
                mbar_init(win0 + kDFull + (i * 2 + h) * 8, 1);
                mbar_init(win0 + kDEmpty + (i * 2 + h) * 8, 4);
            }
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(win0 + kXFull + i * 8, 4);
            mbar_init(win0 + kXEmpty + i * 8, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 12) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(win0 + 8u), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_ptr;
    auto a_cols = [&](int h, uint32_t slot) { return tmem + (uint32_t)(h * 2 + (int)slot) * 64u; };
    auto d_cols = [&](uint32_t buf, int h) { return tmem + 256u + (buf * 2u + (uint32_t)h) * 64u; };
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp < 8) {
        // ============================================================ dequantise, read slices back, store
        // registers of the four warpgroups: 192 + 192 + 80 + 48 = 4 x the 128 of the launch
        asm volatile("setmaxnreg.inc.sync.aligned.u32 192;");
        const int h = warp >> 2, q = warp & 3;
        const int g = lane >> 2, t = lane & 3;
        const uint32_t lanes = (uint32_t)(32 * q) << 16;
        Codebook cb = {0u, 0u, 0u, 0u};
        if (kLut) {
            const uint4 v = *reinterpret_cast<const uint4 *>(BITS == 3 ? P.hdr->lut_prmt : P.hdr->lut2_prmt);
            cb = {v.x, v.y, v.z, v.w};
        }
        const float s_w = P.hdr->s;
        float acc[NC];
        bool ok = true;
        uint32_t cnt = 0, step = 0, wst = 0, wph = 0;       // slices, A buffers filled, ring stage and its phase
        uint32_t grp = 0;                                   // groups handed over
        bool open = false;                                  // the last of them is not in the running sums yet
        uint32_t next_xi = 0, open_xi = 0;                  // inverse activation scales of the next group and of that one
        // the last complete group from its accumulator into the running sums
        auto flush = [&]() {
            if (!open) return;
            open = false;
            const uint32_t n = grp - 1u;
            if (ok) ok = wait_warp(win0 + kDFull + ((n & 1u) * 2u + (uint32_t)h) * 8u, (n >> 1) & 1u, abort_flag, budget);
            if (!ok) return;
            tc_fence_after();
            const uint32_t d = d_cols(n & 1u, h) + lanes;
            constexpr int kBatch = NC == 64 ? 32 : NC;      // columns read at once
#pragma unroll
            for (int c = 0; c < NC; c += kBatch) {
                float v[kBatch / 16][16];
#pragma unroll
                for (int i = 0; i < kBatch / 16; ++i) tmem_ld16(d + (uint32_t)(c + 16 * i), v[i]);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < kBatch; i += 4) {
                    const uint4 x = lds_v4(open_xi + (uint32_t)(c + i) * 4u);
                    acc[c + i] = fmaf(v[i / 16][i % 16], __uint_as_float(x.x), acc[c + i]);
                    acc[c + i + 1] = fmaf(v[i / 16][i % 16 + 1], __uint_as_float(x.y), acc[c + i + 1]);
                    acc[c + i + 2] = fmaf(v[i / 16][i % 16 + 2], __uint_as_float(x.z), acc[c + i + 2]);
                    acc[c + i + 3] = fmaf(v[i / 16][i % 16 + 3], __uint_as_float(x.w), acc[c + i + 3]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(win0 + kDEmpty + ((n & 1u) * 2u + (uint32_t)h) * 8u);
        };
        auto a_slot = [&]() -> uint32_t {                   // the next A buffer, free
            const uint32_t slot = step & 1u;
            ok = wait_warp(win0 + kAEmpty + ((uint32_t)h * 2u + slot) * 8u, ((step >> 1) & 1u) ^ 1u, abort_flag, budget);
            tc_fence_after();
            return slot;
        };
        // The activations' inverse scales of the slice, read in flush, are visible after this.  It comes before the slice's first
        // step is handed over: until then the barrier cannot be a phase further.
        auto see_scales = [&]() { ok = wait_warp(win0 + kXFull + (cnt & 1u) * 8u, (cnt >> 1) & 1u, abort_flag, budget); };
        // its stores have landed: to the MMA warp.  `st` of `nsteps`: the step inside the slice.  The group before is read back
        // after the first step of a group.
        auto a_done = [&](uint32_t slot, int st, int nsteps) {
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(win0 + kAFull + ((uint32_t)h * 2u + slot) * 8u);
            ++step;
            if (st % C::kGroupSteps == 0) flush();
            if ((st + 1) % C::kGroupSteps == 0 || st + 1 == nsteps) {
                ++grp;
                open = true;
                open_xi = next_xi;
                if (kLut) next_xi += 4u * kXinvGroup;
            }
        };
        for (int tile = first_tile; tile < ntiles && ok; tile += tile_stride) {
            if (h >= halves(tile)) continue;
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] = 0.0f;
            for (int sl = s0; sl < s1 && ok; ++sl, ++cnt) {
                const int ng = groups(sl);
                next_xi = win0 + kXinvOff + (cnt & 3u) * 16u * kXinvGroup;
                if constexpr (kLut) {
                    // Index words and scales of this warp's 32 rows: four atoms.  Scales of the slice and words of one half of it at a time
                    // are held in registers, and the halves are a loop: unrolled over the slice the code outgrows the instruction
                    // cache and the registers leave the scheduler too little to interleave (34816x5120 LUT3 batch 64: 96 us so, 80 this way).
                    uint2 s8[2][2];
                    ok = wait_warp(win0 + kWFull + ((uint32_t)h * 4u + wst) * 8u, wph, abort_flag, budget);
                    if (!ok) break;
                    const uint32_t base = win0 + kRingOff + ((uint32_t)h * S + wst) * C::kStageBytes + (uint32_t)q * 4u * C::kAtom;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int rh = 0; rh < 2; ++rh)
                            s8[j][rh] = lds_v2(base + (uint32_t)(j * 2 + rh) * C::kAtom + (C::kAtom - kLutAtomScaleBytes) + (uint32_t)lane * 8u);
#pragma unroll 1
                    for (int hw = 0; hw < 2 && ok; ++hw) {
                    uint2 w[2][2][BITS];
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int rh = 0; rh < 2; ++rh)
#pragma unroll
                            for (int p = 0; p < BITS; ++p)
                                w[j][rh][p] = lds_v2(base + (uint32_t)(j * 2 + rh) * C::kAtom + (uint32_t)p * 512u + (uint32_t)lane * 16u + (uint32_t)hw * 8u);
                    if (hw == 1) {                          // everything of the stage is in registers
                        __syncwarp();
                        if (lane == 0) mbar_arrive(win0 + kWEmpty + ((uint32_t)h * 4u + wst) * 8u);
                        if (++wst == S) { wst = 0; wph ^= 1u; }
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int wi = 2 * hw + k;
                        if (wi >= ng) continue;
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t slot = 0;
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                uint32_t hi[16], lo[16];
#pragma unroll
                                for (int rh = 0; rh < 2; ++rh) {
                                    uint32_t wd[BITS], sel[4];
#pragma unroll
                                    for (int p = 0; p < BITS; ++p) {
                                        wd[p] = k ? w[j][rh][p].y : w[j][rh][p].x;
                                    }
                                    lut_selectors<BITS>(wd, sel);
                                    // scales of blocks 4 hf .. 4 hf + 3 of the word group: lane wi of the quad holds the group's
                                    const uint32_t sc = __shfl_sync(0xffffffffu, hf ? s8[j][rh].y : s8[j][rh].x, (lane & ~3) | wi);
                                    const uint32_t d01 = e4m3x2_to_f16x2(sc), d23 = e4m3x2_to_f16x2(sc >> 16);
#pragma unroll
                                    for (int b = 0; b < 4; ++b) {
                                        const uint32_t sw = sel[2 * hf + (b >> 1)], u = (b & 1) ? sw >> 16 : sw;
                                        const uint32_t l8 = prmt(cb.tl0, cb.tl1, u), h8 = prmt(cb.th0, cb.th1, u);
                                        const uint32_t g01 = prmt(l8, h8, 0x5140u), g23 = prmt(l8, h8, 0x7362u);
                                        const uint32_t dd = (b & 1) ? both_hi(b < 2 ? d01 : d23) : both_lo(b < 2 ? d01 : d23);
                                        hi[4 * b + 2 * rh] = hmul2(g01, dd);
                                        hi[4 * b + 2 * rh + 1] = hmul2(g23, dd);
                                        lo[4 * b + 2 * rh] = hfms2(g01, dd, hi[4 * b + 2 * rh]);
                                        lo[4 * b + 2 * rh + 1] = hfms2(g23, dd, hi[4 * b + 2 * rh + 1]);
                                    }
                                }
                                if (j == 0) slot = a_slot();
                                if (!ok) break;
                                const uint32_t a = a_cols(h, slot) + lanes + ((uint32_t)(16 * j) << 16);
                                tmem_st_x4(a, hi);
                                tmem_st_x4(a + 32u, lo);
                            }
                            if (!ok) break;
                            if (wi == 0 && hf == 0) { see_scales(); if (!ok) break; }
                            a_done(slot, 2 * wi + hf, 2 * ng);
                            if (!ok) break;
                        }
                        if (!ok) break;
                    }
                    }
                } else {
                    see_scales();
#pragma unroll 1
                    for (int gi = 0; gi < ng && ok; ++gi) {
                        const int part = gi & 1;            // 128-weight group of the ring stage
                        if (part == 0) {
                            ok = wait_warp(win0 + kWFull + ((uint32_t)h * 4u + wst) * 8u, wph, abort_flag, budget);
                            if (!ok) break;
                        }
                        const uint32_t base = win0 + kRingOff + ((uint32_t)h * S + wst) * C::kStageBytes;
                        uint32_t r[2][32];
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int rh = 0; rh < 2; ++rh) {
                                // lane (g, t): weights 32 t .. 32 t + 31 of row g; MMA i contracts weights 4 i .. 4 i + 3 of every lane
                                const uint32_t rr = (uint32_t)(16 * j + 8 * rh + g);
                                const uint4 c = lds_v4(base + (uint32_t)part * 8192u + ((uint32_t)(32 * q) + rr) * 64u + (uint32_t)t * 16u);
                                const uint32_t d2 = e4m3x2_to_f16x2(lds_u16(base + 16384u + (uint32_t)(2 * part + (t >> 1)) * 512u + rr * 16u +
                                                                            (uint32_t)q * 4u + (uint32_t)(t & 1) * 2u));
                                const uint32_t dA = both_lo(d2), dB = both_hi(d2);
                                const uint32_t cw[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                                for (int m = 0; m < 4; ++m) {
                                    uint32_t p[4];
                                    e2m1x8_to_f16(cw[m], p);
                                    const uint32_t dd = m < 2 ? dA : dB;
                                    r[j][8 * m + 2 * rh] = hmul2(p[0], dd);
                                    r[j][8 * m + 2 * rh + 1] = hmul2(p[1], dd);
                                    r[j][8 * m + 4 + 2 * rh] = hmul2(p[2], dd);
                                    r[j][8 * m + 4 + 2 * rh + 1] = hmul2(p[3], dd);
                                }
                            }
                        if (part == 1 || gi + 1 == ng) {    // last group of the stage is in registers
                            __syncwarp();
                            if (lane == 0) mbar_arrive(win0 + kWEmpty + ((uint32_t)h * 4u + wst) * 8u);
                            if (++wst == S) { wst = 0; wph ^= 1u; }
                        }
                        const uint32_t slot = a_slot();
                        if (!ok) break;
                        const uint32_t a = a_cols(h, slot) + lanes;
                        tmem_st_x8(a, r[0]);
                        tmem_st_x8(a + (16u << 16), r[1]);
                        a_done(slot, gi, ng);
                    }
                }
            }
            if (ok) flush();
            if (ok && csize == 1) {
                const int row = tile * 256 + h * 128 + 32 * q + lane;
                if (row < P.N) {
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        if (c < P.cols) P.Y[(int64_t)(P.b0 + c) * P.ldy + row] = __float2bfloat16_rn(acc[c] * s_w);
                }
            }
        }
        if (csize > 1) {
            // One tile per cluster.  Group of four columns i goes to CTA i % csize; everybody's copies, MMAs and reads are over
            // after the first barrier, so the ring and X area takes the partial sums: [source][group of this CTA][256 rows].
            cluster_sync();
            const int per = (NC / 4 + csize - 1) / csize;
            const uint32_t mine = win0 + kRingOff + (uint32_t)((h * 128 + 32 * q + lane) * 16);
            if (first_tile < ntiles && h < halves(first_tile)) {
#pragma unroll
                for (int i = 0; i < NC / 4; ++i)
                    st_cluster_v4(mine + (uint32_t)((int)rank * per + i / csize) * 4096u, (uint32_t)(i % csize),
                                  make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]));
            }
            cluster_sync();
            const int row = first_tile * 256 + h * 128 + 32 * q + lane;
            if (ok && row < P.N && first_tile < ntiles) {
                for (int i = (int)rank, l = 0; i < NC / 4 && 4 * i < P.cols; i += csize, ++l) {
                    float4 tot = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    for (int src = 0; src < csize; ++src) {
                        const uint4 v = lds_v4(mine + (uint32_t)(src * per + l) * 4096u);
                        tot.x += __uint_as_float(v.x); tot.y += __uint_as_float(v.y);
                        tot.z += __uint_as_float(v.z); tot.w += __uint_as_float(v.w);
                    }
                    __nv_bfloat16 *y = P.Y + (int64_t)(P.b0 + 4 * i) * P.ldy + row;
                    y[0] = __float2bfloat16_rn(tot.x * s_w);
                    if (4 * i + 1 < P.cols) y[P.ldy] = __float2bfloat16_rn(tot.y * s_w);
                    if (4 * i + 2 < P.cols) y[2 * P.ldy] = __float2bfloat16_rn(tot.z * s_w);
                    if (4 * i + 3 < P.cols) y[3 * P.ldy] = __float2bfloat16_rn(tot.w * s_w);
                }
            }
        }
    } else if (warp < 12) {
        // ============================================================ activations
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        asm volatile("griddepcontrol.wait;" ::: "memory");       // X may come from the kernel ahead
        const int sw = warp - 8;
        bool ok = true;
        uint32_t cnt = 0;
        for (int tile = first_tile; tile < ntiles && ok; tile += tile_stride) {
            for (int sl = s0; sl < s1; ++sl, ++cnt) {
                ok = wait_warp(win0 + kXEmpty + (cnt & 1u) * 8u, ((cnt >> 1) & 1u) ^ 1u, abort_flag, budget);
                if (!ok) break;
                const uint32_t xb = win0 + C::kXOff + (cnt & 1u) * C::kXBytes;
                const int live = groups(sl) * 16;            // 16-byte pieces (8 weights) of a column inside K
                uint32_t top = 0;                                // largest magnitude of the warp's columns
                // four columns at a time: eight loads in flight per lane
                for (int c0 = sw; c0 < P.cols; c0 += 16) {
                    uint4 v[4][2];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = c0 + 4 * u;
                        const uint4 *xp = reinterpret_cast<const uint4 *>(P.X + (int64_t)(P.b0 + (c < P.cols ? c : c0)) * P.ldx + sl * kSlice);
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            v[u][i] = (lane + 32 * i < live && c < P.cols) ? __ldg(xp + lane + 32 * i) : make_uint4(0u, 0u, 0u, 0u);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = c0 + 4 * u;
                        if (c >= P.cols) break;
                        uint32_t m = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(v[u][0].x, v[u][0].y), max_abs_bf16x2(v[u][0].z, v[u][0].w)),
                                                    max_abs_bf16x2(max_abs_bf16x2(v[u][1].x, v[u][1].y), max_abs_bf16x2(v[u][1].z, v[u][1].w)));
                        m &= 0x7FFF7FFFu;
                        m = __reduce_max_sync(0xffffffffu, max(m >> 16, m & 0xFFFFu));
                        top = max(top, m);
                        const int ex = max(-100, (int)(m >> 7) - 127);              // floor(log2(max)); -127 for zero / subnormal
                        const float xscale = __uint_as_float((uint32_t)(127 + 14 - ex) << 23);   // 2^(14 - ex)
                        if (lane < (kLut ? 4 : 1)) xinv_s[((cnt & 3u) * 4u + (uint32_t)lane) * kXinvGroup + c] = __uint_as_float((uint32_t)(127 - 14 + ex) << 23);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const uint32_t ww[4] = {v[u][i].x, v[u][i].y, v[u][i].z, v[u][i].w};
                            uint32_t r[4];
#pragma unroll
                            for (int z = 0; z < 4; ++z) {
                                const __half2 hh = __floats2half2_rn(__uint_as_float(ww[z] << 16) * xscale,
                                                                     __uint_as_float(ww[z] & 0xFFFF0000u) * xscale);
                                r[z] = *reinterpret_cast<const uint32_t *>(&hh);
                            }
                            const uint32_t p = (uint32_t)(lane + 32 * i);           // piece: weights 8 p .. 8 p + 7 of the slice
                            const uint32_t col = xb + (uint32_t)c * 16u;
                            if (kLut) {
                                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                                             ::"r"(col + p * C::kXStride), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
                            } else {
                                // weights 32 tt + 4 ii .. + 3 of a 128-weight group are contracted by MMA ii, slots 4 tt ..
                                const uint32_t ii = 2u * (p & 3u), tt = (p >> 2) & 3u, grp = p >> 4;
                                const uint32_t a = col + (grp * 16u + ii * 2u + (tt >> 1)) * C::kXStride + (tt & 1u) * 8u;
                                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(r[0]), "r"(r[1]) : "memory");
                                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + 2u * C::kXStride), "r"(r[2]), "r"(r[3]) : "memory");
                            }
                        }
                    }
                }
                if (kLut && top >= 0x7F80u)
                    stage_infinite(P.X + (int64_t)P.b0 * P.ldx + sl * kSlice, P.ldx, sw, P.cols, live, xb, C::kXStride,
                                   xinv_s + (cnt & 3u) * 4u * kXinvGroup);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");        // the tensor cores read them
                __syncwarp();
                if (lane == 0) mbar_arrive(win0 + kXFull + (cnt & 1u) * 8u);
            }
        }
        if (csize > 1) { cluster_sync(); cluster_sync(); }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
        if (warp == 12) {
            // ======================================================== MMA issue
            // One elected thread for the whole role: with loop, waits and operands inside the branch they are uniform to the compiler
            // and an MMA costs its N / 2 cycles.  With the warp walking the loop and only the MMAs elected every operand
            // is moved to a uniform register first, 45 cycles an MMA, and this role sets the pace
            // (34816x5120 NVFP4 batch 16: 36.0 us so, 32.9 this way).
            if (elect_one()) {
                bool ok = true;
                uint32_t cnt = 0, step = 0, grp = 0;
                for (int tile = first_tile; tile < ntiles && ok; tile += tile_stride) {
                    const int nh = halves(tile);
                    // A last tile without a second half: that half's warps may still be reading the tile before back, with inverse scales
                    // whose place the activations of the fourth slice from then on take.  Steps of half 0 alone would not hold them off.
                    if (nh == 1 && grp > 0) {
                        const uint32_t n = grp - 1u;
                        ok = wait_one(win0 + kDEmpty + ((n & 1u) * 2u + 1u) * 8u, (n >> 1) & 1u, abort_flag, budget);
                    }
                    for (int sl = s0; sl < s1 && ok; ++sl, ++cnt) {
                        const uint32_t xb = cnt & 1u;
                        ok = wait_one(win0 + kXFull + xb * 8u, (cnt >> 1) & 1u, abort_flag, budget);
                        const uint64_t b0 = make_desc_plain(win0 + C::kXOff + xb * C::kXBytes, C::kXStride, 128u);
                        const int nsteps = groups(sl) * (128 / C::kStepK);
                        for (int st = 0; st < nsteps && ok; ++st, ++step) {
                            const uint32_t slot = step & 1u, db = grp & 1u;
                            const bool first = st % C::kGroupSteps == 0, last = (st + 1) % C::kGroupSteps == 0 || st + 1 == nsteps;
                            // 16 weights of X: two pieces of kXStride bytes
                            const uint64_t b = b0 + (uint64_t)((uint32_t)(st * (C::kStepK / 16)) * ((2u * C::kXStride) >> 4));
                            for (int h = 0; h < nh && ok; ++h) {
                                if (first) ok = wait_one(win0 + kDEmpty + (db * 2u + (uint32_t)h) * 8u, ((grp >> 1) & 1u) ^ 1u, abort_flag, budget);
                                if (ok) ok = wait_one(win0 + kAFull + ((uint32_t)h * 2u + slot) * 8u, (step >> 1) & 1u, abort_flag, budget);
                                if (!ok) break;
                                tc_fence_after();
                                const uint32_t a = a_cols(h, slot), d = d_cols(db, h);
#pragma unroll
                                for (int i = 0; i < C::kStepK / 16; ++i) {
                                    const uint64_t bi = b + (uint64_t)((uint32_t)i * ((2u * C::kXStride) >> 4));
                                    mma_f16_ts(d, a + 8u * i, bi, C::kIdesc, !first || i > 0);
                                    if (kLut) mma_f16_ts(d, a + 32u + 8u * i, bi, C::kIdesc, true);
                                }
                                mma_commit(win0 + kAEmpty + ((uint32_t)h * 2u + slot) * 8u);
                                if (last) mma_commit(win0 + kDFull + (db * 2u + (uint32_t)h) * 8u);
                            }
                            if (ok && st + 1 == nsteps) mma_commit(win0 + kXEmpty + xb * 8u);
                            if (last) ++grp;
                        }
                    }
                }
            }
            __syncwarp();
        } else if (warp == 13) {
            // ======================================================== weights
            bool ok = true;
            uint32_t st = 0, ph = 0;
            bool drop = P.drop_first_copy && blockIdx.x == 0;
            for (int tile = first_tile; tile < ntiles && ok; tile += tile_stride) {
                const int nh = halves(tile);
                for (int sl = s0; sl < s1 && ok; ++sl) {
                    const int nst = kLut ? 1 : (groups(sl) + 1) / 2;
                    for (int sub = 0; sub < nst && ok; ++sub) {
                        for (int h = 0; h < nh; ++h) {
                            const uint32_t full = win0 + kWFull + ((uint32_t)h * 4u + st) * 8u;
                            ok = wait_warp(win0 + kWEmpty + ((uint32_t)h * 4u + st) * 8u, ph ^ 1u, abort_flag, budget);
                            if (!ok) break;
                            const uint32_t dst = win0 + kRingOff + ((uint32_t)h * S + st) * C::kStageBytes;
                            if (drop) { drop = false; continue; }
                            if constexpr (kLut) {
                                // 16 atoms: 8 rows x 512 weights each, lanes 0 .. 15 request one each
                                const int t16 = tile * 16 + h * 8 + (lane >> 1), n16 = P.N >> 4;
                                const int have = min(8, n16 - (tile * 16 + h * 8)) * 2;
                                if (lane == 0) mbar_expect_tx(full, (uint32_t)have * C::kAtom);
                                __syncwarp();
                                if (lane < have) {
                                    const size_t atom = (((size_t)t16 * ((P.K + kLutSlice - 1) / kLutSlice) + (sl >> 1)) * 2 + (lane & 1)) * 2 + (sl & 1);
                                    bulk_load(dst + (uint32_t)lane * C::kAtom, P.weights + atom * C::kAtom, C::kAtom, full);
                                }
                                __syncwarp();
                            } else {
                                const int left = groups(sl) - 2 * sub;                      // 128-weight groups of this stage
                                const int katom = sl * (kSlice / 64) + sub * 4, katoms = P.K / 64;
                                const uint32_t sfb = (uint32_t)min(4, katoms - katom) * 512u;
                                const int band = tile * 2 + h;
                                if (elect_one()) {
                                    mbar_expect_tx(full, (left > 1 ? 16384u : 8192u) + sfb);
                                    tma_load_2d(dst, &tmap, katom * 32, band * 128, full);
                                    if (left > 1) tma_load_2d(dst + 8192u, &tmap, katom * 32 + 64, band * 128, full);
                                    bulk_load(dst + 16384u, P.sf + ((size_t)band * katoms + katom) * 512, sfb, full);
                                }
                                __syncwarp();
                            }
                        }
                        if (++st == S) { st = 0; ph ^= 1u; }
                    }
                }
            }
        }
        if (csize > 1) { cluster_sync(); cluster_sync(); }
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // a wait ran out: let copies in flight land before the CTA's shared memory is handed on, then report
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        if (threadIdx.x == 0) {
            atomicExch(&P.status->status, (int)DQ_ERR_TIMEOUT);
            atomicExch(&P.status->detail, 0x3A000 | (int)blockIdx.x);
        }
        __syncthreads();
    }
    if (warp == 12) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}


typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// NVFP4 codes as a byte matrix [N][K/2]; box = 64 bytes (128 weights) x 128 rows, unswizzled, zero fill outside
bool make_codes_tmap(CUtensorMap *tm, const void *ptr, int64_t N, int64_t K)
{
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(gemm_encode_fn());
    if (!enc) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)(K / 2), (cuuint64_t)N};
    cuuint64_t gstride[1] = {(cuuint64_t)(K / 2)};
    cuuint32_t box[2] = {64u, 128u};
    cuuint32_t estr[2] = {1u, 1u};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(ptr), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kMaxCluster = 8;

template <int FMT, int NC>
cudaError_t set_attributes(int dev)
{
    static std::atomic<bool> done[kMaxDevices];
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    auto kernel = decode_tc_kernel<FMT, NC>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<FMT, NC>::kSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return e;
}

template <int FMT, int NC>
cudaLaunchConfig_t launch_config(cudaLaunchAttribute (&attr)[2], int grid, int csize, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<FMT, NC>::kSmem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)csize;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = csize > 1 ? 2 : 1;
    return cfg;
}

// How many clusters of c CTAs a device holds at once: they do not straddle its groups of SMs, so some SMs stay out, on a B200 28 of
// them at eight CTAs.  Every instantiation has an SM to itself, so one answers for all; asked once per size and device, and
// again where the runtime did not answer.
int clusters_that_fit(int dev, int c, int sms)
{
    static std::atomic<int> known[kMaxDevices][kMaxCluster + 1];                 // + 1; 0 = not known
    int fit = known[dev][c].load(std::memory_order_relaxed);
    if (fit == 0) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = launch_config<0, 16>(attr, c * (sms / c), c, nullptr);
        int n = 0;
        if (set_attributes<0, 16>(dev) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, decode_tc_kernel<0, 16>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        fit = n + 1;
        known[dev][c].store(fit, std::memory_order_relaxed);
    }
    return fit - 1;
}

// CTAs per tile: the fewest slices of 512 weights on the busiest CTA, a cluster's exchange counted as half a slice.  Clusters take one
// tile each and must all be resident.
struct TileSplit { int csize; double slices; };
TileSplit split_tiles(int64_t N, int64_t K, int dev, int sms, int force_csize)
{
    const int64_t tiles = (N + 255) / 256, ns = (K + kSlice - 1) / kSlice;
    TileSplit best = {1, (double)((tiles + sms - 1) / sms) * (double)ns};
    for (int c = 2; c <= kMaxCluster && c <= ns && tiles * c <= sms; ++c) {
        if (force_csize > 0 && c != force_csize) continue;
        const double cost = (double)((ns + c - 1) / c) + 0.5;
        if ((force_csize > 0 || cost < best.slices) && tiles <= clusters_that_fit(dev, c, sms)) best = {c, cost};
    }
    return best;
}

template <int FMT, int NC>
cudaError_t launch_one(const CUtensorMap &tmap, TcDecodeArgs P, int force_csize, cudaStream_t stream)
{
    const DeviceInfo *di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    const cudaError_t e = set_attributes<FMT, NC>(di->device);
    if (e != cudaSuccess) return e;
    const int tiles = (P.N + 255) / 256;
    P.csize = split_tiles(P.N, P.K, di->device, di->sms, force_csize).csize;
    if (force_csize > 0 && P.csize != force_csize) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config<FMT, NC>(attr, P.csize > 1 ? tiles * P.csize : (tiles < di->sms ? tiles : di->sms), P.csize, stream);
    return cudaLaunchKernelEx(&cfg, decode_tc_kernel<FMT, NC>, tmap, P);
}

template <int FMT>
cudaError_t launch_cols(const CUtensorMap &tmap, const TcDecodeArgs &P, int force_csize, cudaStream_t stream)
{
    if (P.cols <= 16) return launch_one<FMT, 16>(tmap, P, force_csize, stream);
    if (P.cols <= 32) return launch_one<FMT, 32>(tmap, P, force_csize, stream);
    if (P.cols <= 48) return launch_one<FMT, 48>(tmap, P, force_csize, stream);
    return launch_one<FMT, 64>(tmap, P, force_csize, stream);
}

}  // namespace

// 512-weight slices the busiest CTA of a launch works through, an exchange included.  crowded: clusters of three or five, all or all but one
// that fit: a slice then takes 2.8 to 4.1 us instead of 2.6 (NVFP4, 11296x2816, 45 clusters of three: 11.6; not seen at other sizes)
double decode_tc_slices(int64_t N, int64_t K, bool *crowded)
{
    const DeviceInfo *di = device_info();
    if (!di) return 1e300;
    const TileSplit t = split_tiles(N, K, di->device, di->sms, 0);
    if (crowded) *crowded = (t.csize == 3 || t.csize == 5) && (N + 255) / 256 >= clusters_that_fit(di->device, t.csize, di->sms) - 1;
    return t.slices;
}

cudaError_t launch_decode_tc(const GemvArgs &a, cudaStream_t stream)
{
    TcDecodeArgs P = {};
    P.weights = a.lut;
    P.hdr = a.hdr;
    P.X = reinterpret_cast<const __nv_bfloat16 *>(a.X);
    P.Y = reinterpret_cast<__nv_bfloat16 *>(a.Y);
    P.ldx = a.ldx;
    P.ldy = a.ldy;
    P.cols = (int)a.B;
    P.N = (int)a.N;
    P.K = (int)a.K;
    P.wait_cycles = a.wait_cycles > 0 ? a.wait_cycles : kWaitBudgetCycles;
    P.drop_first_copy = a.drop_first_copy;
    P.status = a.status;
    const CUtensorMap none = {};
    return a.bits == 3 ? launch_cols<3>(none, P, a.force_P, stream) : launch_cols<2>(none, P, a.force_P, stream);
}

cudaError_t launch_decode_tc_nvfp4(const GemvNvArgs &a, int force_csize, cudaStream_t stream)
{
    if (gemm_init_driver_api() != 0) return cudaErrorNotSupported;
    CUtensorMap tmap;
    if (!make_codes_tmap(&tmap, a.codes, a.N, a.K)) return cudaErrorInvalidValue;
    TcDecodeArgs P = {};
    P.sf = a.sf;
    P.hdr = a.hdr;
    P.X = reinterpret_cast<const __nv_bfloat16 *>(a.X);
    P.Y = reinterpret_cast<__nv_bfloat16 *>(a.Y);
    P.ldx = a.ldx;
    P.ldy = a.ldy;
    P.cols = (int)a.B;
    P.N = (int)a.N;
    P.K = (int)a.K;
    P.wait_cycles = kWaitBudgetCycles;
    P.status = a.status;
    return launch_cols<0>(tmap, P, force_csize, stream);
}

}  // namespace dq

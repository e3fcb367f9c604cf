// Weight-only decode on the NVFP4 view (NVFP4A16, Sec. 2.3 / Table 1) through the block-scaled FP4 tensor cores, up to 16 batch
// columns: the stored matrix is the MMA's operand as it lies in HBM, nothing of it is dequantised.
//   Y[b][n] = bf16( s * sum_blk d_blk(n) * sum_{k in blk} e2m1(n,k) * X[b][k] )
//
// Arithmetic.  A bf16 activation is written in twelve digits of base 8 between -4 and 4, whose halves E2M1 holds exactly, under its 16-block's
// power of two: x = 2^(E_blk - 128) sum_p digit_p 8^-p.  E_blk is the largest exponent of the block: the digits hold every element
// within 2^27 of the block's largest exactly and round the rest to 2^-35 of it.  E4M3 block scales carry 2^E_blk relative to the largest of
// the column's 2048 weights (a group), down to 2^-17 of it; blocks below share that exponent (2^-52 of the group's largest).  A batch
// column thus becomes twelve columns of the MMA's other operand.  Products and block scales are exact; the tensor cores sum a group
// (32 instructions, as many as one of decode_tc_kernel's), its twelve sums are put together and added to the running sum by FMA in
// fp32 with the powers of two of the group and, as far as fp32's range allows (scale_exponent), of the tensor scale: without that,
// finite outputs of activations of 2^104 and more were lost.  An infinity or a NaN: the group's products with it, one by one (special_sum).
//
// Work split.  A tile is 256 rows in two halves, the tensor-memory lanes; a step 256 weights.  Where there are too few tiles for the chip
// a cluster of up to 8 CTAs shares one, each taking a range of steps; at the end they exchange partial sums through distributed
// shared memory, every CTA adding a share of the columns in rank order.  One CTA per SM:
//   warp 0     : weights and their scales, TMA and bulk copies into a ring of stages
//   warp 1     : scale copies to tensor memory, tcgen05.mma (M = 128, N = 48 per four columns, K = 64)
//   warps 2-9  : read finished groups back and store the output.  Up to four columns they also make the digits, in the ring's stages, two
//                warps a column in turns.  From five columns on that work, which every tile would repeat, sets the pace (28672x8192 batch 8
//                38.5 us, batch 16 70): there fp4_digits_kernel writes the digits to a workspace once (27.3, 35.1).
//
// Bound by HBM by intent, 5.4 TB/s for a kernel that only reads: a step's MMAs and scale copies take 700 to 1200 cycles, its weights' way from
// HBM 1400 to 1600.  28672x8192: batch 1 27.7 us (36.2 with the mma.sync kernel), batch 4 29.5 (40.1 with decode_tc_kernel), batch 8 27.3 (45.0),
// batch 16 35.1 (46.1); 17408x5120 batch 1 12.0 (14.9); 5120x17408 12.9 (20.1); 2048x2048 5.0 (6.1).  Ring waits are parked in hardware: polling
// took issue slots from the warps that make digits.
#include <atomic>

#include <cuda.h>

#include "dq_common.cuh"
#include "dq_quant.cuh"
#include "dq_tcgen05.cuh"

namespace dq {

namespace {

using namespace tc;

constexpr int kDigits = 12;
constexpr int kGroupSteps = 8;                     // steps summed by the tensor cores
constexpr int kMaxCluster = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kDigitsSmem = 100 * 1024;       // of a CTA of the digits' kernel, which needs none: launched early it would be packed onto the first
                                                   // few SMs that fall free, sixteen CTAs each, and take 9 us instead of 3
constexpr uint32_t kHeadBytes = 1024;              // barriers and scales

// NG: groups of four batch columns, 48 columns of the MMA each; PRE: the digits come from a workspace
template <int NG, bool PRE>
struct Cfg {
    static constexpr int NCOL = 48 * NG;
    static constexpr int kAtoms = (NCOL + 127) / 128;                          // scale atoms of the digits per 64 weights
    static constexpr uint32_t A_BYTES = 32768u, SFA_BYTES = 4096u, B_BYTES = NCOL * 128u, SFB_BYTES = kAtoms * 2048u;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + SFA_BYTES + B_BYTES + SFB_BYTES;
    static constexpr int kFit = (int)((227u * 1024u - 1024u - kHeadBytes) / STAGE_BYTES), S = kFit < 5 ? kFit : 5;
    static constexpr uint32_t SMEM_BYTES = 1024u /*align*/ + kHeadBytes + S * STAGE_BYTES;
    static constexpr uint32_t kDStride = NG == 1 ? 64u : (uint32_t)NCOL;       // accumulator columns of a half
    static constexpr int kAccs = NG <= 2 ? 2 : 1;                              // a group's sums are read while the next one's are made, where they fit
    static constexpr uint32_t kSfBase = kAccs * 2 * kDStride, kSfCols = 32u + 16u * kAtoms;        // two buffers of scales
    static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | ((uint32_t)(NCOL >> 3) << 17) | ((128u >> 4) << 24);
    static constexpr uint32_t X_BYTES = B_BYTES + SFB_BYTES;                   // a step's digits and scales
    static constexpr int kWorkers = 8, kThreads = 64 + 32 * kWorkers;          // warps
    static constexpr int kPerCol = 2;                                          // warps that share a column where they make the digits, step by step
    static_assert(PRE || kPerCol * 4 * NG == kWorkers, "a column per two warps");
    static_assert(S < kGroupSteps, "the scales' slots rely on a full group being longer than the ring");
    static_assert(S >= 3 && STAGE_BYTES % 1024 == 0 && kSfBase + 2 * kSfCols <= kTmemCols, "shared memory, tensor memory");
    static_assert((NG + kMaxCluster) * 4096u <= S * STAGE_BYTES, "partial sums of a cluster must fit the ring");
};

// head of shared memory: barriers, 8 bytes each; then the groups' scales
enum : uint32_t {
    kFull = 0,                   // [S <= 5] weights
    kXFull = 64,                 // [5] digits
    kEmpty = 128,                // [5]
    kDFull = 168,                // [2]
    kDEmpty = 184,               // [2]
    kTmemPtr = 208,
    kAbort = 212,
    kScales = 256,               // [kSlots groups][16 columns] float
    kSpecial = 512,              // [kSlots][16] int: the column's group holds an infinity or a NaN
};
// Groups whose scales and flags are held where the CTAs make the digits: group n's lie in slot n % 3.  They are written with the group's first
// step, when the writer has read the sums of group n - 2, and of n - 1 too where n begins a tile.  Every warp has then read slot n - 3:
//   n begins a tile: the sums of n - 1 exist, so every warp has handed over the first step of n - 1, and reads the sums of n - 3 before that;
//   n does not: n - 1 has eight steps, more than the ring, so the stage that the writer got last held one of its steps but the first.
// Two slots are not enough: group n - 2 is read after the first step of n - 1, which may be the only one (rows of 17, 25, .. steps).
constexpr uint32_t kSlots = 3;

struct Fp4Args {
    const uint8_t *codes, *w_sf;
    const PackedHeader *hdr;
    const __nv_bfloat16 *X;
    __nv_bfloat16 *Y;
    int64_t ldx, ldy;
    int cols, N, K;
    int csize;                   // CTAs that share a tile
    // PRE: the workspace
    uint8_t *digits;             // [steps][X_BYTES]
    uint32_t *group_scale;       // [groups][16 columns] fp32 bits, then the same number of flags: an infinity or a NaN
    int ngroups;
    long long wait_cycles;
    int drop_first_copy;         // test hook: the weights of CTA 0's first step are never requested
    StatusWord *status;
};

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// Digits of eight activations of a block whose largest exponent is eb, the highest first: w[p] holds those of 8^-p, a nibble each.  In bf16
// all of it is exact: a value between -4 and 4 plus 192 is rounded to a whole number, which is the digit; eight times what is left
// is the next value, and never has more than the activation's eight bits.  192 + d has d, as a two's complement nibble, at its low
// end; E2M1 has the halves of -4 .. 4 as sign and magnitude.  Two activations (i and i + 4) share a word: three multiply-adds a digit and
// pair, five operations to put four pairs in order and five to change the sign's form (with the bits cut out of integers and digits looked
// up, four at a time, this was twice as long).
__device__ __forceinline__ void make_digits(const uint4 x, int eb, uint32_t (&w)[kDigits])
{
    const uint32_t k192 = 0x43404340u, k1 = 0x3F803F80u, km1 = 0xBF80BF80u, k8 = 0x41004100u;
    const uint32_t s2 = (uint32_t)(255 - eb) * 0x00800080u;       // 2^(1 - E): the largest is below 4
    uint32_t t[4] = {prmt(x.x, x.z, 0x5410u), prmt(x.x, x.z, 0x7632u), prmt(x.y, x.w, 0x5410u), prmt(x.y, x.w, 0x7632u)};
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = fma_bf16x2(t[i], s2, 0x80008000u);
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        uint32_t f[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[i] = fma_bf16x2(t[i], p ? k8 : k1, k192);
            if (p + 1 < kDigits) t[i] = fma_bf16x2(t[i], p ? k8 : k1, fma_bf16x2(f[i], km1, k192));
        }
        const uint32_t a = (f[0] & 0x0F0F0F0Fu) | ((f[1] << 4) & 0xF0F0F0F0u), b = (f[2] & 0x0F0F0F0Fu) | ((f[3] << 4) & 0xF0F0F0F0u);
        const uint32_t n = prmt(a, b, 0x6240u), sign = n & 0x88888888u, one = sign >> 3;
        w[p] = ((n ^ (sign - one)) & 0x77777777u) + one + sign;
    }
}
// the larger magnitude, per half; the sign is of no use
__device__ __forceinline__ uint32_t max_abs_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.NaN.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t max_magnitude(uint32_t two)       // bf16 bits of the larger half
{
    const uint32_t m = two & 0x7FFF7FFFu;
    return max(m >> 16, m & 0xFFFFu);
}
__device__ __forceinline__ uint32_t max_abs_of(uint4 v) { return max_abs_bf16x2(max_abs_bf16x2(v.x, v.y), max_abs_bf16x2(v.z, v.w)); }

// fp32 bits of a group's power of two, 2^(eg - 135) with eg the largest exponent; a subnormal for the smallest.  0 beside infinities and NaN:
// no sums of the tensor cores
__device__ __forceinline__ uint32_t scale_of_group(uint32_t top, int eg) { return top >= 0x7F80u ? 0u : eg >= 9 ? (uint32_t)(eg - 8) << 23 : 1u << (eg + 14); }
// The part of a tensor scale's power of two, 2^e, that goes with the groups' scales: their product is a number of fp32 whatever the group.  The
// scale is looked at here and not before: it comes from memory, and the first digits are not to wait for it.
__device__ __forceinline__ int scale_exponent(float s)
{
    asm volatile("" : "+f"(s));
    return max(-15, min(8, (int)((__float_as_uint(s) >> 23) & 255u) - 127));
}
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }
// Digits and block scales of a lane's eight activations x; lanes 2i and 2i + 1 share a block, eight lanes the word of four scales
__device__ __forceinline__ void digits_and_scales(const uint4 x, int eg, uint32_t (&w)[kDigits], uint32_t &sf)
{
    const int lane = threadIdx.x & 31;
    uint32_t bm = max_magnitude(max_abs_of(x));
    bm = max(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
    const int eb = max(max((int)(bm >> 7), 1), eg - 17);
    // the block scale is 2^(eb - eg + 8), 2^-9 .. 2^8
    sf = f32_to_e4m3(__uint_as_float((uint32_t)(eb - eg + 135) << 23)) << (8 * ((lane >> 1) & 3));
    sf |= __shfl_xor_sync(0xffffffffu, sf, 2);
    sf |= __shfl_xor_sync(0xffffffffu, sf, 4);
    make_digits(x, eb, w);
}

// Digits of a call to its workspace, as the stages of decode_fp4_kernel want them: grid (groups, columns padded to 16), a warp per step.
// What the batch does not have, and what lies beyond a row's end, becomes zeros.
__global__ void __launch_bounds__(32 * kGroupSteps) fp4_digits_kernel(const __grid_constant__ Fp4Args P, uint32_t x_bytes, uint32_t b_bytes)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");       // X may come from the kernel ahead, which may also still read the workspace
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int group = blockIdx.x, col = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int step = group * kGroupSteps + warp, k = step * 256 + lane * 8;
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (col < P.cols && k < P.K) x = __ldg(reinterpret_cast<const uint4 *>(P.X + (int64_t)col * P.ldx + k));
    __shared__ uint32_t red[kGroupSteps];
    uint32_t top = __reduce_max_sync(0xffffffffu, max_magnitude(max_abs_of(x)));
    if (lane == 0) red[warp] = top;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kGroupSteps; ++i) top = max(top, red[i]);
    const int eg = max((int)(top >> 7), 1);
    if (threadIdx.x == 0) {
        P.group_scale[group * 16 + col] = scale_of_group(top, eg);
        P.group_scale[(P.ngroups + group) * 16 + col] = top >= 0x7F80u;
    }
    if (step * 256 >= P.K) return;
    if (top >= 0x7F80u) x = make_uint4(0u, 0u, 0u, 0u);
    uint32_t w[kDigits], sf;
    digits_and_scales(x, eg, w, sf);
    uint8_t *blk = P.digits + (size_t)step * x_bytes;
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
        const uint32_t n = (uint32_t)(col * kDigits + p);
        *reinterpret_cast<uint32_t *>(blk + n * 128u + ((((uint32_t)lane >> 2) ^ (n & 7u)) << 4) + ((uint32_t)lane & 3u) * 4u) = w[p];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const uint32_t p = ((uint32_t)lane & 7u) + 8u * u, n = (uint32_t)col * kDigits + p, r = n & 127u;
        if (p < kDigits) *reinterpret_cast<uint32_t *>(blk + b_bytes + (n >> 7) * 2048u + ((uint32_t)lane >> 3) * 512u + (r & 31u) * 16u + (r >> 5) * 4u) = sf;
    }
}

// The infinities and NaN of weights k0 .. k1 - 1 of a column times the row's weights; beside them the finite rest of the sum does not matter,
// nor does the magnitude of a weight.
__device__ __noinline__ float special_sum(const uint8_t *codes, const uint8_t *w_sf, const __nv_bfloat16 *x, int row, int k0, int k1, int K)
{
    float sum = 0.0f;
    for (int k = k0; k < k1; ++k) {
        const uint32_t h = reinterpret_cast<const uint16_t *>(x)[k];
        if ((h & 0x7F80u) != 0x7F80u) continue;
        const uint32_t code = codes[(int64_t)row * (K / 2) + (k >> 1)] >> (4 * (k & 1));
        const bool zero = (code & 7u) == 0u || (w_sf[sf_swizzled_offset(row, k >> 4, K)] & 0x7Fu) == 0u;
        sum += (zero ? 0.0f : (code & 8u) ? -1.0f : 1.0f) * __uint_as_float(h << 16);
    }
    return sum;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
                   "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr) : "memory");
}
// Bounded waits whose time hint parks the thread in hardware until the phase completes
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
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t rank, float a, float b, float c, float d)
{
    asm volatile("{\n\t.reg .b32 p;\n\tmapa.shared::cluster.u32 p, %0, %1;\n\tst.shared::cluster.v4.f32 [p], {%2, %3, %4, %5};\n\t}"
                 ::"r"(addr), "r"(rank), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
template <int OFF>
__device__ __forceinline__ void sts_u32_at(uint32_t base, uint32_t v) { asm volatile("st.shared.b32 [%0+%1], %2;" ::"r"(base), "n"(OFF), "r"(v) : "memory"); }
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

template <int NG, bool PRE>
__global__ void __launch_bounds__(Cfg<NG, PRE>::kThreads, 1)
decode_fp4_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ Fp4Args P)
{
    using C = Cfg<NG, PRE>;
    constexpr int S = C::S;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t win0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (win0 - smem_u32(smem_raw));
    const uint32_t ring0 = win0 + kHeadBytes;                 // per stage: weights, their scales, digits, their scales
    auto full_bar = [&](int s) { return win0 + kFull + 8u * s; };
    auto xfull_bar = [&](int s) { return win0 + kXFull + 8u * s; };
    auto empty_bar = [&](int s) { return win0 + kEmpty + 8u * s; };
    auto dfull_bar = [&](uint32_t group) { return win0 + kDFull + 8u * (group % C::kAccs); };
    auto dempty_bar = [&](uint32_t group) { return win0 + kDEmpty + 8u * (group % C::kAccs); };
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kAbort);
    float *scales = reinterpret_cast<float *>(smem + kScales);
    int *specials = reinterpret_cast<int *>(smem + kSpecial);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(xfull_bar(s), C::kWorkers); mbar_init(empty_bar(s), 1); }
        for (uint32_t i = 0; i < 2; ++i) { mbar_init(win0 + kDFull + 8u * i, 1); mbar_init(win0 + kDEmpty + 8u * i, 8); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(win0 + kTmemPtr), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (!PRE) {
        // digits of the columns the batch does not have stay zero
        for (uint32_t i = threadIdx.x; i < S * (C::X_BYTES / 16u); i += C::kThreads) {
            const uint32_t st = i / (C::X_BYTES / 16u), at = i % (C::X_BYTES / 16u);
            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(ring0 + st * C::STAGE_BYTES + C::A_BYTES + C::SFA_BYTES + at * 16u), "r"(0u) : "memory");
        }
        if (threadIdx.x < 16 * kSlots) { scales[threadIdx.x] = 0.0f; specials[threadIdx.x] = 0; }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + kTmemPtr);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int csize = P.csize;
    const uint32_t rank = csize > 1 ? cluster_ctarank() : 0u;
    const int first_tile = (int)blockIdx.x / csize, tile_stride = (int)gridDim.x / csize;
    const int tiles = (P.N + 255) >> 8, ksteps = (P.K + 255) >> 8, katoms = P.K / 64;
    const int k0 = (int)((long long)ksteps * rank / csize), k1 = (int)((long long)ksteps * (rank + 1) / csize);

    if (warp == 0) {
        // -------------------------- weights: constant data, nothing to wait for; digits that the kernel ahead has made
        if (elect_one()) {
            bool drop = P.drop_first_copy && blockIdx.x == 0;
            auto load_w = [&](int stage, int tile, int ks) {
                const uint32_t a = ring0 + stage * C::STAGE_BYTES, sf = (uint32_t)min(4, katoms - 4 * ks) * 512u;
                mbar_expect_tx(full_bar(stage), C::A_BYTES + 2u * sf + (PRE ? C::X_BYTES : 0u));
                if (!drop) tma_load_2d(a, &tmap_w, ks * 128, tile * 256, full_bar(stage));
                drop = false;
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    bulk_load(a + C::A_BYTES + h * 2048u, P.w_sf + ((size_t)(tile * 2 + h) * katoms + (size_t)ks * 4) * 512, sf, full_bar(stage));
            };
            int early = 0;
            if (PRE) {
                if (first_tile < tiles) {
                    early = min(S, k1 - k0);
                    for (int i = 0; i < early; ++i) load_w(i, first_tile, k0 + i);
                }
                asm volatile("griddepcontrol.wait;" ::: "memory");
            }
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int tile = first_tile; tile < tiles && ok; tile += tile_stride) {
                for (int ks = k0; ks < k1; ++ks) {
                    if (PRE && early > 0) {
                        --early;
                    } else {
                        ok = wait_one(empty_bar(stage), phase ^ 1u, abort_flag, P.wait_cycles);
                        if (!ok) break;
                        load_w(stage, tile, ks);
                    }
                    if (PRE) bulk_load(ring0 + stage * C::STAGE_BYTES + C::A_BYTES + C::SFA_BYTES, P.digits + (size_t)ks * C::X_BYTES, C::X_BYTES, full_bar(stage));
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // -------------------------------------------------------------- MMAs
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0, it = 0, grp = 0;
            int before[2] = {0, 0};                            // stage of the step two before, whose scales the buffer held, and its phase
            uint32_t before_phase[2] = {0, 0};
            bool ok = true;
            for (int tile = first_tile; tile < tiles && ok; tile += tile_stride) {
                int in_group = 0;
                for (int ks = k0; ks < k1; ++ks, ++it) {
                    if (in_group == 0) ok = wait_one(dempty_bar(grp), ((grp / C::kAccs) & 1u) ^ 1u, abort_flag, P.wait_cycles);
                    if (ok && it >= 2) ok = wait_one(empty_bar(before[it & 1u]), before_phase[it & 1u], abort_flag, P.wait_cycles);
                    if (ok) ok = wait_one(full_bar(stage), phase, abort_flag, P.wait_cycles);
                    if (!PRE && ok) ok = wait_one(xfull_bar(stage), phase, abort_flag, P.wait_cycles);
                    if (!ok) break;
                    tc_fence_after();
                    const int nkb = min(4, katoms - 4 * ks);
                    const uint32_t a = ring0 + stage * C::STAGE_BYTES, b = a + C::A_BYTES + C::SFA_BYTES;
                    const uint32_t t_sfa = tmem + C::kSfBase + (it & 1u) * C::kSfCols, t_sfb = t_sfa + 32u;
                    const uint64_t adesc = make_desc_sw128(a), bdesc = make_desc_sw128(b);
                    const uint64_t fadesc = make_desc_sf(a + C::A_BYTES), fbdesc = make_desc_sf(b + C::B_BYTES);
#pragma unroll
                    for (int kb = 0; kb < 4; ++kb) {
                        if (kb < nkb) {
#pragma unroll
                            for (int h = 0; h < 2; ++h) tmem_cp_sf(t_sfa + 16u * h + 4u * kb, fadesc + 128ull * h + 32ull * kb);
#pragma unroll
                            for (int at = 0; at < C::kAtoms; ++at) tmem_cp_sf(t_sfb + 4u * (C::kAtoms * kb + at), fbdesc + 128ull * at + 32ull * kb);
                        }
                    }
#pragma unroll
                    for (int kb = 0; kb < 4; ++kb) {
                        if (kb < nkb) {
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                mma_nvf4(tmem + (grp % C::kAccs * 2u + h) * C::kDStride, adesc + 1024ull * h + 2ull * kb, bdesc + 2ull * kb, C::kIdesc, t_sfa + 16u * h + 4u * kb,
                                         t_sfb + 4u * C::kAtoms * kb, (in_group > 0 || kb > 0) ? 1u : 0u);
                        }
                    }
                    mma_commit(empty_bar(stage));
                    before[it & 1u] = stage;
                    before_phase[it & 1u] = phase;
                    ++in_group;
                    if ((PRE ? (ks + 1) % kGroupSteps == 0 : in_group == kGroupSteps) || ks + 1 == k1) {
                        mma_commit(dfull_bar(grp));
                        ++grp;
                        in_group = 0;
                    }
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else {
        // --------------------------------------- digits, finished groups, output
        const int ww = warp - 2, h = ww >> 2, q = warp & 3;
        const uint32_t lanes = (uint32_t)(32 * q) << 16;
        const int r = h * 128 + 32 * q + lane;                 // row of the tile
        const int col = ww % (4 * NG), turn = ww / (4 * NG);
        const __nv_bfloat16 *xcol = P.X + (int64_t)(col < P.cols ? col : 0) * P.ldx + lane * 8;
        // steps in which the lane has activations of its column: up to the end of this CTA's range, and of the row
        const int live = col < P.cols ? min(k1, (P.K - lane * 8 + 255) / 256) : 0;
        // where the lane's digits go in a stage: rows 12 col + p of 128 bytes, their 16-byte pieces swizzled with the row (12 col mod 8 is 0 or 4),
        // here for rows p = 0 .. 7 without the p * 128; and its scales, of rows 12 col + lane % 8 and + 8
        uint32_t place[8], sf_place[2];
#pragma unroll
        for (int p = 0; p < 8; ++p)
            place[p] = C::A_BYTES + C::SFA_BYTES + (uint32_t)(col * kDigits) * 128u + ((((uint32_t)lane >> 2) ^ ((4u * (uint32_t)col + p) & 7u)) << 4) + ((uint32_t)lane & 3u) * 4u;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t n = (uint32_t)(col * kDigits) + ((uint32_t)lane & 7u) + 8u * u, rr = n & 127u;
            sf_place[u] = C::A_BYTES + C::SFA_BYTES + C::B_BYTES + (n >> 7) * 2048u + ((uint32_t)lane >> 3) * 512u + (rr & 31u) * 16u + (rr >> 5) * 4u;
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");     // X may come from the kernel ahead
        const float s_all = P.hdr->s;
        float acc[4 * NG];
        bool ok = true;
        int stage = 0;
        uint32_t phase = 0, grp = 0, slot = 0;                 // groups whose digits are begun; grp % kSlots
        for (int tile = first_tile; tile < tiles && ok; tile += tile_stride) {
            const int row = tile * 256 + r;
#pragma unroll
            for (int c = 0; c < 4 * NG; ++c) acc[c] = 0.0f;
            // where the group that step ks is in ends: groups of the workspace are counted from the row's start, others from the CTA's first step
            auto group_end = [&](int ks) { return PRE ? (ks / kGroupSteps + 1) * kGroupSteps : ks + kGroupSteps; };
            // group n of the kernel, of steps from ks, its scales in slot sl: from its accumulator into the running sums
            auto flush = [&](uint32_t n, uint32_t sl, int ks) {
                if (ok) ok = wait_warp(dfull_bar(n), (n / C::kAccs) & 1u, abort_flag, P.wait_cycles);
                if (!ok) return;
                tc_fence_after();
                // the columns' powers of two: lane c has column c's
                const int gi = ks / kGroupSteps * 16 + (lane & 15), si = (int)sl * 16 + (lane & 15);
                const float gs = (PRE ? __uint_as_float(__ldcg(P.group_scale + gi)) : scales[si]) * pow2(scale_exponent(s_all));
                const int sp_lane = PRE ? (int)__ldcg(P.group_scale + P.ngroups * 16 + gi) : specials[si];
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    float v[3][16];
#pragma unroll
                    for (int i = 0; i < 3; ++i) tmem_ld16(tmem + (n % C::kAccs * 2u + h) * C::kDStride + lanes + (uint32_t)(48 * g + 16 * i), v[i]);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float x = v[(12 * c + 11) / 16][(12 * c + 11) % 16];
#pragma unroll
                        for (int p = kDigits - 2; p >= 0; --p) x = fmaf(x, 0.125f, v[(12 * c + p) / 16][(12 * c + p) % 16]);
                        acc[4 * g + c] = fmaf(x, __shfl_sync(0xffffffffu, gs, 4 * g + c), acc[4 * g + c]);
                        asm volatile("" : "+f"(acc[4 * g + c]));           // now: the sums of all columns at once would not fit the registers
                    }
                }
                tc_fence_before();
                const uint32_t sp = __ballot_sync(0xffffffffu, lane < 4 * NG && sp_lane != 0);
                if (sp != 0 && row < P.N) {
#pragma unroll
                    for (int c = 0; c < 4 * NG; ++c)
                        if ((sp >> c) & 1u)
                            acc[c] += special_sum(P.codes, P.w_sf, P.X + (int64_t)c * P.ldx, row, ks * 256, min(P.K, min(k1, group_end(ks)) * 256), P.K);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(dempty_bar(n));
            };
            // The lane's eight activations of the warp's steps, one ahead of the one in work, and of the next group's steps, whose largest
            // exponent is wanted before the first of them.
            auto piece = [&](int ks) {
                return ks < live ? __ldg(reinterpret_cast<const uint4 *>(xcol + ks * 256)) : make_uint4(0u, 0u, 0u, 0u);
            };
            uint32_t gm = 0;
            uint4 next = make_uint4(0u, 0u, 0u, 0u);
            if (!PRE) {
#pragma unroll
                for (int s = 0; s < kGroupSteps; ++s) gm = max_abs_bf16x2(gm, max_abs_of(piece(k0 + s)));
                next = piece(k0 + turn);
            }
            for (int kg = k0; PRE && kg < k1 && ok; kg = group_end(kg)) flush(grp++, 0u, kg);
            for (int kg = k0; !PRE && kg < k1 && ok; kg += kGroupSteps, ++grp, slot = slot + 1u == kSlots ? 0u : slot + 1u) {
                const int nk = min(kGroupSteps, k1 - kg);
                const uint32_t top = __reduce_max_sync(0xffffffffu, max_magnitude(gm));
                const bool special = top >= 0x7F80u;
                const int eg = max((int)(top >> 7), 1);
                gm = 0;
#pragma unroll 1
                for (int s = 0; s < nk; ++s) {
                    const uint4 ahead = piece(kg + kGroupSteps + s);
                    ok = wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, P.wait_cycles);
                    if (!ok) break;
                    const uint32_t b = ring0 + stage * C::STAGE_BYTES;
                    if (s == 0 && turn == 0 && lane == 0 && col < P.cols) {
                        scales[slot * 16u + col] = __uint_as_float(scale_of_group(top, eg));
                        specials[slot * 16u + col] = special;
                    }
                    if (col < P.cols && s % C::kPerCol == turn) {
                        const uint4 x = special ? make_uint4(0u, 0u, 0u, 0u) : next;
                        next = piece(kg + s + C::kPerCol);
                        uint32_t w[kDigits], sf;
                        digits_and_scales(x, eg, w, sf);
                        sts_u32_at<0>(b + place[0], w[0]);
                        sts_u32_at<128>(b + place[1], w[1]);
                        sts_u32_at<256>(b + place[2], w[2]);
                        sts_u32_at<384>(b + place[3], w[3]);
                        sts_u32_at<512>(b + place[4], w[4]);
                        sts_u32_at<640>(b + place[5], w[5]);
                        sts_u32_at<768>(b + place[6], w[6]);
                        sts_u32_at<896>(b + place[7], w[7]);
                        sts_u32_at<1024>(b + place[0], w[8]);
                        sts_u32_at<1152>(b + place[1], w[9]);
                        sts_u32_at<1280>(b + place[2], w[10]);
                        sts_u32_at<1408>(b + place[3], w[11]);
                        sts_u32(b + sf_place[0], sf);
                        if ((lane & 7) < kDigits - 8) sts_u32(b + sf_place[1], sf);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");        // the tensor cores read them
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(xfull_bar(stage));
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                    gm = max_abs_bf16x2(gm, max_abs_of(ahead));
                    if (s == 0 && kg > k0) flush(grp - 1u, (slot == 0 ? kSlots : slot) - 1u, kg - kGroupSteps);
                }
            }
            if (!PRE && ok && k1 > k0) flush(grp - 1u, (slot == 0 ? kSlots : slot) - 1u, k0 + (k1 - k0 - 1) / kGroupSteps * kGroupSteps);
            if (ok && csize == 1 && row < P.N) {
                const float s_w = s_all * pow2(-scale_exponent(s_all));        // what the groups' scales have left of it
                __nv_bfloat16 *y = P.Y + row;
#pragma unroll
                for (int c = 0; c < 4 * NG; ++c)
                    if (c < P.cols) y[(int64_t)c * P.ldy] = __float2bfloat16_rn(acc[c] * s_w);
            }
        }
        if (csize > 1) {
            // One tile per cluster.  Four columns i go to CTA i % csize; everybody's copies, MMAs and reads are over
            // after the first barrier, so the ring takes the partial sums: [source][four columns of this CTA][256 rows].
            cluster_sync();
            const int per = (NG + csize - 1) / csize;
            const uint32_t mine = ring0 + (uint32_t)r * 16u;
#pragma unroll
            for (int i = 0; i < NG; ++i)
                st_cluster_v4(mine + (uint32_t)((int)rank * per + i / csize) * 4096u, (uint32_t)(i % csize), acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            cluster_sync();
            const int row = first_tile * 256 + r;
            const float s_w = s_all * pow2(-scale_exponent(s_all));
            if (ok && row < P.N) {
                for (int i = (int)rank, l = 0; i < NG && 4 * i < P.cols; i += csize, ++l) {
                    float tot[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    for (int src = 0; src < csize; ++src) {
                        float4 v;
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                                     : "r"(mine + (uint32_t)(src * per + l) * 4096u) : "memory");
                        tot[0] += v.x; tot[1] += v.y; tot[2] += v.z; tot[3] += v.w;
                    }
                    __nv_bfloat16 *y = P.Y + (int64_t)(4 * i) * P.ldy + row;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (4 * i + c < P.cols) y[(int64_t)c * P.ldy] = __float2bfloat16_rn(tot[c] * s_w);
                }
            }
        }
    }
    __syncwarp();
    if (csize > 1 && warp < 2) { cluster_sync(); cluster_sync(); }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // a wait ran out: give copies in flight time to land, then report
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
        if (threadIdx.x == 0) {
            atomicExch(&P.status->status, (int)DQ_ERR_TIMEOUT);
            atomicExch(&P.status->detail, 0x3E000 | (int)blockIdx.x);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

template <int NG, bool PRE>
cudaError_t set_attributes(int dev)
{
    static std::atomic<bool> done[kMaxDevices];
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    auto kernel = decode_fp4_kernel<NG, PRE>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<NG, PRE>::SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    // the digits' kernel with the same split of an SM's memory: a change has to wait until the SM is empty
    if (PRE && e == cudaSuccess) e = cudaFuncSetAttribute(fp4_digits_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (PRE && e == cudaSuccess) e = cudaFuncSetAttribute(fp4_digits_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDigitsSmem);
    if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return e;
}

template <int NG, bool PRE>
cudaLaunchConfig_t launch_config(cudaLaunchAttribute (&attr)[2], int grid, int csize, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(Cfg<NG, PRE>::kThreads);
    cfg.dynamicSmemBytes = Cfg<NG, PRE>::SMEM_BYTES;
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

// How many clusters of c CTAs the device holds at once (one CTA per SM in every instantiation); asked once per size and device, and again
// where the runtime did not answer: 0 and sure = false then
int clusters_that_fit(int dev, int c, int sms, bool &sure)
{
    static std::atomic<int> known[kMaxDevices][kMaxCluster + 1];                 // + 1; 0 = not known
    int fit = known[dev][c].load(std::memory_order_relaxed);
    if (fit == 0) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = launch_config<1, false>(attr, c * (sms / c), c, nullptr);
        int n = 0;
        if (set_attributes<1, false>(dev) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, decode_fp4_kernel<1, false>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            sure = false;
            return 0;
        }
        fit = n + 1;
        known[dev][c].store(fit, std::memory_order_relaxed);
    }
    return fit - 1;
}

// CTAs per tile, and the steps of the busiest CTA.  Clusters take one tile each and must all be resident.  sure: the runtime has said how many are
struct Split { int csize; int steps; bool sure; };
Split split_tiles(int64_t N, int64_t K, int dev, int sms, int force_csize)
{
    const int64_t tiles = (N + 255) / 256, ksteps = (K + 255) / 256;
    Split best = {1, (int)((tiles + sms - 1) / sms * ksteps), true};
    double cost = (double)best.steps;
    for (int c = 2; c <= kMaxCluster && c <= ksteps && tiles * c <= sms; ++c) {
        if (force_csize > 0 && c != force_csize) continue;
        const int steps = (int)((ksteps + c - 1) / c);
        if ((force_csize > 0 || steps + 0.5 < cost) && tiles <= clusters_that_fit(dev, c, sms, best.sure)) { best = {c, steps, best.sure}; cost = steps + 0.5; }
    }
    return best;
}

// the workspace: digits, then the groups' scales
struct WsLayout { size_t scale_off, total; };
WsLayout ws_layout(int64_t K)
{
    WsLayout L;
    L.scale_off = (size_t)((K + 255) / 256) * Cfg<4, true>::X_BYTES;
    L.total = L.scale_off + (size_t)((K + 256 * kGroupSteps - 1) / (256 * kGroupSteps)) * 2 * 16 * 4;
    return L;
}

template <int NG, bool PRE>
cudaError_t launch_ng(const CUtensorMap &tmap, Fp4Args P, int force_csize, const DeviceInfo *di, cudaStream_t stream)
{
    cudaError_t e = set_attributes<NG, PRE>(di->device);
    if (e != cudaSuccess) return e;
    P.csize = split_tiles(P.N, P.K, di->device, di->sms, force_csize).csize;
    if (force_csize > 0 && P.csize != force_csize) return cudaErrorInvalidValue;
    const int tiles = (P.N + 255) / 256;
    cudaLaunchAttribute attr[2];
    if (PRE) {
        cudaLaunchConfig_t cfg = launch_config<NG, PRE>(attr, 1, 1, stream);
        cfg.gridDim = dim3((unsigned)P.ngroups, (unsigned)(4 * NG));
        cfg.blockDim = dim3(32 * kGroupSteps);
        cfg.dynamicSmemBytes = kDigitsSmem;
        e = cudaLaunchKernelEx(&cfg, fp4_digits_kernel, P, Cfg<NG, PRE>::X_BYTES, Cfg<NG, PRE>::B_BYTES);
        if (e != cudaSuccess) return e;
    }
    const cudaLaunchConfig_t cfg = launch_config<NG, PRE>(attr, P.csize > 1 ? tiles * P.csize : (tiles < di->sms ? tiles : di->sms), P.csize, stream);
    return cudaLaunchKernelEx(&cfg, decode_fp4_kernel<NG, PRE>, tmap, P);
}

}  // namespace

// Against the kernels before it (launch after launch of one matrix; 20038 points from 512 to 34816 rows and 256 to 17408 weights; us, those /
// this).  Up to four columns it is ahead but where a second step holds a half or less and rows are many (16896x384 4.5 / 5.0) and for one column of
// a few long rows (512x14848 7.6 / 8.2): of 6706 points 24 lose more than 2 %, at most 13 %, and on average it is 1.25 times as fast.  From five
// columns on, with the workspace: 4.3 (5.6 above eight) for both launches, 0.51 (0.74) a step of the busiest CTA, 0.078 (0.070) a megabyte, 1.4 for a
// cluster's exchange, against 1.9, 2.75 a slice of 512 and 0.033 a megabyte; its second launch costs the host 3, so that short calls stay
// (1536x8192 batch 8 9.4 / 8.7); clusters of three or five that crowd the chip wait for a free group of SMs (11408x11776 batch 9 27.4 / 33.9).
// The mma.sync kernel is not in it: where this one is taken for five to eight columns it is never the faster (144 points; 23600x10240 batch 5: mma.sync 39.4,
// batch kernel 56.4, this one 28.6).
// sure = false: the answer rests on one that the runtime did not give
bool decode_fp4_is_faster(int64_t N, int64_t K, int64_t B, int sms, bool *sure)
{
    if (sure) *sure = true;
    if (B > 16) return false;
    if (B <= 4) return !(K > 256 && K <= 512 && N >= 9216) && !(B == 1 && K > 10240 && N <= 2304);
    const DeviceInfo *di = device_info();
    if (!di || K <= 1024) return false;
    Split t = split_tiles(N, K, di->device, sms, 0);
    const bool crowded = (t.csize == 3 || t.csize == 5) && (N + 255) / 256 >= clusters_that_fit(di->device, t.csize, sms, t.sure) - 1;
    if (sure) *sure = t.sure;
    if (crowded) return false;
    const double mb = (double)N * (double)K * 0.5625e-6;
    const double here = (B <= 8 ? 4.29 + 0.507 * t.steps + 0.0778 * mb : 5.62 + 0.736 * t.steps + 0.0704 * mb) + (t.csize > 1 ? 1.42 : 0.0);
    const double there = 1.87 + 2.75 * decode_tc_slices(N, K) + 0.033 * mb;
    return there > 14.0 && here < 0.95 * there;
}

size_t decode_fp4_workspace(int64_t K) { return ws_layout(K).total; }

cudaError_t launch_decode_fp4(const GemvNvArgs &a, int force_csize, void *ws, size_t ws_bytes, cudaStream_t stream)
{
    const DeviceInfo *di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    if (a.B > 16 || (a.B > 4 && !ws)) return cudaErrorInvalidValue;
    if (gemm_init_driver_api() != 0) return cudaErrorNotSupported;
    // packed FP4 codes as a byte matrix [N][K/2]; box = 128 bytes x the rows of a tile, 128B swizzle, zero fill outside
    EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(gemm_encode_fn());
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tmap;
    cuuint64_t gdim[2] = {(cuuint64_t)(a.K / 2), (cuuint64_t)a.N};
    cuuint64_t gstride[1] = {(cuuint64_t)(a.K / 2)};
    cuuint32_t box[2] = {128u, 256u};
    cuuint32_t estr[2] = {1u, 1u};
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t *>(a.codes), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    Fp4Args P = {};
    P.codes = a.codes;
    P.w_sf = a.sf;
    P.hdr = a.hdr;
    P.X = reinterpret_cast<const __nv_bfloat16 *>(a.X);
    P.Y = reinterpret_cast<__nv_bfloat16 *>(a.Y);
    P.ldx = a.ldx;
    P.ldy = a.ldy;
    P.cols = (int)a.B;
    P.N = (int)a.N;
    P.K = (int)a.K;
    P.csize = 1;
    P.wait_cycles = a.wait_cycles > 0 ? a.wait_cycles : kWaitBudgetCycles;
    P.drop_first_copy = a.drop_first_copy;
    P.status = a.status;
    if (a.B <= 4) return launch_ng<1, false>(tmap, P, force_csize, di, stream);
    const WsLayout L = ws_layout(a.K);
    if (ws_bytes < L.total) return cudaErrorInvalidValue;
    P.digits = reinterpret_cast<uint8_t *>(ws);
    P.group_scale = reinterpret_cast<uint32_t *>(P.digits + L.scale_off);
    P.ngroups = (int)((a.K + 256 * kGroupSteps - 1) / (256 * kGroupSteps));
    if (a.B <= 8) return launch_ng<2, true>(tmap, P, force_csize, di, stream);
    return launch_ng<4, true>(tmap, P, force_csize, di, stream);
}

}  // namespace dq

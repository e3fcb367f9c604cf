// NVFP4 x NVFP4 block-scaled GEMM for the prefill path on sm_100a (Sec. 2.3;
// App. A.3 "NVFP4": E2M1 values, 16-element blocks, E4M3 block scales, FP32
// tensor scales):
//   Y[m][n] = bf16( s_a * s_w * sum_blk dA[m][blk] dW[n][blk] sum_{k in blk} eA[m][k] eW[n][k] )
//
// One CTA per SM and 128-row tile: the kernel of short prompts, where the weights stream from HBM and what counts is that every
// SM streams its share of them.  Tiles are 128 x 256 or 128 x 128; where there are too few of them for the chip a cluster of up to
// 8 CTAs shares one, each taking a range of k-steps, and they exchange partial sums through distributed shared memory at
// the end (added in rank order; no workspace).  256-element k-steps.  Also the columns that a larger call leaves to it, and gate/up
// matrices whose gating and quantising replaces the output (GATED; clusters only, the sums are then those of the plain call).
//   warp 0      : TMA producer (packed FP4 tiles, 128B swizzle) + bulk copies of the scale atoms; weights that are part of the
//                 handle are requested before the kernel ahead (the activation quantiser) has finished
//   warp 1      : tcgen05.cp of the scales into TMEM and tcgen05.mma (kind::mxf4nvf4, block 16)
//   warps 2..   : epilogue, TMEM -> registers -> bf16 -> global; four warps, or eight beside an exchange (launch_tile)
// The fp32 accumulator lives in TMEM (two of 128 columns or one of 256) beside the scale factors of every stage.  Producer and MMA
// roles are one elected thread each, waits included: see elect_one.  Every mbarrier wait is bounded: when it runs
// out the CTA records DQ_ERR_TIMEOUT in the status word and leaves normally.
// Bound by the weights' way from HBM and the launches: one layer of the 27B-class stack (203 MB) at 77 tokens, quantisers and GEMMs,
// takes 71 us; with lone CTAs on 128 x 256 tiles, 20 to 136 of them, it took 104.
#include <atomic>

#include <cuda.h>

#include "dq_common.cuh"
#include "dq_quant.cuh"
#include "dq_tcgen05.cuh"

namespace dq {

namespace {

using namespace tc;

constexpr int BM = 128;
constexpr int kKbPerStage = 4;                // 64-element MMA k-steps per 256-element stage (128 bytes of FP4: one swizzle row)
constexpr int threads_of(int halves) { return 64 + 128 * halves; }     // `halves` epilogue warps per TMEM lane quarter
constexpr uint32_t kTmemCols = 512;

constexpr int kMaxCluster = 8;
// largest area that the partial sums of a gated tile take: units of 16 gate and 16 up columns go round the CTAs of a cluster, four
// groups of eight columns each
constexpr uint32_t gated_bytes(int units)
{
    uint32_t most = 0;
    for (int c = 2; c <= kMaxCluster; ++c) {
        const uint32_t b = (uint32_t)(c * ((units + c - 1) / c) * 4) * 4096u;
        if (b > most) most = b;
    }
    return most;
}

template <int BN>
struct Cfg {
    static constexpr int kStages = BN == 128 ? 6 : 4;
    static constexpr int kAccs = BN == 128 ? 2 : 1;                    // accumulators
    static constexpr int kSfbAtoms = BN / 128;
    static constexpr uint32_t A_BYTES = BM * 128, B_BYTES = BN * 128;
    static constexpr uint32_t SFA_BYTES = kKbPerStage * 512, SFB_BYTES = kSfbAtoms * kKbPerStage * 512;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES + SFA_BYTES + SFB_BYTES;
    // barriers behind the ring, which an exchange of partial sums uses again; that of a gated tile may reach beyond it
    static constexpr uint32_t GATED_BYTES = gated_bytes(BN / 32);
    static constexpr uint32_t BAR_OFF = kStages * STAGE_BYTES, BAR_OFF_GATED = GATED_BYTES > BAR_OFF ? GATED_BYTES : BAR_OFF;
    static constexpr uint32_t SMEM_BYTES = BAR_OFF + 1024 /*align*/ + 256 /*barriers*/, SMEM_BYTES_GATED = BAR_OFF_GATED + 1024 + 256;
    static constexpr uint32_t kSfBase = kAccs * BN;                    // TMEM columns: accumulators, then scales per stage
    static constexpr uint32_t kSfbCol = 4 * kKbPerStage, kSfCols = kSfbCol + 4 * kKbPerStage * kSfbAtoms;
    static_assert(kSfBase + kStages * kSfCols <= kTmemCols, "scale buffers must fit in TMEM");
    static_assert(STAGE_BYTES % 1024 == 0, "stages must keep 1024-byte alignment for the 128B swizzle");
    static_assert(SMEM_BYTES_GATED <= 227 * 1024, "shared memory");
    static_assert((BN / 8 + 8) * BM * 32 <= kStages * (int)STAGE_BYTES, "partial sums of a cluster must fit the ring");
    // instruction descriptor: dense, A/B = E2M1 (kind::mxf4nvf4), both K-major, scale type UE4M3,
    // N >> 3 at bit 17, M >> 4 at bit 24, scale-factor ids 0, K = 64
    static constexpr uint32_t kInstrDesc = (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
};

// tile index -> (m block, n block): m fastest inside groups of 16 m-blocks so that
// the CTAs running at the same time share A row-blocks and W column-blocks in L2
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int &mb, int &nb)
{
    constexpr int GM = 16;
    const int per_group = GM * tiles_n;
    const int g = t / per_group;
    const int first_m = g * GM;
    const int gsz = min(GM, tiles_m - first_m);
    const int r = t - g * per_group;
    mb = first_m + r % gsz;
    nb = r / gsz;
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
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t rank, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("{\n\t.reg .b32 p;\n\tmapa.shared::cluster.u32 p, %0, %1;\n\tst.shared::cluster.v4.b32 [p], {%2, %3, %4, %5};\n\t}"
                 ::"r"(addr), "r"(rank), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 lds_v4f(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

template <int BN, int HALVES, bool CLOCKS, bool GATED>
__global__ void __launch_bounds__(threads_of(HALVES), 1)
gemm_nvfp4_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                  const uint8_t *__restrict__ a_sf, const uint8_t *__restrict__ w_sf,
                  const PackedHeader *__restrict__ hdr, float act_scale, __nv_bfloat16 *__restrict__ Y, int64_t ldy,
                  int M, int N, int K, int csize, int early_weights, int clocks, StatusWord *status, GatedOut gated)
{
    using C = Cfg<BN>;
    constexpr int kStages = C::kStages, kAccs = C::kAccs;
    constexpr uint32_t kBarOff = GATED ? C::BAR_OFF_GATED : C::BAR_OFF;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    // per stage: [A][B][SFA][SFB]; barriers: full[kStages], empty[kStages], tmem_full[2], tmem_empty[2]; then tmem ptr, abort flag
    const uint32_t bar_base = smem_base + kBarOff;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
    auto tmem_full_bar = [&](int i) { return bar_base + 8u * (2 * kStages + i); };
    auto tmem_empty_bar = [&](int i) { return bar_base + 8u * (2 * kStages + 2 + i); };
    uint32_t *tmem_ptr_smem = reinterpret_cast<uint32_t *>(smem_gen + kBarOff + 8 * (2 * kStages + 4));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_ptr_smem + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tmem_full_bar(i), 1); mbar_init(tmem_empty_bar(i), 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_ptr_smem)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_ptr_smem;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int tiles_m = (M + BM - 1) / BM;
    const int tiles_n = (N + BN - 1) / BN;
    const int num_tiles = tiles_m * tiles_n;
    const int katoms = K / 64;                                // 64-element k atoms in K
    const int num_ks = (katoms + kKbPerStage - 1) / kKbPerStage;
    const uint32_t rank = csize > 1 ? cluster_ctarank() : 0u;
    const int first_tile = (int)blockIdx.x / csize, tile_stride = (int)gridDim.x / csize;
    const int k0 = (int)((long long)num_ks * rank / csize), k1 = (int)((long long)num_ks * (rank + 1) / csize);

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (elect_one()) {
            auto load_w = [&](int stage, int nb, int ks) {
                const int nkb = min(kKbPerStage, katoms - ks * kKbPerStage);
                const uint32_t sB = smem_base + stage * C::STAGE_BYTES + C::A_BYTES, sSFB = sB + C::B_BYTES + C::SFA_BYTES;
                const uint32_t sf_bytes = (uint32_t)nkb * 512u;
                mbar_expect_tx(full_bar(stage), C::A_BYTES + C::B_BYTES + (1u + C::kSfbAtoms) * sf_bytes);
                tma_load_2d(sB, &tmap_w, ks * 128, nb * BN, full_bar(stage));
#pragma unroll
                for (int at = 0; at < C::kSfbAtoms; ++at)
                    bulk_load(sSFB + (uint32_t)at * kKbPerStage * 512u,
                              w_sf + ((size_t)(C::kSfbAtoms * nb + at) * katoms + (size_t)ks * kKbPerStage) * 512, sf_bytes, full_bar(stage));
            };
            auto load_a = [&](int stage, int mb, int ks) {
                const int nkb = min(kKbPerStage, katoms - ks * kKbPerStage);
                const uint32_t sA = smem_base + stage * C::STAGE_BYTES, sSFA = sA + C::A_BYTES + C::B_BYTES;
                tma_load_2d(sA, &tmap_a, ks * 128, mb * BM, full_bar(stage));
                bulk_load(sSFA, a_sf + ((size_t)mb * katoms + (size_t)ks * kKbPerStage) * 512, (uint32_t)nkb * 512u, full_bar(stage));
            };
            // The weights of a handle are constant data: the first stages of them are requested before waiting for the kernel ahead,
            // which makes the activations (weights cast into the workspace for this call are made by it too)
            int early = 0;
            if (early_weights && first_tile < num_tiles) {
                int mb, nb;
                tile_coords(first_tile, tiles_m, tiles_n, mb, nb);
                early = min(kStages, k1 - k0);
                for (int i = 0; i < early; ++i) load_w(i, nb, k0 + i);
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            int stage = 0; uint32_t phase = 0;
            bool ok = true;
            for (int t = first_tile; t < num_tiles && ok; t += tile_stride) {
                int mb, nb;
                tile_coords(t, tiles_m, tiles_n, mb, nb);
                for (int ks = k0; ks < k1; ++ks) {
                    if (early > 0) {
                        --early;
                    } else {
                        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
                        load_w(stage, nb, ks);
                    }
                    load_a(stage, mb, ks);
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        if (elect_one()) {
            int stage = 0; uint32_t phase = 0;
            uint32_t it = 0;                                   // tiles: accumulator it % kAccs
            bool ok = true;
            for (int t = first_tile; t < num_tiles && ok; t += tile_stride, ++it) {
                const uint32_t acc = it % kAccs;
                ok = mbar_wait(tmem_empty_bar(acc), ((it / kAccs) & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int ks = k0; ks < k1; ++ks) {
                    if (!mbar_wait(full_bar(stage), phase, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    const int nkb = min(kKbPerStage, katoms - ks * kKbPerStage);
                    const uint32_t sA = smem_base + stage * C::STAGE_BYTES;
                    const uint32_t sB = sA + C::A_BYTES, sSFA = sB + C::B_BYTES, sSFB = sSFA + C::SFA_BYTES;
                    const uint32_t t_sfa = tmem_base + C::kSfBase + (uint32_t)stage * C::kSfCols;
                    const uint32_t t_sfb = t_sfa + C::kSfbCol;
                    const uint64_t adesc = make_desc_sw128(sA), bdesc = make_desc_sw128(sB);
                    const uint64_t fadesc = make_desc_sf(sSFA), fbdesc = make_desc_sf(sSFB);
#pragma unroll
                    for (int kb = 0; kb < kKbPerStage; ++kb) {
                        if (kb < nkb) {
                            tmem_cp_sf(t_sfa + 4u * kb, fadesc + 32ull * kb);
#pragma unroll
                            for (int at = 0; at < C::kSfbAtoms; ++at)
                                tmem_cp_sf(t_sfb + 4u * C::kSfbAtoms * kb + 4u * at, fbdesc + (uint64_t)(at * (kKbPerStage * 512 >> 4)) + 32ull * kb);
                        }
                    }
#pragma unroll
                    for (int kb = 0; kb < kKbPerStage; ++kb) {
                        // one k-step is 64 elements = 32 bytes inside the 128-byte swizzle row
                        if (kb < nkb)
                            mma_nvf4(d_tmem, adesc + 2ull * kb, bdesc + 2ull * kb, C::kInstrDesc, t_sfa + 4u * kb,
                                     t_sfb + 4u * C::kSfbAtoms * kb, (ks > k0 || kb > 0) ? 1u : 0u);
                    }
                    mma_commit(empty_bar(stage));          // frees the stage once these MMAs have read it
                    if (++stage == kStages) { stage = 0; phase ^= 1u; }
                }
                if (ok) mma_commit(tmem_full_bar(acc));    // accumulator complete
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int wq = warp & 3;                           // TMEM lane quarter this warp may read
        const uint32_t lanes = (uint32_t)(wq * 32) << 16;
        const float alpha = __fmul_rn(act_scale, hdr->s);
        bool ok = true;
        // measurement, as in the pair kernel: SM cycles and global-timer nanoseconds of the first CTA, from the end of the kernel ahead until
        // its first epilogue warp is done; clocks = 1: left in the status word, 2: added to what the launch before it left there
        long long clk0 = 0, ns0 = 0;
        const bool timed = CLOCKS && blockIdx.x == 0 && threadIdx.x == 64;
        if (timed) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            clk0 = clock64();
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns0));
        }
        if (HALVES == 1 && !GATED && csize == 1) {
            uint32_t it = 0;
            for (int t = first_tile; t < num_tiles && ok; t += tile_stride, ++it) {
                const uint32_t acc = it % kAccs;
                int mb, nb;
                tile_coords(t, tiles_m, tiles_n, mb, nb);
                ok = mbar_wait_warp(tmem_full_bar(acc), (it / kAccs) & 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const int row = mb * BM + wq * 32 + lane;
                __nv_bfloat16 *yrow = Y + (int64_t)row * ldy + (int64_t)nb * BN;
                if (mb * BM + wq * 32 < M) {               // whole warps of padding rows read nothing
#pragma unroll 1
                    for (int c = 0; c < BN / 32; ++c) {
                        uint32_t v[32];
                        tmem_ld32(tmem_base + acc * BN + lanes + (uint32_t)(c * 32), v);
                        tmem_ld_wait();
                        if (row < M) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (nb * BN + c * 32 + q * 8 < N) {
                                    uint4 o;
                                    o.x = pack_bf16x2(__uint_as_float(v[8 * q + 0]) * alpha, __uint_as_float(v[8 * q + 1]) * alpha);
                                    o.y = pack_bf16x2(__uint_as_float(v[8 * q + 2]) * alpha, __uint_as_float(v[8 * q + 3]) * alpha);
                                    o.z = pack_bf16x2(__uint_as_float(v[8 * q + 4]) * alpha, __uint_as_float(v[8 * q + 5]) * alpha);
                                    o.w = pack_bf16x2(__uint_as_float(v[8 * q + 6]) * alpha, __uint_as_float(v[8 * q + 7]) * alpha);
                                    *reinterpret_cast<uint4 *>(yrow + c * 32 + q * 8) = o;
                                }
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tmem_empty_bar(acc));
            }
        } else {
            // One tile per cluster.  Eight columns i of the tile go to CTA i % csize; after the first barrier everybody's copies and MMAs
            // are over and the ring takes the partial sums: [source][group of this CTA][128 rows][8 columns].
            int mb, nb;
            tile_coords(first_tile, tiles_m, tiles_n, mb, nb);
            ok = mbar_wait_warp(tmem_full_bar(0), 0u, abort_flag);
            tc_fence_after();
            cluster_sync();
            const int half = HALVES > 1 ? (warp - 2) >> 2 : 0;                        // each takes its part of the columns
            // A gated tile goes out in units of 16 features instead, 16 columns of gate and the 16 of up that lie 64 further on: unit u to
            // CTA u % csize, so that one thread has what a block of the output takes.
            const int per = GATED ? (BN / 32 + csize - 1) / csize * 4 : (BN / 8 + csize - 1) / csize;
            const int row = mb * BM + wq * 32 + lane;
            const uint32_t mine = smem_base + (uint32_t)(wq * 32 + lane) * 16u;       // + 2048 for the second half of a group
            if (ok && mb * BM + wq * 32 < M) {
#pragma unroll 1
                for (int c = half * (BN / 32 / HALVES); c < (half + 1) * (BN / 32 / HALVES); ++c) {
                    uint32_t v[32];
                    tmem_ld32(tmem_base + lanes + (uint32_t)(c * 32), v);
                    tmem_ld_wait();
                    if (row < M) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            // which of the columns' owners, and where in its share
                            const int i = GATED ? (c >> 2) * 4 + (c & 1) * 2 + (q >> 1) : c * 4 + q;
                            const int at = GATED ? i / csize * 4 + ((c >> 1) & 1) * 2 + (q & 1) : i / csize;
                            const uint32_t dst = mine + (uint32_t)((int)rank * per + at) * 4096u;
                            st_cluster_v4(dst, (uint32_t)(i % csize), v[8 * q], v[8 * q + 1], v[8 * q + 2], v[8 * q + 3]);
                            st_cluster_v4(dst + 2048u, (uint32_t)(i % csize), v[8 * q + 4], v[8 * q + 5], v[8 * q + 6], v[8 * q + 7]);
                        }
                    }
                }
            }
            cluster_sync();
            if (GATED) {
                const float rc6 = __frcp_rn(__fmul_rn(6.0f, gated.s));
                if (ok && row < M) {
                    for (int l = half, u = (int)rank + half * csize; u < BN / 32; u += HALVES * csize, l += HALVES) {
                        uint32_t gu[2][8];                                            // gate and up, packed bf16 as the plain epilogue stores them
#pragma unroll
                        for (int sub = 0; sub < 4; ++sub) {
                            float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
                            for (int src = 0; src < csize; ++src) {
                                const uint32_t at = mine + (uint32_t)(src * per + 4 * l + sub) * 4096u;
                                const float4 x = lds_v4f(at), y = lds_v4f(at + 2048u);
                                a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
                                b.x += y.x; b.y += y.y; b.z += y.z; b.w += y.w;
                            }
                            uint32_t *o = &gu[sub >> 1][(sub & 1) * 4];
                            o[0] = pack_bf16x2(a.x * alpha, a.y * alpha);
                            o[1] = pack_bf16x2(a.z * alpha, a.w * alpha);
                            o[2] = pack_bf16x2(b.x * alpha, b.y * alpha);
                            o[3] = pack_bf16x2(b.z * alpha, b.w * alpha);
                        }
                        uint32_t h[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) h[i] = silu_mul_bf16x2(gu[0][i], gu[1][i]);
                        uint2 codes;
                        const uint32_t d8 = quant_block_nvfp4_bf16(h, gated.s, rc6, codes);
                        const int blk = nb * (BN / 32) + u, rr = row & 127;           // 16-feature block of the output row
                        *reinterpret_cast<uint2 *>(gated.codes + ((int64_t)row * (gated.F >> 4) + blk) * 8) = codes;
                        gated.sf[((size_t)(row >> 7) * (size_t)(gated.F >> 6) + (size_t)(blk >> 2)) * 512 +
                                 (size_t)((rr & 31) * 16 + (rr >> 5) * 4 + (blk & 3))] = (uint8_t)d8;
                    }
                }
            } else if (ok && row < M) {
                for (int l = half, i = (int)rank + half * csize; i < BN / 8 && nb * BN + 8 * i < N; i += HALVES * csize, l += HALVES) {
                    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
                    for (int src = 0; src < csize; ++src) {
                        const uint32_t at = mine + (uint32_t)(src * per + l) * 4096u;
                        const float4 x = lds_v4f(at), y = lds_v4f(at + 2048u);
                        a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
                        b.x += y.x; b.y += y.y; b.z += y.z; b.w += y.w;
                    }
                    uint4 o;
                    o.x = pack_bf16x2(a.x * alpha, a.y * alpha);
                    o.y = pack_bf16x2(a.z * alpha, a.w * alpha);
                    o.z = pack_bf16x2(b.x * alpha, b.y * alpha);
                    o.w = pack_bf16x2(b.z * alpha, b.w * alpha);
                    *reinterpret_cast<uint4 *>(Y + (int64_t)row * ldy + (int64_t)nb * BN + 8 * i) = o;
                }
            }
        }
        if (timed) {
            long long ns1;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns1));
            status->gemm_cycles = (unsigned long long)(clock64() - clk0) + (clocks == 2 ? status->gemm_cycles : 0ull);
            status->gemm_ns = (unsigned long long)(ns1 - ns0) + (clocks == 2 ? status->gemm_ns : 0ull);
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
            atomicExch(&status->status, (int)DQ_ERR_TIMEOUT);
            atomicExch(&status->detail, (int)blockIdx.x);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

// packed FP4 codes as a byte matrix [rows][K/2]; box = 128 bytes x box_rows, 128B swizzle, zero fill outside
bool make_codes_tmap(CUtensorMap *tm, const void *ptr, int64_t rows, int64_t K, uint32_t box_rows)
{
    cuuint64_t gdim[2] = {(cuuint64_t)(K / 2), (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)(K / 2)};
    cuuint32_t box[2] = {128u, box_rows};
    cuuint32_t estr[2] = {1u, 1u};
    CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(ptr), gdim, gstride, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

struct Split { int csize; double cost; };

template <int BN, int HALVES, bool GATED>
cudaLaunchConfig_t launch_config(cudaLaunchAttribute (&attr)[2], int grid, int csize, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads_of(HALVES));
    cfg.dynamicSmemBytes = GATED ? Cfg<BN>::SMEM_BYTES_GATED : Cfg<BN>::SMEM_BYTES;
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

template <int BN, int HALVES, bool CLOCKS, bool GATED>
cudaError_t set_attributes(int dev)
{
    static std::atomic<bool> done[kMaxDevices];
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(gemm_nvfp4_kernel<BN, HALVES, CLOCKS, GATED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)(GATED ? Cfg<BN>::SMEM_BYTES_GATED : Cfg<BN>::SMEM_BYTES));
    if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return e;
}

// Whether clusters of c CTAs may share the tiles of 128 x BN: each takes one tile and at least one k-step, and all must be resident.  How
// many of a size fit is asked once per device, and again where the runtime did not answer.
template <int BN>
bool clusters_fit(int64_t tiles, int num_ks, int c, int dev, int sms)
{
    static std::atomic<int> known[kMaxDevices][kMaxCluster + 1];                 // + 1; 0 = not known
    if (c > kMaxCluster || c > num_ks || tiles * c > sms) return false;
    int fit = known[dev][c].load(std::memory_order_relaxed);
    if (fit == 0) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = launch_config<BN, 1, false>(attr, c * (sms / c), c, nullptr);
        int n = 0;
        if (set_attributes<BN, 1, false, false>(dev) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, gemm_nvfp4_kernel<BN, 1, false, false>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        fit = n + 1;
        known[dev][c].store(fit, std::memory_order_relaxed);
    }
    return tiles <= fit - 1;
}

// CTAs per tile of 128 x BN: bytes of weights (rows x k-steps) that the busiest CTA streams, the activation tile of a step counted
// as 48 rows (it comes from L2) and a cluster's exchange as 600.
// Against the pair kernel, above one tile of rows, the output counts as well: a round takes no less than its epilogue and half its k-steps
// (34816 columns, 16384 rows: 2.3 us a round at K = 128, 2.9 at 1024), the exchange of full row tiles up to 1500 more where few
// k-steps hide it (512x1536, 793 rows: 9.6 us against 8.2 in the pair kernel; 5120x17408, 300 rows: 25.2 with it, 27.0 without), and the ramp is 600 shorter than the pair kernel's.
template <int BN>
Split choose_split(int64_t M, int64_t N, int64_t K, int dev, int sms)
{
    const int64_t tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    const int num_ks = (int)((K / 64 + kKbPerStage - 1) / kKbPerStage);
    const double step = BN + 48.0;
    const double rounds = (double)((tiles + sms - 1) / sms), stream = num_ks * step, output = 0.54 * stream + 1290.0 * (BN / 128);
    const bool many = M > BM;
    Split best = {1, many ? rounds * (stream > output ? stream : output) - 600.0 : rounds * stream};
    // the more CTAs the fewer k-steps each: the largest cluster that fits, less the CTAs that make no step fewer
    int c = num_ks < kMaxCluster ? num_ks : kMaxCluster;
    while (c > 1 && !clusters_fit<BN>(tiles, num_ks, c, dev, sms)) --c;
    if (c > 1) {
        const int steps = (num_ks + c - 1) / c;
        c = (num_ks + steps - 1) / steps;
        const double cost = steps * step + 600.0 + (many && num_ks < 50 ? 1500.0 - 30.0 * num_ks : 0.0);
        if (cost < best.cost) best = {c, cost};
    }
    return best;
}

template <int BN, int HALVES, bool CLOCKS, bool GATED>
cudaError_t launch_with(const GemmArgs &a, const Split &sp, int sms, cudaStream_t stream)
{
    const DeviceInfo *di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    cudaError_t e = set_attributes<BN, HALVES, CLOCKS, GATED>(di->device);
    if (e != cudaSuccess) return e;
    CUtensorMap tmap_a, tmap_w;
    if (!make_codes_tmap(&tmap_a, a.a_codes, a.M, a.K, BM)) return cudaErrorInvalidValue;
    if (!make_codes_tmap(&tmap_w, a.w_codes, a.N, a.K, BN)) return cudaErrorInvalidValue;
    const int64_t tiles = ((a.M + BM - 1) / BM) * ((a.N + BN - 1) / BN);
    const int grid = (int)(sp.csize > 1 ? tiles * sp.csize : (tiles < sms ? tiles : sms));
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config<BN, HALVES, GATED>(attr, grid, sp.csize, stream);
    return cudaLaunchKernelEx(&cfg, gemm_nvfp4_kernel<BN, HALVES, CLOCKS, GATED>, tmap_a, tmap_w, a.a_sf, a.w_sf, a.hdr, a.act_scale,
                              reinterpret_cast<__nv_bfloat16 *>(a.Y), (int64_t)a.ldy, (int)a.M, (int)a.N, (int)a.K, sp.csize,
                              a.w_const ? 1 : 0, a.clocks, a.status, a.gated);
}

// An exchange whose row tile leaves a lane quarter empty hangs on the one to three warps that have rows: two warps a quarter then save
// 0.2 to 1 us (5120x17408, 1 row: 16.7 -> 15.9; 10240x5120, 1 / 16 / 77 / 96 rows: 13.7 / 14.0 / 14.2 / 14.5 -> 12.7 / 13.1 / 13.7 /
// 14.2).  With all four quarters busy, or no exchange, the extra warps gain 0.2 us at best and cost up to 0.5 (2048x1024, 128 rows:
// 6.5 -> 7.0; 34816x5120, 128 rows: 26.3 -> 26.9).  The count is a template parameter: as a variable it cost the four-warp form 1 %.
template <int BN>
cudaError_t launch_tile(const GemmArgs &a, const Split &sp, int sms, cudaStream_t stream)
{
    // SiLU and quantiser are worth a second warp a quarter where a CTA has more than one unit of the tile (gate/up 3328x8192, 129 tokens:
    // 18.6 -> 13.7; with one unit, 1024x4096: 8.9 -> 9.5; in the pair kernel 29.7 and 25.0)
    if (a.gated.codes) return BN / 32 > sp.csize ? launch_with<BN, 2, true, true>(a, sp, sms, stream) : launch_with<BN, 1, true, true>(a, sp, sms, stream);
    if (a.clocks) return launch_with<BN, 1, true, false>(a, sp, sms, stream);       // above 128 tokens
    return sp.csize > 1 && a.M <= 3 * 32 ? launch_with<BN, 2, false, false>(a, sp, sms, stream) : launch_with<BN, 1, false, false>(a, sp, sms, stream);
}

}  // namespace

int gemm_init_driver_api()
{
    if (g_encode) return 0;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || fn == nullptr) return 1;
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    return 0;
}

void *gemm_encode_fn() { return reinterpret_cast<void *>(g_encode); }

// Kernel and tile of a GEMM: the pair kernel for the first `head` columns, tiles of 128 x bn with clusters of sp.csize for the rest
struct Plan { int64_t head; int bn; Split sp; };

static Plan choose_plan(int64_t M, int64_t N, int64_t K, int dev, int sms)
{
    const Split s128 = choose_split<128>(M, N, K, dev, sms), s256 = choose_split<256>(M, N, K, dev, sms);
    const Plan tiles_only = s128.cost < s256.cost ? Plan{0, 128, s128} : Plan{0, 256, s256};
    if (M <= BM) return tiles_only;
    // CTA pairs on 256 x 256 tiles move half as many bytes per flop but have few tiles to share out: 0.36 us per k-step and round
    // and 1 us per tile against 1.75 ns per unit of the other cost, and no less than the output of a round on short rows
    // (34816x256, 16384 rows: 293 us here, 568 with the other kernel; 5120x1024, 2048 rows 13.3 / 16.7).  Measured (us, quantiser included, pair / here): 5120x17408
    // 200 tokens 29.7 / 21.7, 300 tokens 31.3 / 26.0, 512 tokens 32.7 / 37.3; 6144x4096 256 tokens 12.6 / 11.5, 512 tokens
    // 14.1 / 15.2; 10240x5120 256 tokens 15.2 / 17.7, 300 tokens 22.3 / 17.9; 34816x5120 129 tokens 28.3 / 32.9.
    const int64_t tiles = ((M + 255) / 256) * ((N + 255) / 256);
    const int64_t rounds = (tiles + sms / 2 - 1) / (sms / 2), num_ks = (K + 255) / 256;
    const auto pair_cost = [&](int64_t r) {
        const double stream = (double)num_ks * 206.0 + 571.0, output = (double)num_ks * 150.0 + 900.0;
        return (double)r * (stream > output ? stream : output);
    };
    // Where the last round would be nearly empty its columns go to the cluster kernel in a launch of their own, about 7 us of
    // ramp before its k-steps count (5120x17408, 1000 tokens, 80 tiles on 74 pairs: 59.6 -> 50.0 us; 10240x5120,
    // where a round is 9 us, would lose: 31.7 -> 37.3)
    const int64_t tiles_m = (M + 255) / 256, head = (rounds - 1) * (sms / 2) / tiles_m;      // 256-column blocks of the full rounds
    if (rounds > 1 && head > 0 && head * 256 < N) {
        const int64_t rest = N - head * 256;
        const Split t128 = choose_split<128>(M, rest, K, dev, sms), t256 = choose_split<256>(M, rest, K, dev, sms);
        const double tail_cost = (t128.cost < t256.cost ? t128.cost : t256.cost) + 4000.0;
        const double split_cost = pair_cost(rounds - 1) + tail_cost;
        if (split_cost < pair_cost(rounds) && split_cost < s128.cost && split_cost < s256.cost)
            return t128.cost < t256.cost ? Plan{head * 256, 128, t128} : Plan{head * 256, 256, t256};
    }
    if (pair_cost(rounds) <= s128.cost && pair_cost(rounds) <= s256.cost) return {N, 256, {1, 0.0}};
    return tiles_only;
}

// The plan a test asks for; false where it does not fit
static bool forced_plan(const GemmArgs &a, int dev, int sms, Plan &p)
{
    const int c = a.force_csize > 1 ? a.force_csize : 1;
    p = {0, a.force_kernel == 3 ? 256 : 128, {c, 0.0}};
    if (a.force_kernel == 1) p.head = a.N;
    if (a.force_kernel == 4) p.head = (a.N - 1) / 256 * 256;
    const int64_t tiles = (a.M + BM - 1) / BM * ((a.N - p.head + p.bn - 1) / p.bn);
    const int num_ks = (int)((a.K / 64 + kKbPerStage - 1) / kKbPerStage);
    if (a.force_kernel == 1 || c == 1) return a.force_kernel != 4 || p.head > 0;
    return (a.force_kernel != 4 || p.head > 0) && (p.bn == 128 ? clusters_fit<128>(tiles, num_ks, c, dev, sms) : clusters_fit<256>(tiles, num_ks, c, dev, sms));
}

cudaError_t launch_gemm_nvfp4(GemmArgs &a, cudaStream_t stream)
{
    if (gemm_init_driver_api() != 0) return cudaErrorNotSupported;
    const DeviceInfo *di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    if (a.plan_rows == 0) a.plan_rows = a.M;
    a.clocks = a.plan_rows > BM ? 1 : 0;
    Plan p = {a.N, 256, {1, 0.0}};
    // The measurement mode exists in the pair kernel only, and up to 128 tokens the gated epilogue too.  Above, a gated call adds its
    // products up as the plain call does: clusters where that takes clusters.  A lone CTA's sums are those of the pair kernel bit
    // for bit, k-step after k-step, so there the gated call keeps to the pair kernel, whose epilogue overlaps.
    if (a.force_kernel != 0) {
        if (!forced_plan(a, di->device, di->sms, p)) return cudaErrorInvalidValue;
    } else if (!a.mma_only && !(a.gated.codes && a.plan_rows <= BM)) {
        p = choose_plan(a.plan_rows, a.N, a.K, di->device, di->sms);
    }
    if (a.gated.codes && p.sp.csize == 1) p.head = a.N;
    if (p.head > 0) {
        const int64_t rest = a.N - p.head;
        a.N = p.head;
        const cudaError_t e = launch_gemm_nvfp4_pair(a, reinterpret_cast<void *>(g_encode), stream);
        if (e != cudaSuccess || rest == 0) return e;
        a.N = rest;
        a.w_codes += p.head * (a.K / 2);
        a.w_sf += p.head * (a.K / kBlock);
        a.clocks = 2;
        if (a.gated.codes) {                                      // half as many features
            a.gated.codes += p.head / 4;
            a.gated.sf += p.head / 128 * 512;                     // 64 features to an atom
        } else {
            a.Y = reinterpret_cast<__nv_bfloat16 *>(a.Y) + p.head;
        }
    }
    return p.bn == 128 ? launch_tile<128>(a, p.sp, di->sms, stream) : launch_tile<256>(a, p.sp, di->sms, stream);
}

}  // namespace dq

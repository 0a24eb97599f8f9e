// Block-scaled FP8 product on the tensor cores' own block-scaled path (the Blackwell half of
// ScaledMatMul): out[M,N] = A W^T (+ bias) with BOTH operands given as (8-bit element codes, one E8M0
// scale byte per 32 consecutive k).  Two kernels:
//
//  quantise_mx_kernel      bf16 activations -> (codes, scales) by the microscaling rule: per block of 32,
//                          shared exponent floor(log2 max|x|) - emax(format), elements rounded to the
//                          nearest even code with saturation.  Every step is exact (powers of two) except
//                          the final rounding, which is the hardware's round-to-nearest-even conversion.
//
//  gemm_mx_tcgen05_kernel  tcgen05.mma.kind::mxf8f6f4.block_scale: the tensor core multiplies the 8-bit
//                          elements and applies scale_A[row, k/32] * scale_B[col, k/32] per 32-wide
//                          k-group itself; the scale bytes have to sit in tensor memory.  One persistent CTA
//                          per SM walks the 128 x BN output tiles, fourteen warps:
//    warp 0 (1 lane)   TMA: 128 x 128-byte operand tiles (128 k per stage, 128-byte swizzle)
//    warp 1            MMA issue: per stage two or three tcgen05.cp of the stage's scale words from shared into
//                      tensor memory, then four instructions (K = 32 each), scale byte selected by the
//                      instruction descriptor's scale-id fields
//    warps 2..5        scale feed: the 32-bit scale words (4 k-groups each) of the stage's rows into shared memory
//                      in the order the instruction expects: row l of 32 holds rows l, 32 + l, 64 + l and 96 + l of
//                      the operand, 16 bytes; tcgen05.cp.32x128b.warpx4 replicates it in all four lane quarters
//    warps 6..13       epilogue, one lane quarter x one half of the columns each
//  BN = 192 where N allows (a tile moves 40 KB of operands per 384 tensor-core cycles), else 128 (32 KB per 256).
//  Accumulators are double-buffered in tensor memory, so that one tile's epilogue overlaps the next main loop.
//  Scale words are handed over four k-blocks at a time, through two slots with barriers of their own; one commit per
//  stage frees its operands.
//  What bounds it: the operands.  36736 x 384 x 1536 moves 275 MB from L2 in 21 us, 13.1 TB/s; all SMs loading and nothing else
//  drew 13.2 (32749 x 3072 x 768 in bf16).  128 x 384 tiles (220 MB; three stages, one accumulator) took as long there and longer
//  at fewer rows (20000 x 384 x 1536 15.9 / 19.9).  A scale word is
//  loaded once per tile, four k-blocks per 16-byte load where the row pitch allows; with each of four warps loading
//  all of a stage's words one by one and writing its own quarter (12 loads of 32 rows each per warp and stage) those
//  loads took longer than the operands.
// All mbarrier waits are bounded; on expiry the CTA sets the status bit and leaves.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcmx {

using namespace rlx::tc;

constexpr int kThreads = 448;           // TMA, MMA, 4 scale warps, 8 epilogue warps
constexpr int kTileM = 128;
constexpr int kBlockK = 128;            // 8-bit elements per stage row = 128 bytes = one swizzle row
constexpr int kOperandBytes = kTileM * kBlockK;
constexpr int kSfGroup = 512;           // scale words of 128 operand rows of one k-block
constexpr int kSfAhead = 4;             // k-blocks whose scale words are handed over together

template <int BN> struct MxCfg {
    static_assert((BN == 128 || BN == 192) && kSfAhead == 4, "");
    static constexpr int STAGES = kSfAhead;                     // stage = k-block modulo kSfAhead, from a tile's first on
    static constexpr int STAGE_BYTES = kOperandBytes + BN * kBlockK;
    static constexpr int W_GROUPS = (BN + 127) / 128;           // 128-row groups of W's scale words; the last may be half used
    static constexpr int SF_BYTES = (1 + W_GROUPS) * kSfGroup;  // one k-block's scale words
    static constexpr int SF_SLOT_BYTES = kSfAhead * SF_BYTES;
    static constexpr int SF_COLS = 4 * (1 + W_GROUPS);
    static constexpr int ACC_COLS = 2 * BN;
    static constexpr int STAGING = 8 * kStageBufBytes;          // one 2 KB chunk buffer per epilogue warp (TMA-store source)
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 2 * SF_SLOT_BYTES + STAGING + 256 + 1024;
    static_assert(ACC_COLS + 2 * kSfAhead * SF_COLS <= 512 && SMEM_BYTES <= 232448, "");
};

// element format ids of the instruction descriptor
constexpr int kFmtE4M3 = 0, kFmtE5M2 = 1;

// Instruction descriptor of kind::mxf8f6f4 with block scaling: [4,6) scale id of B, [7,10) A format,
// [10,13) B format, [15] / [16] A / B major (0 = K-major), [17,23) N >> 3, [23] scale format (1 = E8M0),
// [24,29) M >> 4, [29,31) scale id of A.  fp32 accumulation is implied.
template <int BN>
__device__ __forceinline__ uint32_t idesc_mx(int a_fmt, int b_fmt, int sf_id) {
    return ((uint32_t)sf_id << 4) | ((uint32_t)a_fmt << 7) | ((uint32_t)b_fmt << 10) | ((uint32_t)(BN >> 3) << 17) |
           (1u << 23) | ((uint32_t)(kTileM >> 4) << 24) | ((uint32_t)sf_id << 29);
}
// The issuing instructions take the elected lane as a predicate instead of standing under a branch: in converged code
// the compiler keeps their operands in uniform registers, under a branch it moves each one there again for every
// instruction.
__device__ __forceinline__ void umma_mx(uint32_t elected, uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t tmem_sfa, uint32_t tmem_sfb, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %6, 0;\n"
        "setp.ne.b32 q, %7, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%4], [%5], p;\n"
        "}\n" ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(tmem_sfa), "r"(tmem_sfb), "r"(accumulate), "r"(elected)
        : "memory");
}
// 32 rows of 16 bytes (8-row groups 128 bytes apart, no swizzle) into four tensor-memory columns of every lane quarter
__device__ __forceinline__ void copy_scales(uint32_t elected, uint32_t tmem_dst, uint32_t smem_src) {
    const uint64_t desc = (uint64_t)((smem_src & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %2, 0;\n"
        "@q tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;\n"
        "}\n" ::"r"(tmem_dst), "l"(desc), "r"(elected) : "memory");
}
__device__ __forceinline__ void commit_if(uint32_t elected, uint32_t bar) {
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar), "r"(elected) : "memory");
}

struct MxParams {
    const uint8_t* sfa;     // [M, K/32] scale bytes of A
    const uint8_t* sfw;     // [N, K/32] scale bytes of W
    const float* bias;      // [N] or nullptr
    __nv_bfloat16* out;     // [M, N]
    int M, N, K;
    int a_fmt, w_fmt;       // kFmtE4M3 / kFmtE5M2
    int32_t* status;
};

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
gemm_mx_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                       const __grid_constant__ CUtensorMap tmap_out, MxParams p) {
    using C = MxCfg<BN>;
    constexpr int ST = C::STAGES;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t staging = base + ST * C::STAGE_BYTES;
    constexpr int kSfOff = ST * C::STAGE_BYTES + C::STAGING;
    const uint32_t scales = base + kSfOff;
    const uint32_t bars = scales + 2 * C::SF_SLOT_BYTES;
    const uint32_t full = bars, empty = full + 8 * ST, tfull = empty + 8 * ST, tempty = tfull + 16;
    const uint32_t sfull = tempty + 16, sempty = sfull + 16;   // scale words of kSfAhead k-blocks, two slots
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + kSfOff + 2 * C::SF_SLOT_BYTES + 8 * (2 * ST + 8));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int n_tiles = p.N / BN, m_tiles = (p.M + kTileM - 1) / kTileM, num_tiles = n_tiles * m_tiles;
    const int nkb = p.K / kBlockK;

    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) { mbar_init(full + 8 * i, 1); mbar_init(empty + 8 * i, 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull + 8 * i, 1); mbar_init(tempty + 8 * i, 8);
            mbar_init(sfull + 8 * i, 4); mbar_init(sempty + 8 * i, 1);
        }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap_a);
        prefetch_tmap(&tmap_w);
        prefetch_tmap(&tmap_out);
    }
    if (warp == 1) {
        tmem_alloc<1>(smem_u32(tmem_slot), 512);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);
    pdl_wait();   // codes and scales come from the kernel in front

    // Stage u of the ring holds the k-blocks u, u + 4, ... of every tile (a tile of fewer leaves some out), so that stage
    // addresses are constants of the unrolled loops.  With the addresses formed per stage, under a branch for the elected
    // lane and behind a blocking wait, a stage took the issuing warp 700 cycles (340 of them the four products and their
    // commit) where the tensor core needs 256 or 384; in this form 36736 x 384 x 1536 with its quantiser 57.2 -> 55.6 us.
    if (warp == 0) {
        uint32_t ph = 0xFu;   // one bit per stage; a fresh barrier passes the wait for the phase before its first
        bool ok = true;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
            const int m0 = (tile / n_tiles) * kTileM, n0 = (tile % n_tiles) * BN;
            for (int kb0 = 0; kb0 < nkb && ok; kb0 += ST) {
#pragma unroll
                for (int u = 0; u < ST; ++u) {
                    if (kb0 + u < nkb && ok) {
                        ok = mbar_wait_warp(empty + 8 * u, ph >> u & 1, abort_flag);
                        ph ^= 1u << u;
                        if (ok && elect_one()) {
                            const uint32_t dst = base + u * C::STAGE_BYTES;
                            mbar_expect_tx(full + 8 * u, C::STAGE_BYTES);
                            tma_load_2d(dst, &tmap_a, (kb0 + u) * kBlockK, m0, full + 8 * u);
                            tma_load_2d(dst + kOperandBytes, &tmap_w, (kb0 + u) * kBlockK, n0, full + 8 * u);
                        }
                        __syncwarp();
                    }
                }
            }
        }
    } else if (warp == 1) {
        const uint32_t elected = elect_one() ? 1u : 0u;
        const uint64_t adesc0 = make_smem_desc(base), bdesc0 = make_smem_desc(base + kOperandBytes);
        const uint32_t idesc0 = idesc_mx<BN>(p.a_fmt, p.w_fmt, 0);
        uint32_t ph = 0, tcount = 0, ss = 0, sph = 0;
        // A group of four k-blocks' scale words goes to tensor memory at once, and a group ahead of its products where the words are
        // there: copies and products run in the order they are issued, and a product right behind the copy that it needs waits for
        // all of that copy's latency (product alone, 36736 x 384 x 1536 23.0 -> 21.4 us, 20000 rows 18.8 -> 16.8).  That order is also
        // all that keeps a copy into a slot behind the products of the group before last, which read it: `sempty` frees the words
        // in shared memory, once they are copied.
        auto copy_group = [&](uint32_t slot) {
#pragma unroll
            for (int u = 0; u < ST; ++u)
#pragma unroll
                for (int g = 0; g <= C::W_GROUPS; ++g)
                    copy_scales(elected, tmem + C::ACC_COLS + (slot * ST + u) * C::SF_COLS + 4 * g, scales + slot * C::SF_SLOT_BYTES + u * C::SF_BYTES + g * kSfGroup);
            commit_if(elected, sempty + 8 * slot);
        };
        // the next wait's outcome is asked for before the current stage is issued: a round to a barrier takes 100-150 cycles
        bool ok = true, ready = false, copied = false;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++tcount) {
            const uint32_t as = tcount & 1, ause = tcount >> 1;
            if (ause >= 1 && !(ok = mbar_wait_warp(tempty + 8 * as, (ause - 1) & 1, abort_flag))) break;
            const uint32_t acc = tmem + as * BN;
            for (int kb0 = 0; kb0 < nkb && ok; kb0 += ST) {
                if (!copied) {
                    if (!(ok = mbar_wait_warp(sfull + 8 * ss, sph, abort_flag))) break;
                    tc_fence_after();
                    copy_group(ss);
                }
                const uint32_t sf = tmem + C::ACC_COLS + ss * (kSfAhead * C::SF_COLS);
                ss ^= 1; sph ^= ss ^ 1;
                copied = (kb0 + ST < nkb || tile + (int)gridDim.x < num_tiles) && __all_sync(0xffffffffu, mbar_test_wait(sfull + 8 * ss, sph)) != 0;
                if (copied) {
                    tc_fence_after();
                    copy_group(ss);
                }
#pragma unroll
                for (int u = 0; u < ST; ++u) {
                    if (kb0 + u < nkb && ok) {
                        if (!__all_sync(0xffffffffu, ready)) ok = mbar_wait_warp(full + 8 * u, ph >> u & 1, abort_flag);
                        ph ^= 1u << u;
                        tc_fence_after();
                        const bool last = kb0 + u == nkb - 1;
                        const int nu = last ? 0 : (u + 1) % ST;
                        ready = mbar_test_wait(full + 8 * nu, ph >> nu & 1);
                        if (!ok) break;
#pragma unroll
                        for (int k = 0; k < kBlockK / 32; ++k)   // 32 bytes of k per instruction: descriptor start + 2
                            umma_mx(elected, acc, adesc0 + (u * (C::STAGE_BYTES >> 4) + 2 * k), bdesc0 + (u * (C::STAGE_BYTES >> 4) + 2 * k),
                                    idesc0 + ((uint32_t)k << 4 | (uint32_t)k << 29), sf + u * C::SF_COLS, sf + u * C::SF_COLS + 4,
                                    (u | k) != 0 ? 1u : (kb0 != 0 ? 1u : 0u));
                        commit_if(elected, empty + 8 * u);
                        if (last) commit_if(elected, tfull + 8 * as);
                    }
                }
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------ scale feed: 32 rows of every 128 per warp
        // Four k-blocks of a row at a time, requested as soon as the four before them are handed over, across tiles too.
        const int q = warp - 2;
        const int ld = p.K / 128;                      // scale words per row
        const bool vec = (ld & 3) == 0;                // 16-byte loads: rows start on 16 bytes
        const uint32_t* sfa = reinterpret_cast<const uint32_t*>(p.sfa);
        const uint32_t* sfw = reinterpret_cast<const uint32_t*>(p.sfw);
        auto load4 = [&](const uint32_t* row, int kb0, uint32_t (&r)[kSfAhead]) {
            if (vec) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + kb0));
                r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
            } else {
#pragma unroll
                for (int u = 0; u < kSfAhead; ++u)
                    if (kb0 + u < nkb) r[u] = __ldg(row + kb0 + u);
            }
        };
        auto fetch = [&](int tile, int kb0, uint32_t (&r)[1 + C::W_GROUPS][kSfAhead]) {
            const int ar = (tile / n_tiles) * kTileM + 32 * q + lane, n0 = (tile % n_tiles) * BN;
            // rows past M are zero-filled operand rows: any finite scale will do
            if (ar < p.M) load4(sfa + (size_t)ar * ld, kb0, r[0]);
            else r[0][0] = r[0][1] = r[0][2] = r[0][3] = 0x7F7F7F7Fu;
#pragma unroll
            for (int g = 0; g < C::W_GROUPS; ++g)
                if (128 * g + 32 * q < BN) load4(sfw + (size_t)(n0 + 128 * g + 32 * q + lane) * ld, kb0, r[1 + g]);
        };
        uint32_t cur[1 + C::W_GROUPS][kSfAhead] = {};
        const uint32_t slot_addr = scales + lane * 16 + q * 4;
        uint32_t ss = 0, sph = 1;
        int tile = blockIdx.x, kb0 = 0;
        bool ok = true;
        if (tile < num_tiles) fetch(tile, 0, cur);
        while (tile < num_tiles && ok) {
            if (!(ok = mbar_wait(sempty + 8 * ss, sph, abort_flag))) break;
#pragma unroll
            for (int u = 0; u < kSfAhead; ++u)
#pragma unroll
                for (int g = 0; g <= C::W_GROUPS; ++g)
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(slot_addr + ss * C::SF_SLOT_BYTES + u * C::SF_BYTES + g * kSfGroup), "r"(cur[g][u]) : "memory");
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(sfull + 8 * ss);
            ss ^= 1; sph ^= ss ^ 1;
            kb0 += kSfAhead;
            if (kb0 >= nkb) { tile += gridDim.x; kb0 = 0; }
            if (tile < num_tiles) fetch(tile, kb0, cur);   // behind the fence, which would wait for it
        }
    } else {
        // ------------------------------------------------------------ epilogue: lane quarter x half of the columns
        // the bf16 GEMM's epilogue tile: all chunks to registers, accumulator handed back, bias, one
        // TMA store per 32 x 32 chunk out of the warp's swizzled staging buffer
        constexpr int NC = BN / 64;
        const int quad = warp & 3, half = (warp - 6) >> 2, ew = warp - 6;
        const uint32_t stg = staging + ew * kStageBufBytes;
        Params gp = {};
        gp.bias = p.bias; gp.out = p.out; gp.M = p.M; gp.N = p.N; gp.K = p.K; gp.status = p.status;
        uint32_t tcount = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++tcount) {
            const int m_row0 = (tile / n_tiles) * kTileM + quad * 32, n0 = (tile % n_tiles) * BN + half * (BN / 2);
            const uint32_t as = tcount & 1;
            if (!(ok = mbar_wait(tfull + 8 * as, (tcount >> 1) & 1, abort_flag))) break;
            tc_fence_after();
            EpilogueTile<0, NC> et;
            et.template drain<1>(gp, &tmap_out, p.M, m_row0, n0, tmem + ((uint32_t)(quad * 32) << 16) + as * BN + half * (BN / 2),
                                 stg, lane, tempty + 8 * as, 0u);
        }
        EpilogueTile<0, NC>::finish(lane);
    }
    // ---------------------------------------------------------------- teardown
    if (*abort_flag) {
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, RLX_DEVSTAT_TIMEOUT_BIT);
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, 512);
    }
}

// ---------------------------------------------------------------------------- activation quantiser
template <bool E5M2>
__device__ __forceinline__ uint16_t cvt_fp8x2(float lo, float hi) {
    uint16_t r;
    if (E5M2) asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    else      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

constexpr int kQuantThreads = 256;
constexpr int kQuantIters = 4;                                       // 16-byte loads in flight per lane
constexpr int kQuantWarpBlocks = 8 * kQuantIters;                    // 32-element blocks per warp
constexpr int kQuantCtaBlocks = kQuantThreads / 32 * kQuantWarpBlocks;

// x bf16 [M, K] -> codes [M, K] bytes, scales [M, K/32] bytes.  Bound by DRAM: 2 bytes in and 1 + 1/32 out per element.
// Four lanes share a block of 32, so that a warp's loads (16 bytes a lane) and its stores (8 bytes) are contiguous, and
// the shared exponent comes from the exponent field of the packed maximum; the warp's 32 scale bytes leave as one store.
// (One thread per block of 64 bytes, with ilogbf and scalbnf per element, took 46 us for 36736 x 1536.)
template <bool E5M2>
__global__ void __launch_bounds__(kQuantThreads)
quantise_mx_kernel(const __nv_bfloat16* __restrict__ x, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                   long long blocks) {
    constexpr int kEmax = E5M2 ? 15 : 8;
    pdl_launch_dependents();   // a product behind it sets itself up meanwhile
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long b0 = (long long)blockIdx.x * kQuantCtaBlocks + warp * kQuantWarpBlocks;
    uint4 in[kQuantIters];
#pragma unroll
    for (int i = 0; i < kQuantIters; ++i) {
        const long long b = b0 + 8 * i + (lane >> 2);
        in[i] = b < blocks ? __ldcs(reinterpret_cast<const uint4*>(x + b * 32) + (lane & 3)) : make_uint4(0, 0, 0, 0);
    }
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < kQuantIters; ++i) {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(&in[i]);
        // packed maximum of the magnitudes; a NaN loses against any number, as in fmaxf
        __nv_bfloat162 m2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t a = w[j] & 0x7FFF7FFFu;
            m2 = __hmax2(m2, *reinterpret_cast<const __nv_bfloat162*>(&a));
        }
        uint32_t m = *reinterpret_cast<uint32_t*>(&m2);
        m = max(m & 0xFFFFu, m >> 16);                 // non-negative numbers: their bits order as they do
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const int e = (int)(m >> 7);                   // exponent field; zero for a subnormal maximum
        int s = m == 0 ? 0 : e == 255 ? 127 : max(e - 127 - kEmax, -127);   // infinity takes the largest scale
        // 2^-s; 2^-127 is subnormal
        const float f = s == 127 ? __uint_as_float(0x00400000u) : __uint_as_float((uint32_t)(127 - s) << 23);
        uint2 o;
        o.x = cvt_fp8x2<E5M2>(bf16lo(w[0]) * f, bf16hi(w[0]) * f) | (uint32_t)cvt_fp8x2<E5M2>(bf16lo(w[1]) * f, bf16hi(w[1]) * f) << 16;
        o.y = cvt_fp8x2<E5M2>(bf16lo(w[2]) * f, bf16hi(w[2]) * f) | (uint32_t)cvt_fp8x2<E5M2>(bf16lo(w[3]) * f, bf16hi(w[3]) * f) << 16;
        const long long b = b0 + 8 * i + (lane >> 2);
        if (b < blocks) *(reinterpret_cast<uint2*>(codes + b * 32) + (lane & 3)) = o;
        // lane l keeps the byte of block 8 (l & 3) + (l >> 2): its own four-lane group's, of iteration l & 3
        if ((lane & 3) == i) mine = (uint32_t)(s + 127);
    }
    const long long b = b0 + 8 * (lane & 3) + (lane >> 2);
    if (b < blocks) scales[b] = (uint8_t)mine;
}

}  // namespace tcmx
}  // namespace rlx

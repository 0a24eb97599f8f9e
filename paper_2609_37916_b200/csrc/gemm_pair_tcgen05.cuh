// bf16 "Linear" GEMM of a CTA pair whose tile width is chosen on the device: out[M,N] = epilogue(A[M,K] W[N,K]^T + bias), K from
// 1536 on, N a multiple of 384 (the feed-forward down products).
//
// A packed batch has fewer rows than the host knows of (its padded count), and how wide a tile should be depends on them: as wide
// as possible while all tiles run beside each other, narrower where that fills pairs that would idle.  61 sequences of
// up to 203 at N = 384: 29 row blocks are 58 tiles of 192 columns, one round of 74 pairs, or 87 of 128, two; with every position
// valid 49 are 98 or 147, two rounds each, and the narrow ones are shorter.
// So the width is a variable here; the rest is gemm_tcgen05.cuh's pair kernel, with its stages of each width (192 columns in three
// stages of two k-blocks instead of seven of one: 12 x 768, 20 x 512 with all positions valid 2477 us where the fixed kernel took 2424, now 2441).  The loops of
// the producer and the issuer are compiled for each width, nothing is divided, and shared memory is left for the CTAs of the next
// kernel: where the width comes out as the fixed kernel's, that much less is lost (us fixed / chosen, 6 x 384, before and now: 50 x 128 with
// half of the positions valid 272.7 / 276.4 and 273.4 / 274.0, 64 x 128 288.1 / 292.4 and 288.6 / 290.9, 24 x 400 384.4 / 390.2 and 385.9 / 389.2).
// The order along K does not depend on the width: the bits are the same with each.
#pragma once
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcpw {

using namespace rlx::tc;

constexpr int kMaxBN = 192, kMaxStages = 7;
constexpr int kABytes = BLOCK_M * BLOCK_K * 2;
constexpr int kEpiWarps = 12, kThreads = 64 + 32 * kEpiWarps;
constexpr int kBarBytes = 8 * (2 * kMaxStages + 4) + 16;
template <int EPI>
struct Cfg {
    static constexpr bool VEC = EPI >= 3;
    static constexpr int VEC_BYTES = VEC ? kEpiWarps * 384 : 0;
    static constexpr int RING_BYTES = kMaxStages * (kABytes + 96 * BLOCK_K * 2);   // seven k-blocks at 192 columns, four pairs of them at 128
    static constexpr int STG_OFF = RING_BYTES, VEC_OFF = STG_OFF + kEpiWarps * kStageBufBytes, BAR_OFF = VEC_OFF + VEC_BYTES, SMEM_BYTES = BAR_OFF + kBarBytes + 1024;
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");
};
struct Widths {
    CUtensorMap a1;               // A by single k-blocks
    CUtensorMap w[3];             // W, boxes of 32, 64 and 96 rows: a CTA's half of a tile of 64, 128 (pairs of k-blocks) and 192 columns (single ones)
    int n_tiles[3];               // tiles of a row block at each width
    uint32_t inv[3], inv_pairs;   // reciprocals of those and of the number of pairs, see div_by
};
// x / n by the reciprocal 2^32 / n + 1 (2^32 / n for a power of two; n > 1): exact for x < 2^32 / n.  A division by a variable is forty instructions that a kernel of one
// tile per pair fetches for the first time, in front of its first load.
__host__ __device__ __forceinline__ uint32_t reciprocal(uint32_t n) { return 0xffffffffu / n + 1u; }
__device__ __forceinline__ int div_by(uint32_t x, uint32_t inv) { return (int)__umulhi(x, inv); }

// Columns of a tile, in units of 64, for `blocks` 256-row blocks: the least rounds times the clocks that a k-block takes (measured:
// operands at 70 bytes a clock and SM, at N = 64 the round to the barriers).
__device__ __forceinline__ int pick_width(const Widths& wm, int blocks, int pairs) {
    int best = 3, cost = 0x7fffffff;
#pragma unroll
    for (int w = 3; w >= 1; --w) {
        const int c = div_by(blocks * wm.n_tiles[w - 1] + pairs - 1, wm.inv_pairs) * (w == 3 ? 410 : w == 2 ? 351 : 310);
        if (c < cost) { cost = c; best = w; }
    }
    return best;
}

// k-blocks of a stage, as in gemm_tcgen05.cuh's Cfg: narrow tiles take two behind one barrier round, wide ones a deeper ring.
constexpr int kps(int width) { return width == 3 ? 1 : 2; }

// The loops of the producer and of the issuer, for each width: with stage size, box and instruction shape as variables a stage takes
// the issuing thread longer than its products.
template <int EPI, int WIDTH>
struct Loop {
    static constexpr int KPS = kps(WIDTH), BN = 64 * WIDTH, B_ROWS = 32 * WIDTH, B_BYTES = B_ROWS * BLOCK_K * 2, STAGE_BYTES = KPS * (kABytes + B_BYTES);
    static constexpr int FIT = Cfg<EPI>::RING_BYTES / STAGE_BYTES, STAGES = FIT < kMaxStages ? FIT : kMaxStages;
    static_assert(STAGES >= 4, "ring too shallow");

    static __device__ __forceinline__ void produce(const CUtensorMap* map_a, const CUtensorMap* map_w, uint32_t base, uint32_t full_bar,
                                                   uint32_t empty_bar, int n_tiles, uint32_t inv, int num_tiles, int num_kb, int pairs, uint32_t cta_rank,
                                                   volatile int* abort_flag) {
        int stage = 0;
        uint32_t phase = 1;
        for (int tile = blockIdx.x / 2; tile < num_tiles; tile += pairs) {
            const int m_blk = div_by(tile, inv);
            const int arow = m_blk * 256 + (int)cta_rank * BLOCK_M, brow = (tile - m_blk * n_tiles) * BN + (int)cta_rank * B_ROWS;
            for (int kb = 0; kb < num_kb; kb += KPS) {
                if (!mbar_wait_warp(empty_bar + 8 * stage, phase, abort_flag)) return;
                if (elect_one()) {
                    const uint32_t st = base + stage * STAGE_BYTES, lead_full = map_to_cta(full_bar + 8 * stage, 0);
                    if (cta_rank == 0) mbar_expect_tx(full_bar + 8 * stage, 2 * STAGE_BYTES);
                    tma_load_3d_cg2(st, map_a, 0, arow, kb, lead_full);
                    tma_load_3d_cg2(st + KPS * kABytes, map_w, 0, brow, kb, lead_full);
                }
                __syncwarp();
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
    }

    static __device__ __forceinline__ void issue(uint32_t tmem, uint32_t base, uint32_t full_bar, uint32_t empty_bar, uint32_t tfull_bar,
                                                 uint32_t tempty_bar, int num_tiles, int num_kb, int pairs, volatile int* abort_flag) {
        constexpr uint32_t idesc = make_idesc(256, BN);
        const uint64_t ad0 = make_smem_desc(base), bd0 = make_smem_desc(base + KPS * kABytes);
        uint32_t stage = 0, phase = 0;
        int it = 0;
        for (int tile = blockIdx.x / 2; tile < num_tiles; tile += pairs, ++it) {
            const int as = it & 1;
            if (!mbar_wait_warp(tempty_bar + 8 * as, ((it >> 1) & 1) ^ 1, abort_flag)) return;
            tc_fence_after();
            const uint32_t acc = tmem + as * kMaxBN;
            for (int kb = 0; kb < num_kb; kb += KPS) {
                if (!mbar_wait_warp(full_bar + 8 * stage, phase, abort_flag)) return;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t ad = ad0 + stage * (STAGE_BYTES >> 4), bd = bd0 + stage * (STAGE_BYTES >> 4);
#pragma unroll
                    for (int i = 0; i < KPS; ++i)
#pragma unroll
                        for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                            umma_bf16<2>(acc, ad + (i * (kABytes >> 4) + 2 * k), bd + (i * (B_BYTES >> 4) + 2 * k), idesc, (kb | i | k) != 0 ? 1u : 0u);
                    umma_commit<2>(empty_bar + 8 * stage);
                }
                __syncwarp();
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (elect_one()) umma_commit<2>(tfull_bar + 8 * as);
            __syncwarp();
        }
    }
};

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
gemm_pair_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ Widths wm,
                         const __grid_constant__ CUtensorMap tmap_out, const Params p) {
    using C = Cfg<EPI>;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t full_bar = base + C::BAR_OFF, empty_bar = full_bar + 8 * kMaxStages;
    const uint32_t tfull_bar = empty_bar + 8 * kMaxStages, tempty_bar = tfull_bar + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + C::BAR_OFF + 8 * (2 * kMaxStages + 4));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t cta_rank = warp_uniform(cluster_ctarank());   // rank 0 leads the pair
    pdl_launch_dependents();

    int M = p.M;
    if (p.m_ptr != nullptr) M = min(M, ld_early(p.m_ptr));
    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(full_bar + 8 * i, 1); mbar_init(empty_bar + 8 * i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull_bar + 8 * i, 1); mbar_init(tempty_bar + 8 * i, 2 * kEpiWarps); }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap_a);
        prefetch_tmap(&wm.a1);
        prefetch_tmap(&tmap_out);
    }
    if (warp == 1) {
        tmem_alloc<2>(smem_u32(tmem_slot), 512);
        tmem_relinquish<2>();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);

    const int pairs = gridDim.x / 2, m_tiles = (M + 255) / 256, num_kb = p.K / BLOCK_K;
    const int width = (int)warp_uniform((uint32_t)pick_width(wm, m_tiles, pairs)), bn = 64 * width;
    const int n_tiles = width == 3 ? wm.n_tiles[2] : width == 2 ? wm.n_tiles[1] : wm.n_tiles[0], num_tiles = n_tiles * m_tiles;
    const uint32_t inv = width == 3 ? wm.inv[2] : width == 2 ? wm.inv[1] : wm.inv[0];

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
        const CUtensorMap* map_w = &wm.w[width - 1];
        if (lane == 0) prefetch_tmap(map_w);
        __syncwarp();
        pdl_wait();
        if (width == 3) Loop<EPI, 3>::produce(&wm.a1, map_w, base, full_bar, empty_bar, n_tiles, inv, num_tiles, num_kb, pairs, cta_rank, abort_flag);
        else if (width == 2) Loop<EPI, 2>::produce(&tmap_a, map_w, base, full_bar, empty_bar, n_tiles, inv, num_tiles, num_kb, pairs, cta_rank, abort_flag);
        else Loop<EPI, 1>::produce(&tmap_a, map_w, base, full_bar, empty_bar, n_tiles, inv, num_tiles, num_kb, pairs, cta_rank, abort_flag);
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader CTA, whole warp, one lane issues)
        if (cta_rank == 0) {
            if (width == 3) Loop<EPI, 3>::issue(tmem, base, full_bar, empty_bar, tfull_bar, tempty_bar, num_tiles, num_kb, pairs, abort_flag);
            else if (width == 2) Loop<EPI, 2>::issue(tmem, base, full_bar, empty_bar, tfull_bar, tempty_bar, num_tiles, num_kb, pairs, abort_flag);
            else Loop<EPI, 1>::issue(tmem, base, full_bar, empty_bar, tfull_bar, tempty_bar, num_tiles, num_kb, pairs, abort_flag);
        }
    } else {
        // ------------------------------------------------------------ epilogue warps: 32 rows x 64 columns, as many groups as the tile has
        const int ew = warp - 2, quad = warp & 3, half = ew >> 2;
        const uint32_t stg = base + C::STG_OFF + ew * kStageBufBytes;
        using ET = EpilogueTile<EPI, 2, C::VEC>;
        if ((int)blockIdx.x / 2 < num_tiles && half < width) ET::prefetch_bias(p, ((int)blockIdx.x / 2 - div_by(blockIdx.x / 2, inv) * n_tiles) * bn + half * 64);
        pdl_wait();
        int it = 0;
        bool ok = true;
        for (int tile = blockIdx.x / 2; tile < num_tiles && ok; tile += pairs, ++it) {
            const int as = it & 1;
            const uint32_t ph = (it >> 1) & 1;
            if (half >= width) {                     // columns that this width does not have
                if (tile + 2 * pairs >= num_tiles) break;   // nobody waits for this accumulator again
                if (!(ok = mbar_wait_warp(tfull_bar + 8 * as, ph, abort_flag))) break;
                if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(tempty_bar + 8 * as, 0));
                continue;
            }
            const int m_blk = div_by(tile, inv);
            const int m_row0 = m_blk * 256 + (int)cta_rank * BLOCK_M + quad * 32, n0 = (tile - m_blk * n_tiles) * bn + half * 64;
            const int next = tile + pairs;
            if (next < num_tiles) ET::prefetch_bias(p, (next - div_by(next, inv) * n_tiles) * bn + half * 64);
            ET et;
            et.load_vectors(p, n0, base + C::VEC_OFF + ew * 384);
            et.prefetch(p, M, m_row0 + lane, n0);
            if (!(ok = mbar_wait_warp(tfull_bar + 8 * as, ph, abort_flag))) break;
            tc_fence_after();
            et.template drain<2>(p, &tmap_out, M, m_row0, n0, tmem + ((uint32_t)(quad * 32) << 16) + as * kMaxBN + half * 64, stg, lane,
                                 tempty_bar + 8 * as, cta_rank);
        }
        ET::finish(lane);
    }
    // ---------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        if (threadIdx.x == 0 && p.status) atomicOr(p.status, RLX_DEVSTAT_TIMEOUT_BIT);
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();      // neither CTA leaves while the pair still uses its memory
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<2>(tmem, 512);
    }
}

}  // namespace tcpw
}  // namespace rlx

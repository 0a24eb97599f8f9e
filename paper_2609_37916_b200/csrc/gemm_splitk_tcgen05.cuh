// bf16 "Linear" GEMM for few rows and a long contraction: out[M,N] = epilogue(A[M,K] W[N,K]^T + bias), split along K
// over a cluster.
//
// `S` CTAs, a cluster or a part of one, take one 128 x 64 tile and K / S of its contraction each (TMA -> tcgen05, as in
// gemm_tcgen05.cuh; the W tiles are requested in front of the wait for the previous kernel). The tile's
// 32 x 32 units are dealt out to the CTAs: every CTA sends its partial sums of a unit to the unit's owner with
// st.async (data and arrival in one, no fence), and the owner adds them in rank order -- the result does not
// depend on timing -- and runs the ordinary epilogue. Only units with rows that exist are sent.
// Only the 32-row groups of A that exist are loaded.
//
// What bounds it: with one CTA per tile the operands of a 128 x 64 x 1536 tile are 590 KB through one SM's L2 port at
// 80 bytes per clock, 4.6 us of a 7.3 us kernel; four CTAs need 1.2 us and the exchange about 0.7.
// All waits are bounded.
#pragma once
#include "gemm_cln_tcgen05.cuh"
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcsk {

using namespace rlx::tc;
using rlx::tccl::mbar_wait_cluster;

constexpr int kBN = 64;
constexpr int kMaxSplit = 4;
constexpr int kUnitBytes = 32 * 32 * 4;        // fp32 partial sums of a 32 x 32 unit
constexpr int kStages = 3;                     // of two 64-wide k-blocks each: a quarter of K = 1536 without reuse
constexpr int kKps = 2;
constexpr int kABytes = BLOCK_M * BLOCK_K * 2, kBBytes = kBN * BLOCK_K * 2;
constexpr int kStageBytes = kKps * (kABytes + kBBytes);
constexpr int kEpiWarps = 8;                   // (quadrant, column half)
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kXchOff = kStages * kStageBytes; // partial sums received: [local unit][source rank]
constexpr int kXchBytes = 8 * kUnitBytes;      // 8 / S units from S sources
constexpr int kStagingOff = kXchOff + kXchBytes;
constexpr int kVecOff = kStagingOff + kEpiWarps * kStageBufBytes;   // per-column vectors, see EpilogueTile
constexpr int kBarOff = kVecOff + kEpiWarps * 384;
constexpr int kSmemBytes = kBarOff + 8 * (2 * kStages + 2) + 16 + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, const uint32_t* v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];"
                 ::"r"(addr), "r"(bar), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
gemm_splitk_tcgen05_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                           const __grid_constant__ CUtensorMap tmap_out, const Params p) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t full_bar = base + kBarOff, empty_bar = full_bar + 8 * kStages, acc_bar = empty_bar + 8 * kStages;
    const uint32_t xch_bar = acc_bar + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + kBarOff + 8 * (2 * kStages + 2));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_launch_dependents();

    int M = p.M;
    if (p.m_ptr != nullptr) M = min(M, ld_early(p.m_ptr));
    const int n_tiles = p.N / kBN;
    // CTAs per tile: as many as there are in a cluster, fewer when the tiles that exist (the host knows the padded row count
    // only) would not all run beside each other; the cluster then holds several tiles.
    const int existing = (M + BLOCK_M - 1) / BLOCK_M * n_tiles, crank = (int)warp_uniform(cluster_ctarank());
    int S = (int)tccl::cluster_nctarank();
    if (S == 4 && existing > p.split_tiles4) S = 2;
    if (S == 2 && existing > p.split_tiles2) S = 1;
    const int rank = crank % S, first = crank - rank;        // rank among the tile's CTAs, cluster rank of its first one
    const int tile = blockIdx.x / S, m_blk = tile / n_tiles, n_blk = tile % n_tiles;
    const int rows = min(BLOCK_M, M - m_blk * BLOCK_M);      // rows of this tile that exist (<= 0: none)
    const int groups = rows > 0 ? (rows + 31) / 32 : 0;      // 32-row groups
    const int units = 2 * groups;                            // unit u = (group u / 2, column half u % 2), owner u % S
    const int mine = units > rank ? (units - rank + S - 1) / S : 0;
    const int num_kb = (p.K + BLOCK_K - 1) / BLOCK_K, per = (num_kb + S - 1) / S;
    const int kb0 = min(rank * per, num_kb), kb1 = min(kb0 + per, num_kb);

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(full_bar + 8 * i, 1); mbar_init(empty_bar + 8 * i, 1); }
        mbar_init(acc_bar, 1);
        mbar_init(xch_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap_a);
        prefetch_tmap(&tmap_b);
        prefetch_tmap(&tmap_out);
        if (mine > 0) mbar_expect_tx(xch_bar, (uint32_t)(mine * S * kUnitBytes));
    }
    if (warp == 1) {
        tmem_alloc<1>(smem_u32(tmem_slot), 64);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();      // the peers' barriers exist before anything is sent to them
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
        auto load_w = [&](int kb, int stage) {
            const int cnt = min(kKps, kb1 - kb);
            mbar_expect_tx(full_bar + 8 * stage, (uint32_t)(cnt * (kBBytes + groups * 32 * BLOCK_K * 2)));
            for (int i = 0; i < cnt; ++i)
                tma_load_2d(base + stage * kStageBytes + kKps * kABytes + i * kBBytes, &tmap_b, (kb + i) * BLOCK_K, n_blk * kBN, full_bar + 8 * stage);
        };
        auto load_a = [&](int kb, int stage) {
            const int cnt = min(kKps, kb1 - kb);
            for (int i = 0; i < cnt; ++i)
                for (int g = 0; g < groups; ++g)
                    tma_load_2d(base + stage * kStageBytes + i * kABytes + g * 32 * BLOCK_K * 2, &tmap_a, (kb + i) * BLOCK_K,
                                m_blk * BLOCK_M + g * 32, full_bar + 8 * stage);
        };
        int early = 0;
        if (groups > 0)
            for (; early < kStages && kb0 + early * kKps < kb1; ++early) {
                if (elect_one()) load_w(kb0 + early * kKps, early);
                __syncwarp();
            }
        pdl_wait();
        if (groups > 0) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; kb += kKps) {
                if (early > 0) {
                    --early;
                    if (elect_one()) load_a(kb, stage);
                } else {
                    if (!mbar_wait_warp(empty_bar + 8 * stage, phase ^ 1, abort_flag)) break;
                    if (elect_one()) { load_w(kb, stage); load_a(kb, stage); }
                }
                __syncwarp();
                if (++stage == kStages) { stage = 0; phase ^= 1; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
        if (groups > 0) {
            constexpr uint32_t idesc = make_idesc(BLOCK_M, kBN);
            const uint64_t adesc0 = make_smem_desc(base), bdesc0 = make_smem_desc(base + kKps * kABytes);
            uint32_t stage = 0, phase = 0;
            bool ok = true, ready = false;
            for (int kb = kb0; kb < kb1; kb += kKps) {
                const int cnt = min(kKps, kb1 - kb);
                if (!__all_sync(0xffffffffu, ready) && !(ok = mbar_wait_warp(full_bar + 8 * stage, phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t cur = stage;
                if (++stage == kStages) { stage = 0; phase ^= 1; }
                ready = mbar_test_wait(full_bar + 8 * stage, phase);
                if (elect_one()) {
                    const uint64_t ad0 = adesc0 + cur * (kStageBytes >> 4), bd0 = bdesc0 + cur * (kStageBytes >> 4);
#pragma unroll
                    for (int i = 0; i < kKps; ++i)
                        if (i < cnt)
#pragma unroll
                            for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                                umma_bf16<1>(tmem, ad0 + (i * (kABytes >> 4) + 2 * k), bd0 + (i * (kBBytes >> 4) + 2 * k), idesc,
                                             (kb != kb0 || (i | k) != 0) ? 1u : 0u);
                    umma_commit<1>(empty_bar + 8 * cur);
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit<1>(acc_bar);
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------ exchange, then the epilogue of this CTA's units
        const int e = warp - 2, quad = warp & 3, half = e >> 2;
        const int unit = 2 * quad + half;
        // the unit this warp finishes, if it does
        const int u = rank + e * S, ug = u / 2, uh = u % 2;
        const bool finish = e < mine;
        const int m_row0 = m_blk * BLOCK_M + ug * 32, n0 = n_blk * kBN + uh * 32;
        const uint32_t stg = base + kStagingOff + e * kStageBufBytes;
        using ET = EpilogueTile<EPI, 1, true>;
        ET et;
        if (finish) et.load_vectors(p, n0, base + kVecOff + e * 384);
        pdl_wait();
        if (finish) et.prefetch(p, M, m_row0 + lane, n0);
        bool ok = true;
        if (unit < units) {
            ok = mbar_wait_warp(acc_bar, 0, abort_flag);
            if (ok) {
                tc_fence_after();
                uint32_t r[32];
                tmem_ld_32x32(tmem + ((uint32_t)(quad * 32) << 16) + half * 32, r);
                tmem_ld_wait();
                if (kb0 >= kb1)
#pragma unroll
                    for (int i = 0; i < 32; ++i) r[i] = 0;
                const uint32_t dst = map_to_cta(base + kXchOff + ((unit / S) * S + rank) * kUnitBytes + lane * 16, first + unit % S);
                const uint32_t bar = map_to_cta(xch_bar, first + unit % S);
#pragma unroll
                for (int i = 0; i < 8; ++i) st_async_v4(dst + i * 512, bar, r + 4 * i);   // [column quad][row]: no bank conflicts
                tc_fence_before();
            }
        }
        if (finish && ok && mbar_wait_cluster(xch_bar, 0, abort_flag)) {
            const uint32_t src = base + kXchOff + e * S * kUnitBytes + lane * 16;
            float acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint4 q = ld_shared_v4(src + s * kUnitBytes + i * 512);
                    acc[4 * i + 0] += __uint_as_float(q.x); acc[4 * i + 1] += __uint_as_float(q.y);
                    acc[4 * i + 2] += __uint_as_float(q.z); acc[4 * i + 3] += __uint_as_float(q.w);
                }
            uint32_t a[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) a[i] = __float_as_uint(acc[i]);
            const int m = m_row0 + lane;
            uint4 q[4];
            et.compute_chunk(p, a, n0, 0, m, m < M, p.bias + n0, q);
            ET::store_chunk(p, &tmap_out, q, n0, m_row0, stg, lane, lane * 64, (uint32_t)((lane >> 1) & 3));
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
    cluster_sync_all();      // no CTA leaves while a peer may still write into it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, 64);
    }
}

}  // namespace tcsk
}  // namespace rlx

// Packed-sequence attention on the 5th-generation tensor cores: any length, head_dim 32 / 64 / 128, all keys / causal /
// sliding window, plain and grouped-query heads, optional rotary q and k.
//
// A work item is a PAIR of 128-row query tiles that walk the same 128-key blocks, so that the two softmax groups
// of a CTA take turns on the exponential units while the tensor cores work for the other one:
//   PAIR         the same rows of two neighbouring heads with a K / V head each (head_dim 32 / 64; the two heads'
//                columns are neighbours in memory, so one tile brings q, k or v of both)
//   otherwise    the same rows of two query heads of one K / V head (grouped-query layouts), or two consecutive
//                row tiles of one head (everything else: "rows mode")
// Items are numbered with the last row tiles first (under the causal mask these are the long ones), one CTA of the
// grid per item; a CTA that has finished takes over the next one that has not been launched yet
// (clusterlaunchcontrol), so tensor memory and barriers are set up once per SM, the loads of the next item run
// behind the current one, and no counter in global memory is needed: calls on several streams do not meet.
//
//   warps 0..3, 4..7  softmax of tile 0 / tile 1, one thread per query row (no shuffles): 128 scores of a block
//                     from tensor memory to registers, block maximum, exponentials, P (bf16) back over the
//                     scores; at the end of an item O / row sum -> global
//   warp 8            items and TMA: Q tiles, then K and V blocks through one ring
//   warp 9            MMA issue:  S_t = Q_t K^T, O_t += P_t V (P read from tensor memory, V MN-major);
//                     in the order PV_0(j) S_0(j+1) PV_1(j) S_1(j+1), across item boundaries too
//   warps 12..15      (rotary form only) rotate the Q tiles and K blocks in shared memory before they are used
//
// The reference maximum of a row stays the one of its first block unless a later block exceeds it by more than 2^8
// (then P <= 256 is still exact in range); only then is the row of O rescaled in tensor memory.  S_t(j+1) is issued
// behind PV_t(j) by the same thread, so a warp that has seen S_t(j+1) may read and write O_t.
// All mbarrier waits are bounded.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "epilogue.cuh"
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcat {

using namespace rlx::tc;

constexpr int kTile = 128;       // query rows per tile and keys per block
constexpr int kItemRing = 4;
constexpr float kRescaleAbove = 8.f;   // exp2 units

__host__ __device__ constexpr uint32_t idesc_attn(int m, int n, int b_mn) {
    // fp32 accumulate, bf16 operands, A K-major (or tensor memory), B K-major (0) or MN-major (1)
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Work stealing: ask for a CTA of this grid that has not been launched; the answer (16 bytes) lands in shared memory.
__device__ __forceinline__ void steal_request(uint32_t smem_answer, uint32_t bar) {
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(smem_answer), "r"(bar) : "memory");
}
__device__ __forceinline__ int steal_answer(uint32_t smem_answer) {   // block index taken over, or -1
    uint32_t ok, x = 0;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b128 h;\n"
        "ld.shared.b128 h, [%2];\n"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "mov.u32 %1, 0;\n"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, h;\n"
        "}\n"
        : "=r"(ok), "=r"(x) : "r"(smem_answer) : "memory");
    return ok ? (int)x : -1;
}

template <int D, bool PAIR>
struct Cfg {
    static constexpr int W = PAIR ? 2 * D : D;                // columns of a q / k / v tile
    static constexpr int COLS = W > 64 ? 64 : W;              // columns of a TMA box (one swizzle span)
    static constexpr int ROWB = COLS * 2;
    static constexpr int NSUB = W / COLS;
    static constexpr int SUB = kTile * ROWB;
    static constexpr int TILE = NSUB * SUB;
    static constexpr int QB = PAIR ? TILE : 2 * TILE;         // Q of an item
    static constexpr int QST = QB > 32768 ? 1 : 2;
    static constexpr int NST = TILE == 32768 ? 5 : 8;         // K / V ring
    static constexpr int NV = (PAIR && D == 32) ? 64 : D;     // accumulator columns (N = 32 costs the tensor pipe what N = 64 does)
    static constexpr int RING_OFF = QST * QB;
    static constexpr int ITEM_OFF = RING_OFF + NST * TILE;
    static constexpr int ANS_OFF = ITEM_OFF + kItemRing * 32;
    static constexpr int BAR_OFF = ANS_OFF + 16;
    static constexpr int NBAR = 3 * QST + 3 * NST + 6 + 2 * kItemRing + 1;
    static constexpr int SMEM_BYTES = BAR_OFF + 8 * NBAR + 16 + 1024;
    static constexpr uint64_t SWZ = ROWB == 128 ? 2 : 4;
    static_assert(ROWB == 128 || ROWB == 64, "swizzle span");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");

    // Q / K operand tile: K-major rows of ROWB bytes
    static __device__ __forceinline__ uint64_t desc_k(uint32_t a) {
        return (uint64_t)((a & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)((8 * ROWB) >> 4) << 32 | (uint64_t)1 << 46 | SWZ << 61;
    }
    // V: the head dimension is contiguous (N), keys run over rows; the second 64 columns are SUB bytes away
    static __device__ __forceinline__ uint64_t desc_v(uint32_t a) {
        return (uint64_t)((a & 0x3FFFFu) >> 4) | (uint64_t)(NV > COLS ? SUB >> 4 : 1) << 16 | (uint64_t)((8 * ROWB) >> 4) << 32 |
               (uint64_t)1 << 46 | SWZ << 61;
    }
    // byte offset of the first column of 16-column step k of tile t's head inside a q / k tile
    static __device__ __forceinline__ constexpr uint32_t koff(int t, int k) {
        const int c = (PAIR ? t * D : 0) + 16 * k;
        return (uint32_t)((c / COLS) * SUB + (c % COLS) * 2);
    }
};

struct Params {
    const int32_t *seq_start, *seq_len;
    __nv_bfloat16* ctx;
    const float *rope_cos, *rope_sin;   // [max_len, D/2]
    int32_t* status;
    int H, Hkv;                         // widths of the q and of the k block
    int batch, qtiles, units;           // items = qtiles * batch * units
    int kv_group;                       // q heads per k / v head
    int rows_mode;                      // shared K/V: 1 = two row tiles of one head, 0 = two heads
    int positional, window;             // key k visible to query i iff i - window < k <= i
    float scale_log2e;
};

template <bool ROPE>
struct Threads {
    static constexpr int N = ROPE ? 512 : 384;
    // 256 softmax threads and the rest share what the launch holds: 512 x 128 = 256 x (200 + 56), 384 x 168 > 256 x 208 + 128 x 80
    static constexpr int REG_SOFTMAX = ROPE ? 200 : 208;
    static constexpr int REG_REST = ROPE ? 56 : 80;
};

struct Item {
    int valid, unit, q0, len, row0, j0, nb, hi;
};

template <int D, bool PAIR, bool ROPE>
__global__ void __launch_bounds__(Threads<ROPE>::N, 1)
attention_fwd_kernel(const __grid_constant__ CUtensorMap tmap, const Params p) {
    using C = Cfg<D, PAIR>;
    constexpr int NST = C::NST, QST = C::QST, NV = C::NV;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t ring = base + C::RING_OFF;
    volatile int4* items = reinterpret_cast<volatile int4*>(gbase + C::ITEM_OFF);
    const uint32_t bars = base + C::BAR_OFF;
    const uint32_t q_full = bars, q_free = q_full + 8 * QST, q_rot = q_free + 8 * QST;
    const uint32_t kv_full = q_rot + 8 * QST, kv_free = kv_full + 8 * NST, kv_rot = kv_free + 8 * NST;
    const uint32_t s_full = kv_rot + 8 * NST, p_ready = s_full + 16, o_full = p_ready + 16;
    const uint32_t item_full = o_full + 16, item_free = item_full + 8 * kItemRing, ans_bar = item_free + 8 * kItemRing;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + C::BAR_OFF + 8 * C::NBAR);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int i = 0; i < QST; ++i) { mbar_init(q_full + 8 * i, 1); mbar_init(q_free + 8 * i, 1); mbar_init(q_rot + 8 * i, 4); }
        for (int i = 0; i < NST; ++i) { mbar_init(kv_full + 8 * i, 1); mbar_init(kv_free + 8 * i, 1); mbar_init(kv_rot + 8 * i, 4); }
        for (int i = 0; i < 2; ++i) { mbar_init(s_full + 8 * i, 1); mbar_init(p_ready + 8 * i, 4); mbar_init(o_full + 8 * i, 1); }
        for (int i = 0; i < kItemRing; ++i) { mbar_init(item_full + 8 * i, 1); mbar_init(item_free + 8 * i, ROPE ? 13 : 9); }
        mbar_init(ans_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap);
    }
    if (warp == 9) {
        tmem_alloc<1>(smem_u32(tmem_slot), 512);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();

    // A consumer's next item: 1 ready, 0 end of the list, -1 a wait ran out.  All lanes of a warp call.
    auto next_item = [&](uint32_t n, Item& it) -> int {
        const uint32_t slot = n % kItemRing;
        if (!mbar_wait_warp(item_full + 8 * slot, (n / kItemRing) & 1, abort_flag)) return -1;
        const int4 a = {items[2 * slot].x, items[2 * slot].y, items[2 * slot].z, items[2 * slot].w};
        const int4 b = {items[2 * slot + 1].x, items[2 * slot + 1].y, items[2 * slot + 1].z, items[2 * slot + 1].w};
        it = Item{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        __syncwarp();
        if (lane == 0) mbar_arrive(item_free + 8 * slot);
        return it.valid;
    };

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Threads<ROPE>::REG_REST));
        if (warp == 8) {
            // -------------------------------------------------------- items and TMA
            if (lane == 0) {
                const uint32_t ans = base + C::ANS_OFF;
                const int per_tile = p.batch * p.units;
                int cand = (int)blockIdx.x;
                uint32_t n = 0, g = 0, n_ans = 0;   // items published, ring slots used, answers read
                bool ok = true;
                mbar_expect_tx(ans_bar, 16);
                steal_request(ans, ans_bar);
                while (ok) {
                    Item it{};
                    if (cand >= 0) {
                        const int qt = p.qtiles - 1 - cand / per_tile, rem = cand % per_tile;
                        const int b = rem / p.units;
                        const int rows = p.rows_mode ? 2 * kTile : kTile;
                        it.unit = rem % p.units;
                        it.q0 = qt * rows;
                        it.len = __ldg(p.seq_len + b);
                        it.valid = it.q0 < it.len;
                        it.row0 = __ldg(p.seq_start + b);
                        it.hi = p.positional ? min(it.len, it.q0 + rows) : it.len;
                        it.j0 = p.positional ? max(0, it.q0 - p.window + 1) / kTile : 0;
                        it.nb = (it.hi + kTile - 1) / kTile;
                    }
                    if (it.valid || cand < 0) {
                        const uint32_t slot = n % kItemRing;
                        if (n >= kItemRing && !(ok = mbar_wait(item_free + 8 * slot, ((n / kItemRing) - 1) & 1, abort_flag))) break;
                        items[2 * slot].x = it.valid; items[2 * slot].y = it.unit; items[2 * slot].z = it.q0; items[2 * slot].w = it.len;
                        items[2 * slot + 1].x = it.row0; items[2 * slot + 1].y = it.j0; items[2 * slot + 1].z = it.nb; items[2 * slot + 1].w = it.hi;
                        mbar_arrive(item_full + 8 * slot);   // release: orders the stores above
                    }
                    if (cand < 0) break;
                    if (it.valid) {
                        const uint32_t qs = n % QST;
                        if (n >= QST && !(ok = mbar_wait(q_free + 8 * qs, ((n / QST) - 1) & 1, abort_flag))) break;
                        const int head0 = (PAIR || !p.rows_mode) ? 2 * it.unit : it.unit;
                        const int kvh = PAIR ? head0 : head0 / p.kv_group;
                        mbar_expect_tx(q_full + 8 * qs, C::QB);
#pragma unroll
                        for (int t = 0; t < (PAIR ? 1 : 2); ++t)
#pragma unroll
                            for (int s = 0; s < C::NSUB; ++s)
                                tma_load_2d(base + qs * C::QB + t * C::TILE + s * C::SUB, &tmap,
                                            (head0 + (p.rows_mode ? 0 : t)) * D + s * C::COLS, it.row0 + it.q0 + (p.rows_mode ? t * kTile : 0),
                                            q_full + 8 * qs);
                        for (int j = it.j0; j < it.nb && ok; ++j) {
#pragma unroll
                            for (int kv = 0; kv < 2; ++kv) {
                                const uint32_t st = g % NST, use = g / NST;
                                if (use >= 1 && !(ok = mbar_wait(kv_free + 8 * st, (use - 1) & 1, abort_flag))) break;
                                mbar_expect_tx(kv_full + 8 * st, C::TILE);
#pragma unroll
                                for (int s = 0; s < C::NSUB; ++s)
                                    tma_load_2d(ring + st * C::TILE + s * C::SUB, &tmap, p.H + kv * p.Hkv + kvh * D + s * C::COLS,
                                                it.row0 + j * kTile, kv_full + 8 * st);
                                ++g;
                            }
                        }
                        if (!ok) break;
                        ++n;
                    }
                    if (!(ok = mbar_wait(ans_bar, n_ans & 1, abort_flag))) break;
                    ++n_ans;
                    cand = steal_answer(ans);
                    if (cand >= 0) {
                        fence_proxy_async();   // the answer has been read before the next one may land on it
                        mbar_expect_tx(ans_bar, 16);
                        steal_request(ans, ans_bar);
                    }
                }
            }
        } else if (warp == 9) {
            // -------------------------------------------------------- MMA issue (whole warp, one lane issues)
            const uint32_t kv_rdy = ROPE ? kv_rot : kv_full, q_rdy = ROPE ? q_rot : q_full;
            constexpr uint32_t idesc_o = idesc_attn(kTile, NV, 1);
            Item it, nx;
            uint32_t n = 0, slot = 0;       // items opened; ring slots consumed
            uint32_t gp = 0;                // blocks whose P has been awaited
            bool ok = true;
            int state = next_item(0, it);
            // S of block j of `w` (item number m) for tile t; K in ring slot `ks`
            auto issue_s = [&](const Item& w, uint32_t m, int j, uint32_t ks, int t) {
                const int keys = min(kTile, w.hi - j * kTile);
                const uint32_t idesc = idesc_attn(kTile, (keys + 15) & ~15, 0);
                const uint32_t q = base + (m % QST) * C::QB + (PAIR ? 0 : t * C::TILE);
                const uint64_t qd = C::desc_k(q), kd = C::desc_k(ring + ks * C::TILE);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        umma_bf16<1>(tmem + t * kTile, qd + (C::koff(t, k) >> 4), kd + (C::koff(PAIR ? t : 0, k) >> 4), idesc, k != 0);
                    umma_commit<1>(s_full + 8 * t);
                }
                __syncwarp();
            };
            auto wait_slot = [&]() -> bool {
                const bool r = mbar_wait_warp(kv_rdy + 8 * (slot % NST), (slot / NST) & 1, abort_flag);
                tc_fence_after();
                return r;
            };
            if (state == 1) {
                ok = mbar_wait_warp(q_rdy, 0, abort_flag) && wait_slot();
                if (ok) {
                    issue_s(it, 0, it.j0, 0, 0);
                    issue_s(it, 0, it.j0, 0, 1);
                    if (elect_one()) {
                        umma_commit<1>(kv_free);
                        if (it.j0 + 1 == it.nb) umma_commit<1>(q_free);
                    }
                    __syncwarp();
                    slot = 1;
                }
            }
            int j = state == 1 ? it.j0 : 0;
            while (ok && state == 1) {
                const uint32_t vs = slot % NST;
                const uint32_t vt = ring + vs * C::TILE;
                const int keys = min(kTile, it.hi - j * kTile), kpad = (keys + 15) & ~15;
                const bool last = j + 1 == it.nb;
                if (!(ok = wait_slot())) break;
                ++slot;
                if (keys < kpad) {
                    // rows past the end of the sequence get probability 0, but whatever lies behind them in memory must
                    // not turn that into a NaN: clear them
                    for (int i = lane; i < (kpad - keys) * (C::ROWB / 16) * C::NSUB; i += 32) {
                        const int s = i / ((kpad - keys) * (C::ROWB / 16)), o = i % ((kpad - keys) * (C::ROWB / 16));
                        st_shared_v4(vt + s * C::SUB + keys * C::ROWB + o * 16, make_uint4(0, 0, 0, 0));
                    }
                    fence_proxy_async();
                    __syncwarp();
                }
                // the block after this one: of this item or of the next
                uint32_t ks = 0;
                int nstate = 1, nj = j + 1;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (!(ok = mbar_wait_warp(p_ready + 8 * t, gp & 1, abort_flag))) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t vd = C::desc_v(vt + (PAIR && D == 64 ? t * C::SUB : 0));
                        for (int kk = 0; kk < kpad / 16; ++kk)
                            umma_ts(tmem + 256 + t * kTile, tmem + t * kTile + kk * 8, vd + (uint64_t)((16 * C::ROWB) >> 4) * kk, idesc_o,
                                    (j != it.j0 || kk != 0) ? 1u : 0u);
                        if (last) umma_commit<1>(o_full + 8 * t);
                        if (t == 1) umma_commit<1>(kv_free + 8 * vs);
                    }
                    __syncwarp();
                    if (t == 0) {
                        nx = it;
                        if (last) {
                            ++n;
                            nstate = next_item(n, nx);
                            nj = nx.j0;
                            if (nstate == 1 && !mbar_wait_warp(q_rdy + 8 * (n % QST), (n / QST) & 1, abort_flag)) nstate = -1;
                        }
                        if (nstate == 1) {
                            ks = slot % NST;
                            if (!wait_slot()) nstate = -1;
                            ++slot;
                        }
                        if (nstate < 0) { ok = false; break; }
                    }
                    if (nstate == 1) {
                        issue_s(nx, n, nj, ks, t);
                        if (t == 1 && elect_one()) {
                            umma_commit<1>(kv_free + 8 * ks);
                            if (nj + 1 == nx.nb) umma_commit<1>(q_free + 8 * (n % QST));
                        }
                        __syncwarp();
                    }
                }
                ++gp;
                it = nx;
                j = nj;
                state = nstate;
            }
        } else if (ROPE && warp >= 12) {
            // -------------------------------------------------------- rotary embedding of Q tiles and K blocks
            constexpr int HEADS = PAIR ? 2 : 1, CPR = D / 16;   // heads per tile; (lo, hi) 16-byte chunk pairs per head row
            const int rt = threadIdx.x - 12 * 32;
            // rows first_pos + r, r < 128, of a tile; positions at or past `len` are left alone
            auto rotate = [&](uint32_t tile, int first_pos, int len) {
                for (int i = rt; i < kTile * HEADS * CPR; i += 128) {
                    const int r = i / (HEADS * CPR), c = i % (HEADS * CPR);
                    const int hd = c / CPR, cc = c % CPR, pos = first_pos + r;
                    if (pos >= len) continue;
                    const int lo_col = hd * D + cc * 8, hi_col = lo_col + D / 2;
                    const uint32_t swz = C::ROWB == 128 ? (uint32_t)(r & 7) : (uint32_t)((r >> 1) & 3);
                    const uint32_t a = tile + (lo_col / C::COLS) * C::SUB + r * C::ROWB + ((((uint32_t)(lo_col % C::COLS) / 8) ^ swz) << 4);
                    const uint32_t b = tile + (hi_col / C::COLS) * C::SUB + r * C::ROWB + ((((uint32_t)(hi_col % C::COLS) / 8) ^ swz) << 4);
                    const float4* pc = reinterpret_cast<const float4*>(p.rope_cos + (size_t)pos * (D / 2) + cc * 8);
                    const float4* ps = reinterpret_cast<const float4*>(p.rope_sin + (size_t)pos * (D / 2) + cc * 8);
                    uint4 lo = ld_shared_v4(a), hi = ld_shared_v4(b);
                    rope_rotate8(lo, hi, __ldg(pc), __ldg(pc + 1), __ldg(ps), __ldg(ps + 1));
                    st_shared_v4(a, lo);
                    st_shared_v4(b, hi);
                }
                fence_proxy_async();
                __syncwarp();
            };
            Item it;
            uint32_t slot = 0;
            bool ok = true;
            for (uint32_t n = 0; ok; ++n) {
                if (next_item(n, it) != 1) break;
                const uint32_t qs = n % QST;
                if (!mbar_wait_warp(q_full + 8 * qs, (n / QST) & 1, abort_flag)) break;
                rotate(base + qs * C::QB, it.q0, it.len);
                if (!PAIR) rotate(base + qs * C::QB + C::TILE, it.q0 + (p.rows_mode ? kTile : 0), it.len);
                if (lane == 0) mbar_arrive(q_rot + 8 * qs);
                for (int j = it.j0; j < it.nb && ok; ++j)
                    for (int kv = 0; kv < 2; ++kv, ++slot) {
                        const uint32_t st = slot % NST;
                        if (!(ok = mbar_wait_warp(kv_full + 8 * st, (slot / NST) & 1, abort_flag))) break;
                        if (kv == 0) rotate(ring + st * C::TILE, j * kTile, it.len);
                        if (lane == 0) mbar_arrive(kv_rot + 8 * st);
                    }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax (thread = query row)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Threads<ROPE>::REG_SOFTMAX));
        const int t = warp >> 2, quad = warp & 3;
        const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t s_col = tl + t * kTile, o_col = tl + 256 + t * kTile + ((PAIR && D == 32) ? t * 32 : 0);
        const float scale = p.scale_log2e;
        uint32_t gb = 0;    // blocks seen
        bool ok = true;
        Item it;
        for (uint32_t n = 0; ok; ++n) {
            if (next_item(n, it) != 1) break;
            const int q0 = it.q0 + (p.rows_mode ? t * kTile : 0);
            const int wr0 = q0 + quad * 32, row = wr0 + lane;      // rows of this warp, of this thread (position in the sequence)
            const bool live = wr0 < it.len;
            const int head = (PAIR || !p.rows_mode) ? 2 * it.unit + t : it.unit;
            float m_ref = -INFINITY;
            uint64_t l2[2] = {0, 0};
            for (int j = it.j0; j < it.nb; ++j, ++gb) {
                if (!(ok = mbar_wait_warp(s_full + 8 * t, gb & 1, abort_flag))) break;
                if (live) {
                    tc_fence_after();
                    const int k0 = j * kTile;
                    uint32_t s[4][32];
                    // 32-key chunks with a key that some row of the warp can see
                    const int c_lo = p.positional ? max(0, (wr0 - p.window + 1 - k0) >> 5) : 0;
                    const int c_hi = (min(it.hi, p.positional ? wr0 + 32 : it.hi) - k0 + 31) >> 5;   // one past the last
                    const bool whole = k0 + kTile <= it.hi &&
                                       (!p.positional || (k0 + kTile - 1 <= wr0 && k0 > wr0 + 31 - p.window));
                    const int n_store = (min(kTile, it.hi - k0) + 31) >> 5;
                    if (whole) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) tmem_ld_32x32(s_col + 32 * c, s[c]);
                        tmem_ld_wait();
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (c >= c_lo && c < c_hi) tmem_ld_32x32(s_col + 32 * c, s[c]);
                        tmem_ld_wait();
                        const int first = p.positional ? row - p.window + 1 - k0 : 0;
                        const int lim = min(it.hi - 1, p.positional ? row : it.hi) - k0;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const bool on = c >= c_lo && c < c_hi;
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (!on || 32 * c + i < first || 32 * c + i > lim) s[c][i] = 0xFF800000u;   // -inf
                        }
                    }
                    float m_blk;
                    {
                        float mx[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            mx[c] = fmaxf(__uint_as_float(s[c][0]), __uint_as_float(s[c][1]));
#pragma unroll
                            for (int i = 2; i < 32; i += 2) mx[c] = max3f(mx[c], __uint_as_float(s[c][i]), __uint_as_float(s[c][i + 1]));
                        }
                        m_blk = fmaxf(max3f(mx[0], mx[1], mx[2]), mx[3]) * scale;
                    }
                    if (j == it.j0) {
                        m_ref = m_blk;
                    } else {
                        const bool need = m_blk > m_ref + kRescaleAbove;
                        if (__any_sync(0xffffffffu, need)) {
                            const float alpha = need ? ex2f(m_ref - m_blk) : 1.f;
                            if (need) m_ref = m_blk;
                            const uint64_t a2 = pack_f32x2(alpha, alpha);
                            l2[0] = mul_f32x2(l2[0], a2);
                            l2[1] = mul_f32x2(l2[1], a2);
#pragma unroll
                            for (int c0 = 0; c0 < D; c0 += 16) {
                                uint32_t o[16];
                                tmem_ld_32x16(o_col + c0, o);
                                tmem_ld_wait();
#pragma unroll
                                for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                                tmem_st_32x16(o_col + c0, o);
                            }
                        }
                    }
                    const float neg = m_ref == -INFINITY ? 0.f : -m_ref;
                    const uint64_t sc2 = pack_f32x2(scale, scale), ng2 = pack_f32x2(neg, neg);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c >= n_store) break;
                        uint32_t pk[16];
                        if (whole || (c >= c_lo && c < c_hi)) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                float x0, x1;
                                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c][2 * i]), __uint_as_float(s[c][2 * i + 1])), sc2, ng2), x0, x1);
                                x0 = ex2f(x0);
                                x1 = ex2f(x1);
                                l2[i & 1] = add_f32x2(l2[i & 1], pack_f32x2(x0, x1));
                                pk[i] = pack_bf16(x0, x1);
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i) pk[i] = 0;
                        }
                        tmem_st_32x16(s_col + 16 * c, pk);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(p_ready + 8 * t);
            }
            if (!ok) break;
            // ---- O / row sum -> bf16 -> global ----
            if (!(ok = mbar_wait_warp(o_full + 8 * t, n & 1, abort_flag))) break;
            if (live) {
                tc_fence_after();
                float a0, a1, b0, b1;
                unpack_f32x2(l2[0], a0, a1);
                unpack_f32x2(l2[1], b0, b1);
                const float l = (a0 + a1) + (b0 + b1);
                const float inv = l > 0.f ? 1.0f / l : 0.f;
                __nv_bfloat16* orow = p.ctx + (size_t)(it.row0 + row) * p.H + head * D;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld_32x32(o_col + 32 * c, o);
                    tmem_ld_wait();
                    if (row < it.len) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint4 q;
                            q.x = pack_bf16(__uint_as_float(o[8 * i + 0]) * inv, __uint_as_float(o[8 * i + 1]) * inv);
                            q.y = pack_bf16(__uint_as_float(o[8 * i + 2]) * inv, __uint_as_float(o[8 * i + 3]) * inv);
                            q.z = pack_bf16(__uint_as_float(o[8 * i + 4]) * inv, __uint_as_float(o[8 * i + 5]) * inv);
                            q.w = pack_bf16(__uint_as_float(o[8 * i + 6]) * inv, __uint_as_float(o[8 * i + 7]) * inv);
                            *(reinterpret_cast<uint4*>(orow + 32 * c) + i) = q;
                        }
                    }
                }
                tc_fence_before();   // the next item's products overwrite O behind this warp's next arrival
            }
        }
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
    if (warp == 9) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, 512);
    }
}

}  // namespace tcat
}  // namespace rlx

// QKV projection and attention of short sequences in one kernel: ctx = attention(x Wqkv^T + b), or with the LayerNorm in front
// folded in (epilogue mode 3 of gemm_tcgen05.cuh).
//
// A CTA takes a bin (consecutive whole sequences with at most 128 packed rows together, see pack_sequences_kernel) and HPC
// heads: it multiplies the bin's rows with those heads' rows of Wqkv (TMA -> tcgen05, accumulators in tensor memory), puts q,
// k and v as bf16 where the operand ring was, and attends from there with mma.sync, a warp per 16 rows of a sequence.  Every
// number is formed as the two separate kernels form it (same order along K, same epilogue, same softmax steps), so the
// result is bit for bit theirs, and a sequence's does not depend on its bin.
//
// What bounds it: latency, as everything in a small forward; the point is the link that is not there.  A kernel boundary
// costs the store of q, k, v, the hand-over and the round trip of the loads behind it.
//
// With OUT (few bins, heads of 32, one per CTA) the CTAs of a bin's heads are a cluster that goes on to the attention output:
// y = ctx Wo^T + bias + residual, with its row statistics, epilogue modes 5 / 6.  Every CTA sends its head's context rows to all of
// them (st.async: data and arrival in one) and multiplies the whole rows with 32 rows of Wo, which have been there since the
// start.  An SM takes in 16.5 bytes a clock from its peers behind 700 cycles of latency: 32 / 64 / 128 rows of context 1.8 / 3.0 /
// 5.4 thousand cycles, where another kernel's link costs eight thousand.
//
// All waits are bounded.
#pragma once
#include "attention.cuh"
#include "gemm_cln_tcgen05.cuh"
#include "gemm_splitk_tcgen05.cuh"
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcqa {

using namespace rlx::tc;
using rlx::tccl::mbar_wait_cluster;
using rlx::tcsk::st_async_v4;

constexpr int kRows = kBinRows;
constexpr int kMaxOutHeads = 12;              // CTAs of a cluster, with OUT
constexpr int kChunk = kRows * 16;            // 8 columns of the context rows: [column chunk][row][16 B], the layout without swizzle
constexpr int kEpiWarps = 12;                 // a 32-row quadrant of q, of k or of v each; then they attend
constexpr int kMaxTasks = kRows / 16 + kBinSeqs;   // 16-row groups of a bin's sequences

template <int D, int HPC, bool OUT = false>
struct Cfg {
    static constexpr int WARPS = HPC == 2 ? 16 : kEpiWarps;   // that attend: two heads of a full bin are sixteen groups of 16 rows
    static constexpr int THREADS = 64 + 32 * WARPS;
    static constexpr int N = 3 * D * HPC;                     // columns: q of the heads, then k, then v
    static constexpr int NC = N / 96;                         // 32-column chunks of a warp
    static constexpr int KPS = N == 96 ? 2 : 1;               // k-blocks per stage
    static constexpr int STAGES = N == 96 ? 3 : 5;
    static constexpr int A_BYTES = kRows * BLOCK_K * 2, B_BYTES = N * BLOCK_K * 2, KB_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGE_BYTES = KPS * KB_BYTES;
    static constexpr int TMEM_COLS = N <= 128 ? 128 : 256;
    static constexpr int STR = D + 8;                         // elements per q / k / v row: conflict-free ldmatrix
    // OUT: the context rows lie over the ring, behind q, k and v; Wo's rows have room of their own
    static constexpr int CTX_OFF = 65536, WO_OFF = STAGES * STAGE_BYTES, WO_BYTES = OUT ? kMaxOutHeads * 32 * 32 * 2 : 0;
    static constexpr int VEC_OFF = WO_OFF + WO_BYTES;
    static constexpr int ZERO_OFF = VEC_OFF + kEpiWarps * 384;   // a row of zeros, read in place of v past a sequence's end
    static constexpr int TASK_OFF = ZERO_OFF + (STR * 2 + 15) / 16 * 16;
    static constexpr int BAR_OFF = TASK_OFF + kMaxTasks * 16;
    static constexpr int NBAR = 2 * STAGES + 5;
    static constexpr int SMEM_BYTES = BAR_OFF + 8 * NBAR + 16 + 1024;
    static_assert(!OUT || (D == 32 && HPC == 1 && 3 * kRows * STR * 2 <= CTX_OFF && CTX_OFF + kMaxOutHeads * 4 * kChunk <= WO_OFF), "context rows");
    static_assert(N == 96 || N == 192, "tile");
    static_assert(3 * HPC * kRows * STR * 2 <= STAGES * STAGE_BYTES, "q, k and v over the ring");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");
};

// Attention of 16 query rows of one sequence, as attention_bf16_kernel computes it: online softmax in steps of 32 (heads of 32) or
// 64 keys.  q: the first query row, k / v: the sequence's first key, all with STR elements per row; keys: length of the
// sequence, rows: query rows that exist.  The result replaces the q rows.
template <int D, int STR>
__device__ __forceinline__ void attend16(__nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, uint32_t zero_row, int keys,
                                         int rows, float scale_log2e) {
    constexpr int KT = D / 16, ND = D / 8, KS = D == 32 ? 32 : 64, NT = KS / 8;
    const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3, mi = lane >> 3;
    uint32_t qf[KT][4];
#pragma unroll
    for (int kt = 0; kt < KT; ++kt)
        ldmatrix_x4(smem_u32(q + ((lane & 7) + (mi & 1) * 8) * STR + kt * 16 + (lane >> 4) * 8), qf[kt][0], qf[kt][1], qf[kt][2], qf[kt][3]);
    float o[ND][4];
#pragma unroll
    for (int i = 0; i < ND; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }
    float m_run[2] = {-INFINITY, -INFINITY};
    float l_acc[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr uint32_t kOnesBf16x2 = 0x3F803F80u;
#pragma unroll 1
    for (int k0 = 0; k0 < keys; k0 += KS) {
        float s[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
            for (int kp = 0; kp < KT / 2; ++kp) {
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4(smem_u32(k + (k0 + nt * 8 + (lane & 7)) * STR + kp * 32 + (mi & 1) * 8 + (mi >> 1) * 16), b0, b1, b2, b3);
                mma_bf16_16816(s[nt], qf[2 * kp][0], qf[2 * kp][1], qf[2 * kp][2], qf[2 * kp][3], b0, b1);
                mma_bf16_16816(s[nt], qf[2 * kp + 1][0], qf[2 * kp + 1][1], qf[2 * kp + 1][2], qf[2 * kp + 1][3], b2, b3);
            }
        }
        if (k0 + KS > keys) {
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const int kk = k0 + nt * 8 + 2 * t4;
                if (kk >= keys) { s[nt][0] = -INFINITY; s[nt][2] = -INFINITY; }
                if (kk + 1 >= keys) { s[nt][1] = -INFINITY; s[nt][3] = -INFINITY; }
            }
        }
        float mx[2] = {fmaxf(s[0][0], s[0][1]), fmaxf(s[0][2], s[0][3])};
#pragma unroll
        for (int nt = 1; nt < NT; ++nt) {
            mx[0] = fmax3(mx[0], s[nt][0], s[nt][1]);
            mx[1] = fmax3(mx[1], s[nt][2], s[nt][3]);
        }
        float alpha[2], msub[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
            mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
            const float m_new = fmaxf(m_run[r], mx[r] * scale_log2e);
            msub[r] = (m_new == -INFINITY) ? 0.f : m_new;
            alpha[r] = fast_exp2(m_run[r] - msub[r]);
            m_run[r] = m_new;
        }
        const uint64_t a0 = att_pack2(alpha[0], alpha[0]), a1 = att_pack2(alpha[1], alpha[1]);
#pragma unroll
        for (int nd = 0; nd < ND; ++nd) {
            att_unpack2(att_mul2(att_pack2(o[nd][0], o[nd][1]), a0), o[nd][0], o[nd][1]);
            att_unpack2(att_mul2(att_pack2(o[nd][2], o[nd][3]), a1), o[nd][2], o[nd][3]);
        }
        l_acc[0] *= alpha[0];
        l_acc[2] *= alpha[1];
        uint32_t pf[NT / 2][4];
        const uint64_t c2 = att_pack2(scale_log2e, scale_log2e);
        const uint64_t nm0 = att_pack2(-msub[0], -msub[0]), nm1 = att_pack2(-msub[1], -msub[1]);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float x0, x1, x2, x3;
            att_unpack2(att_fma2(att_pack2(s[nt][0], s[nt][1]), c2, nm0), x0, x1);
            att_unpack2(att_fma2(att_pack2(s[nt][2], s[nt][3]), c2, nm1), x2, x3);
            pf[nt >> 1][(nt & 1) * 2 + 0] = pack_bf16(fast_exp2(x0), fast_exp2(x1));
            pf[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(fast_exp2(x2), fast_exp2(x3));
        }
#pragma unroll
        for (int kk = 0; kk < NT / 2; ++kk) {
            mma_bf16_16816(l_acc, pf[kk][0], pf[kk][1], pf[kk][2], pf[kk][3], kOnesBf16x2, kOnesBf16x2);
            // behind the sequence's end lie another's rows: probability 0 times whatever they hold must stay 0
            const int r = k0 + kk * 16 + (mi & 1) * 8 + (lane & 7);
            const uint32_t vrow = r < keys ? smem_u32(v + r * STR) : zero_row;
#pragma unroll
            for (int np = 0; np < ND / 2; ++np) {
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4_trans(vrow + (np * 16 + (mi >> 1) * 8) * 2, b0, b1, b2, b3);
                mma_bf16_16816(o[2 * np], pf[kk][0], pf[kk][1], pf[kk][2], pf[kk][3], b0, b1);
                mma_bf16_16816(o[2 * np + 1], pf[kk][0], pf[kk][1], pf[kk][2], pf[kk][3], b2, b3);
            }
        }
    }
    float l_run[2] = {l_acc[0], l_acc[2]};
#pragma unroll
    for (int r = 0; r < 2; ++r) l_run[r] = l_run[r] > 0.f ? 1.0f / l_run[r] : 0.f;
    // rows past the sequence's end are the next one's queries: left alone
#pragma unroll
    for (int nd = 0; nd < ND; ++nd) {
        if (g < rows) *reinterpret_cast<uint32_t*>(q + g * STR + nd * 8 + 2 * t4) = pack_bf16(o[nd][0] * l_run[0], o[nd][1] * l_run[0]);
        if (g + 8 < rows)
            *reinterpret_cast<uint32_t*>(q + (g + 8) * STR + nd * 8 + 2 * t4) = pack_bf16(o[nd][2] * l_run[1], o[nd][3] * l_run[1]);
    }
    __syncwarp();
}

struct RowMaps {
    CUtensorMap m[4];                  // x as k-blocks, boxes of 32, 64, 96 and 128 rows: only the 32-row groups that a bin has are loaded
};
struct AttParams {
    const int32_t *bins, *seq_start;   // pack_sequences_kernel's
    __nv_bfloat16* ctx;                // [rows, H]
    float scale_log2e;
    int first;                         // the kernel in front wrote the tables: nothing may be read ahead of it, not by the next kernel either
};

// grid (heads / HPC, bins that there can be); tmap_w: Wqkv as [q | k | v][row][column], boxes of 3 x D HPC x 64.  p: bias / folding vectors and row statistics of the product, K = H.
// OUT: tmap_wo: Wo as k-blocks, boxes of 32 x H; po: the attention output's epilogue, its result to po.out.
template <int D, int HPC, int EPI, bool OUT>
__global__ void __launch_bounds__((Cfg<D, HPC, OUT>::THREADS), 1)
qkv_attention_kernel(const __grid_constant__ RowMaps tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                     const __grid_constant__ CUtensorMap tmap_wo, const Params p, const Params po, const AttParams ap) {
    using C = Cfg<D, HPC, OUT>;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t full_bar = base + C::BAR_OFF, empty_bar = full_bar + 8 * C::STAGES, acc_bar = empty_bar + 8 * C::STAGES;
    const uint32_t wo_bar = acc_bar + 8, ctx_bar = wo_bar + 8, free_bar = ctx_bar + 8, out_bar = free_bar + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + C::BAR_OFF + 8 * C::NBAR);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int4* tasks = reinterpret_cast<int4*>(gbase + C::TASK_OFF);   // first row in the bin, query row offset, length
    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int bin = blockIdx.y, head0 = blockIdx.x * HPC, H = p.K, num_kb = H / BLOCK_K;
    if (!ap.first) pdl_launch_dependents();

    if (threadIdx.x == 0) {
        for (int i = 0; i < C::STAGES; ++i) { mbar_init(full_bar + 8 * i, 1); mbar_init(empty_bar + 8 * i, 1); }
        mbar_init(acc_bar, 1);
        if (OUT) {
            mbar_init(wo_bar, 1);
            mbar_init(ctx_bar, 1);
            mbar_init(free_bar, gridDim.x);
            mbar_init(out_bar, 1);
        }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap_w);
    }
    if (warp == 1) {
        tmem_alloc<1>(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish<1>();
    }
    if (ap.first) {
        pdl_wait();
        pdl_launch_dependents();
    }
    const bool exists = bin < ld_early(ap.bins);
    const int b0 = exists ? ld_early(ap.bins + 1 + bin) : 0, b1 = exists ? ld_early(ap.bins + 2 + bin) : 0;
    const int row0 = exists ? ld_early(ap.seq_start + b0) : 0, rows = exists ? ld_early(ap.seq_start + b1) - row0 : 0;
    tc_fence_before();
    __syncthreads();
    if constexpr (OUT) cluster_sync_all();   // the peers' barriers exist before anything is sent to them
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);
    const int groups = (rows + 31) / 32, a_kb = groups * (C::A_BYTES / 4);   // 32-row groups; bytes of a k-block of them

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
        auto load_w = [&](int kb, int stage) {
            mbar_expect_tx(full_bar + 8 * stage, (uint32_t)(C::KPS * (a_kb + C::B_BYTES)));
            for (int i = 0; i < C::KPS; ++i)
                tma_load_3d(base + stage * C::STAGE_BYTES + C::KPS * C::A_BYTES + i * C::B_BYTES, &tmap_w, (kb + i) * BLOCK_K, head0 * D, 0,
                            full_bar + 8 * stage);
        };
        auto load_a = [&](int kb, int stage) { tma_load_3d(base + stage * C::STAGE_BYTES, tmap_a.m + groups - 1, 0, row0, kb, full_bar + 8 * stage); };
        int early = 0;   // weights do not come from the previous kernel
        if (rows > 0)
            for (; early < C::STAGES && early * C::KPS < num_kb; ++early) {
                if (elect_one()) load_w(early * C::KPS, early);
                __syncwarp();
            }
        if constexpr (OUT)
            if (rows > 0 && elect_one()) {
                mbar_expect_tx(wo_bar, (uint32_t)(num_kb * 32 * 128));
                tma_load_3d(base + C::WO_OFF, &tmap_wo, 0, head0 * D, 0, wo_bar);
            }
        __syncwarp();
        pdl_wait();
        if (rows > 0) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < num_kb; kb += C::KPS) {
                if (early > 0) {
                    --early;
                    if (elect_one()) load_a(kb, stage);
                } else {
                    if (!mbar_wait_warp(empty_bar + 8 * stage, phase ^ 1, abort_flag)) break;
                    if (elect_one()) { load_w(kb, stage); load_a(kb, stage); }
                }
                __syncwarp();
                if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
        if (rows > 0) {
            constexpr uint32_t idesc = make_idesc(kRows, C::N);
            const uint64_t adesc0 = make_smem_desc(base), bdesc0 = make_smem_desc(base + C::KPS * C::A_BYTES);
            uint32_t stage = 0, phase = 0;
            bool ok = true, ready = false;
            for (int kb = 0; kb < num_kb; kb += C::KPS) {
                if (!__all_sync(0xffffffffu, ready) && !(ok = mbar_wait_warp(full_bar + 8 * stage, phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t cur = stage;
                if (++stage == C::STAGES) { stage = 0; phase ^= 1; }
                ready = mbar_test_wait(full_bar + 8 * stage, phase);
                if (elect_one()) {
                    const uint64_t ad0 = adesc0 + cur * (C::STAGE_BYTES >> 4), bd0 = bdesc0 + cur * (C::STAGE_BYTES >> 4);
#pragma unroll
                    for (int i = 0; i < C::KPS; ++i)
#pragma unroll
                        for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                            umma_bf16<1>(tmem, ad0 + (i * (uint32_t)(a_kb >> 4) + 2 * k), bd0 + (i * (C::B_BYTES >> 4) + 2 * k), idesc,
                                         (kb | i | k) != 0 ? 1u : 0u);
                    umma_commit<1>(empty_bar + 8 * cur);
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit<1>(acc_bar);
            __syncwarp();
            if constexpr (OUT) {
                // the attention output: 32 columns, once all heads' context rows are here
                if (elect_one()) mbar_expect_tx(ctx_bar, (uint32_t)(rows * H * 2));
                __syncwarp();
                ok = ok && mbar_wait_warp(wo_bar, 0, abort_flag) && __all_sync(0xffffffffu, mbar_wait_cluster(ctx_bar, 0, abort_flag)) != 0;
                asm volatile("fence.proxy.async;" ::: "memory");   // the peers' stores, for the tensor core
                tc_fence_after();
                if (ok && elect_one()) {
                    // K-major without swizzle: the 16-byte chunks of a K = 16 step are kChunk apart, 8-row groups 128 bytes
                    const uint64_t cd = (uint64_t)((base + C::CTX_OFF & 0x3FFFFu) >> 4) | (uint64_t)(kChunk >> 4) << 16 | (uint64_t)(128 >> 4) << 32 |
                                        (uint64_t)1 << 46;
                    const uint64_t wd = make_smem_desc(base + C::WO_OFF);
                    for (int kb = 0; kb < num_kb; ++kb)
#pragma unroll
                        for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                            umma_bf16<1>(tmem + C::N, cd + (kb * 4 + k) * (2 * kChunk >> 4), wd + (kb * (32 * 128 >> 4) + 2 * k), make_idesc(kRows, 32),
                                         (kb | k) != 0 ? 1u : 0u);
                    umma_commit<1>(out_bar);
                }
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------ q, k, v, then attention
        const int e = warp - 2, quad = warp & 3, part = e >> 2;
        const int n0 = part * H + head0 * D;      // part 3: warps that only attend
        using ET = EpilogueTile<EPI, C::NC, true>;
        ET et;
        if (part < 3) et.load_vectors(p, n0, base + C::VEC_OFF + e * 384);
        // the bin's row groups and the row of zeros
        int ntasks = 0;
        {
            const int i = b0 + lane, nseq = b1 - b0;
            const int first = lane < nseq ? ld_early(ap.seq_start + i) - row0 : 0;
            const int len = lane < nseq ? ld_early(ap.seq_start + i + 1) - row0 - first : 0;
            const int mine = (len + 15) / 16;
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += n;
            }
            ntasks = __shfl_sync(0xffffffffu, incl, 31);
            if (e == 0)
                for (int j = 0; j < mine; ++j) tasks[incl - mine + j] = make_int4(first, 16 * j, len, 0);
            if (e == 1 && lane < (C::STR * 2 + 15) / 16) st_shared_v4(base + C::ZERO_OFF + lane * 16, make_uint4(0, 0, 0, 0));
        }
        pdl_wait();
        const int row = quad * 32 + lane;
        const bool live = quad * 32 < rows && part < 3;
        bool ok = true;
        if (live) {
            et.prefetch(p, row0 + rows, row0 + row, n0);
            ok = mbar_wait_warp(acc_bar, 0, abort_flag);
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < C::NC; ++c) {
                uint32_t r[32];
                tmem_ld_32x32(tmem + ((uint32_t)(quad * 32) << 16) + part * (D * HPC) + c * 32, r);
                tmem_ld_wait();
                uint4 v[4];
                et.compute_chunk(p, r, n0 + c * 32, c, row0 + row, row < rows, p.bias + n0 + c * 32, v);
                // column c * 32 of the part: head c (heads of 32), or column 32 c of the one head
                const int hh = D == 32 ? c : 0, col = D == 32 ? 0 : c * 32;
                const uint32_t dst = base + (uint32_t)(((part * HPC + hh) * kRows + row) * C::STR + col) * 2;
#pragma unroll
                for (int i = 0; i < 4; ++i) st_shared_v4(dst + 16 * i, v[i]);
            }
            tc_fence_before();
        } else if (rows > 0) {
            ok = mbar_wait_warp(acc_bar, 0, abort_flag);   // the ring is free
        }
        if constexpr (OUT) {
            // this CTA's ring is free: its peers may send context rows.  They write where this CTA's products have read, so the
            // release reaches them: cluster scope.  The warp has no store to global memory outstanding that it would wait for.
            if (ok && rows > 0 && e == 0 && lane < (int)gridDim.x) mbar_arrive_cluster(map_to_cta(free_bar, lane));
            __syncwarp();
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * C::WARPS) : "memory");
        if (ok) {
            __nv_bfloat16* qkv = reinterpret_cast<__nv_bfloat16*>(gbase);
            for (int t = e; t < ntasks * HPC; t += C::WARPS) {
                const int hh = t / ntasks;
                const int4 task = tasks[t - hh * ntasks];
                __nv_bfloat16* qh = qkv + hh * kRows * C::STR;
                const int first = task.x + task.y, n = min(16, task.z - task.y);   // query rows, in the bin
                attend16<D, C::STR>(qh + first * C::STR, qh + (HPC * kRows + task.x) * C::STR, qh + (2 * HPC * kRows + task.x) * C::STR,
                                    base + C::ZERO_OFF, task.z, n, ap.scale_log2e);
                if constexpr (!OUT) {
                    constexpr int CH = D / 8;
                    __nv_bfloat16* out = ap.ctx + (size_t)(row0 + first) * H + (head0 + hh) * D;
                    for (int i = lane; i < 16 * CH; i += 32) {
                        const int r = i / CH, c = i % CH;
                        if (r < n)
                            *reinterpret_cast<uint4*>(out + (size_t)r * H + c * 8) = *reinterpret_cast<const uint4*>(qh + (first + r) * C::STR + c * 8);
                    }
                }
            }
        }
        if constexpr (OUT) {
            // a warp per peer: a warp's stores to different CTAs go out one behind the other
            asm volatile("bar.sync 1, %0;" ::"n"(32 * C::WARPS) : "memory");
            const int peer = head0 + e < (int)gridDim.x ? head0 + e : head0 + e - (int)gridDim.x;   // not all to the same one at once
            if (rows > 0 && e < (int)gridDim.x) ok = ok && __all_sync(0xffffffffu, mbar_wait_cluster(free_bar, 0, abort_flag)) != 0;
            if (ok && e < (int)gridDim.x) {
                const uint32_t dst = map_to_cta(base + C::CTX_OFF + head0 * 4 * kChunk, peer), bar = map_to_cta(ctx_bar, peer);
                for (int r = lane; r < rows; r += 32)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint4 a = ld_shared_v4(base + (uint32_t)(r * C::STR + c * 8) * 2);
                        const uint32_t w[4] = {a.x, a.y, a.z, a.w};
                        st_async_v4(dst + c * kChunk + r * 16, bar, w);
                    }
            }
            __syncwarp();
            if (part == 0 && live) {
                using EO = EpilogueTile<EPI == 0 ? 5 : 6, 1, true>;
                EO eo;
                eo.load_vectors(po, head0 * D, base + C::VEC_OFF + e * 384);
                eo.prefetch(po, row0 + rows, row0 + row, head0 * D);
                ok = ok && mbar_wait_warp(out_bar, 0, abort_flag);
                tc_fence_after();
                uint32_t r[32];
                tmem_ld_32x32(tmem + ((uint32_t)(quad * 32) << 16) + C::N, r);
                tmem_ld_wait();
                uint4 v[4];
                eo.compute_chunk(po, r, head0 * D, 0, row0 + row, ok && row < rows, po.bias + head0 * D, v);
                if (ok && row < rows) {   // the rows behind are another bin's
                    uint4* y = reinterpret_cast<uint4*>(po.out + (size_t)(row0 + row) * H + head0 * D);
#pragma unroll
                    for (int i = 0; i < 4; ++i) y[i] = v[i];
                }
                tc_fence_before();
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
    if constexpr (OUT) cluster_sync_all();   // no CTA leaves while a peer may still write into it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<1>(tmem, C::TMEM_COLS);
    }
}

}  // namespace tcqa
}  // namespace rlx

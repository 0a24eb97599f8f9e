// Packed-sequence attention on the 5th-generation tensor cores: any length, head_dim 32 / 64 / 128, all keys / causal /
// sliding window, plain and grouped-query heads, optional rotary q and k.
//
// A work item is a PAIR of 128-row query tiles that walk the same 128-key blocks, so that the two softmax groups
// of a CTA take turns on the exponential units while the tensor cores work for the other one:
//   PAIR         the same rows of two neighbouring heads with a K / V head each (head_dim 32 / 64; the two heads'
//                columns are neighbours in memory, so one tile brings q, k or v of both)
//   otherwise    the same rows of two query heads of one K / V head (grouped-query layouts), or two consecutive
//                row tiles of one head (everything else: "rows mode")
// The CTAs (one per SM) walk the items that exist with a fixed stride, last row tiles first (under the causal mask these
// are the long ones): a warp scans the sequence lengths 32 at a time, so tiles past a sequence's end cost nothing and
// no counter in global memory is needed (calls on several streams do not meet).
//
//   warps 0..3, 4..7  softmax of tile 0 / tile 1, one thread per query row (no shuffles): the scores of a block from
//                     tensor memory to registers, block maximum, exponentials, P (bf16) back over the scores; at the
//                     end of an item O / row sum -> global
//   warp 8            TMA: Q tiles, K and V blocks through a ring each
//   warp 9             issues S(q) = Q_t K^T: score jobs q = 2 * block + tile go round the score buffers, across item
//                     boundaries too, so the scores run ahead of the softmax.  Heads of 32 and 64 have three buffers, and P
//                     is written over the scores.  Heads of 128 leave room for one, which is free again as soon as a
//                     softmax group has its scores in registers, and a buffer for each tile's P: with 64-key blocks and
//                     four buffers instead, S came as 16 products of N = 64 per 128 keys, which take the tensor core 46
//                     cycles each where N = 128 takes 63 (32 q / 8 kv heads, 8 x 2048: 465 -> 429 us)
//   warp 11            issues O_t += P(q) V (P read from tensor memory, V MN-major) and hands the buffer back
//                     One warp for both was the pace-maker: 1750 cycles per job, of which 640 to 770 are tensor time and
//                     the rest its own scalar code; the softmax takes about 2400 per job and tile
//   warp 10           items
//   warps 12..15      (rotary form only) rotate the Q tiles and K blocks in shared memory before they are used
//
// The reference maximum of a row stays the one of its first block unless a later block exceeds it by more than 2^8
// (then P <= 256 is still exact in range); only then does the warp wait for PV_t(j-1) and rescale its rows of O in
// tensor memory.  Waits that skip completions of a barrier are safe because either issuer's products complete in
// order: a group that has seen S(q) knows that S(q - 1), PV(q - 3) and everything before them are complete (heads of 128 wait
// for the tile's previous PV in every block).
// All mbarrier waits are bounded: a CTA whose wait runs out records RLX_DEVSTAT_TIMEOUT, drains, frees its tensor memory and
// leaves NaN in its rows.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "epilogue.cuh"
#include "gemm_tcgen05.cuh"

namespace rlx {
namespace tcat {

using namespace rlx::tc;

constexpr int kTile = 128;     // query rows per tile
constexpr int kItemRing = 2;
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
__device__ __forceinline__ void tmem_ld_32x1(uint32_t taddr, uint32_t& r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_32x1(uint32_t taddr, uint32_t r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(r) : "memory");
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
// lo += low half of v, hi += high half
__device__ __forceinline__ void add_bf16x2(float& lo, float& hi, uint32_t v) {
    asm("{\n"
        ".reg .b16 a, b;\n"
        "mov.b32 {a, b}, %2;\n"
        "add.rn.f32.bf16 %0, a, %0;\n"
        "add.rn.f32.bf16 %1, b, %1;\n"
        "}\n" : "+f"(lo), "+f"(hi) : "r"(v));
}
template <int D, bool PAIR>
struct Cfg {
    static constexpr int KB = kTile;                          // keys per block
    // The accumulators take 2 * D columns of tensor memory.  Heads of 128 leave room for one score buffer and a buffer for
    // P per tile (APART); otherwise three score buffers, over which P is written.
    static constexpr bool APART = D == 128;
    static constexpr int NSB = APART ? 1 : 3;
    static constexpr int NPB = APART ? 2 : NSB;               // P buffers, in order of use
    static constexpr int W = PAIR ? 2 * D : D;                // columns of a q / k / v tile
    static constexpr int COLS = W > 64 ? 64 : W;              // columns of a TMA box (one swizzle span)
    static constexpr int ROWB = COLS * 2;
    static constexpr int NSUB = W / COLS;
    static constexpr int QSUB = kTile * ROWB, QTILE = NSUB * QSUB;
    static constexpr int SUB = KB * ROWB, TILE = NSUB * SUB;  // a K or V block
    static constexpr int QB = PAIR ? QTILE : 2 * QTILE;       // Q of an item
    static constexpr int QST = QB > 32768 ? 1 : 2;
    static constexpr int KST = TILE == 32768 ? 3 : 4;         // K ring
    static constexpr int VST = TILE == 32768 ? 2 : 4;         // V ring
    // Heads of 32 leave tensor memory for 16 more accumulator columns, and N = 48 costs the tensor pipe what N = 32 does: the
    // row sums come as further columns of P V, whose V columns are ones.  V tiles then have one head's columns each.
    static constexpr bool SUMS = D == 32;
    static constexpr int NV = SUMS ? D + 16 : D;              // accumulator columns
    static constexpr int VROWB = SUMS ? 2 * D : ROWB;         // bytes of a row of a V tile
    static constexpr int VCOLS = VROWB / 2, VSUBS = W / VCOLS, VSUB = KB * VROWB;
    static constexpr int ONES_BYTES = SUMS ? 16 * VROWB : 0;  // 16 keys: what one product reads
    static constexpr int P_COL = APART ? KB : 0, P_STRIDE = APART ? KB / 2 : KB;
    static constexpr int O_COL = APART ? 2 * KB : NSB * KB, O_STRIDE = NV;
    static constexpr int RING_OFF = QST * QB;
    static constexpr int VRING_OFF = RING_OFF + KST * TILE;
    static constexpr int ONES_OFF = VRING_OFF + VST * TILE;
    static constexpr int ITEM_OFF = ONES_OFF + ONES_BYTES;
    static constexpr int BAR_OFF = ITEM_OFF + kItemRing * 32;
    static constexpr int NBAR = 3 * QST + 3 * KST + 2 * VST + 2 * NPB + NSB + 2 + 2 + 2 * kItemRing;
    static constexpr int SMEM_BYTES = BAR_OFF + 8 * NBAR + 16 + 1024;
    static constexpr uint64_t SWZ = ROWB == 128 ? 2 : 4;
    static_assert(ROWB == 128 || ROWB == 64, "swizzle span");
    static_assert(VSUBS * VSUB == TILE, "V tile");
    static_assert(O_COL + 2 * O_STRIDE <= 512, "tensor memory");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");

    // Q / K operand tile: K-major rows of ROWB bytes
    static __device__ __forceinline__ uint64_t desc_k(uint32_t a) {
        return (uint64_t)((a & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)((8 * ROWB) >> 4) << 32 | (uint64_t)1 << 46 | SWZ << 61;
    }
    // V: the head dimension is contiguous (N), keys run over rows; the columns behind a tile's are SUB bytes away, or the ones
    static __device__ __forceinline__ uint64_t desc_v(uint32_t a) {
        constexpr uint64_t lbo = SUMS ? (ONES_OFF - VRING_OFF) >> 4 : NV > VCOLS ? VSUB >> 4 : 1;
        return (uint64_t)((a & 0x3FFFFu) >> 4) | lbo << 16 | (uint64_t)((8 * VROWB) >> 4) << 32 | (uint64_t)1 << 46 |
               (uint64_t)(VROWB == 128 ? 2 : 4) << 61;
    }
    // the descriptor `bytes` further on in the ring; the ones stay where they are
    static __device__ __forceinline__ uint64_t desc_step(uint32_t bytes) {
        const uint64_t d = bytes >> 4;
        return SUMS ? d - (d << 16) : d;
    }
    // byte offset of column c of a q / k tile with `sub` bytes per COLS columns
    static __device__ __forceinline__ constexpr uint32_t koff(int sub, int c) { return (uint32_t)((c / COLS) * sub + (c % COLS) * 2); }
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
    // 256 softmax threads and the rest share what the launch holds: 512 x 128 = 256 x (176 + 80), 384 x 168 > 256 x 208 + 128 x 80
    // (with 192 + 64 the rotators, and with 168 + 88 the softmax, spilled: windowed prompts of heads of 64 104.6 -> 100.4 us)
    static constexpr int REG_SOFTMAX = ROPE ? 176 : 208;
    static constexpr int REG_REST = 80;
};

struct Item {
    int valid, unit, q0, len, row0, j0, nb, hi;
};
// Two row tiles of one head walk the item's blocks j0 .. nb - 1 together, but a block that no row of a tile can see is not
// multiplied for it: a non-finite v there would reach it (0 x inf).  Tile 0 has the blocks in front of the first one's end, tile 1
// those from the second one's start on.
__device__ __forceinline__ int tile0_end(const Params& p, const Item& it) {
    return p.rows_mode && p.positional ? min(it.nb, it.q0 / kTile + 1) : it.nb;
}
__device__ __forceinline__ int tile1_begin(const Params& p, const Item& it) {
    if (!p.rows_mode) return it.j0;
    if (it.len <= it.q0 + kTile) return it.nb;   // no row of it exists
    return p.positional ? max(0, it.q0 + kTile - p.window + 1) / kTile : it.j0;
}

// A CTA that gave up leaves NaN in every row of its items, written before or not: its callers need not hold a status word.
// `cols`: columns of ctx that belong to an item.
// Out of line and with its arguments by value: in place it changed the softmax loop, 32 q / 8 kv heads of 128, causal: 1021 -> 1084 us.
__device__ __noinline__ void fill_nan(__nv_bfloat16* ctx, int H, const int32_t* seq_start, const int32_t* seq_len, int batch, int qtiles,
                                      int units, int rows, int cols) {
    const int vecs = cols / 8;                // 16-byte pieces of a row
    long long i = blockIdx.x, tiles = 0;      // next item of this CTA; row tiles that exist so far, in the order of the items
    for (int qt = qtiles - 1; qt >= 0; --qt)
        for (int b = 0; b < batch; ++b) {
            const int n = min(rows, __ldg(seq_len + b) - qt * rows);
            if (n <= 0) continue;
            ++tiles;
            for (; i < tiles * units; i += gridDim.x) {
                __nv_bfloat16* o = ctx + ((size_t)__ldg(seq_start + b) + qt * rows) * H + (i % units) * cols;
                for (int k = threadIdx.x; k < n * vecs; k += blockDim.x)
                    *reinterpret_cast<uint4*>(o + (size_t)(k / vecs) * H + k % vecs * 8) =
                        make_uint4(0x7FFF7FFFu, 0x7FFF7FFFu, 0x7FFF7FFFu, 0x7FFF7FFFu);
            }
        }
}

template <int D, bool PAIR, bool ROPE>
__global__ void __launch_bounds__(Threads<ROPE>::N, 1)
attention_fwd_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap tmap_v, const Params p) {
    using C = Cfg<D, PAIR>;
    constexpr int KST = C::KST, VST = C::VST, QST = C::QST, NV = C::NV, NSB = C::NSB, NPB = C::NPB, KB = C::KB;
    constexpr bool APART = C::APART;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - raw);
    const uint32_t kring = base + C::RING_OFF, vring = base + C::VRING_OFF;
    volatile int4* items = reinterpret_cast<volatile int4*>(gbase + C::ITEM_OFF);
    const uint32_t bars = base + C::BAR_OFF;
    const uint32_t q_full = bars, q_free = q_full + 8 * QST, q_rot = q_free + 8 * QST;
    const uint32_t k_full = q_rot + 8 * QST, k_free = k_full + 8 * KST, k_rot = k_free + 8 * KST;
    const uint32_t v_full = k_rot + 8 * KST, v_free = v_full + 8 * VST;
    const uint32_t s_full = v_free + 8 * VST, p_ready = s_full + 8 * NPB, buf_free = p_ready + 8 * NPB, o_full = buf_free + 8 * NSB;
    const uint32_t item_full = o_full + 16, item_free = item_full + 8 * kItemRing, p_free = item_free + 8 * kItemRing;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + C::BAR_OFF + 8 * C::NBAR);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int i = 0; i < QST; ++i) { mbar_init(q_full + 8 * i, 1); mbar_init(q_free + 8 * i, 1); mbar_init(q_rot + 8 * i, 4); }
        for (int i = 0; i < KST; ++i) { mbar_init(k_full + 8 * i, 1); mbar_init(k_free + 8 * i, 1); mbar_init(k_rot + 8 * i, 4); }
        for (int i = 0; i < VST; ++i) { mbar_init(v_full + 8 * i, 1); mbar_init(v_free + 8 * i, 1); }
        for (int i = 0; i < NPB; ++i) { mbar_init(s_full + 8 * i, 1); mbar_init(p_ready + 8 * i, 4); }
        for (int i = 0; i < NSB; ++i) mbar_init(buf_free + 8 * i, APART ? 4 : 1);
        for (int i = 0; i < 2; ++i) mbar_init(o_full + 8 * i, 1);
        for (int i = 0; i < 2; ++i) mbar_init(p_free + 8 * i, 1);
        for (int i = 0; i < kItemRing; ++i) { mbar_init(item_full + 8 * i, 1); mbar_init(item_free + 8 * i, ROPE ? 15 : 11); }
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tmap);
        prefetch_tmap(&tmap_v);
    }
    if (C::SUMS && warp == 11) {
        for (int i = lane; i < C::ONES_BYTES / 16; i += 32)
            st_shared_v4(base + C::ONES_OFF + 16 * i, make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u));
        fence_proxy_async();
    }
    if (warp == 9) {
        tmem_alloc<1>(smem_u32(tmem_slot), 512);
        tmem_relinquish<1>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = warp_uniform(*tmem_slot);
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
        if (warp == 10) {
            // -------------------------------------------------------- items (whole warp)
            const int rows = p.rows_mode ? 2 * kTile : kTile;
            int qt = p.qtiles - 1, b0 = 0;          // scan position: row tile, first of 32 sequences
            long long before = 0;                   // tiles that exist in front of it
            uint32_t n = 0;
            for (long long i = blockIdx.x;; i += gridDim.x, ++n) {
                const long long want = i / p.units;
                int len = 0;
                unsigned mask = 0;
                for (; qt >= 0;) {
                    const int b = b0 + lane;
                    len = b < p.batch ? __ldg(p.seq_len + b) : 0;
                    mask = __ballot_sync(0xffffffffu, len > qt * rows);
                    if (want < before + __popc(mask)) break;
                    before += __popc(mask);
                    b0 += 32;
                    if (b0 >= p.batch) { b0 = 0; --qt; }
                }
                Item it{};
                if (qt >= 0) {
                    const bool mine = ((mask >> lane) & 1) && __popc(mask & ((1u << lane) - 1u)) == (int)(want - before);
                    const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
                    it.valid = 1;
                    it.unit = (int)(i % p.units);
                    it.q0 = qt * rows;
                    it.len = __shfl_sync(0xffffffffu, len, src);
                    it.row0 = __ldg(p.seq_start + b0 + src);
                    it.hi = p.positional ? min(it.len, it.q0 + rows) : it.len;
                    it.j0 = p.positional ? max(0, it.q0 - p.window + 1) / KB : 0;
                    it.nb = (it.hi + KB - 1) / KB;
                }
                const uint32_t slot = n % kItemRing;
                if (n >= kItemRing && !mbar_wait_warp(item_free + 8 * slot, ((n / kItemRing) - 1) & 1, abort_flag)) break;
                if (lane == 0) {
                    items[2 * slot].x = it.valid; items[2 * slot].y = it.unit; items[2 * slot].z = it.q0; items[2 * slot].w = it.len;
                    items[2 * slot + 1].x = it.row0; items[2 * slot + 1].y = it.j0; items[2 * slot + 1].z = it.nb; items[2 * slot + 1].w = it.hi;
                    mbar_arrive(item_full + 8 * slot);   // release: orders the stores above
                }
                if (!it.valid) break;
            }
        } else if (warp == 8) {
            // -------------------------------------------------------- TMA (whole warp, one lane issues)
            uint32_t kst = 0, kph = 1, vst = 0, vph = 1;   // ring positions and the parities of their free barriers
            bool ok = true;
            Item it;
            for (uint32_t n = 0; ok; ++n) {
                if (next_item(n, it) != 1) break;
                const uint32_t qs = n % QST;
                if (n >= QST && !mbar_wait_warp(q_free + 8 * qs, ((n / QST) - 1) & 1, abort_flag)) break;
                const int head0 = (PAIR || !p.rows_mode) ? 2 * it.unit : it.unit;
                const int kvh = PAIR ? head0 : head0 / p.kv_group;
                if (elect_one()) {
                    mbar_expect_tx(q_full + 8 * qs, C::QB);
#pragma unroll
                    for (int t = 0; t < (PAIR ? 1 : 2); ++t)
#pragma unroll
                        for (int s = 0; s < C::NSUB; ++s)
#pragma unroll
                            for (int r = 0; r < kTile; r += KB)
                                tma_load_2d(base + qs * C::QB + t * C::QTILE + s * C::QSUB + r * C::ROWB, &tmap,
                                            (head0 + (p.rows_mode ? 0 : t)) * D + s * C::COLS,
                                            it.row0 + it.q0 + (p.rows_mode ? t * kTile : 0) + r, q_full + 8 * qs);
                }
                __syncwarp();
                for (int j = it.j0; j < it.nb && ok; ++j) {
                    if (!(ok = mbar_wait_warp(k_free + 8 * kst, kph, abort_flag))) break;
                    if (elect_one()) {
                        mbar_expect_tx(k_full + 8 * kst, C::TILE);
#pragma unroll
                        for (int s = 0; s < C::NSUB; ++s)
                            tma_load_2d(kring + kst * C::TILE + s * C::SUB, &tmap, p.H + kvh * D + s * C::COLS, it.row0 + j * KB, k_full + 8 * kst);
                    }
                    __syncwarp();
                    if (++kst == KST) { kst = 0; kph ^= 1; }
                    if (!(ok = mbar_wait_warp(v_free + 8 * vst, vph, abort_flag))) break;
                    if (elect_one()) {
                        mbar_expect_tx(v_full + 8 * vst, C::TILE);
#pragma unroll
                        for (int s = 0; s < C::VSUBS; ++s)
                            tma_load_2d(vring + vst * C::TILE + s * C::VSUB, &tmap_v, p.H + p.Hkv + kvh * D + s * C::VCOLS, it.row0 + j * KB,
                                        v_full + 8 * vst);
                    }
                    __syncwarp();
                    if (++vst == VST) { vst = 0; vph ^= 1; }
                }
            }
        } else if (warp == 9) {
            // -------------------------------------------------------- scores (whole warp, one lane issues)
            const uint32_t k_rdy = ROPE ? k_rot : k_full, q_rdy = ROPE ? q_rot : q_full;
            constexpr uint32_t idesc_s = idesc_attn(kTile, KB, 0);
            const uint64_t kd0 = C::desc_k(kring), qd0 = C::desc_k(base);
            uint32_t sbuf = 0, bph = 1, kst = 0, kph = 0, qst = 0, qph = 0;
            bool ok = true;
            Item it;
            for (uint32_t n = 0; ok; ++n) {
                if (next_item(n, it) != 1 || !mbar_wait_warp(q_rdy + 8 * qst, qph, abort_flag)) break;
                const uint64_t qd1 = qd0 + (uint64_t)((qst * C::QB) >> 4);
                const int end0 = tile0_end(p, it), begin1 = tile1_begin(p, it);
                for (int left = it.nb - it.j0; left > 0 && ok; --left) {
                    if (!(ok = mbar_wait_warp(k_rdy + 8 * kst, kph, abort_flag))) break;
                    const uint64_t kd1 = kd0 + (uint64_t)((kst * C::TILE) >> 4);
                    const uint32_t idesc = left == 1 ? idesc_attn(kTile, (it.hi - (it.nb - 1) * KB + 15) & ~15, 0) : idesc_s;
#pragma unroll 1
                    for (uint32_t t = 0; t < 2; ++t) {
                        if (!(ok = mbar_wait_warp(buf_free + 8 * sbuf, bph, abort_flag))) break;
                        tc_fence_after();
                        const uint64_t qd = qd1 + (uint64_t)((t * (PAIR ? C::koff(C::QSUB, D) : C::QTILE)) >> 4);
                        const uint64_t kd = kd1 + (uint64_t)((PAIR ? t * C::koff(C::SUB, D) : 0) >> 4);
                        const uint32_t acc = tmem + sbuf * KB;
                        const bool seen = t ? it.nb - left >= begin1 : it.nb - left < end0;
                        if (elect_one()) {
                            if (seen) {
#pragma unroll
                                for (int k = 0; k < D / 16; ++k)
                                    umma_bf16<1>(acc, qd + (C::koff(C::QSUB, 16 * k) >> 4), kd + (C::koff(C::SUB, 16 * k) >> 4), idesc, k != 0);
                            }
                            umma_commit<1>(s_full + 8 * (APART ? t : sbuf));
                            if (t) {
                                umma_commit<1>(k_free + 8 * kst);
                                if (left == 1) umma_commit<1>(q_free + 8 * qst);
                            }
                        }
                        __syncwarp();
                        if (++sbuf == NSB) { sbuf = 0; bph ^= 1; }
                    }
                    if (++kst == KST) { kst = 0; kph ^= 1; }
                }
                if (++qst == QST) { qst = 0; qph ^= 1; }
            }
        } else if (warp == 11) {
            // -------------------------------------------------------- O += P V (whole warp, one lane issues)
            constexpr uint32_t idesc_o = idesc_attn(kTile, NV, 1);
            const uint64_t vd0 = C::desc_v(vring);
            uint32_t vbuf = 0, pph = 0, vst = 0, vph = 0;
            bool ok = true;
            Item it;
            for (uint32_t n = 0; ok; ++n) {
                if (next_item(n, it) != 1) break;
                const int end0 = tile0_end(p, it), begin1 = tile1_begin(p, it);
                for (int left = it.nb - it.j0; left > 0 && ok; --left) {
                    const bool last = left == 1;
                    const int keys = last ? it.hi - (it.nb - 1) * KB : KB, kpad = (keys + 15) & ~15;
                    if (!(ok = mbar_wait_warp(v_full + 8 * vst, vph, abort_flag))) break;
                    if (keys < kpad) {
                        // rows past the end of the sequence get probability 0, but whatever lies behind them in memory must
                        // not turn that into a NaN: clear them
                        const uint32_t vtile = vring + vst * C::TILE;
                        const int chunks = (kpad - keys) * (C::VROWB / 16);
                        for (int i = lane; i < chunks * C::VSUBS; i += 32)
                            st_shared_v4(vtile + (i / chunks) * C::VSUB + keys * C::VROWB + (i % chunks) * 16, make_uint4(0, 0, 0, 0));
                        fence_proxy_async();
                        __syncwarp();
                    }
#pragma unroll 1
                    for (uint32_t t = 0; t < 2; ++t) {
                        const uint64_t vd = vd0 + C::desc_step(vst * C::TILE + (PAIR ? t * C::VSUB : 0));
                        const uint32_t pa = tmem + C::P_COL + vbuf * C::P_STRIDE, oa = tmem + C::O_COL + t * C::O_STRIDE;
                        if (!(ok = mbar_wait_warp(p_ready + 8 * vbuf, pph, abort_flag))) break;
                        tc_fence_after();
                        const int j = it.nb - left;
                        if (elect_one()) {
                            if (t ? j >= begin1 : j < end0) {
                                umma_ts(oa, pa, vd, idesc_o, j == (t ? begin1 : it.j0) ? 0u : 1u);
#pragma unroll
                                for (int kk = 1; kk < KB / 16; ++kk)
                                    if (kk * 16 < kpad) umma_ts(oa, pa + kk * 8, vd + C::desc_step(16 * C::VROWB * kk), idesc_o, 1u);
                            }
                            umma_commit<1>((APART ? p_free : buf_free) + 8 * vbuf);
                            if (last) umma_commit<1>(o_full + 8 * t);
                            if (t) umma_commit<1>(v_free + 8 * vst);
                        }
                        __syncwarp();
                        if (++vbuf == NPB) { vbuf = 0; pph ^= 1; }
                    }
                    if (++vst == VST) { vst = 0; vph ^= 1; }
                }
            }
        } else if (ROPE && warp >= 12) {
            // -------------------------------------------------------- rotary embedding of Q tiles and K blocks
            constexpr int HEADS = PAIR ? 2 : 1, CPR = D / 16;   // heads per tile; (lo, hi) 16-byte chunk pairs per head row
            // A thread keeps to one chunk pair and walks over rows, with the next row's cosines and sines requested before the
            // current one is rotated (both heads of a pair share them): 64 KB of tables per 128 x 64 block come from L2.
            constexpr int STEP = 128 / CPR;                      // rows between a thread's tasks
            const int rt = threadIdx.x - 12 * 32, cc = rt % CPR, r0 = rt / CPR;
            // rows first_pos + r, r < rows, of a tile with `sub` bytes per COLS columns; positions at or past `len` are left alone
            auto rotate = [&](uint32_t tile, int sub, int rows, int first_pos, int len) {
                const int end = min(rows, len - first_pos);
                const float4* pc = reinterpret_cast<const float4*>(p.rope_cos + (size_t)(first_pos + r0) * (D / 2) + cc * 8);
                const float4* ps = reinterpret_cast<const float4*>(p.rope_sin + (size_t)(first_pos + r0) * (D / 2) + cc * 8);
                float4 c0, c1, s0, s1;
                if (r0 < end) { c0 = __ldg(pc); c1 = __ldg(pc + 1); s0 = __ldg(ps); s1 = __ldg(ps + 1); }
#pragma unroll 1
                for (int r = r0; r < end; r += STEP) {
                    float4 n0 = c0, n1 = c1, m0 = s0, m1 = s1;
                    pc += STEP * (D / 8);
                    ps += STEP * (D / 8);
                    if (r + STEP < end) { n0 = __ldg(pc); n1 = __ldg(pc + 1); m0 = __ldg(ps); m1 = __ldg(ps + 1); }
                    const uint32_t swz = C::ROWB == 128 ? (uint32_t)(r & 7) : (uint32_t)((r >> 1) & 3);
#pragma unroll
                    for (int hd = 0; hd < HEADS; ++hd) {
                        const int lo_col = hd * D + cc * 8, hi_col = lo_col + D / 2;
                        const uint32_t a = tile + (lo_col / C::COLS) * sub + r * C::ROWB + ((((uint32_t)(lo_col % C::COLS) / 8) ^ swz) << 4);
                        const uint32_t b = tile + (hi_col / C::COLS) * sub + r * C::ROWB + ((((uint32_t)(hi_col % C::COLS) / 8) ^ swz) << 4);
                        uint4 lo = ld_shared_v4(a), hi = ld_shared_v4(b);
                        rope_rotate8(lo, hi, c0, c1, s0, s1);
                        st_shared_v4(a, lo);
                        st_shared_v4(b, hi);
                    }
                    c0 = n0; c1 = n1; s0 = m0; s1 = m1;
                }
                fence_proxy_async();
                __syncwarp();
            };
            Item it;
            uint32_t kst = 0, kph = 0;
            bool ok = true;
            for (uint32_t n = 0; ok; ++n) {
                if (next_item(n, it) != 1) break;
                const uint32_t qs = n % QST;
                if (!mbar_wait_warp(q_full + 8 * qs, (n / QST) & 1, abort_flag)) break;
                rotate(base + qs * C::QB, C::QSUB, kTile, it.q0, it.len);
                if (!PAIR) rotate(base + qs * C::QB + C::QTILE, C::QSUB, kTile, it.q0 + (p.rows_mode ? kTile : 0), it.len);
                if (lane == 0) mbar_arrive(q_rot + 8 * qs);
                for (int j = it.j0; j < it.nb; ++j) {
                    if (!(ok = mbar_wait_warp(k_full + 8 * kst, kph, abort_flag))) break;
                    rotate(kring + kst * C::TILE, C::SUB, KB, j * KB, it.len);
                    if (lane == 0) mbar_arrive(k_rot + 8 * kst);
                    if (++kst == KST) { kst = 0; kph ^= 1; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ softmax (thread = query row)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Threads<ROPE>::REG_SOFTMAX));
        const int t = warp >> 2, quad = warp & 3;
        const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t o_col = tl + C::O_COL + t * C::O_STRIDE;
        constexpr int NCH = KB / 32;         // 32-key chunks per block
        const float scale = p.scale_log2e;
        uint32_t buf = t, sph = 0;   // score buffer and its parity; jobs t, t + 2, t + 4, ..
        uint32_t pbuf = 0, pph = 0;  // the same of this tile's previous block
        bool ok = true;
        Item it;
        for (uint32_t n = 0; ok; ++n) {
            if (next_item(n, it) != 1) break;
            const int q0 = it.q0 + (p.rows_mode ? t * kTile : 0);
            const int wr0 = q0 + quad * 32, row = wr0 + lane;      // rows of this warp, of this thread (position in the sequence)
            const bool live = wr0 < it.len;
            const int head = (PAIR || !p.rows_mode) ? 2 * it.unit + t : it.unit;
            const int jb = t ? tile1_begin(p, it) : it.j0, je = t ? it.nb : tile0_end(p, it);
            float m_ref = -INFINITY;
            float l4[4] = {0.f, 0.f, 0.f, 0.f};
            uint64_t any2[2] = {0, 0};
            for (int j = it.j0; j < it.nb; ++j) {
                if (!(ok = mbar_wait_warp(s_full + 8 * buf, sph, abort_flag))) break;
                const bool seen = live && j >= jb && j < je;
                if (APART && !seen) {
                    if (lane == 0) mbar_arrive(buf_free);
                    if (!(ok = mbar_wait_warp(p_free + 8 * t, sph ^ 1, abort_flag))) break;
                }
                if (seen) {
                    tc_fence_after();
                    const uint32_t s_col = tl + (APART ? 0 : buf * KB);
                    const uint32_t p_col = APART ? tl + C::P_COL + t * C::P_STRIDE : s_col;
                    const int k0 = j * KB;
                    uint32_t s[NCH][32];
#pragma unroll
                    for (int c = 0; c < NCH; ++c) tmem_ld_32x32(s_col + 32 * c, s[c]);
                    tmem_ld_wait();
                    bool p_done = false;
                    if (APART) {
                        // the scores are in registers: their buffer is the other tile's
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(buf_free);
                        // this tile's previous product: P's buffer is free and O complete (asked for ahead of its use)
                        p_done = mbar_test_wait(p_free + 8 * t, sph ^ 1);
                    }
                    const bool whole = k0 + KB <= it.hi && (!p.positional || (k0 + KB - 1 <= wr0 && k0 > wr0 + 31 - p.window));
                    if (!whole) {
                        // visible keys of this row: columns first .. lim; one bit per column
                        const int first = p.positional ? row - p.window + 1 - k0 : 0;
                        const int lim = min(it.hi - 1, p.positional ? row : it.hi) - k0;
#pragma unroll
                        for (int c = 0; c < NCH; ++c) {
                            const int a = min(max(first - 32 * c, 0), 32), e = min(max(lim + 1 - 32 * c, 0), 32);
                            const uint32_t bits = (e > a ? (uint32_t)((1ull << e) - 1) & ~(uint32_t)((1ull << a) - 1) : 0u);
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (!((bits >> i) & 1)) s[c][i] = 0xFF800000u;   // -inf
                        }
                    }
                    float m_blk;
                    {
                        float mx[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            constexpr int R = KB / 4;     // scores per partial maximum
                            mx[c] = fmaxf(__uint_as_float(s[c * R / 32][c * R % 32]), __uint_as_float(s[c * R / 32][c * R % 32 + 1]));
#pragma unroll
                            for (int i = 2; i < R; i += 2)
                                mx[c] = max3f(mx[c], __uint_as_float(s[c * R / 32][c * R % 32 + i]), __uint_as_float(s[c * R / 32][c * R % 32 + i + 1]));
                        }
                        m_blk = fmaxf(max3f(mx[0], mx[1], mx[2]), mx[3]) * scale;
                    }
                    if (APART) {
                        if (!__all_sync(0xffffffffu, p_done) && !(ok = mbar_wait_warp(p_free + 8 * t, sph ^ 1, abort_flag))) break;
                        tc_fence_after();
                    }
                    if (j == jb) {
                        m_ref = m_blk;
                    } else {
                        const bool need = m_blk > m_ref + kRescaleAbove;
                        if (__any_sync(0xffffffffu, need)) {
                            // the products issued so far must have landed in O
                            if (!APART && !(ok = mbar_wait_warp(buf_free + 8 * pbuf, pph, abort_flag))) break;
                            tc_fence_after();
                            const float alpha = need ? ex2f(m_ref - m_blk) : 1.f;
                            if (need) m_ref = m_blk;
#pragma unroll
                            for (int i = 0; i < 4; ++i) l4[i] *= alpha;
                            if (C::SUMS) {
                                uint32_t l;
                                tmem_ld_32x1(o_col + D, l);
                                tmem_ld_wait();
                                tmem_st_32x1(o_col + D, __float_as_uint(__uint_as_float(l) * alpha));
                            }
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
                    // straight line over all chunks, masked ones included: a branch per chunk drains the exponential unit
                    // each time, and a second copy of the code costs more in instruction fetches than it saves
                    // The row sum adds the ROUNDED probabilities, those that P V multiplies, so that a weight's rounding changes
                    // numerator and denominator alike: with the sum of the unrounded ones the error against 64 bits was 1 to 2 %
                    // larger for v around zero and 7 % for v with a mean of four deviations.
                    // The unrounded sum is kept as well: it says whether a row saw any key, and with it the compiler orders the
                    // loop far better, even where it is one instruction more (12 heads of 32, 256 sequences of 32..256: 71.8 us
                    // without it, 62.3 with; 32 q / 8 kv heads of 64, window 300 over 1024..4096: 306 / 293; of 128, causal: 1078 / 1054).
#pragma unroll
                    for (int c = 0; c < NCH; ++c) {
                        uint32_t pk[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            float x0, x1;
                            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c][2 * i]), __uint_as_float(s[c][2 * i + 1])), sc2, ng2), x0, x1);
                            x0 = ex2f(x0);
                            x1 = ex2f(x1);
                            any2[i & 1] = add_f32x2(any2[i & 1], pack_f32x2(x0, x1));
                            pk[i] = pack_bf16(x0, x1);
                            if (!C::SUMS) add_bf16x2(l4[2 * (i & 1)], l4[2 * (i & 1) + 1], pk[i]);
                        }
                        tmem_st_32x16(p_col + 16 * c, pk);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(p_ready + 8 * buf);
                pbuf = buf;
                pph = sph;
                if (!APART) buf += 2;
                if (APART) sph ^= 1;
                else if (buf >= NSB) { buf -= NSB; sph ^= 1; }
            }
            if (!ok) break;
            // ---- O / row sum -> bf16 -> global ----
            if (!(ok = mbar_wait_warp(o_full + 8 * t, n & 1, abort_flag))) break;
            if (live) {
                tc_fence_after();
                float l = (l4[0] + l4[1]) + (l4[2] + l4[3]);
                if (C::SUMS) {
                    uint32_t sum;
                    tmem_ld_32x1(o_col + D, sum);
                    tmem_ld_wait();
                    l = __uint_as_float(sum);
                }
                float a0, a1, b0, b1;
                unpack_f32x2(any2[0], a0, a1);
                unpack_f32x2(any2[1], b0, b1);
                const float inv = (a0 + a1) + (b0 + b1) > 0.f ? 1.0f / l : 0.f;
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
    if (*abort_flag) fill_nan(p.ctx, p.H, p.seq_start, p.seq_len, p.batch, p.qtiles, p.units, p.rows_mode ? 2 * kTile : kTile, p.rows_mode ? D : 2 * D);
}

}  // namespace tcat
}  // namespace rlx

// Persistent tcgen05 GPTQ matmul for 17 token rows and more.
//
// As in gptq_umma.cuh, the 128 columns of a panel are the MMA's rows, dequantised into a ring of A stages in tensor memory, and a tile of
// token rows is its N.  An item (128 rows of K of a panel, 8 KB of packed weights) is the unit of every hand-over.  What differs:
//   * One CTA per SM works through its tiles without leaving the kernel.  Tensor memory holds two accumulators of up to 160
//     token rows beside the A stages, so the epilogue of a tile (four warps of its own) runs under the main loop of the next
//     one, and the rings never drain between tiles.  The last tile, with nothing to hide under, is shared out over all 20
//     epilogue and dequant warps.
//   * The number of token rows of a tile is a run-time multiple of 16, so that tiles and waves come out even: 300 rows on 96
//     panels are three tiles of 112 in two waves, where tiles of 256 cost two waves of 256.
//   * Four sets of four dequant warps take every fourth item each: a set's pass takes about 1000 clocks, most of it latency.
//   * x lands on the barrier that the item's dequant warps arrive on, so the MMA thread has one wait per item.  These barriers are
//     a ring of 16, so x may be requested further ahead than there are A stages: an x tile arrives 1500 clocks after its request,
//     and with tiles of 160 rows, which have three A stages, four slots of x instead of three give 1 to 4 % (2048 x 4096 x 12288
//     149 -> 143 us).  Weights run ahead in a ring of their own (and start before the previous kernel has finished).
//   * Where tiles are few, clusters of two or four CTAs share the K range of a tile (one tile per cluster then).
// What bounds it.  From 128 token rows per tile the MMA: 572 clocks per item of 512 at full rate (qkv M = 512), and then the
// power limit (1.45-1.5 GHz in that loop).  With fewer rows instruction issue: about 520 clocks per item, for four dequant
// warps on every scheduler and the MMA thread among them (a second MMA thread with an accumulator of its own made it 560).  The
// MMA thread pays for every instruction it fetches between theirs, hence its short loop (765 -> 589 clocks per item against a
// warp that elects for every item, o M = 512) and the rolled dequant loop.  Stages of a tile of 176 or 192 rows (only two fit beside the accumulators) made the hand-over the
// limit: 811 clocks per item of 704.
// Measured (7B layer of four matmuls in a chain, us, kernel of gptq_umma.cuh alone -> this where it is chosen): M = 17
// 59.4 -> 51.5, M = 64 71.6 -> 55.7, M = 128 82 -> 68.6, M = 300 177 -> 122, M = 512 212 -> 172; 8-bit M = 128 124 -> 102,
// M = 300 232 -> 167.
#pragma once
#include "gptq_decode.cuh"      // waits with a CTA-wide flag

namespace gptq {

constexpr int kPrefillSets = 4;                                      // dequant warp sets
constexpr int kPrefillMaxTok = 160;
// warps: x producer, MMA, epilogue x 4, dequant x 16, weight producer
constexpr int kPrefillXWarp = 0, kPrefillFirstEpi = 2, kPrefillFirstDq = 6, kPrefillWWarp = kPrefillFirstDq + 4 * kPrefillSets;
constexpr int kPrefillThreads = 32 * (kPrefillWWarp + 1);
constexpr int kPrefillStage = 4 * 32 * 64;                           // epilogue: 32 tokens x 64 bytes per warp
// A stages (of one item, 64 columns) and columns of an accumulator: tensor memory holds 2 x 128 + 4 x 64 or 2 x 160 + 3 x 64
__host__ __device__ constexpr int prefill_a_stages(int tok) { return tok <= 128 ? 4 : 3; }
__host__ __device__ constexpr int prefill_acc_columns(int tok) { return tok <= 128 ? 128 : 160; }
// Fewest items of a tile that a CTA works through alone (without a split of K).  The dequant warps take part in the epilogue of
// the CTA's last tile only, and wait for its accumulator by parity without having waited for the tile before the last but one,
// which used the same accumulator: if that were still being multiplied, the wait would pass at once.  It is not: a set's last
// item, one of the CTA's last kPrefillSets, has waited for the MMAs of the item an A ring earlier, and two tiles lie behind.
constexpr int kPrefillMinItems = 4;
static_assert(2 * kPrefillMinItems + 1 > kPrefillSets + prefill_a_stages(0), "a dequant warp's wait for the last tile's accumulator would be ambiguous");
// Slots of x, at most.  4096 x 22016 with three / four / eight, us: 64 rows 22.3 / 21.1 / 21.0, 96 rows 24.6 / 22.2 / 22.0; 112 rows
// 25.7 / 23.0 / 22.8 (five fit), 128 rows 27.1 / 24.4 (four fit).
constexpr int kPrefillXSlots = 4;
static_assert(kPrefillXSlots <= kUmmaDoneRing, "x would be requested onto a barrier whose last item has not been multiplied");
// Weight slots.  A set's parity wait on a slot needs the slot's previous item to be in: with this many that is known, the
// set's last pass (four items ago) has waited for the MMAs of the item that had its A stage before.  With 8-bit weights
// (16 KB per slot) five, and the set asks.
__host__ __device__ constexpr int prefill_w_slots(int tok, bool w8) { return w8 ? 5 : kPrefillSets + prefill_a_stages(tok); }
// bytes of the epilogue's stage and the weight ring, and x slots of tok * 256 bytes that fit behind them (2 KB: barriers, alignment)
__host__ __device__ constexpr int prefill_ring_bytes(int tok, bool w8) { return kPrefillStage + prefill_w_slots(tok, w8) * (w8 ? 2 : 1) * kItemWBytes; }
__host__ __device__ constexpr int prefill_x_slots(int tok, bool w8)
{
    const int fit = (227 * 1024 - 2048 - prefill_ring_bytes(tok, w8)) / (tok * 256);
    return fit < kPrefillXSlots ? fit : kPrefillXSlots;
}

// 16 lanes x 32 columns of tensor memory as four 8-column groups: r[4 g], r[4 g + 1] are lane T / 4, columns 8 g + 2 (T % 4) and
// the next one, r[4 g + 2], r[4 g + 3] the same of lane T / 4 + 8 (T: thread of the warp)
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, const uint32_t (&r)[4])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
                 : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// bulk copy from this CTA's shared memory to a CTA of the cluster, completion counted in bytes on that CTA's mbarrier
__device__ __forceinline__ void bulk_s2s_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src),
                 "r"(bytes), "r"(bar)
                 : "memory");
}
// 16 bytes into the shared memory of a CTA of the cluster, counted on that CTA's mbarrier
__device__ __forceinline__ void st_async_b32x4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
template <bool BF>
__device__ __forceinline__ uint32_t pack_out16(float2 v)
{
    if constexpr (BF) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
        return *reinterpret_cast<const uint32_t *>(&b);
    } else {
        const __half2 h = __floats2half2_rn(v.x, v.y);
        return *reinterpret_cast<const uint32_t *>(&h);
    }
}

// Tiles of at most this many token rows exchange their parts by stores into the owners' shared memory, taller ones by bulk copies
// (what both take with 4-bit weights: see prefill_kernel).  8-bit weights, copies / stores, us: clusters of four, 4096 x 4096, 17 rows
// 9.7 / 9.4, 64 rows 12.4 / 12.3, 80 rows 12.8 / 12.7, 96 rows 13.1 / 13.5; 11008 x 4096, 17 to 64 rows the same, 112 rows 22.4 / 23.1;
// 2048 x 2048, 64 rows 8.1 / 8.0, 112 rows 9.4 / 9.6; clusters of two, 4096 x 5120, 17 rows 12.5 / 11.7, 64 rows 14.9 / 14.7, 112 rows 16.3 / 16.3.
__host__ __device__ constexpr int prefill_push_rows(bool w8) { return w8 ? 64 : 112; }
// bytes of a sender's part: 128 / S columns of the tile's rows, a column an odd number of 16-byte pieces
__host__ __device__ constexpr int prefill_part_bytes(int tok, int S) { return kPanel / S * (tok + 4) * 4; }
// The others' parts land in the epilogue's stage and the weight ring, the own one in the x ring.
constexpr bool prefill_parts_fit(bool w8)
{
    for (int S = 2; S <= 4; S *= 2)
        for (int tok = 32; tok <= prefill_push_rows(w8); tok += 16)
            if ((S - 1) * prefill_part_bytes(tok, S) > prefill_ring_bytes(tok, w8) || prefill_part_bytes(tok, S) > prefill_x_slots(tok, w8) * tok * 256)
                return false;
    return true;
}
static_assert(prefill_parts_fit(false) && prefill_parts_fit(true), "stored parts would run over what a CTA still uses");

struct PrefillArgs {
    const uint8_t *scales, *qzeros;   // tiled
    __half *y;
    int M, N, G;                      // G: 128-row items of K (of one plane with 8-bit weights)
    int S;                            // CTAs (a cluster) that share the K range of a tile; then every cluster has one tile
    int tok, tiles, x_slots;          // token rows per tile; tiles; depth of the x ring in items
    const TiledTrailer *trailer;
    int fuse;
    const __half *bias, *residual;
    int trace_slot;
    const int32_t *out_index;
};

// SPLIT: K shared by a cluster, the partial tiles parked and copied, or stored into the owners' shared memory
constexpr int kParkParts = 1, kPushParts = 2;
template <int SUB, bool BF, bool W8, int SPLIT>
__global__ void __launch_bounds__(kPrefillThreads, 1)
prefill_kernel(const PrefillArgs a, const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap x_map)
{
    extern __shared__ uint8_t smem_raw[];
    constexpr int PL = W8 ? 2 : 1;                            // nibble planes
    const uint32_t flags = __ldg(&a.trailer->flags);          // needed late: requested first
    if (threadIdx.x == 0) {
        GPTQ_TRACE_MIN(a.trace_slot, first_entry);
        GPTQ_TRACE_MAX(a.trace_slot, last_entry);
        if (blockIdx.x == 0) {
            GPTQ_TRACE_SET(a.trace_slot, kernel_and_ctas, (2ull << 32) | gridDim.x);
        }
    }
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // wfull[s]: packed weights of a ring slot have landed; afull[n mod 16]: the A operand of the CTA's n-th item has been written and
    // its x has landed; done[n mod 16]: the MMAs of the CTA's n-th item have completed; dfull / dempty: accumulators
    const uint32_t bar_wfull = base, bar_afull = base + 384, bar_done = base + 192, bar_dfull = base + 320,
                   bar_dempty = base + 336;
    const uint32_t tmem_slot = base + 352, flag = base + 356, bar_recv = base + 360, bar_ready = base + 368;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int S = SPLIT ? a.S : 1, rank = SPLIT ? (int)blockIdx.x % S : 0, tile0 = SPLIT ? (int)blockIdx.x / S : (int)blockIdx.x;
    const int tile_step = SPLIT ? (int)gridDim.x / S : (int)gridDim.x;
    const int g0 = SPLIT ? a.G * rank / S : 0, G = SPLIT ? a.G * (rank + 1) / S - g0 : a.G;           // items of a tile that are this CTA's
    const int tok = a.tok, panels = a.N / kPanel, XS = a.x_slots;
    const int PS = prefill_a_stages(tok), WS = prefill_w_slots(tok, W8), acc = prefill_acc_columns(tok);
    constexpr uint32_t kWSlot = PL * kItemWBytes;
    const uint32_t x_half = (uint32_t)tok * 128, x_slot = 2 * x_half;       // an item's x: two K64 tiles
    const uint32_t stg0 = base + 1024, w_ring = stg0 + kPrefillStage, x_ring = w_ring + WS * kWSlot;

    if (threadIdx.x == 0) {
        for (int s = 0; s < WS; ++s) mbar_init(bar_wfull + 8 * s, 1);
        for (int s = 0; s < kUmmaDoneRing; ++s) {
            mbar_init(bar_afull + 8 * s, 5);
            mbar_init(bar_done + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_dfull + 8 * s, 1);
            mbar_init(bar_dempty + 8 * s, 4);
        }
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(0u) : "memory");
        if (SPLIT) mbar_init(bar_recv, 1);
        if (SPLIT == kPushParts) mbar_init(bar_ready, 4 * kPrefillSets * S);
        fence_barrier_init();
        if (SPLIT) {
            const int m0 = tile0 / panels * tok, rows = (a.M - m0) < tok ? (a.M - m0) : tok;
            mbar_arrive_expect_tx(bar_recv, (uint32_t)((S - 1) * (kPanel / S) * (SPLIT == kPushParts ? (rows + 3) & ~3 : rows) * 4));
        }
        fence_proxy_async();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, lds32(tmem_slot), 0);
    if (SPLIT == kPushParts) cluster_arrive_release();        // "my barriers are set up"
    pdl_launch_dependents();

    const bool is_dq = warp >= kPrefillFirstDq && warp < kPrefillWWarp, is_epi = warp >= kPrefillFirstEpi && warp < kPrefillFirstDq;
    auto wait_done = [&](int n) { decode_wait(bar_done + 8 * (n & (kUmmaDoneRing - 1)), (uint32_t)(n / kUmmaDoneRing) & 1u, flag); };

    if (warp == kPrefillXWarp || warp == kPrefillWWarp) {
        // ---------------------------------------------------------------- TMA producers (one thread issues): x tiles and
        // packed weights by a warp each
        const bool xw = warp == kPrefillXWarp;
        if (elect_one()) tma_prefetch_descriptor(xw ? &x_map : &w_map);
        if (xw) {
            pdl_wait();                  // weights do not depend on earlier kernels
            GPTQ_TRACE_MIN(a.trace_slot, first_wait_done);
            GPTQ_TRACE_MAX(a.trace_slot, last_wait_done);
        } else {
            GPTQ_TRACE_MIN(a.trace_slot, first_weight_issue);
        }
        const int NS = xw ? XS : WS;
        int s = 0, n = 0;
        for (int tile = tile0; tile < a.tiles; tile += tile_step) {
            const int mt = tile / panels, p = tile - mt * panels;       // neighbouring CTAs share the x tile
            for (int t = 0; t < G; ++t, ++n) {
                if (n >= NS) wait_done(n - NS);
                if (elect_one()) {
                    if (xw) {
                        // (item n - 16, the last on this barrier, has been multiplied: there are at most 16 slots)
                        const uint32_t bar = bar_afull + 8 * (n & (kUmmaDoneRing - 1));
                        mbar_arrive_expect_tx(bar, x_slot);
                        tma_load_3d(x_ring + s * x_slot, &x_map, 0, mt * tok, 2 * (g0 + t), bar);     // rows >= M read as zero
                    } else {
                        // packed weights as rows of 64 bytes, 128 to an item
                        mbar_arrive_expect_tx(bar_wfull + 8 * s, kWSlot);
#pragma unroll
                        for (int pl = 0; pl < PL; ++pl)
                            tma_load_2d(w_ring + s * kWSlot + pl * kItemWBytes, &w_map, 0, (a.G * (PL * p + pl) + g0 + t) * 128, bar_wfull + 8 * s);
                    }
                }
                __syncwarp();
                if (++s == NS) s = 0;
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA (one thread issues)
        const uint32_t idesc = umma_idesc_f16(128, tok) | (BF ? kUmmaIdescBf16 : 0u);
        if (elect_one()) {
            const uint64_t desc0 = umma_desc_k_major_sw128(x_ring);
            const uint32_t desc_lo = (uint32_t)desc0, desc_hi = (uint32_t)(desc0 >> 32);      // (the address field is in the low word)
            const uint32_t x_step = x_slot >> 4, half_step = x_half >> 4, x_end = XS * x_step, a0 = tmem_base + 2 * acc;
            uint32_t xo = 0, n = 0, sa = 0;
            for (int tile = tile0, it = 0; tile < a.tiles; tile += tile_step, ++it) {
                const uint32_t d = it & 1, d_tmem = tmem_base + d * acc;
                decode_wait(bar_dempty + 8 * d, ((uint32_t)(it >> 1) & 1u) ^ 1u, flag);
                uint32_t accumulate = 0;
                for (int t = G; t > 0; --t, ++n) {
                    decode_wait(bar_afull + 8 * (n & (kUmmaDoneRing - 1)), n / kUmmaDoneRing & 1u, flag);
                    tc_fence_after_sync();
                    if (n == 0) GPTQ_TRACE_MIN(a.trace_slot, first_data);
                    const uint32_t a_tmem = a0 + sa * 64;
                    const uint32_t b0 = desc_lo + xo, b1 = b0 + half_step;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {     // 16 k per MMA: 8 columns of A, 32 bytes of each x row
                        umma_f16_ts(d_tmem, a_tmem + kk * 8, (uint64_t)desc_hi << 32 | ((kk < 4 ? b0 : b1) + (kk & 3) * 2), idesc, accumulate);
                        accumulate = 1;
                    }
                    umma_commit(bar_done + 8 * (n & (kUmmaDoneRing - 1)));
                    xo += x_step;
                    if (xo == x_end) xo = 0;
                    if (++sa == (uint32_t)PS) sa = 0;
                }
                umma_commit(bar_dfull + 8 * d);
            }
        }
        __syncwarp();
    } else if (is_dq) {
        // ---------------------------------------------------------------- dequant warps: a set's pass takes an item
        const int q = warp & 3, set = (warp - kPrefillFirstDq) >> 2;
        const int n_col = 32 * q + lane, u = n_col >> 4, g = n_col & 7, h = (n_col >> 3) & 1;
        uint32_t w_rd[4];               // the column's 8 bytes (rows +0..7, +32..39) in the four chunks of a K64 block
#pragma unroll
        for (int t4 = 0; t4 < 4; ++t4) w_rd[t4] = w_ring + (u * 8 + g) * 64 + ((uint32_t)(t4 ^ (g >> 1)) << 4) + 8 * h;
        const uint32_t z_add = flags & kFormatZerosMinusOne;
        const uint32_t a_base = tmem_base + ((uint32_t)(32 * q) << 16) + 2 * acc;
        constexpr uint32_t MAGIC_LO = 0x64006400u;
        // Scales and zero points of the column (SUB of each per item) straight from global memory, one pass ahead.
        const uint8_t *const s_col = a.scales + (16 * u + 2 * g + h) * 2, *const z_col = a.qzeros + 8 * u + g;
        const size_t s_plane = (size_t)a.G * SUB * kItemSBytes, z_plane = (size_t)a.G * SUB * kItemZBytes;
        const uint8_t *s_at = s_col, *z_at = z_col;
        auto sz_seek = [&](int p, int t) {           // to item t of panel p
            const size_t sub = ((size_t)(p * PL) * a.G + g0 + t) * SUB;
            s_at = s_col + sub * kItemSBytes + (PL - 1) * s_plane;
            z_at = z_col + sub * kItemZBytes;
        };
        uint32_t sc_next[SUB] = {}, zb_next[SUB] = {}, zl_next[SUB] = {};
        auto load_sz = [&]() {
#pragma unroll
            for (int e = 0; e < SUB; ++e) {
                sc_next[e] = __ldcg(reinterpret_cast<const unsigned short *>(s_at + e * kItemSBytes));
                zb_next[e] = __ldcg(z_at + e * kItemZBytes);
                if (W8) zl_next[e] = __ldcg(z_at + z_plane + e * kItemZBytes);
            }
        };
        // the set's items: every fourth of the CTA's, across its tiles
        int tile = tile0, t = set, n = set, s = set, sa = set < PS ? set : set - PS;
        uint32_t ph = 0;
        while (t >= G && tile < a.tiles) { t -= G; tile += tile_step; }
        if (tile < a.tiles) {
            sz_seek(tile % panels, t);
            load_sz();
        }
        while (tile < a.tiles) {
            uint32_t s2[SUB], zlo[SUB], zhi[SUB];
#pragma unroll
            for (int e = 0; e < SUB; ++e) {
                s2[e] = sc_next[e] * 0x00010001u;
                zhi[e] = 0;
                const int sh = h ? 4 : 0;
                if constexpr (W8) zlo[e] = ((zb_next[e] >> sh & 15u) << 4 | (zl_next[e] >> sh & 15u)) * 0x00010001u | MAGIC_LO;   // 1024 + z, z < 256
                else zero_constants<BF>((zb_next[e] >> sh & 15u) + z_add, zlo[e], zhi[e]);
            }
            // the next item of this set
            t += kPrefillSets;
            if (t >= G) {
                do {
                    t -= G;
                    tile += tile_step;
                } while (t >= G);
                sz_seek(tile % panels, t);
            } else {
                s_at += kPrefillSets * SUB * kItemSBytes;
                z_at += kPrefillSets * SUB * kItemZBytes;
            }
            if (tile < a.tiles) load_sz();
            if (W8 && n >= WS) wait_done(n - WS);
            decode_wait(bar_wfull + 8 * s, ph, flag);
#pragma unroll 1        // (unrolled, the code of the dequant warps evicts that of the MMA warp from the instruction cache)
            for (int half = 0; half < 2; ++half) {
                const uint32_t wofs = s * kWSlot + half * kUmmaWBlockBytes;
                uint2 wv[4], wl[4];
#pragma unroll
                for (int t4 = 0; t4 < 4; ++t4) wv[t4] = lds64(wofs + w_rd[t4]);
                if constexpr (W8) {
#pragma unroll
                    for (int t4 = 0; t4 < 4; ++t4) wl[t4] = lds64(wofs + kItemWBytes + w_rd[t4]);
                }
                uint32_t r[32];
#pragma unroll
                for (int jj = 0; jj < 2; ++jj)
#pragma unroll
                    for (int t4 = 0; t4 < 4; ++t4) {
                        const int e0 = SUB == 4 ? jj : 0;
                        const uint32_t w = jj ? wv[t4].y : wv[t4].x;       // rows 32 jj + 8 t4 + (0..7), TMEM columns 16 jj + 4 t4 + (0..3)
                        uint32_t o[4];
                        if constexpr (W8) {
                            // bytes 16 hi + lo: nibbles 0, 2, 4, 6 and 1, 3, 5, 7 of both planes; 1024 + byte is an exact
                            // fp16 number, so is q - z; one rounding with the scale
                            const uint32_t l = jj ? wl[t4].y : wl[t4].x;
                            const uint32_t even = (l & 0x0f0f0f0fu) | ((w << 4) & 0xf0f0f0f0u), odd = ((l >> 4) & 0x0f0f0f0fu) | (w & 0xf0f0f0f0u);
                            o[0] = hsub2_u32(prmt(even, MAGIC_LO, 0x7270), zlo[e0]);
                            o[1] = hsub2_u32(prmt(odd, MAGIC_LO, 0x7270), zlo[e0]);
                            o[2] = hsub2_u32(prmt(even, MAGIC_LO, 0x7371), zlo[e0]);
                            o[3] = hsub2_u32(prmt(odd, MAGIC_LO, 0x7371), zlo[e0]);
                        } else {
                            nibble_pairs_minus_zero<BF>(w, zlo[e0], zhi[e0], o);
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) r[16 * jj + 4 * t4 + e] = BF ? bmul2_u32(o[e], s2[e0]) : hmul2_u32(o[e], s2[e0]);
                    }
                if (half == 0 && n >= PS) {
                    wait_done(n - PS);
                    tc_fence_after_sync();
                }
                __syncwarp();
                tmem_st_32x32(a_base + sa * 64 + half * 32, r);
                if constexpr (SUB > 1) {             // the second half's groups
#pragma unroll
                    for (int e = 0; e < SUB / 2; ++e) {
                        s2[e] = s2[SUB / 2 + e];
                        zlo[e] = zlo[SUB / 2 + e];
                        zhi[e] = zhi[SUB / 2 + e];
                    }
                }
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_afull + 8 * (n & (kUmmaDoneRing - 1)));       // (item n - 16 has been multiplied: n - PS has)
            n += kPrefillSets;
            sa += kPrefillSets;
            while (sa >= PS) sa -= PS;
            s += kPrefillSets;
            if (s >= WS) {
                s -= WS;
                ph ^= 1u;
            }
        }
    }
    if constexpr (SPLIT) {
        // ---------------------------------------------------------------- the cluster's partial tiles
        // A CTA owns 128 / S neighbouring columns; the owner adds the CTAs' parts in rank order.
        const bool layout_ok = ((flags & kFormatGateUp) != 0) == (a.fuse != 0) && ((flags & kFormatBf16) != 0) == BF;
        if (!layout_ok && threadIdx.x == 32 * kPrefillFirstEpi) atomicMax(&g_device_status, (int)kStatusLayoutMismatch);
        const int group = is_epi ? 0 : 1 + ((warp - kPrefillFirstDq) >> 2), n_groups = 1 + kPrefillSets;
        const int mt = tile0 / panels, p = tile0 - mt * panels, m0 = mt * tok, W = kPanel / S;
        const int rows = (a.M - m0) < tok ? (a.M - m0) : tok;
        if constexpr (SPLIT == kPushParts) {
            __syncwarp();
            cluster_wait_acquire();
            // Once the dequant warps of all CTAs have read their last weights, the owners' stages and weight rings take the other
            // CTAs' parts, [sender][own column][token] floats, straight from the registers of the threads that read the accumulator;
            // the own part waits in the idle x ring.  A CTA that has all parts needs the others no more.  What bounds it is
            // latency and, for tall tiles, the 16-byte stores.  K = 4096 on 32 panels, bulk copies and two barriers of the cluster
            // -> this, us: 17 rows 8.4 -> 7.6, 64 rows 9.5 -> 8.8, 100 rows 10.4 -> 10.1, 112 rows 10.6 -> 10.5, 128 rows
            // 11.1 -> 11.1, 160 rows 12.3 -> 12.5; K = 11008, 64 rows 13.9 -> 13.1; 64 panels, 50 rows 11.3 -> 10.2; 8-bit weights
            // 17 rows 9.7 -> 9.4, 64 rows 12.3 -> 12.3, 100 rows 13.3 -> 13.6.
            if (is_dq && lane < S) mbar_arrive_release_cluster(map_to_cluster_rank(bar_ready, (uint32_t)lane));
            if (is_dq || is_epi) {
                const int quads = (rows + 3) >> 2, w_shift = S == 4 ? 5 : 6;
                const uint32_t pitch = (uint32_t)(tok + 4) * 4, part = (uint32_t)prefill_part_bytes(tok, S);      // of a column, of a sender
                pdl_wait();
                decode_wait(bar_dfull, 0, flag);
                decode_wait_cluster(bar_ready, 0, flag);
                __syncwarp();
                tc_fence_after_sync();
                const bool ok = layout_ok && lds32(flag) == 0;
                {
                    const int q = warp & 3, n = 32 * q + lane, owner = n >> w_shift, lc = n & (W - 1);
                    const uint32_t dst = map_to_cluster_rank(stg0 + (rank < owner ? rank : rank - 1) * part + lc * pitch, (uint32_t)owner);
                    const uint32_t dbar = map_to_cluster_rank(bar_recv, (uint32_t)owner), own = x_ring + lc * pitch;
#pragma unroll 1
                    for (int c0 = 16 * group; c0 < rows; c0 += 16 * n_groups) {
                        uint32_t r[16];
                        tmem_ld_32x16(tmem_base + ((uint32_t)(32 * q) << 16) + c0, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (c0 + 4 * k >= rows || !ok) break;
                            if (owner == rank) sts128(own + (c0 + 4 * k) * 4, make_uint4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]));
                            else st_async_b32x4(dst + (c0 + 4 * k) * 4, r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3], dbar);
                        }
                        __syncwarp();
                    }
                }
                named_bar_sync(1, 128 * n_groups);                      // the own part is there
                if (ok) decode_wait_cluster(bar_recv, 0, flag);
                if (ok && lds32(flag) == 0) {
                    // a thread takes a column of four rows
                    for (int idx = threadIdx.x - 32 * kPrefillFirstEpi; idx < quads * W; idx += 128 * n_groups) {
                        const int c = idx & (W - 1), m = 4 * (idx >> w_shift);
                        const size_t col = (size_t)p * kPanel + rank * W + c, at = (size_t)(m0 + m) * a.N + col;
                        float v[4] = {};
                        for (int k = 0; k < S; ++k) {
                            const uint4 u = lds128((k == rank ? x_ring : stg0 + (k < rank ? k : k - 1) * part) + c * pitch + m * 4);
                            v[0] += __uint_as_float(u.x);
                            v[1] += __uint_as_float(u.y);
                            v[2] += __uint_as_float(u.z);
                            v[3] += __uint_as_float(u.w);
                        }
                        const float bias = a.bias ? __half2float(a.bias[col]) : 0.f;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (m + e >= rows) break;
                            float f = v[e] + bias;
                            if (a.residual) f += __half2float(a.residual[at + (size_t)e * a.N]);
                            store_out16<BF>(a.y + at + (size_t)e * a.N, f);
                        }
                    }
                }
            }
        } else {
            // After its main loop a CTA's rings are idle: it parks its partial sums there as [owner][token][own column] floats.  Once
            // every CTA has, bulk copies through distributed shared memory bring each owner its part, [sender][token][own column]
            // behind the parked tile.
            const uint32_t part = (uint32_t)(rows * W * 4), park = w_ring, recv = park + (uint32_t)((rows + 31) & ~31) * (kPanel * 4);
            if (is_dq || is_epi) {
                const int q = warp & 3, n = 32 * q + lane, owner = n / W, lc = n - owner * W;
                pdl_wait();
                decode_wait(bar_dfull, 0, flag);
                __syncwarp();
                tc_fence_after_sync();
                const uint32_t at = park + owner * part + (uint32_t)lc * 4u;
#pragma unroll 1
                for (int c0 = 32 * group; c0 < rows; c0 += 32 * n_groups) {
                    uint32_t r[32];
                    tmem_ld_32x32(tmem_base + ((uint32_t)(32 * q) << 16) + c0, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c0 + i < rows) sts_f32(at + (uint32_t)((c0 + i) * W) * 4u, __uint_as_float(r[i]));
                }
                fence_proxy_async();
            }
            __syncwarp();
            cluster_arrive_release();
            cluster_wait_acquire();
            const bool ok = layout_ok && lds32(flag) == 0;
            if (warp == kPrefillXWarp && ok && elect_one()) {
                for (int k = 1; k < S; ++k) {
                    const int to = rank + k < S ? rank + k : rank + k - S;
                    const int slot = rank < to ? rank : rank - 1;              // (nobody sends to itself)
                    bulk_s2s_cluster(map_to_cluster_rank(recv + slot * part, (uint32_t)to), park + to * part, part,
                                     map_to_cluster_rank(bar_recv, (uint32_t)to));
                }
            }
            __syncwarp();
            if ((is_dq || is_epi) && ok) {
                decode_wait_cluster(bar_recv, 0, flag);
                if (lds32(flag) == 0) {
                    const int w4 = W >> 2;
                    for (int idx = threadIdx.x - 32 * kPrefillFirstEpi; idx < rows * w4; idx += 128 * n_groups) {
                        const int m = idx / w4, c = 4 * (idx - m * w4);
                        const size_t col = (size_t)p * kPanel + rank * W + c, at = (size_t)(m0 + m) * a.N + col;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int k = 0; k < S; ++k) {
                            const uint32_t from = k == rank ? park + rank * part : recv + (k < rank ? k : k - 1) * part;
                            const uint4 u = lds128(from + (uint32_t)(m * W + c) * 4u);
                            v.x += __uint_as_float(u.x);
                            v.y += __uint_as_float(u.y);
                            v.z += __uint_as_float(u.z);
                            v.w += __uint_as_float(u.w);
                        }
                        auto add4 = [&](const __half *from) {
                            const uint2 b = *reinterpret_cast<const uint2 *>(from);
                            const float2 b0 = __half22float2(*reinterpret_cast<const __half2 *>(&b.x));
                            const float2 b1 = __half22float2(*reinterpret_cast<const __half2 *>(&b.y));
                            v.x += b0.x, v.y += b0.y, v.z += b1.x, v.w += b1.y;
                        };
                        if (a.bias) add4(a.bias + col);
                        if (a.residual) add4(a.residual + at);
                        *reinterpret_cast<uint2 *>(a.y + at) = make_uint2(pack_out16<BF>(make_float2(v.x, v.y)), pack_out16<BF>(make_float2(v.z, v.w)));
                    }
                }
            }
            // no CTA may leave while its parked sums are being read; what it sent has landed once all have received
            __syncwarp();
            cluster_arrive_release();
            cluster_wait_acquire();
        }
    } else if (is_dq || is_epi) {
        // ---------------------------------------------------------------- epilogue
        // A warp reads its 32 lanes (columns of y) x 32 tokens as 8 x 8 fragments, rounds them and transposes them with
        // stmatrix into rows of 64 bytes in shared memory (16-byte chunks swizzled over pairs of rows), to be stored 16 bytes
        // per lane.  A residual takes the way back through the same rows (ldmatrix) and joins the fp32 sum.
        // The CTA's last tile, which nothing runs over any more, is shared out over the epilogue and the dequant warps, 32
        // tokens at a time.
        const bool layout_ok = ((flags & kFormatGateUp) != 0) == (a.fuse != 0) && ((flags & kFormatBf16) != 0) == BF;
        if (!layout_ok && threadIdx.x == 32 * kPrefillFirstEpi) atomicMax(&g_device_status, (int)kStatusLayoutMismatch);
        const int group = is_epi ? 0 : 1 + ((warp - kPrefillFirstDq) >> 2), n_groups = 1 + kPrefillSets;
        const int q = warp & 3;
        // (the ring is idle by then; with the gate/up epilogue a gate warp has the room of its up warp too)
        const uint32_t stg = (is_epi ? stg0 : w_ring + (group - 1) * kPrefillStage) + (a.fuse ? (q & 1) * 4096 : q * (32 * 64));
        const uint32_t mrow = lane & 7, mchunk = lane >> 3;       // row and chunk that this lane addresses in a fragment store
        const uint32_t frag = stg + mrow * 64 + ((mchunk ^ (mrow >> 1)) << 4);          // token block i: + 512 i
        const uint32_t prow = lane >> 2, pchunk = lane & 3;       // row (+ 8 t) and chunk of its 16-byte pieces
        const uint32_t piece = stg + prow * 64 + ((pchunk ^ (prow >> 1)) << 4);
        const bool has_bias = a.bias != nullptr, has_res = a.residual != nullptr;
        pdl_wait();
        const int my_tiles = (a.tiles - tile0 + tile_step - 1) / tile_step;
        for (int it = is_epi ? 0 : my_tiles - 1; it < my_tiles; ++it) {
            const bool last = it == my_tiles - 1;
            const int tile = tile0 + it * tile_step, d = it & 1;
            const uint32_t ph = (uint32_t)(it >> 1) & 1u;
            const int mt = tile / panels, p = tile - mt * panels, m0 = mt * tok;
            const int rows = (a.M - m0) < tok ? (a.M - m0) : tok;
            float bv[4] = {};                        // columns lane / 4 + 8 j of the warp's 32
            if (has_bias) {
#pragma unroll
                for (int j = 0; j < 4; ++j) bv[j] = __half2float(a.bias[(size_t)p * kPanel + 32 * q + 8 * j + (lane >> 2)]);
            }
            decode_wait(bar_dfull + 8 * d, ph, flag);        // (unambiguous for the dequant warps too: kPrefillMinItems)
            __syncwarp();
            tc_fence_after_sync();
            const bool ok = layout_ok && lds32(flag) == 0;
            const uint32_t src = tmem_base + ((uint32_t)(32 * q) << 16) + d * acc;
            const size_t y_at = (size_t)(m0 + prow) * a.N + (size_t)p * kPanel + 32 * q + 8 * pchunk;
#pragma unroll 1
            for (int c0 = last ? 32 * group : 0; c0 < rows; c0 += last ? 32 * n_groups : 32) {
                uint32_t r0[16], r1[16];             // lanes 0..15 and 16..31 (columns behind the tile's: read, not looked at)
                tmem_ld_16x256b_x4(src + c0, r0);
                tmem_ld_16x256b_x4(src + (16u << 16) + c0, r1);
                const int nr = rows - c0;
                if (has_res) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (prow + 8 * t < nr) sts128(piece + 512 * t, *reinterpret_cast<const uint4 *>(a.residual + y_at + (size_t)(c0 + 8 * t) * a.N));
                    __syncwarp();
                }
                tmem_wait_ld();
                if (a.fuse) {
                    // The up warps hand their fp32 sums to the gate warps, which hold the same fragments 64 columns lower:
                    // [value][lane] words in the gate warp's part of the stage.
                    const uint32_t at = stg + lane * 4;
                    if (q >= 2) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) sts_f32(at + e * 128, __uint_as_float(r0[e]));
#pragma unroll
                        for (int e = 0; e < 16; ++e) sts_f32(at + 2048 + e * 128, __uint_as_float(r1[e]));
                    }
                    named_bar_sync(1 + group, 128);
                    if (q < 2) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) r0[e] = __float_as_uint(silu_mul(__uint_as_float(r0[e]), lds_f32(at + e * 128)));
#pragma unroll
                        for (int e = 0; e < 16; ++e) r1[e] = __float_as_uint(silu_mul(__uint_as_float(r1[e]), lds_f32(at + 2048 + e * 128)));
                        __syncwarp();
                    }
                }
                if (!a.fuse || q < 2) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float2 v[4];                 // tokens 8 i + 2 (lane % 4) + (0, 1); columns lane / 4 + 8 j
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            v[e] = make_float2(__uint_as_float(r0[4 * i + 2 * e]), __uint_as_float(r0[4 * i + 2 * e + 1]));
                            v[2 + e] = make_float2(__uint_as_float(r1[4 * i + 2 * e]), __uint_as_float(r1[4 * i + 2 * e + 1]));
                        }
                        if (has_bias) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) v[j].x += bv[j], v[j].y += bv[j];
                        }
                        if (has_res) {
                            uint32_t rr[4];
                            ldmatrix_x4_trans(frag + 512 * i, rr);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&rr[j]));
                                v[j].x += f.x, v[j].y += f.y;
                            }
                            __syncwarp();
                        }
                        uint32_t o[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) o[j] = pack_out16<BF>(v[j]);
                        stmatrix_x4_trans(frag + 512 * i, o);
                    }
                    __syncwarp();
                }
                if (!a.fuse) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (ok && (int)prow + 8 * t < nr) *reinterpret_cast<uint4 *>(a.y + y_at + (size_t)(c0 + 8 * t) * a.N) = lds128(piece + 512 * t);
                    __syncwarp();
                } else {
                    if (q < 2 && ok) {
                        const int oc = p * 64 + 32 * q + 8 * pchunk;
#pragma unroll 1
                        for (int t = 0; t < 4; ++t) {
                            if ((int)prow + 8 * t >= nr) break;
                            const uint4 ov = lds128(piece + 512 * t);
                            __half *orow = a.y + (size_t)(m0 + c0 + prow + 8 * t) * (a.N / 2);
                            if (a.out_index == nullptr) {
                                *reinterpret_cast<uint4 *>(orow + oc) = ov;
                            } else {
                                // scattered columns: eight destinations (two 16-byte index loads), eight 2-byte stores
                                const int4 ia = *reinterpret_cast<const int4 *>(a.out_index + oc);
                                const int4 ib = *reinterpret_cast<const int4 *>(a.out_index + oc + 4);
                                const int dst[8] = {ia.x, ia.y, ia.z, ia.w, ib.x, ib.y, ib.z, ib.w};
                                const uint32_t ow[4] = {ov.x, ov.y, ov.z, ov.w};
#pragma unroll
                                for (int e = 0; e < 8; ++e)
                                    orow[dst[e]] = __ushort_as_half((unsigned short)(ow[e >> 1] >> (16 * (e & 1))));
                            }
                        }
                    }
                    named_bar_sync(1 + group, 128);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (!last && lane == 0) mbar_arrive(bar_dempty + 8 * d);
        }
        if (threadIdx.x == 32 * kPrefillFirstEpi) GPTQ_TRACE_MAX(a.trace_slot, last_exit);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (lds32(flag) != 0) {
        // A wait gave up: leave time for the copies in flight to land.
        const uint64_t start = global_timer_ns();
        while (global_timer_ns() - start < 200000ull) { }
        __syncthreads();
        if (SPLIT == kPushParts) {        // ... and stay until the other CTAs of the cluster have left or come here too: they may still send
            cluster_arrive_release();
            cluster_wait_acquire();
        }
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

struct PrefillPlan {
    bool use;
    int S, tok, tiles, ctas, x_slots, smem_bytes;
};

// Token rows per tile and CTAs per tile with the smallest number of clocks: waves of tiles x items x the slower of the MMA
// (4 clocks per token row) and what an item costs at any size (dequantisation and the MMA thread), plus a part per wave; of
// equals the larger tile, which dequantises less.  A split of K over clusters of two or four CTAs (one tile per cluster) costs
// about 6000 clocks for the exchange; it wins where tiles are few: K = 11008, 32 panels, M = 100 15.6 us against 19.7 on the
// kernel of gptq_umma.cuh and 27 without a split.
//
// The kernel is used unless that one is estimated faster: it splits K finer and puts several CTAs on an SM.  Its planner's
// estimate is scaled to clocks by what was measured per kernel variant (K = 2048 to 11008, 8 to 216 panels).  Both sides, us,
// this kernel without a split: K = 11008, M = 64: 64 panels 27.2 here, 24.2 there; 80 panels 28.5 / 38.7.  K = 4096, M = 64:
// 32 panels 10.6 / 9.5, 40 panels 10.8 / 11.6.  K = 4096, M = 256: 16 panels 13.6 / 15.6.  M = 16 (the mma.sync kernel's) on
// 96 panels 11.4 / 11.1, on 32 panels 10.0 / 5.8.
inline PrefillPlan plan_prefill(int M, int N, int K, int group_size, int sm_count, bool w8, bool may_split)
{
    PrefillPlan pl{};
    const int panels = N / kPanel, G = K / kGroup;
    if (G < kPrefillMinItems) return pl;     // (a condition of correctness, see there)
    long long best = -1, best_waves = 0;
    for (int S = 1; S <= (may_split ? 4 : 1); S *= 2) {
        for (int most = kPrefillMaxTok; most >= 32; most -= 16) {
            const int t = (M + most - 1) / most;
            const int tok = ((M + t - 1) / t + 15) & ~15;
            const long long tiles = (long long)panels * t, waves = S > 1 ? 1 : (tiles + sm_count - 1) / sm_count;
            if (tiles >= (1 << 30) || (S > 1 && tiles > decode_max_clusters(S, sm_count))) continue;
            const int any = w8 ? (tok > 128 ? 800 : 670) : 520, mma = 4 * tok + 60;
            const long long clocks = waves * ((long long)((G + S - 1) / S) * (mma > any ? mma : any) + 1500) + 900 + (S > 1 ? 6000 : 0);
            if (best < 0 || clocks < best) {
                best = clocks;
                best_waves = waves;
                pl.S = S;
                pl.tok = tok;
                pl.tiles = (int)tiles;
            }
        }
    }
    if (best < 0) return pl;
    const UmmaPlan split = plan_umma(M, N, K, sm_count, w8);
    const int percent = (split.tok <= 64 ? 100 : split.tok == 128 ? 117 : 150) * (w8 ? (split.tok <= 128 ? 18 : 13) : 10) / 10;
    if (split.one_wave && 6500 + split.estimate * 243 * percent / 1000 < best) return pl;
    // Groups of 32 rows cost this kernel about 0.25 us per item beside the MMA, which tiles of 256 rows pay half as often.  Both
    // kernels' times in us, fitted to 208 problems of 150 rows and more (K = 1408 to 13824, N = 2048 to 27648): the choice is
    // 0.6 % off the better one on average, this kernel always 3.8 %.  There / here: 13824 x 27648, 200 rows 155 / 237, 1000 rows
    // 676 / 802; 11008 x 4096, 900 rows 71 / 86; 4096 x 4096, 900 rows 27 / 31; 5120 x 15360, 320 rows 62 / 41.
    if (group_size == 32 && !w8 && may_split && split.tok == 256) {
        const int tail = split.tail_tiles > 0, waves = (split.ctas + sm_count - 1) / sm_count + tail;
        const int items = split.S > 1 ? (G + split.S - 1) / split.S : (waves - tail) * G + (tail ? (G + split.tail_S - 1) / split.tail_S : 0);
        const double there = 0.85 * items + 4.5 * waves - 5.3 + (split.S > 1 || tail ? 6.5 : 0);
        const double here = (double)best_waves * (((G + pl.S - 1) / pl.S) * (0.00208 * pl.tok + 0.25) + 0.45) - 1.2 + (pl.S > 1 ? 5.7 : 0);
        if (1.05 * there < here) return pl;
    }
    pl.use = true;
    pl.ctas = pl.S > 1 ? pl.tiles * pl.S : pl.tiles < sm_count ? pl.tiles : sm_count;
    pl.x_slots = prefill_x_slots(pl.tok, w8);
    pl.smem_bytes = 2048 + prefill_ring_bytes(pl.tok, w8) + pl.x_slots * pl.tok * 256;
    const int floor_one_per_sm = (227 * 1024) / 2 + 512;                 // the CTA owns all tensor memory
    if (pl.smem_bytes < floor_one_per_sm) pl.smem_bytes = floor_one_per_sm;
    return pl;
}

template <int SUB, bool BF, bool W8, int SPLIT>
static int launch_prefill_split(const PrefillArgs &args, const CUtensorMap &w_map, const CUtensorMap &x_map, const PrefillPlan &plan,
                              cudaStream_t s)
{
    static int configured_smem[64] = {};
    const int cfg_st = ensure_dynamic_smem((const void *)prefill_kernel<SUB, BF, W8, SPLIT>, configured_smem, plan.smem_bytes);
    if (cfg_st) return cfg_st;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)plan.ctas);
    cfg.blockDim = dim3(kPrefillThreads);
    cfg.dynamicSmemBytes = (size_t)plan.smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)args.S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SPLIT ? 2 : 1;        // (a launch with clusters of one took 0.4 us longer)
    return record_cuda_error(cudaLaunchKernelEx(&cfg, prefill_kernel<SUB, BF, W8, SPLIT>, args, w_map, x_map));
}

template <int SUB, bool BF, bool W8>
static int launch_prefill_sub(const PrefillArgs &args, const CUtensorMap &w_map, const CUtensorMap &x_map, const PrefillPlan &plan,
                              cudaStream_t s)
{
    // (a template: with the number of CTAs per tile known only at run time, launches without a split were 7 % slower; with both
    // kinds of exchange in one kernel registers spilled)
    if (plan.S == 1) return launch_prefill_split<SUB, BF, W8, 0>(args, w_map, x_map, plan, s);
    return plan.tok <= prefill_push_rows(W8) ? launch_prefill_split<SUB, BF, W8, kPushParts>(args, w_map, x_map, plan, s)
                                             : launch_prefill_split<SUB, BF, W8, kParkParts>(args, w_map, x_map, plan, s);
}

int launch_prefill(const __half *x, const void *qweight, const void *qzeros, const void *scales, __half *y, int M, int N, int K,
                   int group_size, const PrefillPlan &plan, int fuse, const __half *bias, const __half *residual,
                   const int32_t *out_index, int bf16, int w8, cudaStream_t s)
{
    PrefillArgs args;
    args.scales = (const uint8_t *)scales;
    args.qzeros = (const uint8_t *)qzeros;
    args.y = y;
    args.M = M;
    args.N = N;
    args.G = K / kGroup;
    args.S = plan.S;
    args.tok = plan.tok;
    args.tiles = plan.tiles;
    args.x_slots = plan.x_slots;
    args.trailer = reinterpret_cast<const TiledTrailer *>((const uint8_t *)qzeros + tiled_zero_bytes(N, w8 ? 2 * K : K, group_size));
    args.fuse = fuse;
    args.bias = bias;
    args.residual = residual;
    args.trace_slot = next_trace_slot();
    args.out_index = out_index;
    CUtensorMap w_map, x_map;
    int st = make_tensor_map_2d(&w_map, CU_TENSOR_MAP_DATA_TYPE_UINT32, qweight, 16, (uint64_t)K * N * (w8 ? 2 : 1) / 2 / 64, 64, 16, 128,
                                CU_TENSOR_MAP_SWIZZLE_64B);
    if (st) return st;
    st = make_tensor_map_ktiles(&x_map, x, (uint64_t)K, (uint64_t)M, (uint32_t)plan.tok, 2);
    if (st) return st;
    switch (kGroup / group_size + (w8 ? 20 : bf16 ? 10 : 0)) {
    case 1: return launch_prefill_sub<1, false, false>(args, w_map, x_map, plan, s);
    case 2: return launch_prefill_sub<2, false, false>(args, w_map, x_map, plan, s);
    case 4: return launch_prefill_sub<4, false, false>(args, w_map, x_map, plan, s);
    case 11: return launch_prefill_sub<1, true, false>(args, w_map, x_map, plan, s);
    case 12: return launch_prefill_sub<2, true, false>(args, w_map, x_map, plan, s);
    case 14: return launch_prefill_sub<4, true, false>(args, w_map, x_map, plan, s);
    case 21: return launch_prefill_sub<1, false, true>(args, w_map, x_map, plan, s);
    case 22: return launch_prefill_sub<2, false, true>(args, w_map, x_map, plan, s);
    case 24: return launch_prefill_sub<4, false, true>(args, w_map, x_map, plan, s);
    default: return GPTQ_ERR_UNSUPPORTED;
    }
}

}  // namespace gptq

// GPTQ matmul for few token rows (fp16): HBM-bound streaming on byte-wide tcgen05 operands, one CTA per SM and launch.
//
// Swap-AB as in gptq_umma.cuh: the 128 columns of a panel are the MMA's 128 rows (TMEM lanes), the token rows its N.  The
// unit of work is an item (panel, 128 K rows); the S CTAs of a cluster share panels along K and a cluster works through
// panels cl, cl + clusters, ... without leaving the kernel, so one launch is one CTA per SM whatever the layer's size.
//
// Operands.  A packed nibble IS an e4m3 number: the bytes 0x00 .. 0x0f read as e4m3 are q * 2^-9, so `w & 0x0f0f0f0f` and
// `(w >> 4) & 0x0f0f0f0f` are A operands of tcgen05.mma kind::f8f6f4 - three instructions per eight weights where q - z as
// fp16 takes nine (and twice the tensor memory).  The activations are split without error into four e5m2 pieces: the upper
// byte of an fp16 number is its e5m2 truncation p0, (x - p0) * 8 is again an fp16 number, and after four steps nothing is
// left: x = p0 + p1 / 8 + p2 / 64 + p3 / 512.  Two tokens are eight rows of the B operand.  Products and sums are exact to fp32
// (measured: 8e-8 of the sum of magnitudes).  An infinity or NaN in x makes every sum of its row NaN: such outputs are formed at
// the end, from those activations alone.  Every quantisation group has an accumulator of its
// own; the drain warps recombine the pieces, subtract z * sum(x) and apply the scale in fp32.
//
// Warp roles, each with its own pace:
//   weights   tensor-map loads of packed weights (8 KB per item) into a ring, bulk copies of scales and zero points for
//             several items; depends on nothing and so runs ahead into the previous launch's time
//   MMA       the MMAs and one commit per step (two items where tensor memory has room)
//   dequant   two sets of four warps, alternate steps: packed words -> bytes -> tcgen05.st into an A stage per set.  When
//             both stages are full and x exists, all eight split it, once per launch, into B tiles that hold the CTA's K range
//   drain     four warps: accumulators -> registers, and at a panel's end st.async to the columns' owners in the cluster
//   finish    one warp: sums the cluster's slices in rank order, epilogue, store y - while the others are in the next panel
//
// What bounds it: between the weights' arrival and the MMA a step passes several hands, and a warp issues an instruction
// every five to seven clocks (an SM holds one or two warps of a role per scheduler), so instructions per step and hand-overs
// set the pace: 250-300 clocks per item and CTA, where the 8.5 KB of an item take 370 at the HBM rate if all SMs stream.  A
// dequant warp needs 115 clocks per item of ALU time alone (half-rate pipe).  The rest is the launch boundary: the first MMA
// runs 1.3 us after the previous launch has ended (x from L2, its split), the cluster exchange takes about 1 us.
//
// A CTA takes at most half of an SM's shared memory and tensor memory: the next launch's CTAs become resident beside it
// (programmatic dependent launch), fill their weight rings and their A stages before x exists, which keeps HBM busy across
// the launch boundary - once this launch has asked for all of its own weights: with the dependents released at the start the
// next launch's prefetch queued in front of this one's loads (4096 x 22016 at M = 1: 15.1 instead of 12.2 us).
//
// Measured at M = 1 in a chain of launches on distinct weights, against the mma.sync kernel: 4096 x 4096 3.95 / 4.6 us,
// 4096 x 12288 7.4 / 8.3, 11008 x 4096 7.7 / 8.3, 4096 x 22016 11.4 / 12.8 (4.1 TB/s), 5120 x 27648 15.2 / 17.1 (4.8 TB/s).
#pragma once
#include "gptq_umma.cuh"

namespace gptq {

constexpr int kDecodeDequantWarps = 8, kDecodeDrainWarps = 4;
constexpr int kDecodeFirstDq = 2;                                              // warp 0: weights, warp 1: MMA + TMEM
constexpr int kDecodeFirstDrain = kDecodeFirstDq + kDecodeDequantWarps;        // 10
constexpr int kDecodeFinishWarp = kDecodeFirstDrain + kDecodeDrainWarps;       // 14
// Steps still to be requested when the next launch may start.  7B layer of four matmuls in a chain, M = 1 / 2, us: 1 28.7 / 29.5,
// 3 27.6 / 28.5, 5 26.4 / 27.7; from the start of the launch on 37.7 (M = 1).
constexpr int kDecodeLead = 5;
constexpr int kDecodeThreads = 32 * (kDecodeFinishWarp + 1);
constexpr int kDecodeMetaBufs = 3;
constexpr int kDecodeMetaItems = 8;          // items (of SUB = 1) whose scales and zero points travel together
constexpr int kDecodeMetaBytes = kDecodeMetaItems * (kItemSBytes + kItemZBytes);
constexpr int kDecodeMaxWSlots = 16, kDecodeMaxItems = 32;       // of a CTA: its weight ring, its K range
constexpr int kDecodeMaxXPasses = 16;
constexpr uint32_t kDecodeCols = 256;        // tensor-memory columns of a CTA: two launches share the SM's 512
constexpr int kDecodeACols = 32;             // of an item's A operand

struct DecodeArgs {
    const uint8_t *qweight, *scales, *qzeros;   // tiled
    const __half *x;                  // [M, K]
    __half *y;
    int M, N, G;
    int S, clusters;                // CTAs per panel; clusters in the grid
    int w_slots;                    // weight ring (steps)
    int x_tiles;                    // B tiles: items of the widest K range
    uint32_t m_inverse;             // 2^16 / M, rounded up: u / M = u * m_inverse >> 16 for u < 2^10
    const TiledTrailer *trailer;
    int fuse;
    const __half *bias, *residual;
    int trace_slot;
    const int32_t *out_index;
    unsigned long long slice_lo;    // column slices of the owners, as in SplitKArgs
    int slice_max;
};

constexpr int kDecodeMaxRows = 2;            // token rows of a tile: eight B rows
// MMA N (the eight B rows are read as sixteen: the accumulator columns of the rows behind them are never looked at),
// accumulator columns of an item, items per step (two A stages, and two accumulators at least), and accumulators in 256
// columns.
constexpr int kDecodeN = 16;
__host__ __device__ constexpr int decode_d_cols(int SUB) { return SUB * kDecodeN; }
__host__ __device__ constexpr int decode_step_items(int SUB)
{
    return 4 * (kDecodeACols + decode_d_cols(SUB)) <= (int)kDecodeCols ? 2 : 1;
}
__host__ __device__ constexpr int decode_d_stages(int SUB)
{
    const int p = decode_step_items(SUB);
    return ((int)kDecodeCols - 2 * p * kDecodeACols) / (p * decode_d_cols(SUB)) >= 4 ? 4 : 2;
}
constexpr int kDecodeXTile = kDecodeMaxRows * 512;      // bytes of an item's B tile
__host__ __device__ constexpr int decode_sum_bytes(int SUB, int items) { return (items * SUB * kDecodeMaxRows * 4 + 127) & ~127; }

__host__ __device__ inline int decode_recv_bytes(int M, int fuse, int S, int slice_max)      // of one of the two buffers
{
    return (S * (fuse ? 2 : 1) * slice_max * M * 4 + 127) & ~127;
}

__device__ __forceinline__ void st_async_f32x2(uint32_t addr, float2 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void umma_f8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// kind::f8f6f4, A e4m3, B e5m2, both K-major, fp32 accumulator (K = 32)
__host__ __device__ constexpr uint32_t umma_idesc_e4m3_e5m2(int M, int N) { return umma_idesc_f16(M, N) | (1u << 10); }
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ uint4 ldg128_cg(const void *p)
{
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// two fp32 lanes in a 64-bit register
__device__ __forceinline__ uint64_t pack_f32x2(uint32_t lo, uint32_t hi)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
    return v;
}
__device__ __forceinline__ float2 unpack_f32x2(uint64_t v)
{
    uint32_t lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
    return make_float2(__uint_as_float(lo), __uint_as_float(hi));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t lds_f32x2(uint32_t addr)
{
    uint64_t v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
// Bits of the CTA's flag word
constexpr uint32_t kDecodeGaveUp = 1u;      // a wait gave up
constexpr uint32_t kDecodeNotFinite = 2u;   // outputs whose sum is NaN have not been stored yet
__device__ __forceinline__ void raise_flag(uint32_t flag, uint32_t bits)
{
    asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(flag), "r"(bits) : "memory");
}
// A wait without a result.  One that gives up raises the CTA's flag, and from then on no wait of the CTA waits: everything
// runs through on whatever data there is, the status word tells the host, and the CTA leaves after a pause that covers
// its copies in flight.
__device__ __noinline__ void decode_wait_slow(uint32_t bar, uint32_t parity, uint32_t flag)
{
    for (int it = 0; it < kWaitTries; ++it)
        if (mbar_try_wait(bar, parity)) return;
    const uint64_t start = global_timer_ns();
    while ((lds32(flag) & kDecodeGaveUp) == 0) {
        if (mbar_try_wait(bar, parity)) return;
        if (global_timer_ns() - start > kWaitLimitNs) {
            raise_flag(flag, kDecodeGaveUp);
            atomicMax(&g_device_status, (int)kStatusWaitTimeout);
        }
    }
}
__device__ __forceinline__ void decode_wait(uint32_t bar, uint32_t parity, uint32_t flag)
{
    if (!mbar_try_wait(bar, parity)) decode_wait_slow(bar, parity, flag);
}
// the same, observing arrivals and stores from other CTAs of the cluster
__device__ __noinline__ void decode_wait_cluster(uint32_t bar, uint32_t parity, uint32_t flag)
{
    for (int it = 0; it < kWaitTries; ++it)
        if (mbar_try_wait_cluster(bar, parity)) return;
    const uint64_t start = global_timer_ns();
    while ((lds32(flag) & kDecodeGaveUp) == 0) {
        if (mbar_try_wait_cluster(bar, parity)) return;
        if (global_timer_ns() - start > kWaitLimitNs) {
            raise_flag(flag, kDecodeGaveUp);
            atomicMax(&g_device_status, (int)kStatusWaitTimeout);
        }
    }
}
// The eight activations of `v` (k = 8 kc .. 8 kc + 7 of an item, one token) split into pieces and stored in the swizzled B
// tile at `tile`: piece p of token t is row 8 (t / 2) + 2 p + t % 2, bytes in the order of the weights' nibbles (K rows 0, 4,
// 1, 5 and 2, 6, 3, 7).
__device__ __forceinline__ void decode_store_pieces(uint32_t tile, int token, int kc, uint4 v)
{
    uint32_t r[4] = {v.x, v.y, v.z, v.w};
    const uint32_t rows = tile + (token >> 1) * 1024 + (token & 1) * 128 + (kc & 1) * 8, c16 = (uint32_t)(kc >> 1) ^ (token & 1);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        uint32_t b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            b[i] = r[i] & 0xff00ff00u;
            if (p < 3) r[i] = hmul2_u32(hsub2_u32(r[i], b[i]), 0x48004800u);      // (x - piece) * 8, exact
        }
        sts64(rows + p * 256 + ((c16 ^ (2 * p)) << 4), prmt(b[0], b[2], 0x7351), prmt(b[1], b[3], 0x7351));
    }
}

__device__ __forceinline__ void tmem_ld_8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// nonzero if one of the two fp16 numbers is an infinity or NaN
__device__ __forceinline__ uint32_t half2_not_finite(uint32_t v) { return ((v & 0x7c007c00u) + 0x04000400u) & 0x80008000u; }

// Sum of token m and tiled column n as the mma.sync kernel forms it, s * sum((q - z) x) per quantisation group, for outputs
// that come out as NaN.  Unless `all`, only what decides about them is looked at: infinities and NaNs of x, and groups whose
// scale is one; `met` is set if there are any (what the rest would add is finite).
template <int SUB>
__device__ __forceinline__ float decode_sum_not_finite(const DecodeArgs &a, int m, int n, uint32_t z_plus, bool all, bool &met)
{
    constexpr int kRows = kGroup / SUB;
    const __half *const x = a.x + (size_t)m * a.G * kGroup;
    float run = 0.f;
#pragma unroll 1
    for (int group = 0; group < a.G * SUB; ++group) {
        const float s = __half2float(__ldcg(reinterpret_cast<const __half *>(a.scales) + repacked_scale_index(group, n, a.G * SUB)));
        const bool whole = all || !(fabsf(s) <= 65504.f);
        uint32_t found = whole;
#pragma unroll 1
        for (int j = 0; j < kRows / 8; ++j) {
            const uint4 v = ldg128_cg(x + group * kRows + 8 * j);
            found |= half2_not_finite(v.x) | half2_not_finite(v.y) | half2_not_finite(v.z) | half2_not_finite(v.w);
        }
        if (!found) continue;
        met = true;
        int hi, slot;
        const uint32_t zb = __ldcg(a.qzeros + repacked_zero_byte(group, n, a.G * SUB, &hi));
        const float z = (float)((hi ? zb >> 4 : zb & 15u) + z_plus);
        float v = 0.f;
#pragma unroll 1
        for (int i = group * kRows; i < (group + 1) * kRows; ++i) {
            const float xi = __half2float(__ldcg(x + i));
            if (!whole && fabsf(xi) <= 65504.f) continue;
            const size_t at = repacked_word_offset(i, n, a.G, &slot);
            v += ((float)(__ldcg(reinterpret_cast<const uint32_t *>(a.qweight + at)) >> (4 * slot) & 15u) - z) * xi;
        }
        run += s * v;
    }
    return run;
}
// The outputs of the panels cl, cl + clusters, ... and own columns [lo, lo + hw) of a run whose sum is NaN (the finish warp has
// not stored them): an infinity or NaN in x, or a scale that is one.  A call that works out everything again: values kept for
// it in registers, or a branch to it in the finish warp's loop, made every launch slower (M = 1 2 %, M = 2 5 to 20 %).
template <int SUB>
__device__ __noinline__ void decode_store_not_finite(const DecodeArgs &a)
{
    pdl_wait();                                 // (x is read: long since through)
    const uint32_t z_plus = a.trailer->flags & kFormatZerosMinusOne;
    const int S = a.S, cl = blockIdx.x / S, rank = blockIdx.x - cl * S, n_panels = (a.N / kPanel - cl + a.clusters - 1) / a.clusters;
    const int lo = (int)((a.slice_lo >> (8 * rank)) & 255);
    const int hw = (rank + 1 < S ? (int)((a.slice_lo >> (8 * (rank + 1))) & 255) : a.fuse ? 64 : kPanel) - lo;
#pragma unroll 1
    for (int idx = threadIdx.x; idx < n_panels * a.M * hw; idx += kDecodeThreads) {
        const int pi = idx / (a.M * hw), rest = idx - pi * a.M * hw, m = rest / hw, c = lo + rest - m * hw;
        const int p = cl + pi * a.clusters, n = p * kPanel + c;
        bool met = false, met_up = false, all = false;
        float v = 0.f, up = 0.f;
#pragma unroll 1
        for (int k = 0; k < (a.fuse ? 4 : 1); ++k) {        // sum of the column, of the matching up column; whatever of the two has been left out
            if (k >= 2 && !all) break;
            bool &seen = k & 1 ? met_up : met;
            if (k >= 2 && seen) continue;
            const float f = decode_sum_not_finite<SUB>(a, m, n + 64 * (k & 1), z_plus, all, seen);
            if (k & 1) up = f;
            else v = f;
            if (k == 1) all = met || met_up;
        }
        if (!met && !met_up) continue;
        if (!a.fuse) {
            if (a.bias) v += __half2float(a.bias[n]);
            __half *const y = a.y + (size_t)m * a.N + n;
            if (a.residual) v += __half2float(a.residual[(size_t)m * a.N + n]);
            *y = __float2half_rn(v);
        } else {
            const int oc = p * 64 + c;
            a.y[(size_t)m * (a.N / 2) + (a.out_index ? a.out_index[oc] : oc)] = __float2half_rn(silu_mul(v, up));
        }
    }
}

// SUB: quantisation groups per item
template <int SUB>
__global__ void __launch_bounds__(kDecodeThreads, 2)
decode_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ CUtensorMap w_map)
{
    extern __shared__ uint8_t smem_raw[];
    constexpr int P = decode_step_items(SUB);                 // items per step
    constexpr int ND = decode_d_stages(SUB);              // accumulators (A stages: two, one per dequant set)
    constexpr int kN = kDecodeN, kDCols = decode_d_cols(SUB);      // columns per item
    constexpr int kWSlot = P * kItemWBytes, kXTile = kDecodeXTile, NX = kDecodeMaxRows;
    static_assert(P * (2 * kDecodeACols + ND * kDCols) <= (int)kDecodeCols, "tensor memory");
    constexpr int MC = kDecodeMetaItems / SUB;                // items per metadata chunk (whole steps)
    constexpr uint32_t kOffZ = kDecodeMetaItems * kItemSBytes;

    const uint32_t flags = __ldg(&a.trailer->flags);          // needed late: requested first
    if (threadIdx.x == 0) {
        GPTQ_TRACE_MIN(a.trace_slot, first_entry);
        GPTQ_TRACE_MAX(a.trace_slot, last_entry);
        if (blockIdx.x == 0) {
            GPTQ_TRACE_SET(a.trace_slot, kernel_and_ctas, (2ull << 32) | gridDim.x);
        }
    }
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar_wfull = base, bar_wempty = base + 128, bar_xfull = base + 256;
    const uint32_t bar_afull = base + 512, bar_done = base + 528, bar_drained = base + 560, bar_mfull = base + 592;
    const uint32_t bar_mempty = base + 624, bar_recv = base + 656, bar_free = base + 672, tmem_slot = base + 688, flag = base + 692;
    const uint32_t wring = base + 1024;
    const int NW = a.w_slots;
    const uint32_t xtiles = wring + NW * kWSlot;
    const uint32_t meta = xtiles + a.x_tiles * kXTile;
    const uint32_t sums = meta + kDecodeMetaBufs * kDecodeMetaBytes;
    const uint32_t recv = sums + decode_sum_bytes(SUB, a.x_tiles);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int S = a.S, cl = blockIdx.x / S, rank = blockIdx.x - cl * S;
    const int panels = a.N / kPanel;
    const int g0 = rank * a.G / S, ng = (rank + 1) * a.G / S - g0;      // this CTA's items of a panel
    const int n_panels = (panels - cl + a.clusters - 1) / a.clusters;
    const int spp = (ng + P - 1) / P;                                   // steps per panel (a step lies in one panel)
    const int hsh = a.fuse ? 6 : 7, runs = a.fuse ? 2 : 1;              // `runs` runs of 2^hsh columns
    const int lo = (int)((a.slice_lo >> (8 * rank)) & 255);             // own columns of a run: [lo, lo + hw)
    const int hw = (rank + 1 < S ? (int)((a.slice_lo >> (8 * (rank + 1))) & 255) : (1 << hsh)) - lo;
    const int wide = runs * a.slice_max;
    const uint32_t recv_tx = (uint32_t)(S * runs * hw * a.M * 4);
    const uint32_t recv_bytes = (uint32_t)decode_recv_bytes(a.M, a.fuse, S, a.slice_max);
    // the split of x goes in passes of 16 units (a unit: the 128 k of an item for one token, half a warp)
    constexpr int kUnits = kDecodeDequantWarps * 2;
    const int x_units = ng * a.M, x_passes = (x_units + kUnits - 1) / kUnits;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NW; ++s) {
            mbar_init(bar_wfull + 8 * s, 1);
            mbar_init(bar_wempty + 8 * s, 4);
        }
        for (int s = 0; s < x_passes; ++s) mbar_init(bar_xfull + 8 * s, kDecodeDequantWarps);
        for (int s = 0; s < 2; ++s) mbar_init(bar_afull + 8 * s, 4);
        for (int s = 0; s < ND; ++s) {
            mbar_init(bar_done + 8 * s, 1);
            mbar_init(bar_drained + 8 * s, kDecodeDrainWarps);
        }
        for (int s = 0; s < kDecodeMetaBufs; ++s) {
            mbar_init(bar_mfull + 8 * s, 1);
            mbar_init(bar_mempty + 8 * s, kDecodeDrainWarps);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_recv + 8 * s, 1);
            mbar_init(bar_free + 8 * s, S);
        }
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(flag), "r"(0u) : "memory");
        fence_barrier_init();
        fence_proxy_async();
        mbar_arrive_expect_tx(bar_recv, recv_tx);
        mbar_arrive_expect_tx(bar_recv + 8, recv_tx);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kDecodeCols);
        tmem_relinquish();
    }
    // The weights warp, which set up the barriers, does not wait for the others: its first copies leave while tensor memory is
    // still being allocated.
    if (warp == 0) {
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"r"(kDecodeThreads) : "memory");
    } else {
        tc_fence_before_sync();
        asm volatile("bar.sync 1, %0;" ::"r"(kDecodeThreads) : "memory");
        tc_fence_after_sync();
    }
    cluster_arrive_release();           // "my receive barriers are armed"; waited for before the first send
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, lds32(tmem_slot), 0);      // (not read by the weights warp)
    const uint32_t d_base = tmem_base + 2 * P * kDecodeACols;

    if (warp == 0) {
        // ---------------------------------------------------------------- weights (one thread issues)
        if (elect_one()) tma_prefetch_descriptor(&w_map);
        GPTQ_TRACE_MIN(a.trace_slot, first_weight_issue);
        // The next launch may start when the last kDecodeLead steps are about to be requested: earlier its prefetch would queue
        // in front of this launch's own loads, later it would not be under way before this launch has ended.
        int s = 0, mb = 0, left = n_panels * spp;
        uint32_t eph = 1, mph = 1;  // parities that pass in the first round
        for (int p = cl; p < panels; p += a.clusters) {
            for (int c0 = 0; c0 < ng; c0 += MC) {
                const int nc = (ng - c0) < MC ? (ng - c0) : MC;
                const int t = p * a.G + g0 + c0;
                decode_wait(bar_mempty + 8 * mb, mph, flag);
                if (elect_one()) {
                    const uint32_t md = meta + mb * kDecodeMetaBytes, bar = bar_mfull + 8 * mb;
                    mbar_arrive_expect_tx(bar, (uint32_t)(nc * SUB * (kItemSBytes + kItemZBytes)));
                    bulk_g2s(md, a.scales + (size_t)t * (SUB * kItemSBytes), nc * SUB * kItemSBytes, bar);
                    bulk_g2s(md + kOffZ, a.qzeros + (size_t)t * (SUB * kItemZBytes), nc * SUB * kItemZBytes, bar);
                }
                __syncwarp();
                for (int i = 0; i < nc; i += P) {
                    if (left-- == kDecodeLead) pdl_launch_dependents();
                    decode_wait(bar_wempty + 8 * s, eph, flag);
                    fence_proxy_async();        // the copies stay behind the dequant warps' loads, as in mbar_wait_stage_free
                    if (elect_one()) {
                        const bool two = P == 2 && i + 1 < nc;
                        mbar_arrive_expect_tx(bar_wfull + 8 * s, two ? 2 * kItemWBytes : kItemWBytes);
                        // packed weights as rows of 64 bytes, 128 rows per item
                        tma_load_2d(wring + s * kWSlot, &w_map, 0, (t + i) * 128, bar_wfull + 8 * s);
                        if (two) tma_load_2d(wring + s * kWSlot + kItemWBytes, &w_map, 0, (t + i + 1) * 128, bar_wfull + 8 * s);
                    }
                    __syncwarp();
                    if (++s == NW) { s = 0; eph ^= 1u; }
                }
                if (++mb == kDecodeMetaBufs) { mb = 0; mph ^= 1u; }
            }
        }
        if (n_panels * spp < kDecodeLead) pdl_launch_dependents();
        cluster_wait_acquire();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA (one thread issues)
        constexpr uint32_t idesc = umma_idesc_e4m3_e5m2(128, kN);
        const uint64_t bdesc0 = umma_desc_k_major_sw128(xtiles);
        uint32_t sa = 0, pha = 0, sd = 0, phd = 1;
        int x_have = 0;             // passes of the split of x that have been waited for
        for (int pi = 0; pi < n_panels; ++pi) {
            uint64_t b0 = bdesc0;
            for (int i = 0; i < ng; i += P) {
                const bool two = P == 2 && i + 1 < ng;
                if (pi == 0) {
                    for (const int need = ((i + (two ? 2 : 1)) * a.M - 1) / kUnits; x_have <= need; ++x_have)
                        decode_wait(bar_xfull + 8 * x_have, 0, flag);
                }
                decode_wait(bar_drained + 8 * sd, phd, flag);
                decode_wait(bar_afull + 8 * sa, pha, flag);
                tc_fence_after_sync();
                if (pi == 0 && i == 0) GPTQ_TRACE_MIN(a.trace_slot, first_data);
                if (elect_one()) {
                    const uint32_t d0 = d_base + sd * (P * kDCols), a0 = tmem_base + sa * (P * kDecodeACols);
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)       // 32 k each: 8 columns of A, 32 bytes of each B row
                        umma_f8_ts(d0 + (k4 * SUB / 4) * kN, a0 + k4 * 8, b0 + (uint64_t)(k4 * 2), idesc, k4 * SUB % 4 != 0);
                    if (two) {
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)
                            umma_f8_ts(d0 + kDCols + (k4 * SUB / 4) * kN, a0 + kDecodeACols + k4 * 8,
                                       b0 + (uint64_t)(kXTile / 16 + k4 * 2), idesc, k4 * SUB % 4 != 0);
                    }
                    umma_commit(bar_done + 8 * sd);
                }
                __syncwarp();
                b0 += (uint64_t)(P * kXTile / 16);
                pha ^= sa;
                sa ^= 1u;
                if (++sd == ND) { sd = 0; phd ^= 1u; }
            }
        }
        cluster_wait_acquire();
    } else if (warp < kDecodeFirstDrain) {
        // ---------------------------------------------------------------- dequant warps
        const int q = warp & 3, set = (warp - kDecodeFirstDq) >> 2;
        const int n_col = 32 * q + lane, u = n_col >> 4, g = n_col & 7, h = (n_col >> 3) & 1;
        // x -> pieces in the B tiles and the groups' sums, once: a thread takes eight consecutive k of a token
        auto split_x = [&]() {
            const int tid = threadIdx.x - 32 * kDecodeFirstDq, kc = tid & 15;
            pdl_wait();
            if (tid == 0) {
                GPTQ_TRACE_MIN(a.trace_slot, first_wait_done);
                GPTQ_TRACE_MAX(a.trace_slot, last_wait_done);
            }
            const __half *x0 = a.x + (size_t)g0 * kGroup + 8 * kc;
            const int K = a.G * kGroup;
            constexpr int kBatch = 4;
            for (int b0 = 0; b0 < x_passes; b0 += kBatch) {
                uint4 v[kBatch];
                int item[kBatch], token[kBatch];
#pragma unroll
                for (int b = 0; b < kBatch; ++b) {
                    const int unit = (b0 + b) * kUnits + (tid >> 4);
                    item[b] = (int)((uint32_t)unit * a.m_inverse >> 16);
                    token[b] = unit - item[b] * a.M;
                    v[b] = make_uint4(0, 0, 0, 0);
                    if (unit < x_units) v[b] = ldg128_cg(x0 + (size_t)token[b] * K + item[b] * kGroup);
                }
#pragma unroll
                for (int b = 0; b < kBatch; ++b) {
                    if (b0 + b >= x_passes) break;
                    const bool live = (b0 + b) * kUnits + (tid >> 4) < x_units;
                    if (live) decode_store_pieces(xtiles + item[b] * kXTile, token[b], kc, v[b]);
                    const float2 f0 = pair_to_float2<false>(v[b].x), f1 = pair_to_float2<false>(v[b].y);
                    const float2 f2 = pair_to_float2<false>(v[b].z), f3 = pair_to_float2<false>(v[b].w);
                    float sum = ((f0.x + f0.y) + (f1.x + f1.y)) + ((f2.x + f2.y) + (f3.x + f3.y));
#pragma unroll
                    for (int d = 8 / SUB; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
                    if (live && (kc & (16 / SUB - 1)) == 0)
                        sts_f32(sums + (uint32_t)((item[b] * SUB + kc / (16 / SUB)) * NX + token[b]) * 4, sum * (1.f / 512.f));
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_xfull + 8 * (b0 + b));
                }
            }
        };
        uint32_t w_rd[4];               // the column's 8 bytes (rows +0..7, +32..39) in the four chunks of a K64 block
#pragma unroll
        for (int t4 = 0; t4 < 4; ++t4) w_rd[t4] = wring + (u * 8 + g) * 64 + ((uint32_t)(t4 ^ (g >> 1)) << 4) + 8 * h;
        const uint32_t a_dst = tmem_base + ((uint32_t)(32 * q) << 16) + set * (P * kDecodeACols);
        const uint32_t bar_a = bar_afull + 8 * set;
        const int steps = n_panels * spp;
        int s = set, i = set;           // weight slot, step of the panel
        while (i >= spp) i -= spp;
        uint32_t wph = 0, sd = set, dph = 0;    // done[step t - 2]: the accumulator ring's barriers, every other one
        // A set looks at every other step only.  Its parity waits on a weight slot are unambiguous because the step that it
        // has waited for to be multiplied (four back at that point) tells that the slot's previous contents, NW >= 4 steps
        // back, had landed.
        for (int t = set; t < steps; t += 2) {
            const bool two = P == 2 && ((ng & 1) == 0 || i + 1 < spp);
            decode_wait(bar_wfull + 8 * s, wph, flag);
            const uint32_t wofs = s * kWSlot;
            uint2 wv[8];
            uint32_t r[32];             // column 16 blk + 8 j + 2 t4 (+ 1: the odd nibbles)
            auto load_words = [&](int e) {
#pragma unroll
                for (int w = 0; w < 8; ++w) wv[w] = lds64(w_rd[w & 3] + wofs + e * kItemWBytes + (w >> 2) * kBlockWBytes);
            };
            auto to_bytes = [&]() {
#pragma unroll
                for (int w = 0; w < 8; ++w)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t v = j ? wv[w].y : wv[w].x;
                        r[16 * (w >> 2) + 8 * j + 2 * (w & 3)] = v & 0x0f0f0f0fu;
                        r[16 * (w >> 2) + 8 * j + 2 * (w & 3) + 1] = (v >> 4) & 0x0f0f0f0fu;
                    }
            };
            load_words(0);
            to_bytes();
            if (two) load_words(1);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_wempty + 8 * s);          // the step's words are in registers
            if (t >= 2) {               // the A stage's previous step has been multiplied
                decode_wait(bar_done + 8 * sd, dph, flag);
                sd += 2;
                if (sd >= ND) { sd -= ND; dph ^= 1u; }
                __syncwarp();
                tc_fence_after_sync();
            }
            tmem_st_32x32(a_dst, r);
            if (two) {
                to_bytes();
                tmem_st_32x32(a_dst + kDecodeACols, r);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_a);
            s += 2;
            if (s >= NW) { s -= NW; wph ^= 1u; }
            i += 2;
            while (i >= spp) i -= spp;
            if (t == set) split_x();
        }
        if (set >= steps) split_x();    // (a CTA with a single step)
        __syncwarp();
        cluster_wait_acquire();
    } else if (warp < kDecodeFinishWarp) {
        // ---------------------------------------------------------------- drain warps
        const int q = warp & 3;
        const int n_col = 32 * q + lane, u = n_col >> 4, g = n_col & 7, h = (n_col >> 3) & 1;
        const uint32_t s_off = meta + (16 * u + 2 * g + h) * 2, z_off = meta + kOffZ + 8 * u + g;
        const int z_shift = 4 * h;
        const uint32_t d_src = d_base + ((uint32_t)(32 * q) << 16);
        const float z_add = (flags & kFormatZerosMinusOne) ? 8388607.f : 8388608.f;
        const uint64_t eighth = pack_f32x2(0x3e000000u, 0x3e000000u);
        // this column's owner and place in the owner's receive buffer
        const int cc = n_col & ((1 << hsh) - 1), owner = ((cc + 1) * S - 1) >> hsh;
        const int pos = (n_col >> hsh) * a.slice_max + cc - (int)((a.slice_lo >> (8 * owner)) & 255);
        const uint32_t dst = map_to_cluster_rank(recv, (uint32_t)owner) + (uint32_t)((rank * wide + pos) * a.M * 4);
        const uint32_t dbar = map_to_cluster_rank(bar_recv, (uint32_t)owner);
        constexpr uint32_t kSumItem = SUB * NX * 4;
        const uint32_t no_bits = (uint32_t)warp >> 8;       // 0, which the compiler cannot know
        uint32_t mb = 0, mph = 0, sd = 0, dph = 0;
        for (int pi = 0; pi < n_panels; ++pi) {
            uint64_t run = 0;
            uint32_t sum_at = sums;
            for (int c0 = 0; c0 < ng; c0 += MC) {
                const int nc = (ng - c0) < MC ? (ng - c0) : MC;
                uint32_t s_at = s_off + mb * kDecodeMetaBytes, z_at = z_off + mb * kDecodeMetaBytes;
                decode_wait(bar_mfull + 8 * mb, mph, flag);
                for (int i = 0; i < nc; i += P) {
                    const bool two = P == 2 && i + 1 < nc;
                    uint64_t sc[P * SUB], nz[P * SUB];
#pragma unroll
                    for (int e = 0; e < P * SUB; ++e) {     // (a lone last item reads past its own, within the buffer)
                        const uint32_t f = __float_as_uint(pair_to_float2<false>(lds16(s_at + e * kItemSBytes)).x);
                        const uint32_t zb = (lds8(z_at + e * kItemZBytes) >> z_shift) & 15u;
                        const uint32_t z = __float_as_uint(z_add - __uint_as_float(0x4b000000u | zb));   // -z: 2^23 + z is exact
                        sc[e] = pack_f32x2(f, f);
                        nz[e] = pack_f32x2(z, z);
                    }
                    s_at += P * SUB * kItemSBytes;
                    z_at += P * SUB * kItemZBytes;
                    // (the MMA has waited for the items' x: its completion also says that the sums of x are there)
                    decode_wait(bar_done + 8 * sd, dph, flag);
                    __syncwarp();
                    tc_fence_after_sync();
                    const uint32_t d0 = d_src + sd * (P * kDCols);
                    auto drained = [&]() {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_drained + 8 * sd);
                    };
                    auto combine = [&](const uint32_t (&r)[8], int e) {      // group e of the step
                        uint64_t v = fma_f32x2(pack_f32x2(r[6], r[7]), eighth, pack_f32x2(r[4], r[5]));
                        v = fma_f32x2(v, eighth, pack_f32x2(r[2], r[3]));
                        v = fma_f32x2(v, eighth, pack_f32x2(r[0], r[1]));
                        v = fma_f32x2(nz[e], lds_f32x2(sum_at + e * (NX * 4)), v);
                        run = fma_f32x2(sc[e], v, run);
                    };
                    // all groups of the step at once, two at a time (garbage behind a lone last item)
#pragma unroll
                    for (int e = 0; e < P * SUB; e += 2) {
                        uint32_t r0[8], r1[8];
                        tmem_ld_8(d0 + e * kN, r0);
                        tmem_ld_8(d0 + (e + 1) * kN, r1);
                        tmem_wait_ld();
                        if (e + 2 == P * SUB) drained();
                        if (e < SUB || two) combine(r0, e);
                        if (e + 1 < SUB || two) combine(r1, e + 1);
                    }
                    sum_at += P * kSumItem;
                    if (++sd == ND) { sd = 0; dph ^= 1u; }
                }
                // The buffer's next copies must not overtake the loads above.  The arrival's address takes a zero out of the sums, into
                // which all that was loaded has gone.  (A fence, here or in front of the copies: groups of 32 1 to 2 % slower.)
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_mempty + 8 * mb + ((uint32_t)run & no_bits));
                if (++mb == kDecodeMetaBufs) { mb = 0; mph ^= 1u; }
            }
            // ---- send the panel's sums to the columns' owners
            const uint32_t buf = (uint32_t)pi & 1u;
            if (pi == 0) {
                __syncwarp();
                cluster_wait_acquire();             // every CTA of the cluster has armed its receive barriers
            } else if (pi >= 2) {
                decode_wait_cluster(bar_free + 8 * buf, (uint32_t)((pi >> 1) - 1) & 1u, flag);   // the owners have read panel pi - 2
            }
            const float2 f = unpack_f32x2(run);     // nibbles were q * 2^-9
            if (a.M == 2) st_async_f32x2(dst + buf * recv_bytes, make_float2(f.x * 512.f, f.y * 512.f), dbar + 8 * buf);
            else st_async_f32(dst + buf * recv_bytes, f.x * 512.f, dbar + 8 * buf);
        }
    } else {
        // ---------------------------------------------------------------- finish: the own column slice of each panel
        const bool layout_ok = ((flags & kFormatGateUp) != 0) == (a.fuse != 0) && (flags & kFormatBf16) == 0;
        if (!layout_ok && lane == 0) atomicMax(&g_device_status, (int)kStatusLayoutMismatch);
        pdl_wait();
        cluster_wait_acquire();
        bool any_nan = false;
        for (int pi = 0; pi < n_panels; ++pi) {
            const int p = cl + pi * a.clusters;
            const uint32_t buf = (uint32_t)pi & 1u;
            decode_wait_cluster(bar_recv + 8 * buf, (uint32_t)(pi >> 1) & 1u, flag);
            if (layout_ok && (lds32(flag) & kDecodeGaveUp) == 0) {
                // a thread takes one column (with fuse: a gate column and its up column) of one token
                for (int idx = lane; idx < a.M * hw; idx += 32) {
                    const int j = a.M == 2 ? idx >> 1 : idx, m = a.M == 2 ? idx & 1 : 0;
                    auto slice_sum = [&](int jj) {   // sender order
                        const uint32_t at = recv + buf * recv_bytes + (uint32_t)(jj * a.M + m) * 4u, step = (uint32_t)(wide * a.M) * 4u;
                        float sum = 0.f;
#pragma unroll
                        for (int sdr = 0; sdr < 8; ++sdr) {
                            if (sdr >= S) break;
                            sum += lds_f32(at + sdr * step);
                        }
                        return sum;
                    };
                    if (!a.fuse) {
                        const int n = p * kPanel + lo + j;
                        float v = slice_sum(j);
                        const bool is_nan = isnan(v);
                        if (a.bias || a.residual) {
                            v += (a.bias ? __half2float(a.bias[n]) : 0.f);
                            if (a.residual) v += __half2float(a.residual[(size_t)m * a.N + n]);
                        }
                        if (!is_nan) a.y[(size_t)m * a.N + n] = __float2half_rn(v);
                        any_nan |= is_nan;
                    } else {
                        const int oc = p * 64 + lo + j;
                        const float gate = slice_sum(j), up = slice_sum(a.slice_max + j);
                        const bool is_nan = isnan(gate) || isnan(up);
                        if (!is_nan) a.y[(size_t)m * (a.N / 2) + (a.out_index ? a.out_index[oc] : oc)] = __float2half_rn(silu_mul(gate, up));
                        any_nan |= is_nan;
                    }
                }
            }
            if (pi + 2 < n_panels) {
                __syncwarp();
                if (lane == 0) mbar_arrive_expect_tx(bar_recv + 8 * buf, recv_tx);     // armed before any sender may go on
                __syncwarp();
                if (lane < S) mbar_arrive_release_cluster(map_to_cluster_rank(bar_free + 8 * buf, (uint32_t)lane));
            }
        }
        if (any_nan) raise_flag(flag, kDecodeNotFinite);
        if (lane == 0) GPTQ_TRACE_MAX(a.trace_slot, last_exit);
    }
    tc_fence_before_sync();
    __syncthreads();
    const uint32_t raised = lds32(flag);
    if (raised & kDecodeGaveUp) {
        // A wait gave up: leave time for the copies in flight to land, and stay until the other CTAs of the cluster have
        // left or come here too (they may still send; one that left in order has nothing more to receive).
        const uint64_t start = global_timer_ns();
        while (global_timer_ns() - start < 200000ull) { }
        __syncthreads();
        cluster_arrive_release();
        cluster_wait_acquire();
    } else if (raised) {
        decode_store_not_finite<SUB>(a);
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kDecodeCols);
    }
}

struct DecodePlan {
    bool use;       // else the mma.sync kernel takes the problem
    int sub;
    int S, clusters, ctas;
    int w_slots, x_tiles, smem_bytes;
};

// clusters of S CTAs that fit one CTA per SM (cudaOccupancyMaxActiveClusters on 148 SMs: the GPCs' SM counts are not
// multiples of most sizes), scaled to other SM counts
inline int decode_max_clusters(int S, int sm_count)
{
    static const int at148[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    const int n = at148[S] * sm_count / 148;
    return n > 0 ? n : 1;
}

inline DecodePlan plan_decode(int M, int N, int K, int group_size, int fuse, int bf16, int sm_count)
{
    DecodePlan pl{};
    const int G = K / kGroup, panels = N / kPanel;
    pl.sub = kGroup / group_size;
    if (bf16 || M > kDecodeMaxRows) return pl;
    const int budget = (227 * 1024) / 2 - 1024;                          // two launches share an SM
    const int tile = kDecodeXTile, step = decode_step_items(pl.sub) * kItemWBytes;
    // Estimated times in microseconds, fitted to 80 shapes (K = 1024 .. 13824, N = 1024 .. 27648; the chosen kernel is within
    // 2 % of the better one on average).  Here: the busiest CTA's items.  The mma.sync kernel: the layer's items spread over
    // the SMs, but one CTA's own pace where its grid leaves one CTA per SM.  At M = 1, there and here: 4096 x 6144 5.8 and
    // 6.3 us, 1024 x 3072 2.8 and 3.4; 4096 x 4096 4.7 and 4.1, 4096 x 12288 8.3 and 7.4, 8192 x 2048 8.8 and 5.1,
    // 4096 x 22016 12.8 and 11.4, 13824 x 27648 42.3 and 35.3.
    const double per_item = 0.21, fixed_time = 2.6;
    const SplitKPlan sk = plan_splitk(M, N, K, group_size, sm_count);
    const double spread = 0.0021 * panels * G, serial = sk.ctas <= sm_count ? 0.6 * ((G + sk.S - 1) / sk.S) : 0;
    const double other = 2.2 + (spread > serial ? spread : serial);
    double best = -1;
    int items = 0;      // of the busiest CTA
    for (int S = 1; S <= 8; ++S) {
        if (S > G) break;
        const int most = decode_max_clusters(S, sm_count), c0 = panels < most ? panels : most;
        const int ppc = (panels + c0 - 1) / c0;                          // panels per cluster
        const int ng = (G + S - 1) / S;                                  // items of the busiest CTA, per panel
        // the B tiles of the CTA's K range have to leave four steps of weights
        const int fixed = 2048 + kDecodeMetaBufs * kDecodeMetaBytes + 2 * decode_recv_bytes(M, fuse, S, ((fuse ? 64 : kPanel) + S - 1) / S) +
                          ng * tile + decode_sum_bytes(pl.sub, ng);
        int slots = (budget - fixed) / step;
        if (ng > kDecodeMaxItems || ng * M > 16 * kDecodeMaxXPasses || slots < 4) continue;
        const double t = fixed_time + per_item * ppc * ng + 0.1 * ppc + (S > 1 ? 0.1 : 0);
        if (best < 0 || t < best) {
            best = t;
            items = ppc * ng;
            pl.S = S;
            pl.clusters = (panels + ppc - 1) / ppc;
            pl.x_tiles = ng;
            pl.w_slots = slots < kDecodeMaxWSlots ? slots : kDecodeMaxWSlots;
            pl.smem_bytes = fixed + pl.w_slots * step;
        }
    }
    pl.use = best >= 0 && fixed_time + per_item * items < other;
    pl.ctas = pl.clusters * pl.S;
    const int floor_two_per_sm = (227 * 1024) / 3 + 512;                 // no third CTA: tensor memory holds two
    if (pl.smem_bytes < floor_two_per_sm) pl.smem_bytes = floor_two_per_sm;
    return pl;
}

template <int SUB>
static int launch_decode_sub(const DecodeArgs &args, const CUtensorMap &w_map, const DecodePlan &plan, cudaStream_t s)
{
    static int configured_smem[64] = {};
    const int cfg_st = ensure_dynamic_smem((const void *)decode_kernel<SUB>, configured_smem, plan.smem_bytes);
    if (cfg_st) return cfg_st;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)plan.ctas);
    cfg.blockDim = dim3(kDecodeThreads);
    cfg.dynamicSmemBytes = (size_t)plan.smem_bytes;
    cfg.stream = s;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)plan.S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    attr[2].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
    attr[2].val.clusterSchedulingPolicyPreference = cudaClusterSchedulingPolicyLoadBalancing;
    cfg.attrs = attr;
    cfg.numAttrs = 3;
    return record_cuda_error(cudaLaunchKernelEx(&cfg, decode_kernel<SUB>, args, w_map));
}

int launch_decode(const __half *x, const void *qweight, const void *qzeros, const void *scales, __half *y, int M, int N, int K,
                  const DecodePlan &plan, int fuse, const __half *bias, const __half *residual, const int32_t *out_index,
                  cudaStream_t s)
{
    DecodeArgs args;
    args.qweight = (const uint8_t *)qweight;
    args.scales = (const uint8_t *)scales;
    args.qzeros = (const uint8_t *)qzeros;
    args.x = x;
    args.y = y;
    args.M = M;
    args.N = N;
    args.G = K / kGroup;
    args.S = plan.S;
    args.clusters = plan.clusters;
    args.w_slots = plan.w_slots;
    args.x_tiles = plan.x_tiles;
    args.m_inverse = (65536u + (uint32_t)M - 1) / (uint32_t)M;
    args.trailer = reinterpret_cast<const TiledTrailer *>((const uint8_t *)qzeros + tiled_zero_bytes(N, K, kGroup / plan.sub));
    args.fuse = fuse;
    args.bias = bias;
    args.residual = residual;
    args.trace_slot = next_trace_slot();
    args.out_index = out_index;
    split_columns(fuse, plan.S, &args.slice_lo, &args.slice_max);
    CUtensorMap w_map;
    const int st = make_tensor_map_2d(&w_map, CU_TENSOR_MAP_DATA_TYPE_UINT32, qweight, 16, (uint64_t)K * N / 2 / 64, 64, 16, 128,
                                      CU_TENSOR_MAP_SWIZZLE_64B);
    if (st) return st;
    switch (plan.sub) {
    case 1: return launch_decode_sub<1>(args, w_map, plan, s);
    case 2: return launch_decode_sub<2>(args, w_map, plan, s);
    case 4: return launch_decode_sub<4>(args, w_map, plan, s);
    default: return GPTQ_ERR_UNSUPPORTED;
    }
}

}  // namespace gptq

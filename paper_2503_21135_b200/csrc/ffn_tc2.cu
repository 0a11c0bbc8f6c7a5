// Grouped dequant-GEMM for experts with many tokens (prefill) on PAIRS of SMs: thread-block clusters of two
// CTAs drive one tcgen05.mma.cta_group::2 of M = 256 weight rows x N <= 256 tokens x K = 16.
//
// Why pairs: a tcgen05.mma costs the tensor core at least as long as a 128-token one however few tokens it has,
// and the dequantization of a 256 x 128 weight block costs ~4500 warp instructions however many tokens use
// it.  With M = 256 across two CTAs each CTA dequantizes only ITS 128 rows (8 atoms) per stage, into its own
// tensor memory, for a tile of 256 tokens: half the dequant work per flop of the one-CTA kernel at twice
// the tokens per MMA, so the tensor pipe, not the dequant warps, sets the pace.
//
// Work item of a cluster = (expert, 256-row weight block, tile of <= 256 tokens; an expert's tiles are equal up to the rounding
// to 32 rows, from eight on they are 256 and a rest), K over the whole
// input axis; items are dealt round-robin over the clusters; rings, A buffers, accumulators live across items.
// Per CTA (rank r = 0 leader, 1 peer), 19 warps:
//   warp 16 weights  : ONE thread; bulk copies of the CTA's half block (codes of atoms 8r..8r+7, params of rows 128r..) into a
//                      byte-granular ring of up to eight stages; a place comes free once the stage's warps have expanded
//                      its codes (the first half of them into an A buffer, so that one has to be free).
//   warp 18 operands : bulk copy of ITS half of the token tile (N/2 tokens: the B operand is split across the
//                      pair) into a ring of four 32 KB slots, freed by the MMAs' commit.
//   warps 0-15 dequant: a whole atom (16 rows x 128 k) of every OTHER stage each (eight warps per stage): packed
//                      codes -> full fp16 weight (AND-OR, HSUB2, HFMA2 per register pair, the weight s*q+m rounded
//                      once) -> tcgen05.st into the CTA's tensor memory; then wait for the CTA's operand tile and
//                      arrive on the LEADER's a_full barrier (remote arrive for the peer).
//   warp 17 MMA      : in the leader only: waits for both CTAs' A buffers, issues the eight MMAs of the stage
//                      for the pair as one run, commits (multicast) to both CTAs' done and d_full barriers.
//   epilogue         : warps 0-15 of each CTA read their CTA's 128 accumulator rows x N tokens (tcgen05.ld),
//                      SwiGLU -> fp16 h as the down GEMM's operand tiles, or fp32 rows out; they arrive on the
//                      leader's d_empty barrier with the last load.
// Tensor memory per CTA: columns 0..255 accumulators (128 rows x 256 tokens, or twice 128), 256..511 four A buffers.
// What bounded it (4096 x 14336 experts, 125 rows each; a stage's MMAs run 512 cycles): a stage took 1235 cycles, of which
// the MMA warp spent 700 on issuing with an elect per MMA and 290 on a poll; then the gap between two items, 7 to 17 thousand
// cycles, in which every role found its next item by a chain of global loads and the epilogue stored 4-byte words over eight
// lines.  With the issue as one run, polls asked for early, the experts' table in shared memory and 128-byte stores a stage
// takes 865 cycles and the gap 6 to 7 thousand.  us a pass of the whole layer, passes back to back under the power cap, before
// and now: 500 tokens 542 -> 479, 1000 (skewed) 904 -> 834, 4096 2719 -> 2590, 2048 fine-grained 476 -> 451; short bursts at full
// clock, in which the variants below were compared: 500 tokens 492 -> 416, 4096 2467 -> 2348.  What is left is the epilogue (5
// thousand cycles an item) and the dequant warps' latencies.
// Every wait is bounded; after an expired wait a CTA leaves its loops and meets its peer at the final
// cluster barrier (the peer's own waits expire within the same bound).
#include <cstddef>
#include <type_traits>

#include "common.cuh"
#include "expand.cuh"
#include "layout.cuh"
#include "tcgen05.cuh"

namespace dyn {

constexpr int T2_DEQ_WARPS = 16;
constexpr int T2_W_PROD = 16, T2_W_MMA = 17, T2_W_PRODX = 18;
constexpr int T2_THREADS = 19 * 32;
constexpr int T2_N = 256;                              // tokens per work item (128 per CTA)
constexpr int T2_WHALF_MAX = 17408;                    // half of the largest packed block (8-bit, G = 64)
constexpr int T2_XTILE = 16 * TC_TILE_BYTES;           // 128 tokens x 128 k: 16 row-group tiles
constexpr int T2_POOL_TILES = POOL_GROUP * POOL_TILE_PITCH;       // cached-channel stage: 32 column tiles in a weight slot ...
constexpr int T2_POOL_XG = 16 * 512;                              // ... and their operand tile of 16 row groups in an operand slot
static_assert(T2_POOL_TILES <= T2_WHALF_MAX && T2_POOL_XG <= T2_XTILE, "cached-channel stage does not fit its slots");
// Two rings.  The operand tiles (32 KB slots, read by the MMAs) are freed by the MMAs' commit; the packed weights (read
// only by the dequant warps) lie in a byte-granular ring, up to eight stages of it (four of 8-bit codes), whose places
// come free once the codes are expanded, behind the wait for the stage's A buffer.
constexpr int T2_NW = 8;
constexpr int T2_NX = 4;
constexpr int T2_WRING = 4 * T2_WHALF_MAX;
constexpr int T2_OFF_TAB = 512;                        // experts' table
constexpr int T2_OFF_STAGE = 16384;
constexpr int T2_OFF_XRING = T2_OFF_STAGE + T2_WRING;
constexpr int T2_SMEM_BYTES = T2_OFF_XRING + T2_NX * T2_XTILE;
static_assert(T2_OFF_XRING % 1024 == 0 && T2_XTILE % 1024 == 0, "operand slots must stay 1024-byte aligned");
static_assert(T2_SMEM_BYTES <= 227 * 1024, "shared memory limit of a CTA");
constexpr uint32_t T2_TMEM_COLS = 512;
constexpr uint32_t T2_COL_A = 256;
constexpr int T2_NA = 4;                               // A buffers of 64 columns: the dequant warps run ahead of the MMA
constexpr int T2_SMALL = 128;                          // token tiles up to here leave room for two accumulators

struct T2Params {
    const LayerDev* L;
    WsDev ws;
    int n_rb;       // 256-row weight blocks of this GEMM
    int n_experts;  // experts listed in L->order
    int fills;      // the launch before is the fold kernel's, on the smaller experts: this one starts beside it
};

struct T2Bars {
    uint64_t full[T2_NW], empty[T2_NW];    // per CTA: weight bytes landed / the stage's 8 dequant warps have expanded the codes
    uint64_t fullx[T2_NX];               // per CTA: operand bytes landed
    uint64_t a_full[T2_NA];              // leader only: the 16 dequant warps of the pair that own the stage stored A buffer b
    uint64_t done[T2_NA];                // per CTA: the stage's MMAs are complete (commit): A buffer and operand slot are free
    uint64_t d_full[2];                  // per CTA: the accumulators of an even / odd item are complete (commit)
    uint64_t d_empty[2];                 // leader only: 32 epilogue warps of the pair have read them
    int size[T2_NW];                     // weight producer only: ring bytes of the stage in slot i
    uint32_t tmem_base;
    volatile int poison;
    int off;                             // leader only: an expired wait was on record when the pair started (fills)
};
static_assert(sizeof(T2Bars) <= T2_OFF_TAB, "barrier block overlaps the item table");
static_assert(T2_NA == T2_NX, "one commit frees a stage's A buffer and its operand slot");
// barrier offsets from the CTA's shared-memory base
#define T2_BAR(field, i) (sb + (uint32_t)offsetof(T2Bars, field) + 8u * (uint32_t)(i))

// An expert above the row threshold, gathered once per launch: an item is then found from shared memory alone (a chain of
// five global loads before, which every role waited for between two items: several thousand cycles).
struct T2Expert {
    const uint8_t* w;     // packed blocks
    const uint8_t* pool;  // forward-ready tiles of the cached channels
    int first;            // first item
    int cnt, n_tt, rows;  // rows of the expert, token tiles, rows of a tile
    int row0, bits, blk_bytes, n_it;
};
static_assert(T2_OFF_TAB + (MAX_EXPERTS + 1) * (int)sizeof(T2Expert) <= T2_OFF_STAGE, "expert table overlaps the stage ring");

// One work item of the cluster: (expert, 256-row weight block, token tile).
struct T2Item {
    const T2Expert* t;
    int rb, tile0;        // row block, first row of the tile within the expert's segment
    int n_valid, n_mma;   // rows of the tile; N of the pair's MMA, each CTA holds N/2 token rows of B
    int bits, n_it;       // stages: packed blocks, then cached-channel stages of 32 pool columns
};
__device__ __forceinline__ T2Item t2_item(const T2Expert* tab, int g, int& cursor) {
    while (g >= tab[cursor + 1].first) ++cursor;
    T2Item it;
    it.t = tab + cursor;
    const int local = g - it.t->first, n_tt = it.t->n_tt;
    it.rb = n_tt > 1 ? local / n_tt : local;   // tiles of one weight block are neighbours: concurrent clusters share its L2 lines
    it.tile0 = (local - it.rb * n_tt) * it.t->rows;
    it.n_valid = min(it.t->rows, it.t->cnt - it.tile0);
    it.n_mma = (it.n_valid + 31) & ~31;
    it.bits = it.t->bits;
    it.n_it = it.t->n_it;
    return it;
}

// One (atom, 64-k half) of the CTA's half block -> 32 columns of the A buffer.  prm: the {scale, zero} words of the lane's
// two rows in this half's quantization group.
template <int BITS, int HALF>
__device__ __forceinline__ void t2_dequant_half(const uint32_t (&raw)[16], uint32_t prm0, uint32_t prm1, uint32_t (&regs)[16]) {
    constexpr int BIAS = BITS == 2 ? 4 : (BITS == 3 ? 3 : ((BITS == 4 || BITS == 6) ? 2 : 0));
    constexpr int NOFF = BITS == 2 ? 5 : (BITS == 3 ? 4 : ((BITS == 4 || BITS == 6) ? 2 : 1));  // distinct offsets 0, step, 2*step, ...
    constexpr int OSTEP = (BITS == 4 || BITS == 6) ? 4 : 2;
    const __half2 k1024 = __float2half2_rn(1024.f);
    __half2 S2[2], M2[2][NOFF];
#pragma unroll
    for (int rh = 0; rh < 2; ++rh) {
        const uint32_t pw = rh ? prm1 : prm0;
        const __half2 pp = *reinterpret_cast<const __half2*>(&pw);
        S2[rh] = __hmul2(__low2half2(pp), __half2half2(__ushort_as_half((unsigned short)((15 - BIAS) << 10))));
#pragma unroll
        for (int i = 0; i < NOFF; ++i)  // zero-point times 2^(o - bias), exact
            M2[rh][i] =
                __hmul2(__high2half2(pp), __half2half2(__ushort_as_half((unsigned short)((15 + OSTEP * i - BIAS) << 10))));
    }
    Codes<BITS> cd;
    codes_of<BITS, HALF>(cd, raw);
    auto step = [&](auto S4c) {
        constexpr int S4 = decltype(S4c)::value;
        uint32_t af[4];
        expand<BITS, S4, 0x64006400u>(cd, af);
#pragma unroll
        for (int ri = 0; ri < 4; ++ri) {
            const int oi = code_offset<BITS>(S4, ri >> 1) / OSTEP;
            const __half2 qo = __hsub2(*reinterpret_cast<const __half2*>(&af[ri]), k1024);  // q * 2^o, exact
            const __half2 v = __hfma2(qo, S2[ri & 1], M2[ri & 1][oi]);
            af[ri] = *reinterpret_cast<const uint32_t*>(&v);
        }
        // fragment (rowhalf, h) -> TMEM register order of the 16x256b shape: (row, col pair)
        regs[4 * S4 + 0] = af[0];
        regs[4 * S4 + 1] = af[2];
        regs[4 * S4 + 2] = af[1];
        regs[4 * S4 + 3] = af[3];
    };
    step(std::integral_constant<int, 0>{});
    step(std::integral_constant<int, 1>{});
    step(std::integral_constant<int, 2>{});
    step(std::integral_constant<int, 3>{});
}

// What a dequant warp is: its atom of the CTA's half block, its stages (running number = kh mod 2), its tensor-memory lanes.
struct T2Deq {
    uint32_t sb, a_lanes;
    int a_l, kh, lane, rank;
    volatile int* poison;
    int32_t* status;
};
__device__ __forceinline__ T2Deq t2_deq(uint8_t* smem, uint32_t tbase, int rank, int32_t* status) {
    const int warp = threadIdx.x >> 5;
    T2Deq c;
    c.sb = smem_u32(smem);
    c.kh = warp >> 3;
    c.a_l = 2 * (warp & 3) + ((warp >> 2) & 1);
    c.a_lanes = tbase + T2_COL_A + ((uint32_t)(16 * c.a_l) << 16);
    c.lane = threadIdx.x & 31;
    c.rank = rank;
    c.poison = &reinterpret_cast<T2Bars*>(smem)->poison;
    c.status = status;
    return c;
}

// A stored A buffer is handed to the leader's MMA warp; it also vouches for this CTA's half of the operand tile (the MMA
// reads both CTAs' halves).
__device__ __forceinline__ bool t2_hand_over(const T2Deq& c, uint32_t gis, uint32_t xready) {
    const uint32_t sb = c.sb, b = gis % T2_NA;
    tc_wait_st();
    if (!warp_saw(xready) && !warp_wait(T2_BAR(fullx, b), (gis / T2_NX) & 1, c.poison, c.status, 15, gis))
        return false;
    tc_fence_before();
    __syncwarp();
    if (c.lane == 0) {  // the barrier lives in the leader: a plain arrive there, a remote one from the peer
        if (c.rank == 0) bar_arrive(T2_BAR(a_full, b));
        else bar_arrive_leader(T2_BAR(a_full, b));
    }
    return true;
}

// n stages of an item's packed blocks, gi the running number of the first.  Returns the ring's write offset behind them, -1
// after an expired wait.
// A visit is a chain of barrier polls, shared-memory loads, arithmetic and tensor-memory stores, each hundreds of cycles
// long beside the MMAs' traffic, so polls are asked for early.  Registers are scarce: one half chunk is expanded at a time, and
// what spills in here goes to the L2 and back (the launch took 1.6 times as long).
template <int BITS, int G>
__device__ __forceinline__ int t2_dequant_run(const T2Deq& c, int n, uint32_t gi, int head) {
    constexpr int NG = KC / G;
    constexpr int CODE_HALF = 2048 * BITS, NEED = CODE_HALF + 512 * NG;
    const uint32_t sb = c.sb;
    RingPos pos;
    pos.head = head;
    const uint32_t end = gi + n;
    if (gi < end && (gi & 1) != (uint32_t)c.kh) {
        pos.place(NEED, T2_WRING);
        ++gi;
    }
    uint32_t ready = 0;
#pragma unroll 1
    for (; gi < end; gi += 2) {
        const uint32_t b = gi % T2_NA, dpar = ((gi / T2_NA) & 1) ^ 1;
        if (!warp_saw(ready) &&
            !warp_wait(T2_BAR(full, gi % T2_NW), (gi / T2_NW) & 1, c.poison, c.status, 13, gi))
            return -1;
        const uint32_t st = sb + T2_OFF_STAGE + pos.place(NEED, T2_WRING);
        uint32_t raw[16], prm[2][NG], regs[16];
        load_raw<BITS>(raw, st + c.a_l * (256 * BITS), c.lane);
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            const uint32_t a = st + CODE_HALF + (16 * c.a_l + (c.lane >> 2) + 8 * rh) * (4 * NG);
            if constexpr (NG == 2) {
                const uint2 v = lds64(a);
                prm[rh][0] = v.x;
                prm[rh][1] = v.y;
            } else {
                prm[rh][0] = lds32(a);
            }
        }
        const uint32_t a_free = bar_test(T2_BAR(done, b), dpar);
        ready = bar_test(T2_BAR(full, (gi + 2) % T2_NW), ((gi + 2) / T2_NW) & 1);
        t2_dequant_half<BITS, 0>(raw, prm[0][0], prm[1][0], regs);
        if (!warp_saw(a_free) && !warp_wait(T2_BAR(done, b), dpar, c.poison, c.status, 14, gi)) return -1;
        tc_fence_after();
        tc_st_x4(c.a_lanes + 64 * b, regs);
        t2_dequant_half<BITS, 1>(raw, prm[0][NG - 1], prm[1][NG - 1], regs);
        // the codes are used: their place in the ring can go back to the producer
        __syncwarp();
        if (c.lane == 0) bar_arrive(T2_BAR(empty, gi % T2_NW));
        const uint32_t xready = bar_test(T2_BAR(fullx, b), (gi / T2_NX) & 1);
        tc_st_x4(c.a_lanes + 64 * b + 32, regs);
        if (gi + 1 < end) pos.place(NEED, T2_WRING);
        if (!t2_hand_over(c, gi, xready)) return -1;
    }
    return pos.head;
}

// The same for n cached-channel stages: fp16 tiles [pool column][256 rows] -> A fragments -> tensor memory.
__device__ __forceinline__ int t2_pool_run(const T2Deq& c, int n, uint32_t gi, int head) {
    const uint32_t sb = c.sb;
    RingPos pos;
    pos.head = head;
#pragma unroll 1
    for (const uint32_t end = gi + n; gi < end; ++gi) {
        const uint32_t b = gi % T2_NA, st = sb + T2_OFF_STAGE + pos.place(T2_POOL_TILES, T2_WRING);
        if ((gi & 1) != (uint32_t)c.kh) continue;
        if (!warp_wait(T2_BAR(full, gi % T2_NW), (gi / T2_NW) & 1, c.poison, c.status, 13, gi) ||
            !warp_wait(T2_BAR(done, b), ((gi / T2_NA) & 1) ^ 1, c.poison, c.status, 14, gi))
            return -1;
        tc_fence_after();
        const int mi = c.lane >> 3, r = c.lane & 7;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            uint32_t af[4];
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(af[0]), "=r"(af[1]), "=r"(af[2]), "=r"(af[3])
                         : "r"(st + (j * 16 + (mi >> 1) * 8 + r) * POOL_TILE_PITCH +
                               (16 * (8 * c.rank + c.a_l) + (mi & 1) * 8) * 2)
                         : "memory");
            tc_st_x1(c.a_lanes + 64 * b + 8 * j, af[0], af[2], af[1], af[3]);
        }
        __syncwarp();
        if (c.lane == 0) bar_arrive(T2_BAR(empty, gi % T2_NW));  // the tiles are in registers / tensor memory
        if (!t2_hand_over(c, gi, 0)) return -1;
    }
    return pos.head;
}

// ---- MMA issue: the eight MMAs of a stage as one run behind one elect, operands warp-uniform ------------------------
// A cached-channel stage (main = 0) has two K steps; acc0 = 0: the first step starts from zero.
#define T2_MMA(pred, k, acc)                                        \
    "add.s64 bd, %2, " #k "*16;\n\tadd.s32 aa, %1, " #k "*8;\n\t" \
    "@" pred " tcgen05.mma.cta_group::2.kind::f16 [%0], [aa], bd, %3, " acc ";\n\t"
__device__ __forceinline__ void t2_mma_stage(uint32_t d, uint32_t a, uint64_t bd, uint32_t idesc, uint32_t acc0,
                                             uint32_t main) {
    asm volatile(
        "{\n\t.reg .pred p0, p1, q, m;\n\t.reg .b64 bd;\n\t.reg .b32 aa;\n\telect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 p1, 0, 0;\n\tsetp.ne.and.b32 m, %5, 0, q;\n\t"
        T2_MMA("q", 0, "p0") T2_MMA("q", 1, "p1") T2_MMA("m", 2, "p1") T2_MMA("m", 3, "p1") T2_MMA("m", 4, "p1")
        T2_MMA("m", 5, "p1") T2_MMA("m", 6, "p1") T2_MMA("m", 7, "p1") "}" ::"r"(d),
        "r"(a), "l"(bd), "r"(idesc), "r"(acc0), "r"(main)
        : "memory");
}

// MMA issuer of the pair: one warp of the leader CTA.  Its loop is what paces the pair at small token tiles: the MMAs of a
// stage run 4 cycles per token (512 for 125 rows), so neither a poll (200 to 400 cycles beside tensor-memory traffic even
// when the phase is long complete) nor an elect per MMA (700 cycles a stage) may stand between two stages: it asks for the
// next stage's A buffer before it issues this one's MMAs, and those are one run.  (A function of its own: inlined beside
// the other roles the compiler no longer sees that its operands are warp-uniform.)
__device__ __noinline__ void t2_mma_role(const T2Params& p, const T2Expert* tab, uint32_t sb, uint32_t tbase, int total,
                                         int n_kc, volatile int* poison) {
    int32_t* status = p.ws.status;
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    bool ok = true;
    int cursor = 0;
    uint32_t gi = 0, ic = 0;   // running stage number, items done by this cluster
    uint32_t ready = 0;
    int n_last = 0;            // width of the previous item
    // (the shuffles tell the compiler that the operands are warp-uniform)
    tbase = __shfl_sync(0xffffffffu, tbase, 0);
    sb = __shfl_sync(0xffffffffu, sb, 0);
    n_kc = __shfl_sync(0xffffffffu, n_kc, 0);
    total = __shfl_sync(0xffffffffu, total, 0);
    for (int g = cluster_id; g < total && ok; g += n_clusters, ++ic) {
        const T2Item w = t2_item(tab, g, cursor);
        cursor = __shfl_sync(0xffffffffu, cursor, 0);
        const int n_it = __shfl_sync(0xffffffffu, w.n_it, 0);
        const int n_mma = __shfl_sync(0xffffffffu, w.n_mma, 0);
        const uint32_t idesc = (1u << 4) | ((uint32_t)(n_mma >> 3) << 17) | ((256u >> 4) << 24);
        // Items of up to T2_SMALL tokens take the two halves of the accumulator columns in turn, so that one's epilogue runs
        // beside the other's MMAs; a larger one needs all of them.  Free once every epilogue warp of the pair has read them.
        if (ic >= 2) ok = warp_wait(T2_BAR(d_empty, ic & 1), ((ic - 2) >> 1) & 1, poison, status, 10, ic);
        if (ok && ic && (n_mma > T2_SMALL || n_last > T2_SMALL))
            ok = warp_wait(T2_BAR(d_empty, (ic - 1) & 1), ((ic - 1) >> 1) & 1, poison, status, 11, ic);
        n_last = n_mma;
        const uint32_t acc = tbase + (n_mma <= T2_SMALL && (ic & 1) ? T2_SMALL : 0);
        for (int it = 0; it < n_it && ok; ++it, ++gi) {
            const uint32_t b = gi % T2_NA;
            // A buffer b stored by the 16 dequant warps of the pair that own the stage; each also waited for its CTA's
            // operand tile before it arrived
            if (!warp_saw(ready)) {
                ok = warp_wait(T2_BAR(a_full, b), (gi / T2_NA) & 1, poison, status, 12, gi);
                if (!ok) break;
            }
            tc_fence_after();
            ready = bar_test(T2_BAR(a_full, (gi + 1) % T2_NA), ((gi + 1) / T2_NA) & 1);
            const bool main = it < n_kc;
            const uint32_t a0 = tbase + T2_COL_A + 64 * b;
            // operand tile: [row group][k octet 16][8][8], of a cached-channel stage [row group][k octet 4][8][8]
            const uint32_t xt = sb + T2_OFF_XRING + b * T2_XTILE;
            t2_mma_stage(acc, a0, tc_desc(xt, 128, main ? TC_TILE_BYTES : 512), idesc, it ? 1u : 0u, main ? 1u : 0u);
            tc2_commit_both_elect(T2_BAR(done, b));
        }
        if (ok) tc2_commit_both_elect(T2_BAR(d_full, ic & 1));
    }
}

// ---- epilogues, by the sixteen dequant warps ------------------------------------------------------------------------
// The tensor memory goes back to the leader's MMA warp with a warp's last load of it.  (Taking all accumulators into
// registers first would hand it back at once, but 64 more registers make the dequantization spill, see t2_dequant_run.)
__device__ __forceinline__ void t2_release_acc(uint32_t d_empty, int lane) {
    tc_wait_ld();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) bar_arrive_leader(d_empty);
}
// Gate/up: SwiGLU of one atom's eight hidden units (gate rows 0..7, up rows 8..15) x half `kh` of the tile's 32-token
// blocks -> operand tiles of the down GEMM.
__device__ __forceinline__ bool t2_epilogue_h(const T2Params& p, const T2Expert* tab, int g, int cursor, uint32_t tbase,
                                           uint32_t d_empty, int ic, int a_l, int rank, int kh, int lane) {
    const T2Item w = t2_item(tab, g, cursor);
    uint32_t acc = tbase + (w.n_mma <= T2_SMALL && (ic & 1) ? T2_SMALL : 0);
    bool clamped = false;
    const int nb = w.n_mma >> 5, cb0 = kh ? (nb + 1) >> 1 : 0, ncb = kh ? nb >> 1 : (nb + 1) >> 1;
    acc += ((uint32_t)(16 * a_l) << 16) + 32 * cb0;
    const int gid = lane >> 2, tid4 = lane & 3, odd = gid & 1;
    const int atom_g = 8 * rank + a_l;   // atom within the 256-row block
    const __half2 scl = __float2half2_rn(__uint_as_float((uint32_t)(127 + x_scale_exp(w.bits, 8 * atom_g + gid)) << 23));
    if (ncb == 0) t2_release_acc(d_empty, lane);
    int n_valid = w.n_valid - 32 * cb0 - 2 * tid4;
    const int to_bf16 = p.ws.h_bf16;
    // lanes gid and gid ^ 1 swap one value each, so that every lane stores one 32-bit pair (hidden gid & ~1, gid | 1) of ONE
    // token: even gid token 2 * tid4, odd gid the next one; 128 consecutive bytes a warp
    uint8_t* dst = p.ws.hbuf + tile_off(w.rb, w.t->row0, (w.tile0 >> 3) + 4 * cb0, p.ws.Rcap) + atom_g * 128 +
                   (2 * tid4 + odd) * 16 + (gid & ~1) * 2;
#pragma unroll 1
    for (int cb = 0; cb < ncb; ++cb, acc += 32, n_valid -= 32, dst += 4 * TC_TILE_BYTES) {
        uint32_t r[16];
        tc_ld_x4(acc, r);
        if (cb == ncb - 1) t2_release_acc(d_empty, lane);
        else tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n0 = 8 * j;
            float hs[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float v0 = __uint_as_float(r[4 * j + c]), v1 = __uint_as_float(r[4 * j + 2 + c]);
                float h = __fdividef(v0, 1.f + __expf(-v0)) * v1;
                if (n0 + c < n_valid) h = clamp_act(h, clamped);   // columns past the last token: ignored
                hs[c] = round_operand(h, to_bf16);
            }
            const float got = __shfl_xor_sync(0xffffffffu, odd ? hs[0] : hs[1], 4);   // what the partner does not store
            const __half2 pr = __hmul2(odd ? __floats2half2_rn(got, hs[1]) : __floats2half2_rn(hs[0], got), scl);
            if (n0 + odd < n_valid) *reinterpret_cast<__half2*>(dst + j * TC_TILE_BYTES) = pr;
        }
    }
    return clamped;
}
// Down: fp32 rows out, one weight row per lane (128 consecutive bytes a store), blocks of 16 tokens; cg: which of the four
// warps on this lane quarter.
__device__ __forceinline__ void t2_epilogue_y(const T2Params& p, const T2Expert* tab, int g, int cursor, uint32_t tbase,
                                           uint32_t d_empty, int ic, int q, int rank, int cg, int lane) {
    const T2Item w = t2_item(tab, g, cursor);
    uint32_t acc = tbase + (w.n_mma <= T2_SMALL && (ic & 1) ? T2_SMALL : 0);
    const size_t d = p.L->d;
    acc += ((uint32_t)(32 * q) << 16) + 16 * cg;
    int n_valid = w.n_valid - 16 * cg;
    if (n_valid <= 0) t2_release_acc(d_empty, lane);
    float* y = p.ws.ypart + (size_t)(w.t->row0 + w.tile0 + 16 * cg) * d + w.rb * RB + 128 * rank + 32 * q + lane;
#pragma unroll 1
    for (; n_valid > 0; n_valid -= 64, acc += 64) {
        uint32_t r[16];
        tc_ld_rows16(acc, r);
        if (n_valid <= 64) t2_release_acc(d_empty, lane);
        else tc_wait_ld();
#pragma unroll
        for (int c = 0; c < 16; ++c)
            if (c < n_valid) y[c * d] = __uint_as_float(r[c]);
        y += 64 * d;
    }
}

// ---- dequant warps, then epilogue (a function of its own, see t2_mma_role) ------------------------------------------
// warp -> (TMEM lane quarter q = warp % 4, 16-lane half of it = one atom, stage parity kh): a whole atom of every OTHER
// stage.  In the epilogue kh is the half of the token columns.
template <bool GATEUP, int G>
__device__ __noinline__ void t2_dequant_role(const T2Params& p, uint8_t* smem, uint32_t tbase, int total, int n_kc, int rank,
                                             int warp, int lane) {
    const T2Expert* tab = reinterpret_cast<const T2Expert*>(smem + T2_OFF_TAB);
    volatile int* poison = &reinterpret_cast<T2Bars*>(smem)->poison;
    const uint32_t sb = smem_u32(smem);
    const int q = warp & 3;
    int32_t* status = p.ws.status;
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    const T2Deq c = t2_deq(smem, tbase, rank, status);
    bool ok = true, clamped = false;
    int cursor = 0, cursor_nx = 0;
    uint32_t gi = 0, ic = 0;
    int head = 0;
    // The first stages of the NEXT item are dequantized before this item's epilogue: their A buffers come free while the last
    // MMAs of this item run.  Where both items have accumulators of their own all four buffers are filled, and the MMAs run on
    // through the epilogue; otherwise three, since the fourth comes free only with the last MMA (4096 tokens, short bursts: 2405 us
    // a pass with two, 2348 with three, 2372 with four).
    int lead_done = 0;                       // stages of the item already dequantized (as the previous item's lead)
    for (int g = cluster_id; g < total && ok; g += n_clusters, ++ic) {
        int bits, from = lead_done, to, bits_nx = 0;
        {
            const T2Item w = t2_item(tab, g, cursor);
            bits = w.bits;
            to = w.n_it;
            lead_done = 0;
            if (g + n_clusters < total) {
                const T2Item nx = t2_item(tab, g + n_clusters, cursor_nx);
                lead_done = min(nx.n_it, w.n_mma <= T2_SMALL && nx.n_mma <= T2_SMALL ? T2_NA : 3);
                bits_nx = nx.bits;
            }
        }
#pragma unroll 1
        for (int part = 0; part < 2 && ok; ++part) {
            const int n = min(to, n_kc) - from;
            if (n > 0) {
                switch (bits) {
                    case 2: head = t2_dequant_run<2, G>(c, n, gi, head); break;
                    case 3: head = t2_dequant_run<3, G>(c, n, gi, head); break;
                    case 4: head = t2_dequant_run<4, G>(c, n, gi, head); break;
                    case 6: head = t2_dequant_run<6, G>(c, n, gi, head); break;
                    default: head = t2_dequant_run<8, G>(c, n, gi, head); break;
                }
                gi += n;
            }
            const int n_pool = to - max(from, n_kc);
            if (n_pool > 0 && head >= 0) {
                head = t2_pool_run(c, n_pool, gi, head);
                gi += n_pool;
            }
            ok = head >= 0;
            bits = bits_nx;
            from = 0;
            to = lead_done;
        }
        if (ok) ok = warp_wait(T2_BAR(d_full, ic & 1), (ic >> 1) & 1, poison, status, 16, ic);
        tc_fence_after();
        if (ok) {
            const uint32_t d_empty = T2_BAR(d_empty, ic & 1);
            if constexpr (GATEUP)
                clamped |= t2_epilogue_h(p, tab, g, cursor, tbase, d_empty, ic, 2 * q + ((warp >> 2) & 1), rank, warp >> 3, lane);
            else
                t2_epilogue_y(p, tab, g, cursor, tbase, d_empty, ic, q, rank, warp >> 2, lane);
        }
    }
    if (clamped) atomicOr(status, STATUS_RANGE);
}

template <bool GATEUP, int G>
__device__ __forceinline__ void tc2_cta(const T2Params& p, uint8_t* smem, bool fills) {
    const LayerDev* L = p.L;
    const int K = GATEUP ? L->d : L->f;
    const int n_kc = K / KC;
    const int P_pad = L->P_pad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;

    T2Bars* B = reinterpret_cast<T2Bars*>(smem);
    T2Expert* tab = reinterpret_cast<T2Expert*>(smem + T2_OFF_TAB);
    uint8_t* wring = smem + T2_OFF_STAGE;
    uint8_t* xring = smem + T2_OFF_XRING;

    // After an expired wait nothing new starts.  Both CTAs of a pair read the same word (the preceding kernel has
    // completed, and every cluster of this persistent grid starts at launch), so they leave together, before any
    // barrier or tensor memory exists.  (Beside the fold kernel, which may write the word, the leader's answer holds.)
    if (!fills) {
        if (*p.ws.status & STATUS_TIMEOUT) return;
        pdl_trigger();   // the streaming kernel of the smaller experts may fill the SMs from here on
    }
    // Expert table (identical in both CTAs of the pair): experts above the row threshold contribute (token tiles x row
    // blocks) items.
    for (int i = threadIdx.x; i < p.n_experts; i += T2_THREADS) {
        const int e = L->order[i];
        const ExpertDev& ex = L->ex[e];
        T2Expert t;
        t.cnt = p.ws.counts[e];
        if (t.cnt <= p.ws.tc_min) t.cnt = 0;
        t.n_tt = (t.cnt + T2_N - 1) / T2_N;
        t.rows = t.n_tt > 0 ? ((t.cnt + t.n_tt - 1) / t.n_tt + 31) & ~31 : 0;   // equal tiles: a narrow one costs its dequantization all the same
        t.first = t.n_tt * p.n_rb;
        t.row0 = p.ws.off_pad[e];
        t.bits = ex.bits;
        t.blk_bytes = ex.blk_bytes;
        t.w = GATEUP ? ex.w13 : ex.w2;
        t.pool = reinterpret_cast<const uint8_t*>(ex.pool_hi);
        t.n_it = n_kc + (GATEUP && ex.switchable && L->sig_cnt[e] > 0 ? P_pad >> 5 : 0);
        tab[i] = t;
    }
    __syncthreads();
    if (warp == 0) {   // exclusive scan of the item counts
        int run = 0;
        for (int i0 = 0; i0 < p.n_experts; i0 += 32) {
            const int i = i0 + lane;
            const int n = i < p.n_experts ? tab[i].first : 0;
            int v = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += u;
            }
            if (i < p.n_experts) tab[i].first = run + v - n;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) tab[p.n_experts].first = run;
    }
    __syncthreads();
    int total = tab[p.n_experts].first;
    // Nothing for this pair: both CTAs see the same table and leave together, before the cluster barrier.
    if (cluster_id >= total) return;

    if (threadIdx.x == 0) {
        for (int i = 0; i < T2_NW; ++i) {
            mbar_init(&B->full[i], 1);
            mbar_init(&B->empty[i], T2_DEQ_WARPS / 2);
        }
        for (int i = 0; i < T2_NX; ++i) mbar_init(&B->fullx[i], 1);
        for (int i = 0; i < T2_NA; ++i) {
            mbar_init(&B->a_full[i], T2_DEQ_WARPS);  // 8 warps of each CTA per stage
            mbar_init(&B->done[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&B->d_full[i], 1);
            mbar_init(&B->d_empty[i], 2 * T2_DEQ_WARPS);
        }
        B->poison = 0;
        if (fills) B->off = *p.ws.status & STATUS_TIMEOUT;
        fence_barrier_init();
    }
    if (warp == T2_W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&B->tmem_base)),
                     "r"(T2_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers are initialised before anybody arrives remotely
    tc_fence_after();
    if (fills && ld_leader(&B->off)) total = 0;   // no role finds an item
    const uint32_t tbase = B->tmem_base;
    volatile int* poison = &B->poison;
    int32_t* status = p.ws.status;
    const uint8_t* xbase = GATEUP ? p.ws.xperm : p.ws.hbuf;
    // Every role walks the same items (static round-robin over the clusters) with its own running stage counter.
    int cursor = 0;
    uint32_t gi = 0;

    if (warp == T2_W_PROD) {
        // ---------------- weight producer (each CTA loads its own half block): one thread ----------------
        if (lane == 0) {
            bool ok = true;
            uint32_t tail = 0;
            int free_b = T2_WRING;
            RingPos pos;
            // ring offset of the next stage once it fits behind the oldest stage still in use
            auto acquire = [&](int need) -> int {
                const int pad = pos.head + need > T2_WRING ? T2_WRING - pos.head : 0;
                const int take = min(need + pad, T2_WRING);   // a stage that wraps in its own footprint takes all
                while (free_b < take || tail + T2_NW <= gi) {
                    const int t = tail % T2_NW;
                    if (!mbar_wait_bounded(&B->empty[t], (tail / T2_NW) & 1, poison, status, WAIT_LIMIT_NS, 17, (int)tail))
                        return -1;
                    free_b += B->size[t];
                    ++tail;
                }
                B->size[gi % T2_NW] = take;
                free_b -= take;
                return pos.place(need, T2_WRING);
            };
            for (int g = cluster_id; g < total && ok; g += n_clusters) {
                const T2Item w = t2_item(tab, g, cursor);
                const int code_half = 8 * atom_bytes(w.bits), prm_half = 128 * (KC / G) * 4, blk_bytes = w.t->blk_bytes;
                const uint8_t* blk = w.t->w + (size_t)w.rb * n_kc * blk_bytes;
                for (int it = 0; it < w.n_it; ++it, ++gi, blk += blk_bytes) {
                    const int o = acquire(it < n_kc ? code_half + prm_half : T2_POOL_TILES);
                    if (o < 0) { ok = false; break; }
                    uint8_t* st = wring + o;
                    uint64_t* bar = &B->full[gi % T2_NW];
                    if (it < n_kc) {
                        mbar_arrive_expect_tx(bar, (uint32_t)(code_half + prm_half));
                        bulk_g2s(st, blk + rank * code_half, (uint32_t)code_half, bar);
                        bulk_g2s(st + code_half, blk + block_code_bytes(w.bits) + rank * prm_half, (uint32_t)prm_half, bar);
                    } else {
                        // cached-channel stage: 32 pool columns (whole 256-row tiles: this CTA uses its 128 rows)
                        const int c0 = POOL_GROUP * (it - n_kc);
                        mbar_arrive_expect_tx(bar, (uint32_t)T2_POOL_TILES);
                        bulk_g2s(st, w.t->pool + pool_tile_off(w.rb, c0, P_pad),
                                 (uint32_t)T2_POOL_TILES, bar);
                    }
                }
            }
            if (!ok) {
                // let copies in flight land before the CTA's shared memory goes away
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 2000000ull) {
                }
            }
        }
        __syncwarp();
    } else if (warp == T2_W_PRODX) {
        // ---------------- operand producer: this CTA's half of the token tile, one slot per stage ----------------
        bool ok = true;
        for (int g = cluster_id; g < total && ok; g += n_clusters) {
            const T2Item w = t2_item(tab, g, cursor);
            const int half = w.n_mma >> 1, seg0 = w.t->row0;
            const int n_rg = (max(0, min(half, w.n_valid - rank * half)) + 7) >> 3;   // 8-row groups of this CTA's half that hold rows
            const int rg0 = (w.tile0 + rank * half) >> 3;                             // the first of them in the expert's segment
            for (int it = 0; it < w.n_it && ok; ++it, ++gi) {
                const int s = gi % T2_NX, ph = (gi / T2_NX) & 1;
                uint8_t* st = xring + (size_t)s * T2_XTILE;
                int okl = 1;
                if (lane == 0) okl = mbar_wait_bounded(&B->done[s], ph ^ 1, poison, status) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, okl, 0) != 0;
                if (!ok) break;
                if (lane == 0) {
                    if (it < n_kc) {
                        mbar_arrive_expect_tx(&B->fullx[s], (uint32_t)(n_rg * TC_TILE_BYTES));
                        if (n_rg > 0)
                            bulk_g2s(st, xbase + tile_off(it, seg0, rg0, p.ws.Rcap),
                                     (uint32_t)(n_rg * TC_TILE_BYTES), &B->fullx[s]);
                    } else {
                        mbar_arrive_expect_tx(&B->fullx[s], (uint32_t)(n_rg * 512));
                        if (n_rg > 0)
                            bulk_g2s(st, reinterpret_cast<const uint8_t*>(p.ws.xsig) +
                                             xpool_off(it - n_kc, seg0 + 8 * rg0, p.ws.Rcap),
                                     (uint32_t)(n_rg * 512), &B->fullx[s]);
                    }
                }
                __syncwarp();
            }
        }
        if (!ok && lane == 0) {
            const unsigned long long t0 = globaltimer_ns();
            while (globaltimer_ns() - t0 < 2000000ull) {
            }
        }
    } else if (warp == T2_W_MMA) {
        if (rank == 0) t2_mma_role(p, tab, smem_u32(smem), tbase, total, n_kc, poison);
    } else {
        t2_dequant_role<GATEUP, G>(p, smem, tbase, total, n_kc, rank, warp, lane);
    }
    // No CTA of the pair may exit (or free tensor memory) while its peer can still reach it.
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == T2_W_MMA) {
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(T2_TMEM_COLS) : "memory");
    }
}

template <bool GATEUP, int G>
__global__ void __launch_bounds__(T2_THREADS, 1) ffn_tc2_kernel(const __grid_constant__ T2Params p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    if (p.fills) {
        pdl_trigger();
        pdl_early_start();
    } else {
        pdl_wait();
    }
    tc2_cta<GATEUP, G>(p, smem, p.fills != 0);
    // one pair that waits is enough: the grid completes behind it
    if (p.fills && blockIdx.x < 2) pdl_wait();
}

// Persistent grid: as many CTA pairs as can be resident at once on the current device (pairs must share a TPC; not
// every SM may be pairable), so that the static round-robin over clusters has no second wave.  Also raises the
// kernels' shared-memory limit.  Called once per context at pack time, with the layer's device current.
template <bool GATEUP, int G>
static cudaError_t t2_setup_one(int n_sms, int* clusters_out) {
    cudaError_t err =
        cudaFuncSetAttribute(ffn_tc2_kernel<GATEUP, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, T2_SMEM_BYTES);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_sms & ~1));
    cfg.blockDim = dim3(T2_THREADS);
    cfg.dynamicSmemBytes = T2_SMEM_BYTES;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int m = 0;
    err = cudaOccupancyMaxActiveClusters(&m, ffn_tc2_kernel<GATEUP, G>, &cfg);
    if (err != cudaSuccess) return err;
    if (m < 1) return cudaErrorInvalidConfiguration;
    *clusters_out = m < n_sms / 2 ? m : n_sms / 2;
    return cudaSuccess;
}

// clusters_out[0]: down launch, clusters_out[1]: gate/up launch.
cudaError_t setup_ffn_tc2(int n_sms, int G, int* clusters_out) {
    cudaError_t err = G == 64 ? t2_setup_one<false, 64>(n_sms, &clusters_out[0]) : t2_setup_one<false, 128>(n_sms, &clusters_out[0]);
    if (err != cudaSuccess) return err;
    return G == 64 ? t2_setup_one<true, 64>(n_sms, &clusters_out[1]) : t2_setup_one<true, 128>(n_sms, &clusters_out[1]);
}

// n_rb: 256-row weight blocks; n_experts: experts in L->order; n_clusters: CTA pairs of the persistent grid
// (from setup_ffn_tc2 on this device).
cudaError_t launch_ffn_tc2(const LayerDev* L, const WsDev& ws, int gateup, int n_rb, int n_experts, int n_clusters,
                           int fills, int G, cudaStream_t st) {
    T2Params p;
    p.L = L;
    p.ws = ws;
    p.n_rb = n_rb;
    p.n_experts = n_experts;
    p.fills = fills;
    if (n_clusters < 1) return cudaErrorInvalidConfiguration;
    auto launch = [&](auto kern) {
        return launch_pdl_cluster(kern, dim3((unsigned)(2 * n_clusters)), dim3(T2_THREADS), (size_t)T2_SMEM_BYTES, 2u, st, p);
    };
    if (gateup) return G == 64 ? launch(ffn_tc2_kernel<true, 64>) : launch(ffn_tc2_kernel<true, 128>);
    return G == 64 ? launch(ffn_tc2_kernel<false, 64>) : launch(ffn_tc2_kernel<false, 128>);
}

}  // namespace dyn

// Grouped dequant-GEMM for middle-sized batches (experts of a few dozen rows; beside the pair kernel, which takes popular
// ones): tcgen05 with the INTEGER CODES as the A operand and scale / zero-point folded in once per quantization group.
//
// What bounds it.  A 256 x 128 weight block is 9 to 34 KB; at the copy bandwidth of HBM an SM's share of it takes 390
// (2 bits) to 1440 cycles (8 bits).  Its sixteen MMAs (two tiles of M = 128 rows, K = 16 each) run N / 2 cycles each,
// 160 for 16 tokens and 512 for 64.  Codes become fp16 subnormals q * 2^(o-24) with one logic operation per register
// pair (layout.cuh), a third of the work of forming the fp16 weight s*q + m as the pair kernel does, and the fold is
// two packed FMAs per pair of accumulators.  What is left to bind are the hand-overs: a barrier poll takes 200 to 400
// cycles beside tensor-memory traffic even when its phase is long complete, so the roles ask for their next stage
// before they work on the current one, and the MMAs of a stage are issued as one run behind one elect (an elect per
// MMA costs 34 to 60 cycles each).  About 1150 cycles a stage at 64 tokens, 1340 at 139 (4096 x 14336 layer).
//
// Work item = (expert, 256-row weight block, tile of <= FF_NT tokens, K split of the down GEMM), dealt round-robin over
// one persistent CTA per SM; ring, A buffers and accumulators live across items.  18 warps:
//   warps 0-7 expand  : two groups of four (one warp per lane quarter), a group takes every other stage: the codes of
//                       four atoms (16 rows x 128 k) -> A buffer in tensor memory.
//   warps 8-15 fold   : (lane quarter, row tile) each, one weight row per lane; per quantization group
//                           total += (s * 2^(24-bias)) * acc + m * sum_k x_k          (exact codes, fp32)
//                       and at the end of an item its epilogue: SwiGLU -> h as operand tiles of the down GEMM with
//                       their group sums, or fp32 rows out.
//   warp 16 producer  : ONE thread; per stage one bulk copy of the packed block and one of the operand tile into a
//                       byte-granular ring (up to 16 stages in flight).  The offsets follow from the sizes alone, so
//                       every role computes them itself.
//   warp 17 MMA       : sixteen MMAs and one commit per stage.
// Tensor memory: FF_NA A buffers of 128 columns, then FF_NB accumulator buffers of 2 x FF_NT columns.
// Every wait is bounded; after an expired wait a role leaves its loops and the CTA meets at the final barrier.
#include <cstddef>
#include <type_traits>

#include "common.cuh"
#include "expand.cuh"
#include "layout.cuh"
#include "tcgen05.cuh"

namespace dyn {

constexpr int FF_EXP_WARPS = 8;
constexpr int FF_FOLD_WARPS = 8;
constexpr int FF_W_PROD = FF_EXP_WARPS + FF_FOLD_WARPS, FF_W_MMA = FF_W_PROD + 1;
constexpr int FF_THREADS = (FF_W_MMA + 1) * 32;
constexpr int FF_Q = 16;                  // most stages in flight
constexpr int FF_NT = 64;                   // rows of an expert per pass
constexpr int FF_NA = 2, FF_NB = 2;       // A buffers of 128 columns, accumulator buffers of 2 * FF_NT, in tensor memory
constexpr int FF_HDR = 1024;              // barriers and ring bookkeeping
constexpr int FF_HPITCH = 272;            // bytes per token row of the h tile (128 hidden units fp16 + pad)
constexpr int FF_SMEM = 226 * 1024;
constexpr uint32_t FF_TMEM_COLS = 512;
static_assert(128 * FF_NA + 2 * FF_NT * FF_NB <= (int)FF_TMEM_COLS, "tensor memory");
constexpr int FF_RG = 8 * XROW;   // operand tile of eight rows with its group sums behind it

struct FfParams {
    const LayerDev* L;
    WsDev ws;
    int n_rb;        // 256-row weight blocks of this GEMM
    int n_experts;   // experts listed in L->order
    int ksplit;      // K splits (down GEMM)
    long long split_stride;
    int off_h, off_ring, ring_bytes;   // shared-memory layout behind the header and the expert table
};

struct FfExpert {
    const uint8_t* w;     // packed blocks
    const uint8_t* pool;  // forward-ready tiles of the cached channels
    int first;            // first item
    int cnt, row0, tile_rows, n_tt, bits, blk_bytes, n_pool;
};

struct FfShared {
    uint64_t full[FF_Q];      // block and operand tile landed
    uint64_t empty[FF_Q];     // 8 fold warps are done with the stage (they follow the MMAs, which follow the expand warps)
    uint64_t done[FF_Q];      // the stage's MMAs are complete (commit)
    uint64_t a_full[FF_NA];      // the 4 expand warps of the stage stored A buffer b
    uint64_t acc_empty[FF_NB];   // 8 fold warps have read accumulator buffer i
    uint64_t hready, hfree;   // the item's h tile is written / read by the 8 fold warps
    int size[FF_Q];           // producer only: ring bytes of the stage in slot q
    uint32_t tmem_base;
    volatile int poison;
};
static_assert(sizeof(FfShared) <= FF_HDR, "header too small");

struct FfItem {
    const uint8_t* w;     // first packed block of the item's row block and K split
    const uint8_t* pool;
    int rb, split, n_valid, n_mma, row0, kc0, n_main, n_pool, bits, blk_bytes;
    __device__ __forceinline__ int need() const { return blk_bytes + n_mma * XROW; }   // ring bytes of a main stage
    __device__ __forceinline__ int need_pool() const { return POOL_GROUP * POOL_TILE_PITCH + n_mma * XPOOL_ROW; }
};

__device__ __forceinline__ FfItem ff_item(int ksplit, const FfExpert* tab, int g, int& cur, int n_kc) {
    while (g >= tab[cur + 1].first) ++cur;
    const FfExpert& t = tab[cur];
    const int local = g - t.first;
    const int rs = t.n_tt > 1 ? local / t.n_tt : local, tt = local - rs * t.n_tt;   // tiles of one weight block are neighbours: they share L2 lines
    FfItem it;
    if (ksplit > 1) {
        it.rb = rs / ksplit;
        it.split = rs - it.rb * ksplit;
        it.kc0 = (it.split * n_kc) / ksplit;
        it.n_main = ((it.split + 1) * n_kc) / ksplit - it.kc0;
    } else {
        it.rb = rs;
        it.split = 0;
        it.kc0 = 0;
        it.n_main = n_kc;
    }
    it.n_valid = min(t.tile_rows, t.cnt - tt * t.tile_rows);
    it.n_mma = (it.n_valid + 15) & ~15;
    it.row0 = t.row0 + tt * t.tile_rows;
    it.bits = t.bits;
    it.blk_bytes = t.blk_bytes;
    it.n_pool = t.n_pool;
    it.w = t.w + ((size_t)it.rb * n_kc + it.kc0) * t.blk_bytes;
    it.pool = t.pool;
    return it;
}

__device__ __forceinline__ FfItem ff_item_uni(int ksplit, const FfExpert* tab, int g, int& cur, int n_kc) {
    FfItem it = ff_item(ksplit, tab, g, cur, n_kc);
    cur = __shfl_sync(0xffffffffu, cur, 0);
    it.rb = __shfl_sync(0xffffffffu, it.rb, 0);
    it.split = __shfl_sync(0xffffffffu, it.split, 0);
    it.n_valid = __shfl_sync(0xffffffffu, it.n_valid, 0);
    it.n_mma = __shfl_sync(0xffffffffu, it.n_mma, 0);
    it.row0 = __shfl_sync(0xffffffffu, it.row0, 0);
    it.n_main = __shfl_sync(0xffffffffu, it.n_main, 0);
    it.n_pool = __shfl_sync(0xffffffffu, it.n_pool, 0);
    it.bits = __shfl_sync(0xffffffffu, it.bits, 0);
    it.blk_bytes = __shfl_sync(0xffffffffu, it.blk_bytes, 0);
    return it;
}

// A role's place in a cycle of N barriers: index and parity of the round.  A wait for the round BEFORE (parity ^ 1)
// passes at once in the first round.
template <int N>
struct FfCycle {
    uint32_t i = 0, par = 0;
    __device__ __forceinline__ void next() {
        ++i;
        if (i == N) {
            i = 0;
            par ^= 1;
        }
    }
};
// A role's place in the stage sequence: running stage number (slot si % FF_Q, parity (si / FF_Q) & 1) and ring offset.
struct FfPos : RingPos {
    uint32_t si = 0;
};
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ void lds_sums(uint32_t a, uint64_t& x, uint64_t& y) {   // four fp32 as two pairs
    asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];" : "=l"(x), "=l"(y) : "r"(a) : "memory");
}
// barrier offsets from the CTA's shared-memory base
#define FF_BAR(field, i) (sb + (uint32_t)offsetof(FfShared, field) + 8u * (uint32_t)(i))
// ---- MMA issue: runs of instructions behind one elect, operands warp-uniform ------------------------------------
#define FF_MMA(pred, d, a, k, acc)                                \
    "add.s64 bd, %4, " #k "*16;\n\tadd.s32 aa, " a ", " #k "*8;\n\t" \
    "@" pred " tcgen05.mma.cta_group::1.kind::f16 [" d "], [aa], bd, %5, " acc ";\n\t"
#define FF_MMA8(d0, d1, a, acc4)                                                               \
    FF_MMA("q", d0, a, 0, "p0") FF_MMA("q", d0, a, 1, "p1") FF_MMA("m", d0, a, 2, "p1")        \
    FF_MMA("m", d0, a, 3, "p1") FF_MMA("m", d1, a, 4, acc4) FF_MMA("m", d1, a, 5, "p1")        \
    FF_MMA("m", d1, a, 6, "p1") FF_MMA("m", d1, a, 7, "p1")
#define FF_HEAD \
    "{\n\t.reg .pred p0, p1, pz, q, m;\n\t.reg .b64 bd;\n\t.reg .b32 aa, a1, d2, d3;\n\telect.sync _|q, 0xffffffff;\n\t" \
    "setp.ne.b32 p0, %6, 0;\n\tsetp.eq.b32 p1, 0, 0;\n\tsetp.ne.b32 pz, 0, 0;\n\tsetp.ne.and.b32 m, %7, 0, q;\n\t" \
    "add.s32 a1, %2, 64;\n\tadd.s32 d2, %0, %3;\n\tadd.s32 d3, %1, %3;\n\t"
// The MMAs of a stage: two row tiles (A columns a, a + 64; accumulators d.., d.. + nt) x eight K steps; the first group
// of 64 k goes to d0, the second to d1 (G = 128: d1 = d0, one group).  A cached-channel stage (main = 0) has two K
// steps; acc0 = 0: the first step starts from zero.
template <int G>
__device__ __forceinline__ void ff_mma_stage(uint32_t d0, uint32_t d1, uint32_t a, uint32_t nt, uint64_t bd,
                                             uint32_t idesc, uint32_t acc0, uint32_t main) {
    if constexpr (G == 128) {
        asm volatile(FF_HEAD FF_MMA8("%0", "%1", "%2", "p1") FF_MMA8("d2", "d3", "a1", "p1") "}" ::"r"(d0), "r"(d1), "r"(a),
                     "r"(nt), "l"(bd), "r"(idesc), "r"(acc0), "r"(main)
                     : "memory");
    } else {
        asm volatile(FF_HEAD FF_MMA8("%0", "%1", "%2", "pz") FF_MMA8("d2", "d3", "a1", "pz") "}" ::"r"(d0), "r"(d1), "r"(a),
                     "r"(nt), "l"(bd), "r"(idesc), "r"(acc0), "r"(main)
                     : "memory");
    }
}

// ---- expand: codes of two atoms of every other stage -> A buffer ---------------------------------------------------
template <int BITS>
__device__ __forceinline__ void ff_load_codes(Codes<BITS> (&c)[2], uint32_t atom, int lane) {   // both half chunks
    uint32_t raw[16];
    load_raw<BITS>(raw, atom, lane);
    codes_of<BITS, 0>(c[0], raw);
    codes_of<BITS, 1>(c[1], raw);
}

template <int BITS>
__device__ __forceinline__ void ff_store_atom(const Codes<BITS> (&cd)[2], uint32_t a_cols) {
    uint32_t regs[32];
    auto step = [&](auto S8c) {
        constexpr int S8 = decltype(S8c)::value;
        uint32_t af[4];
        expand<BITS, (S8 & 3)>(cd[S8 >> 2], af);
        // fragment (rowhalf, h) -> TMEM register order of the 16x256b shape: (row, col pair)
        regs[4 * S8 + 0] = af[0];
        regs[4 * S8 + 1] = af[2];
        regs[4 * S8 + 2] = af[1];
        regs[4 * S8 + 3] = af[3];
    };
    step(std::integral_constant<int, 0>{});
    step(std::integral_constant<int, 1>{});
    step(std::integral_constant<int, 2>{});
    step(std::integral_constant<int, 3>{});
    step(std::integral_constant<int, 4>{});
    step(std::integral_constant<int, 5>{});
    step(std::integral_constant<int, 6>{});
    step(std::integral_constant<int, 7>{});
    tc_st_x8(a_cols, regs);
}

// One item on a warp that owns lane quarter q (two atoms) of both row tiles in the stages of parity kh.
template <int BITS>
__device__ __forceinline__ bool ff_expand_item(const FfItem& im, FfShared* S, uint32_t sb, uint32_t ring, int cap,
                                               uint32_t a_lanes, int q, int kh, int lane, FfPos& pos, uint32_t& ready,
                                               int32_t* status) {
    const int n_st = im.n_main + im.n_pool;
    const int need = im.need(), need_pool = im.need_pool();
    for (int it = 0; it < n_st; ++it, ++pos.si) {
        const uint32_t st = ring + pos.place(it < im.n_main ? need : need_pool, cap);
        const uint32_t si = pos.si;
        if ((si & 1) != (uint32_t)kh) continue;
        const uint32_t b = si % FF_NA, u = si - FF_NA;
        if (!warp_saw(ready) &&
            !warp_wait(FF_BAR(full, si % FF_Q), (si / FF_Q) & 1, &S->poison, status, 1, si))
            return false;
        // the MMAs that read this A buffer last must be complete before it is written
        uint32_t a_free = 1;
        if (si >= FF_NA) a_free = bar_test(FF_BAR(done, u % FF_Q), (u / FF_Q) & 1);
        ready = bar_test(FF_BAR(full, (si + 2) % FF_Q), ((si + 2) / FF_Q) & 1);
        const uint32_t a_cols = a_lanes + 128 * b;
        if (it < im.n_main) {
            constexpr int GRP = BITS >= 6 ? 2 : 4;   // atoms whose codes are in registers at a time
#pragma unroll
            for (int a0 = 0; a0 < 4; a0 += GRP) {
                Codes<BITS> cd[GRP][2];
#pragma unroll
                for (int a = 0; a < GRP; ++a)
                    ff_load_codes<BITS>(cd[a], st + (8 * ((a0 + a) >> 1) + 2 * q + (a & 1)) * (256 * BITS), lane);
                if (a0 == 0) {
                    if (!warp_saw(a_free) &&
                        !warp_wait(FF_BAR(done, u % FF_Q), (u / FF_Q) & 1, &S->poison, status, 2, si))
                        return false;
                    tc_fence_after();
                }
#pragma unroll
                for (int a = 0; a < GRP; ++a)
                    ff_store_atom<BITS>(cd[a], a_cols + 64 * ((a0 + a) >> 1) + ((uint32_t)(a & 1) << 20));
            }
        } else {
            // cached-channel stage: fp16 tiles [pool column][256 rows] -> A fragments
            if (!warp_saw(a_free) &&
                !warp_wait(FF_BAR(done, u % FF_Q), (u / FF_Q) & 1, &S->poison, status, 2, si))
                return false;
            tc_fence_after();
            const int mi = lane >> 3, r = lane & 7;
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint32_t af[4];
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(af[0]), "=r"(af[1]), "=r"(af[2]), "=r"(af[3])
                                 : "r"(st + (j * 16 + (mi >> 1) * 8 + r) * POOL_TILE_PITCH +
                                       (16 * (8 * (a >> 1) + 2 * q + (a & 1)) + (mi & 1) * 8) * 2)
                                 : "memory");
                    tc_st_x1(a_cols + 64 * (a >> 1) + ((uint32_t)(a & 1) << 20) + 8 * j, af[0], af[2], af[1], af[3]);
                }
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(FF_BAR(a_full, b));
    }
    return true;
}

// What the roles share.
struct FfRole {
    FfShared* S;
    const FfExpert* tab;
    uint32_t sb, ring, tbase;
    int total, n_kc;
};

// The expand and fold roles are functions of their own: with everything inlined the compiler of the gate/up variant no
// longer saw that the operands of the MMA role are warp-uniform.
__device__ __noinline__ void ff_expand_role(const FfParams& p, FfRole R, int warp, int lane) {
    const int q = warp & 3, kh = warp >> 2;
    const uint32_t a_lanes = R.tbase + ((uint32_t)(32 * q) << 16);
    const int cap = p.ring_bytes;
    int32_t* status = p.ws.status;
    bool ok = true;
    uint32_t ready = 0;
    int cur = 0;
    FfPos pos;
    for (int g = blockIdx.x; g < R.total && ok; g += gridDim.x) {
        const FfItem im = ff_item_uni(p.ksplit, R.tab, g, cur, R.n_kc);
        switch (im.bits) {
            case 2: ok = ff_expand_item<2>(im, R.S, R.sb, R.ring, cap, a_lanes, q, kh, lane, pos, ready, status); break;
            case 3: ok = ff_expand_item<3>(im, R.S, R.sb, R.ring, cap, a_lanes, q, kh, lane, pos, ready, status); break;
            case 4: ok = ff_expand_item<4>(im, R.S, R.sb, R.ring, cap, a_lanes, q, kh, lane, pos, ready, status); break;
            case 6: ok = ff_expand_item<6>(im, R.S, R.sb, R.ring, cap, a_lanes, q, kh, lane, pos, ready, status); break;
            default: ok = ff_expand_item<8>(im, R.S, R.sb, R.ring, cap, a_lanes, q, kh, lane, pos, ready, status); break;
        }
    }
}

// ---- fold: one item on one (lane quarter, row tile) warp, NC columns (n_mma rounded up to an instantiated width) ----
template <bool GATEUP, int NC, int G>
__device__ __forceinline__ bool ff_fold_item(const FfParams& p, const FfItem& im, FfShared* S, uint32_t sb, uint32_t ring,
                                             uint8_t* htile, uint32_t acc_lanes, int q, int mt, int fw, int lane,
                                             int ic, FfPos& pos, FfCycle<FF_NB>& acb, uint32_t& ready, bool& clamped) {
    constexpr int NG = KC / G;
    volatile int* poison = &S->poison;
    int32_t* status = p.ws.status;
    const int row = 128 * mt + 32 * q + lane;   // row of the block
    const float unscale = __uint_as_float((uint32_t)(127 + 24 - x_scale_bias(im.bits)) << 23);
    const uint32_t prm_off = block_code_bytes(im.bits) + row * (NG * 4), sum_off = im.blk_bytes + TC_TILE_BYTES;
    const int need = im.need();
    uint64_t total[NC / 2];
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) total[i] = 0ull;

    for (int it = 0; it < im.n_main; ++it, ++pos.si) {
        const uint32_t st = ring + pos.place(need, p.ring_bytes);
        const uint32_t slot = pos.si % FF_Q, par = (pos.si / FF_Q) & 1;
        // zero-point times the group sums, as soon as the copies have landed
        if (!warp_saw(ready) && !warp_wait(FF_BAR(full, slot), par, poison, status, 3, pos.si)) return false;
        const uint32_t done = bar_test(FF_BAR(done, slot), par);
        ready = bar_test(FF_BAR(full, (pos.si + 1) % FF_Q), ((pos.si + 1) / FF_Q) & 1);
        uint64_t s2[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const uint32_t pw = lds32(st + prm_off + 4 * g);
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&pw));
            const float s = f.x * unscale;
            s2[g] = pack2(s, s);
            const uint64_t m2 = pack2(f.y, f.y);
#pragma unroll
            for (int c = 0; c < NC; c += 4) {
                uint64_t xa, xb;
                lds_sums(st + sum_off + (c >> 3) * FF_RG + g * 32 + (c & 7) * 4, xa, xb);
                total[c / 2] = fma2(m2, xa, total[c / 2]);
                total[c / 2 + 1] = fma2(m2, xb, total[c / 2 + 1]);
            }
        }
        if (!warp_saw(done) && !warp_wait(FF_BAR(done, slot), par, poison, status, 4, pos.si)) return false;
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < NG; ++g, acb.next()) {
            const uint32_t acc = acc_lanes + acb.i * (2 * FF_NT);
            uint32_t r[2][16];
            tc_ld_rows16(acc, r[0]);
#pragma unroll
            for (int c0 = 0; c0 < NC; c0 += 16) {
                tc_wait_ld();
                const uint32_t (&rr)[16] = r[(c0 / 16) & 1];
                if (c0 + 16 < NC) {
                    tc_ld_rows16(acc + c0 + 16, r[(c0 / 16 + 1) & 1]);
                } else {   // the buffer is read: hand it back to the MMA warp, and the stage to the producer
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        bar_arrive(FF_BAR(acc_empty, acb.i));
                        if (g == NG - 1) bar_arrive(FF_BAR(empty, slot));
                    }
                }
#pragma unroll
                for (int c = 0; c < 16; c += 2)
                    total[(c0 + c) / 2] =
                        fma2(s2[g], pack2(__uint_as_float(rr[c]), __uint_as_float(rr[c + 1])), total[(c0 + c) / 2]);
            }
        }
    }
    if constexpr (GATEUP) {
        if (im.n_pool > 0) {
            // all cached-channel stages accumulate into one buffer (values already scaled): one fold after the last
            for (int it = 0; it < im.n_pool; ++it, ++pos.si) {
                const uint32_t slot = pos.si % FF_Q;
                pos.place(im.need_pool(), p.ring_bytes);
                if (!warp_wait(FF_BAR(done, slot), (pos.si / FF_Q) & 1, poison, status, 4, pos.si)) return false;
                if (lane == 0) bar_arrive(FF_BAR(empty, slot));
            }
            ready = 0;
            tc_fence_after();
            const uint32_t acc = acc_lanes + acb.i * (2 * FF_NT);
            const uint64_t one2 = pack2(1.f, 1.f);
#pragma unroll
            for (int c0 = 0; c0 < NC; c0 += 16) {
                uint32_t r[16];
                tc_ld_rows16(acc + c0, r);
                tc_wait_ld();
#pragma unroll
                for (int c = 0; c < 16; c += 2)
                    total[(c0 + c) / 2] =
                        fma2(one2, pack2(__uint_as_float(r[c]), __uint_as_float(r[c + 1])), total[(c0 + c) / 2]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(FF_BAR(acc_empty, acb.i));
            acb.next();
        }
        // SwiGLU.  Lanes l (gate row) and l ^ 8 (the matching up row) split the columns between them: the gate lane
        // takes the first half, the up lane the second, one value each crosses per column.
        if (ic && !warp_wait(FF_BAR(hfree, 0), (ic - 1) & 1, poison, status, 5, ic)) return false;
        const bool up = (lane & 8) != 0;
        const int hid = 64 * mt + 8 * (2 * q + (lane >> 4)) + (lane & 7);   // hidden unit within the block's 128
#pragma unroll
        for (int i = 0; i < NC / 4; ++i) {
            float a[2], b[2];
            unpack2(total[i], a[0], a[1]);
            unpack2(total[i + NC / 4], b[0], b[1]);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float got = __shfl_xor_sync(0xffffffffu, up ? a[c] : b[c], 8);
                const float ga = up ? got : a[c], ua = up ? b[c] : got;
                const int n = 2 * i + c + (up ? NC / 2 : 0);
                float h = __fdividef(ga, 1.f + __expf(-ga)) * ua;
                if (n < im.n_valid) h = clamp_act(h, clamped);   // columns past the last token: ignored
                h = round_operand(h, p.ws.h_bf16);
                if (n < im.n_valid) *reinterpret_cast<__half*>(htile + n * FF_HPITCH + hid * 2) = __float2half_rn(h);
            }
        }
        __syncwarp();
        if (lane == 0) bar_arrive(FF_BAR(hready, 0));
        if (!warp_wait(FF_BAR(hready, 0), ic & 1, poison, status, 6, ic)) return false;
        // h of eight hidden units of one token per thread: operand tile of the down GEMM, scaled for its codes
        const int t = 32 * fw + lane;
        const int oct = t & 15;
        __half2 sc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            sc[i] = __float2half2_rn(__uint_as_float((uint32_t)(127 + x_scale_exp(im.bits, 8 * oct + 2 * i)) << 23));
        for (int n0 = 0; n0 < im.n_valid; n0 += FF_FOLD_WARPS * 2) {
            const int n = n0 + (t >> 4);
            const bool in = n < im.n_valid;
            uint4 hv = make_uint4(0u, 0u, 0u, 0u);
            if (in) hv = *reinterpret_cast<const uint4*>(htile + n * FF_HPITCH + oct * 16);
            __half2* hp = reinterpret_cast<__half2*>(&hv);
            float sum = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(hp[i]);
                sum += f.x + f.y;
                hp[i] = __hmul2(hp[i], sc[i]);
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (G == 128) sum += __shfl_xor_sync(0xffffffffu, sum, 8);
            if (in) {
                const int r = im.row0 + n;
                uint8_t* dst = p.ws.hbuf + act_off(im.rb, r & ~7, p.ws.Rcap);
                *reinterpret_cast<uint4*>(dst + oct * 128 + (r & 7) * 16) = hv;
                if ((oct & 7) == 0) *reinterpret_cast<float*>(dst + TC_TILE_BYTES + (oct >> 3) * 32 + (r & 7) * 4) = sum;
            }
        }
        __syncwarp();
        if (lane == 0) bar_arrive(FF_BAR(hfree, 0));
    } else {
        float* yb = p.ws.ypart + (size_t)im.split * p.split_stride + (size_t)im.row0 * p.L->d + im.rb * RB + row;
        const size_t d = p.L->d;
#pragma unroll
        for (int i = 0; i < NC / 2; ++i) {
            float a, b;
            unpack2(total[i], a, b);
            const int n = 2 * i;
            if (n < im.n_valid) yb[n * d] = a;
            if (n + 1 < im.n_valid) yb[(n + 1) * d] = b;
        }
    }
    return true;
}

template <bool GATEUP, int G>
__device__ __noinline__ void ff_fold_role(const FfParams& p, FfRole R, uint8_t* htile, int fw, int lane) {
    const int q = fw & 3, mt = fw >> 2;
    const uint32_t acc_lanes = R.tbase + 128 * FF_NA + mt * FF_NT + ((uint32_t)(32 * q) << 16);
    bool ok = true, clamped = false;
    FfCycle<FF_NB> acb;
    uint32_t ready = 0;
    int ic = 0, cur = 0;
    FfPos pos;
    for (int g = blockIdx.x; g < R.total && ok; g += gridDim.x, ++ic) {
        const FfItem im = ff_item_uni(p.ksplit, R.tab, g, cur, R.n_kc);
        if (im.n_mma <= 16)
            ok = ff_fold_item<GATEUP, 16, G>(p, im, R.S, R.sb, R.ring, htile, acc_lanes, q, mt, fw, lane, ic, pos, acb, ready, clamped);
        else if (im.n_mma <= 32)
            ok = ff_fold_item<GATEUP, 32, G>(p, im, R.S, R.sb, R.ring, htile, acc_lanes, q, mt, fw, lane, ic, pos, acb, ready, clamped);
        else if (im.n_mma <= 48)
            ok = ff_fold_item<GATEUP, 48, G>(p, im, R.S, R.sb, R.ring, htile, acc_lanes, q, mt, fw, lane, ic, pos, acb, ready, clamped);
        else
            ok = ff_fold_item<GATEUP, FF_NT, G>(p, im, R.S, R.sb, R.ring, htile, acc_lanes, q, mt, fw, lane, ic, pos, acb, ready, clamped);
    }
    if (clamped) atomicOr(p.ws.status, STATUS_RANGE);
}

// ---- MMA issuer (a function of its own, see ff_expand_role) ---------------------------------------------------------
template <int G>
__device__ __noinline__ void ff_mma_role(const FfParams& p, FfRole R) {
    FfShared* S = R.S;
    const FfExpert* tab = R.tab;
    const uint32_t sb = R.sb, ring_a = R.ring, tbase = R.tbase;
    const int total = R.total, n_kc = R.n_kc, cap = p.ring_bytes;
    int32_t* status = p.ws.status;
    volatile int* poison = &S->poison;
    int cur = 0;
    FfPos pos;
    // ---------------- MMA issuer: warp-uniform, one elected lane issues ----------------
    // (A stored A buffer vouches for the stage's operand tile: the expand warps waited for it.)
    bool ok = true;
    FfCycle<FF_NA> ab;
    FfCycle<FF_NB> acb;
    uint32_t ready = 0;   // the next stage's barriers, asked for before this stage's MMAs are issued
    const uint32_t acc0 = tbase + 128 * FF_NA;
    for (int g = blockIdx.x; g < total && ok; g += gridDim.x) {
        const FfItem im = ff_item_uni(p.ksplit, tab, g, cur, n_kc);
        const uint32_t idesc = (1u << 4) | ((uint32_t)(im.n_mma >> 3) << 17) | ((128u >> 4) << 24);
        const int need = im.need(), need_pool = im.need_pool();
        const int n_st = im.n_main + im.n_pool;
        for (int it = 0; it < n_st; ++it, ++pos.si) {
            const bool pool = it >= im.n_main;
            const uint32_t xt = ring_a + (pool ? pos.place(need_pool, cap) + POOL_GROUP * POOL_TILE_PITCH
                                               : pos.place(need, cap) + im.blk_bytes);
            FfCycle<FF_NB> acb1 = acb;
            if (G == 64 && !pool) acb1.next();
            if (!warp_saw(ready)) {
                ok = warp_wait(FF_BAR(acc_empty, acb1.i), acb1.par ^ 1, poison, status, 8, pos.si) &&
                     warp_wait(FF_BAR(a_full, ab.i), ab.par, poison, status, 9, pos.si);
                if (!ok) break;
            }
            tc_fence_after();
            // (the shuffles tell the compiler that the operands are warp-uniform)
            const uint32_t d0 = __shfl_sync(0xffffffffu, acc0 + acb.i * (2 * FF_NT), 0);
            const uint32_t d1 = G == 64 ? __shfl_sync(0xffffffffu, acc0 + acb1.i * (2 * FF_NT), 0) : d0;
            const uint32_t a0 = __shfl_sync(0xffffffffu, tbase + 128 * ab.i, 0);
            const uint32_t xu = __shfl_sync(0xffffffffu, xt, 0);
            const uint32_t done_bar = FF_BAR(done, pos.si % FF_Q);
            const uint32_t acc_flag = it > im.n_main ? 1u : 0u;
            if (G == 64 && !pool) acb.next();
            if (!pool || it == n_st - 1) acb.next();
            ab.next();
            // main and cached-channel stages alike: an upper bound of what the next stage waits for
            FfCycle<FF_NB> nx = acb;
            if (G == 64) nx.next();
            ready = bar_test(FF_BAR(acc_empty, nx.i), nx.par ^ 1) & bar_test(FF_BAR(a_full, ab.i), ab.par);
            // operand tile: main [row group][k octet 16][8][8] + sums, cached channels [row group][k octet 4][8][8]
            ff_mma_stage<G>(d0, d1, a0, FF_NT, tc_desc(xu, 128, pool ? 512 : FF_RG),
                            __shfl_sync(0xffffffffu, idesc, 0), acc_flag, pool ? 0u : 1u);
            asm volatile(
                "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
                "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(done_bar)
                : "memory");
        }
    }
    if (!ok) *poison = 1;
}

template <bool GATEUP, int G>
__global__ void __launch_bounds__(FF_THREADS, 1) ffn_fold_kernel(const __grid_constant__ FfParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    FfShared* S = reinterpret_cast<FfShared*>(smem);
    FfExpert* tab = reinterpret_cast<FfExpert*>(smem + FF_HDR);
    uint8_t* htile = smem + p.off_h;
    uint8_t* ring = smem + p.off_ring;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < FF_Q; ++i) {
            mbar_init(&S->full[i], 1);
            mbar_init(&S->empty[i], FF_FOLD_WARPS);
            mbar_init(&S->done[i], 1);
        }
        for (int i = 0; i < FF_NA; ++i) {
            mbar_init(&S->a_full[i], FF_EXP_WARPS / 2);
        }
        for (int i = 0; i < FF_NB; ++i) mbar_init(&S->acc_empty[i], FF_FOLD_WARPS);
        mbar_init(&S->hready, FF_FOLD_WARPS);
        mbar_init(&S->hfree, FF_FOLD_WARPS);
        S->poison = 0;
        fence_barrier_init();
    }
    if (warp == FF_W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S->tmem_base)),
                     "r"(FF_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // Everything above overlaps the tail of the preceding kernel.
    pdl_wait();
    pdl_trigger();

    const LayerDev* L = p.L;
    int32_t* status = p.ws.status;
    const int n_kc = (GATEUP ? L->d : L->f) / KC;
    const bool off = (*status & STATUS_TIMEOUT) != 0;   // after an expired wait nothing new starts
    for (int i = threadIdx.x; i < p.n_experts; i += FF_THREADS) {
        const int e = L->order[i];
        const ExpertDev& ex = L->ex[e];
        FfExpert t;
        t.cnt = off ? 0 : p.ws.counts[e];
        if (t.cnt > p.ws.tc_min) t.cnt = 0;
        t.n_tt = (t.cnt + FF_NT - 1) / FF_NT;
        t.tile_rows = t.n_tt > 0 ? ((t.cnt + t.n_tt - 1) / t.n_tt + 7) & ~7 : 8;   // even tiles
        t.row0 = p.ws.off_pad[e];
        t.bits = ex.bits;
        t.blk_bytes = ex.blk_bytes;
        t.w = GATEUP ? ex.w13 : ex.w2;
        t.pool = reinterpret_cast<const uint8_t*>(ex.pool_hi);
        t.n_pool = (GATEUP && ex.switchable && L->sig_cnt[e] > 0) ? L->P_pad >> 5 : 0;
        t.first = t.n_tt * p.n_rb * p.ksplit;
        tab[i] = t;
    }
    __syncthreads();
    if (warp == 0) {   // exclusive scan of the item counts
        int run = 0;
        for (int i0 = 0; i0 < p.n_experts; i0 += 32) {
            const int i = i0 + lane;
            const int c = i < p.n_experts ? tab[i].first : 0;
            int v = c;
#pragma unroll
            for (int dd = 1; dd < 32; dd <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, dd);
                if (lane >= dd) v += u;
            }
            if (i < p.n_experts) tab[i].first = run + v - c;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) tab[p.n_experts].first = run;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = __shfl_sync(0xffffffffu, S->tmem_base, 0);
    const int total = __shfl_sync(0xffffffffu, tab[p.n_experts].first, 0);
    volatile int* poison = &S->poison;
    const int cap = p.ring_bytes;
    const uint32_t sb = smem_u32(smem), ring_a = sb + p.off_ring;
    int cur = 0;
    FfPos pos;

    FfRole R;
    R.S = S; R.tab = tab; R.sb = sb; R.ring = ring_a; R.tbase = tbase; R.total = total; R.n_kc = n_kc;
    if (warp < FF_EXP_WARPS) {
        ff_expand_role(p, R, warp, lane);
    } else if (warp < FF_W_PROD) {
        ff_fold_role<GATEUP, G>(p, R, htile, warp - FF_EXP_WARPS, lane);
    } else {
        if (warp == FF_W_PROD) {
            // ---------------- producer: one thread ----------------
            if (lane == 0) {
                bool ok = true;
                uint32_t si = 0, tail = 0;
                int free_b = cap;
                // ring offset of the next stage once it fits behind the oldest stage still in use
                auto acquire = [&](int need) -> int {
                    const int pad = pos.head + need > cap ? cap - pos.head : 0;
                    const int take = need + pad < cap ? need + pad : cap;   // a stage that wraps in its own footprint takes all
                    while (free_b < take || tail + FF_Q <= si) {
                        const int t = tail % FF_Q;
                        if (!mbar_wait_bounded(&S->empty[t], (tail / FF_Q) & 1, poison, status, WAIT_LIMIT_NS, 7, (int)tail))
                            return -1;
                        free_b += S->size[t];
                        ++tail;
                    }
                    S->size[si % FF_Q] = take;
                    free_b -= take;
                    return pos.place(need, cap);
                };
                const uint8_t* xbase = GATEUP ? p.ws.xperm : p.ws.hbuf;
                for (int g = blockIdx.x; g < total && ok; g += gridDim.x) {
                    const FfItem im = ff_item(p.ksplit, tab, g, cur, n_kc);
                    const int n_rg = (im.n_valid + 7) >> 3;   // 8-row groups that hold rows
                    const uint8_t* w = im.w;
                    const uint8_t* x = xbase + act_off(im.kc0, im.row0, p.ws.Rcap);
                    const size_t x_stride = act_off(1, 0, p.ws.Rcap);
                    const uint32_t xb = (uint32_t)(n_rg * FF_RG);
                    for (int it = 0; it < im.n_main; ++it, ++si) {
                        const int o = acquire(im.need());
                        if (o < 0) { ok = false; break; }
                        uint64_t* bar = &S->full[si % FF_Q];
                        mbar_arrive_expect_tx(bar, (uint32_t)im.blk_bytes + xb);
                        bulk_g2s(ring + o, w, (uint32_t)im.blk_bytes, bar);
                        bulk_g2s(ring + o + im.blk_bytes, x, xb, bar);
                        w += im.blk_bytes;
                        x += x_stride;
                    }
                    for (int it = 0; it < im.n_pool && ok; ++it, ++si) {
                        const int o = acquire(im.need_pool());
                        if (o < 0) { ok = false; break; }
                        uint64_t* bar = &S->full[si % FF_Q];
                        mbar_arrive_expect_tx(bar, (uint32_t)(POOL_GROUP * POOL_TILE_PITCH + n_rg * 512));
                        bulk_g2s(ring + o, im.pool + pool_tile_off(im.rb, POOL_GROUP * it, L->P_pad),
                                 (uint32_t)(POOL_GROUP * POOL_TILE_PITCH), bar);
                        bulk_g2s(ring + o + POOL_GROUP * POOL_TILE_PITCH,
                                 reinterpret_cast<const uint8_t*>(p.ws.xsig) + xpool_off(it, im.row0, p.ws.Rcap),
                                 (uint32_t)(n_rg * 512), bar);
                    }
                }
                if (!ok) {   // let copies in flight land before the CTA's shared memory goes away
                    const unsigned long long t0 = globaltimer_ns();
                    while (globaltimer_ns() - t0 < 2000000ull) {
                    }
                }
            }
            __syncwarp();
        } else if (warp == FF_W_MMA) {
            ff_mma_role<G>(p, R);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == FF_W_MMA) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(FF_TMEM_COLS) : "memory");
    }
}

template <bool GATEUP, int G>
static cudaError_t ff_launch(const FfParams& p, int n_ctas, cudaStream_t st) {
    cudaError_t err =
        cudaFuncSetAttribute(ffn_fold_kernel<GATEUP, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, FF_SMEM);
    if (err != cudaSuccess) return err;
    return launch_pdl(ffn_fold_kernel<GATEUP, G>, dim3((unsigned)n_ctas), dim3(FF_THREADS), (size_t)FF_SMEM, st, p);
}

cudaError_t launch_ffn_fold(const LayerDev* L, const WsDev& ws, int gateup, int n_rb, int ksplit, int n_experts,
                            long long split_stride, int n_sms, int G, cudaStream_t st) {
    FfParams p;
    p.L = L;
    p.ws = ws;
    p.n_rb = n_rb;
    p.n_experts = n_experts;
    p.ksplit = ksplit;
    p.split_stride = split_stride;
    auto up = [](int v, int a) { return (v + a - 1) / a * a; };
    p.off_h = up(FF_HDR + (n_experts + 1) * (int)sizeof(FfExpert), 128);
    p.off_ring = up(p.off_h + (gateup ? FF_NT * FF_HPITCH : 0), 1024);
    p.ring_bytes = FF_SMEM - p.off_ring;
    if (gateup) return G == 64 ? ff_launch<true, 64>(p, n_sms, st) : ff_launch<true, 128>(p, n_sms, st);
    return G == 64 ? ff_launch<false, 64>(p, n_sms, st) : ff_launch<false, 128>(p, n_sms, st);
}

}  // namespace dyn

// Routing, permutation, activation gather and weighted combine kernels.
//
// route   : top-k of the router logits per token (ties -> lower expert index), softmax weights.
// scan    : expert histogram -> exclusive scan -> stable counting sort of the (token, slot) pairs
//           (token-ascending inside an expert), warp-ballot ranking: deterministic, no atomics order.
//           Also lays the experts' segments out in PHYSICAL rows (each segment starts at a multiple of 8).
// gather  : expert-contiguous activation rows in fp16, pre-scaled for in-place code use, significant
//           columns zeroed for switchable experts (they are served by the 8-bit path), per-group sums,
//           plus the gathered significant columns; written in the layout of the FFN path the row's
//           expert takes (streaming rows, or 8-row MMA operand tiles).
// combine : y[t] = sum_j w[t,j] * Y[pos(t,j)] + sum_shared Y[pos], fp32, fixed order.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "layout.cuh"
#include "topk_rule.h"

namespace dyn {

// Top-k of one token's logits held across a warp (lane l holds logits l, l+32, ..., NV of them; E <= 32 NV): k largest
// raw logits in the order of topk_rule.h, ties -> lower expert index; weights = softmax over all E restricted to the
// chosen, rescaled to sum 1 if `renorm`.  A round of the selection is two warp reductions in hardware (with ten shuffles and
// eight candidates a lane whatever E is, the front kernel took 24.5 us at 16 tokens, 64 experts, top-6; 13.6 so), and
// the weights are worked out once behind the rounds, a lane each (the pass of those 16 tokens 68.5 -> 65.8 us).
template <int NV>
__device__ __forceinline__ void topk_softmax_store(float (&v)[NV], int lane, int E, int k, int renorm, long long token,
                                                   int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < NV; ++i) mx = fmaxf(mx, v[i]);
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float den = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i)
        if (lane + 32 * i < E) den += expf(v[i] - mx);
#pragma unroll
    for (int o = 16; o; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);

    // The selection works on keys: a taken expert is marked, not given a value that a logit may have, and a NaN has a
    // place in the order, so the k choices are k different experts whatever the logits are (masked with -infinity, NaN).
    uint32_t key[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) key[i] = lane + 32 * i < E ? topk_key(v[i]) : TOPK_TAKEN;
    uint32_t my_key = TOPK_NAN;   // lane j keeps the j-th choice
    int my_i = 0;
    for (int j = 0; j < k; ++j) {
        // local best (value desc, index asc)
        uint32_t bk = key[0];
        int bi = lane;
#pragma unroll
        for (int i = 1; i < NV; ++i)
            if (key[i] > bk) { bk = key[i]; bi = lane + 32 * i; }
        const uint32_t best = __reduce_max_sync(0xffffffffu, bk);
        bi = (int)__reduce_min_sync(0xffffffffu, bk == best ? (uint32_t)bi : 0x7fffffffu);
        // remove the winner from its owner's candidates
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (lane + 32 * i == bi) key[i] = TOPK_TAKEN;
        if (lane == j) {
            my_i = bi;
            my_key = best;
        }
    }
    const float my_w = lane < k ? expf(topk_value(my_key) - mx) / den : 0.f;
    float wsum = 0.f;
    if (renorm)
        for (int j = 0; j < k; ++j) wsum += __shfl_sync(0xffffffffu, my_w, j);   // in the order of the choices
    if (lane < k) {
        topk_idx[token * k + lane] = my_i;
        topk_w[token * k + lane] = renorm ? my_w / wsum : my_w;
    }
}

// Logits l[0 .. E) of one token into a warp's registers, then the selection.
template <int NV>
__device__ __forceinline__ void topk_from_memory(const float* __restrict__ l, int lane, int E, int k, int renorm,
                                                 long long token, int32_t* __restrict__ topk_idx,
                                                 float* __restrict__ topk_w) {
    float v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = lane + 32 * i;
        v[i] = (e < E) ? l[e] : -INFINITY;
    }
    topk_softmax_store<NV>(v, lane, E, k, renorm, token, topk_idx, topk_w);
}
__device__ __forceinline__ void topk_token(const float* __restrict__ l, int lane, int E, int k, int renorm, long long token,
                                           int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
    if (E <= 32) topk_from_memory<1>(l, lane, E, k, renorm, token, topk_idx, topk_w);
    else if (E <= 64) topk_from_memory<2>(l, lane, E, k, renorm, token, topk_idx, topk_w);
    else topk_from_memory<8>(l, lane, E, k, renorm, token, topk_idx, topk_w);
}

// One warp per token.
__global__ void __launch_bounds__(256) route_kernel(const float* __restrict__ logits, int T, int E, int k, int renorm,
                                                    int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
    pdl_prologue();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= T) return;
    topk_token(logits + (long long)warp * E, lane, E, k, renorm, warp, topk_idx, topk_w);
}

// Router GEMM fused with the top-k (Section II-A: the gate scores every expert, the K best are taken):
// logits[t][e] = sum_c x[t][c] * W_r[e][c] (+ bias[e]), bf16 inputs, fp32 accumulate.  One CTA of eight warps per TB
// tokens, which share the loads and the conversion of the router's weights: warp w, lane l take the input indices
// 8*l + 256*(w + 8*i) ..+7, eight experts at a time, the next eight rows of weights on their way meanwhile.  Every warp
// reduces its partial sums over its lanes in the butterfly order (offsets 16, 8, 4, 2, 1), the eight partials are added
// in warp order, so the sum order (hence the fp32 result) is deterministic.  The eight sums of a token are reduced
// together, a lane keeping half of them at each of the first three steps: 9 shuffles instead of 40, the same additions.
// Warp t then selects the top-k of the CTA's token t exactly as route_kernel does.
// 300 tokens, 64 experts, d = 2048: 21.7 us; 37 us with one token per CTA, one expert's shuffles after another and no
// loads ahead.
template <int TB>
__global__ void __launch_bounds__(256) route_gemm_kernel(const __nv_bfloat16* __restrict__ x,
                                                         const __nv_bfloat16* __restrict__ w_router,
                                                         const float* __restrict__ bias, int T, int d, int E, int k,
                                                         int renorm, float* __restrict__ logits_out,
                                                         int32_t* __restrict__ topk_idx, float* __restrict__ topk_w) {
    __shared__ float part[TB][8][MAX_EXPERTS];
    pdl_prologue();
    const int t0 = blockIdx.x * TB, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = 8 * lane + 256 * warp;
    const int n_c = c0 < d ? (d - c0 + 2047) / 2048 : 0;    // this lane's runs of eight input indices
    const int n_cw = (d - 256 * warp + 2047) / 2048;        // the warp's (uniform; some lanes may have one less)
    uint4 wv[8];
    auto load_w = [&](int e0, int i) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            wv[j] = (i < n_c && e0 + j < E)
                        ? *reinterpret_cast<const uint4*>(w_router + (long long)(e0 + j) * d + c0 + 2048 * i)
                        : make_uint4(0u, 0u, 0u, 0u);
    };
    if (n_cw > 0) {
        load_w(0, 0);
        for (int e0 = 0; e0 < E; e0 += 8) {  // eight experts at a time
            float acc[TB][8];
#pragma unroll
            for (int t = 0; t < TB; ++t)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[t][j] = 0.f;
            for (int i = 0; i < n_cw; ++i) {
                uint4 cur[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) cur[j] = wv[j];
                if (i + 1 < n_cw) load_w(e0, i + 1);
                else if (e0 + 8 < E) load_w(e0 + 8, 0);
                float xf[TB][8];
#pragma unroll
                for (int t = 0; t < TB; ++t) {
                    uint4 xv = make_uint4(0u, 0u, 0u, 0u);
                    if (i < n_c && t0 + t < T) xv = *reinterpret_cast<const uint4*>(x + (long long)(t0 + t) * d + c0 + 2048 * i);
                    const __nv_bfloat162* xp = reinterpret_cast<const __nv_bfloat162*>(&xv);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        xf[t][2 * u] = __low2float(xp[u]);
                        xf[t][2 * u + 1] = __high2float(xp[u]);
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const __nv_bfloat162* wp = reinterpret_cast<const __nv_bfloat162*>(&cur[j]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float wl = __low2float(wp[u]), wh = __high2float(wp[u]);
#pragma unroll
                        for (int t = 0; t < TB; ++t) {
                            acc[t][j] = fmaf(xf[t][2 * u], wl, acc[t][j]);
                            acc[t][j] = fmaf(xf[t][2 * u + 1], wh, acc[t][j]);
                        }
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < TB; ++t) {
                // after the steps 16, 8, 4 a lane holds the sum of expert e0 + 4 b4 + 2 b3 + b2 (its lane bits)
                float s4[4], s2[2], s1;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool up = (lane & 16) != 0;
                    const float keep = up ? acc[t][j + 4] : acc[t][j], give = up ? acc[t][j] : acc[t][j + 4];
                    s4[j] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const bool up = (lane & 8) != 0;
                    const float keep = up ? s4[j + 2] : s4[j], give = up ? s4[j] : s4[j + 2];
                    s2[j] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
                }
                {
                    const bool up = (lane & 4) != 0;
                    const float keep = up ? s2[1] : s2[0], give = up ? s2[0] : s2[1];
                    s1 = keep + __shfl_xor_sync(0xffffffffu, give, 4);
                }
                s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
                s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
                const int e = e0 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
                if ((lane & 3) == 0 && e < E) part[t][warp][e] = s1;
            }
        }
    } else {
        for (int e = lane; e < E; e += 32)
#pragma unroll
            for (int t = 0; t < TB; ++t) part[t][warp][e] = 0.f;
    }
    __syncthreads();
    const int token = t0 + warp;
    if (warp >= TB || token >= T) return;
    auto select = [&](auto nvc) {
        constexpr int NV = decltype(nvc)::value;
        float v[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = lane + 32 * i;
            v[i] = -INFINITY;
            if (e < E) {
                float sum = part[warp][0][e];
#pragma unroll
                for (int w = 1; w < 8; ++w) sum += part[warp][w][e];
                v[i] = sum + (bias ? bias[e] : 0.f);
                if (logits_out) logits_out[(long long)token * E + e] = v[i];
            }
        }
        topk_softmax_store<NV>(v, lane, E, k, renorm, token, topk_idx, topk_w);
    };
    if (E <= 32) select(std::integral_constant<int, 1>{});
    else if (E <= 64) select(std::integral_constant<int, 2>{});
    else select(std::integral_constant<int, 8>{});
}

// The pair array (pair i = t*k + j, ascending in t) is cut into contiguous segments, one per warp of a CTA.  Pass 1:
// each warp histograms its segment per expert (lanes holding the same expert find one another with match.any; the
// lowest lane of each group adds the group's size).  An exclusive scan over segments turns the histograms into each
// segment's first rank within the expert; pass 2 walks the segment again and ranks each pair = segment base + pairs of
// that expert seen so far in the segment + position within the 32-pair batch.  Segments and lanes ascend in i and
// a token holds an expert at most once, so the rank is the stable order.
// Large pair arrays: gridDim.x CTAs, each of which histograms the whole array (a few loads a thread) and ranks only its
// own run of segments, so no CTA waits for another; the loads of pass 1 are issued four batches at a time.  One CTA
// that walked 12288 pairs twice, a dependent load per 32 of them, took 26.4 us (2048 tokens, top-6), eight take 15.2.
// offsets/perm are the logical (unpadded) permutation; pos/row_token/row_expert use physical rows.
__global__ void __launch_bounds__(1024) scan_kernel(WsDev ws, int E, int Es, int k) {
    __shared__ int s_hist[32][MAX_EXPERTS];
    __shared__ int s_count[MAX_EXPERTS + 1];
    __shared__ int s_off[MAX_EXPERTS + 1];
    __shared__ int s_pad[MAX_EXPERTS + 1];
    pdl_prologue();
    const int T = ws.T, n_pairs = T * k;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int kk = k + Es;
    // work-queue counters of this forward's streaming launches (callers that only route pass no status block)
    if (ws.status && blockIdx.x == 0 && threadIdx.x < 4) ws.status[4 + threadIdx.x] = 0;
    const int per_warp = ((n_pairs + 31) / 32 + nwarps - 1) / nwarps * 32;  // whole 32-pair batches per segment
    const int seg_lo = min(n_pairs, warp * per_warp), seg_hi = min(n_pairs, seg_lo + per_warp);
    const unsigned lt = (1u << lane) - 1;
    for (int e = lane; e < E; e += 32) s_hist[warp][e] = 0;
    __syncwarp();
    for (int base = seg_lo; base < seg_hi; base += 128) {
        int ev[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = base + 32 * u + lane;
            ev[u] = i < seg_hi ? ws.topk_idx[i] : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned m = __match_any_sync(0xffffffffu, ev[u]);
            if (ev[u] >= 0 && (m & lt) == 0) s_hist[warp][ev[u]] += __popc(m);
            __syncwarp();
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E + Es; e += blockDim.x) {
        int acc = 0;
        if (e < E) {
#pragma unroll 8
            for (int w = 0; w < nwarps; ++w) {
                const int c = s_hist[w][e];
                s_hist[w][e] = acc;
                acc += c;
            }
        } else {
            acc = T;
        }
        s_count[e] = acc;
    }
    __syncthreads();
    if (warp == 0) {
        int run = 0, run_pad = 0;
        for (int e0 = 0; e0 < E + Es; e0 += 32) {
            const int e = e0 + lane;
            const int c = e < E + Es ? s_count[e] : 0;
            int v = c, vp = (c + 7) & ~7;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, d), up = __shfl_up_sync(0xffffffffu, vp, d);
                if (lane >= d) {
                    v += u;
                    vp += up;
                }
            }
            if (e < E + Es) {
                s_off[e] = run + v - c;
                s_pad[e] = run_pad + vp - ((c + 7) & ~7);
            }
            run += __shfl_sync(0xffffffffu, v, 31);
            run_pad += __shfl_sync(0xffffffffu, vp, 31);
        }
        if (lane == 0) {
            s_off[E + Es] = run;
            s_pad[E + Es] = run_pad;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0) {
        for (int e = threadIdx.x; e <= E + Es; e += blockDim.x) {
            ws.offsets[e] = s_off[e];
            ws.off_pad[e] = s_pad[e];
            if (e < E + Es) ws.counts[e] = s_count[e];
        }
        // padding rows of each routed expert's segment
        for (int e = threadIdx.x; e < E; e += blockDim.x) {
            const int c = s_count[e], po = s_pad[e];
            for (int r = c; r < ((c + 7) & ~7); ++r) {
                ws.row_token[po + r] = -1;
                ws.row_expert[po + r] = e;
            }
        }
    }
    // pass 2: this CTA's run of segments (gridDim.x divides the warp count), one warp each
    if (warp / (nwarps / (int)gridDim.x) == (int)blockIdx.x) {
        int next = seg_lo + lane < seg_hi ? ws.topk_idx[seg_lo + lane] : -1;
        for (int base = seg_lo; base < seg_hi; base += 32) {
            const int i = base + lane, e = next;
            next = i + 32 < seg_hi ? ws.topk_idx[i + 32] : -1;
            const bool valid = e >= 0;
            const unsigned m = __match_any_sync(0xffffffffu, e);
            const int start = valid ? s_hist[warp][e] : 0;
            __syncwarp();
            if (valid && (m & lt) == 0) s_hist[warp][e] = start + __popc(m);
            __syncwarp();
            if (valid) {
                const int r = start + __popc(m & lt);
                const int t = i / k, j = i - t * k;
                const int po = s_pad[e];
                ws.perm[s_off[e] + r] = i;
                ws.pos[t * kk + j] = po + r;
                ws.row_token[po + r] = t;
                ws.row_expert[po + r] = e;
            }
        }
    }
    // shared experts: every token, natural order
    const int padded = (T + 7) & ~7;
    for (int s = 0; s < Es; ++s) {
        const int po = s_pad[E + s];
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < padded; t += gridDim.x * blockDim.x) {
            if (t < T) ws.pos[t * kk + k + s] = po + t;
            ws.row_token[po + t] = t < T ? t : -1;
            ws.row_expert[po + t] = E + s;
        }
    }
}

// One physical row; part p of n converts the 128-k chunks p, p + n, ...  Forwards of 17 to 64 tokens give each row a CTA of
// eight warps (eight rows per CTA with one warp per row: +18 us on the 64-token step).  The fp16 activations are stored
// multiplied by 2^x_scale_exp(bits of the row's expert, k) so that the FFN kernels can use packed codes
// in place; the per-group sums are of the unscaled fp16 values.
enum : int { LAY_ROWS, LAY_TILES };   // which kernel reads the row: streaming, pair
__device__ __forceinline__ void gather_row(const LayerDev* __restrict__ L, const WsDev& ws,
                                           const __nv_bfloat16* __restrict__ x, int row, int t, int e, int seg0, int lay, int part, int n_parts) {
    const bool tc = lay != LAY_ROWS;
    const int lane = threadIdx.x & 31;
    if (t < 0 && !tc) return;  // padding rows matter only as zero rows of an MMA operand tile
    const int d = L->d;
    const int n_kc = d / KC;
    const int bits = L->ex[e].bits;
    const bool sw = L->ex[e].switchable != 0;
    const uint32_t* mask = sw ? (L->sigmask + (long long)e * (d / 32)) : nullptr;
    const __nv_bfloat16* xr = x + (long long)(t < 0 ? 0 : t) * d;
    const float sc0 = __uint_as_float((uint32_t)(127 + x_scale_exp(bits, 4 * lane)) << 23);
    const float sc1 = __uint_as_float((uint32_t)(127 + x_scale_exp(bits, 4 * lane + 2)) << 23);
    const int rg = row >> 3, rr = row & 7;
    bool clamped = false;
    // four chunks at a time, their loads in flight together: a chunk's load, mask and sum are a chain of latencies
    for (int c0 = part; c0 < n_kc; c0 += 4 * n_parts) {
        uint2 raw[4];
        uint32_t mw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * n_parts, k0 = c * KC + lane * 4;
            raw[u] = make_uint2(0u, 0u);
            mw[u] = 0u;
            if (c < n_kc && t >= 0) {
                raw[u] = *reinterpret_cast<const uint2*>(xr + k0);
                if (sw) mw[u] = __ldg(mask + (k0 >> 5)) >> (k0 & 31);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + u * n_parts;
            if (c >= n_kc) break;
            const __nv_bfloat162 p0 = *reinterpret_cast<const __nv_bfloat162*>(&raw[u].x);
            const __nv_bfloat162 p1 = *reinterpret_cast<const __nv_bfloat162*>(&raw[u].y);
            float v[4] = {__low2float(p0), __high2float(p0), __low2float(p1), __high2float(p1)};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                v[i] = clamp_act(v[i], clamped);
                if ((mw[u] >> i) & 1u) v[i] = 0.f;
            }
            float hv[4];
            float sum = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                hv[i] = __half2float(__float2half_rn(v[i]));
                sum += hv[i];
            }
            // sum over the 16 lanes of each half chunk (64 k), fixed butterfly order
#pragma unroll
            for (int o = 8; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            const __half2 oa = __floats2half2_rn(hv[0] * sc0, hv[1] * sc0), ob = __floats2half2_rn(hv[2] * sc1, hv[3] * sc1);
            uint2 packed;
            packed.x = *reinterpret_cast<const uint32_t*>(&oa);
            packed.y = *reinterpret_cast<const uint32_t*>(&ob);
            if (!tc) {
                uint8_t* out = ws.xperm + act_off(c, row, ws.Rcap);
                *reinterpret_cast<uint2*>(out + lane * 8) = packed;
                if ((lane & 15) == 0) *reinterpret_cast<float*>(out + XROW_SUM_OFF + (lane >> 4) * 4) = sum;
            } else {
                uint8_t* out = ws.xperm + tile_off(c, seg0, (row - seg0) >> 3, ws.Rcap);
                *reinterpret_cast<uint2*>(out + (lane >> 1) * 128 + rr * 16 + (lane & 1) * 8) = packed;
            }
        }
    }
    if (clamped && ws.status) atomicOr(ws.status, STATUS_RANGE);
    // Activations of ALL cached channels of the row's expert, unscaled, zero where the channel is not
    // currently significant: the FFN kernels multiply them with the contiguous 8-bit-valued tiles of the
    // whole cache pool, so a switch only has to flip mask bits.
    if (!sw) return;
    const int P = L->P, P_pad = L->P_pad;
    const int32_t* ci = L->cache_idx + (long long)e * P;
    uint8_t* xp = reinterpret_cast<uint8_t*>(ws.xsig);
    for (int j = 32 * part + lane; j < P_pad; j += 32 * n_parts) {
        const int pq = j >> 5, col = j & 31;
        if (!tc) {
            float v = 0.f;
            if (j < P) {
                const int ch = ci[j];
                if ((mask[ch >> 5] >> (ch & 31)) & 1u) v = clamp_act(__bfloat162float(xr[ch]), clamped);
            }
            *reinterpret_cast<__half*>(xp + xpool_off(pq, row, ws.Rcap) + col * 2) = __float2half_rn(v);
        } else {
            // operand position kp of a 16-column step holds pool column 16*step + sigma(kp): the A tile reaches
            // TMEM through an ldmatrix fragment whose k pairs (2t, 2t+1 | 2t+8, 2t+9) land on TMEM k 4t .. 4t+3.
            const int step = col >> 4, kp = col & 15;
            const int pj = pq * 32 + step * 16 + 2 * (kp >> 2) + (kp & 1) + ((kp & 2) ? 8 : 0);
            float v = 0.f;
            if (t >= 0 && pj < P) {
                const int ch = ci[pj];
                if ((mask[ch >> 5] >> (ch & 31)) & 1u) v = clamp_act(__bfloat162float(xr[ch]), clamped);
            }
            // 8-row operand tile of group pq: [k-octet 4][row 8][8 k] fp16 = 512 B
            *reinterpret_cast<__half*>(xp + xpool_off(pq, 8 * rg, ws.Rcap) + (col >> 3) * 128 + rr * 16 + (col & 7) * 2) =
                __float2half_rn(v);
        }
    }
}

__global__ void __launch_bounds__(256) gather_kernel(const LayerDev* __restrict__ L, WsDev ws,
                                                     const __nv_bfloat16* __restrict__ x) {
    pdl_wait();   // no early start for the next kernel: see front_kernel
    const int row = blockIdx.x;
    if (row >= ws.off_pad[L->E + L->Es]) return;
    const int e = ws.row_expert[row];
    gather_row(L, ws, x, row, ws.row_token[row], e, ws.off_pad[e], LAY_ROWS, threadIdx.x >> 5, 8);
}

// Forwards whose experts (most of them) read operand tiles: one CTA per 8-row group, all of one expert.  A warp takes
// whole 128-k chunks of the group: lane (row rr, octet o of 8 k) reads 16 bytes of its row and writes 16 bytes of the
// tile, so that four lanes read 64 consecutive bytes of a row and a warp writes 512 consecutive bytes; the chain of
// loads that finds a row's expert and token is paid once per group.  One CTA per row wrote every 128-byte line of a
// tile from eight CTAs and took 59 us at 2048 fine-grained tokens (16.9 k rows of 2048), this 36.3.  grid.y cuts the chunks of a
// group where there are few groups.
__global__ void __launch_bounds__(256) gather_group_kernel(const LayerDev* __restrict__ L, WsDev ws,
                                                           const __nv_bfloat16* __restrict__ x) {
    pdl_prologue();
    const int row0 = 8 * blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (row0 >= ws.off_pad[L->E + L->Es]) return;
    const int e = ws.row_expert[row0], seg0 = ws.off_pad[e];
    const bool small = ws.counts[e] <= ws.tc_min, fold = small && ws.fold;
    if (small && !fold) {   // a warp per row
        gather_row(L, ws, x, row0 + warp, ws.row_token[row0 + warp], e, seg0, LAY_ROWS, blockIdx.y, gridDim.y);
        return;
    }
    const int rr = lane & 7, o = lane >> 3;
    const int t = ws.row_token[row0 + rr];
    const int d = L->d, n_kc = d / KC, G = L->G;
    const int bits = L->ex[e].bits;
    const bool sw = L->ex[e].switchable != 0;
    const uint32_t* mask = L->sigmask + (long long)e * (d / 32);
    const __nv_bfloat16* xr = x + (long long)(t < 0 ? 0 : t) * d;
    float sc[2][2];   // scale of k pairs 0, 2 | 1, 3 of octet o, o + 4 of a half chunk
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            sc[u][h] = __uint_as_float((uint32_t)(127 + x_scale_exp(bits, 8 * (o + 4 * u) + 2 * h)) << 23);
    bool clamped = false;
    for (int c = warp + 8 * blockIdx.y; c < n_kc; c += 8 * gridDim.y) {
        uint4 raw[4];
        uint32_t mw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // q = 2 * half + (octet >= 4)
            const int k0 = c * KC + 64 * (q >> 1) + 8 * (o + 4 * (q & 1));
            raw[q] = t >= 0 ? *reinterpret_cast<const uint4*>(xr + k0) : make_uint4(0u, 0u, 0u, 0u);
            mw[q] = sw ? mask[k0 >> 5] >> (k0 & 31) : 0u;
        }
        uint8_t* out = ws.xperm + (fold ? act_off(c, row0, ws.Rcap) : tile_off(c, seg0, (row0 - seg0) >> 3, ws.Rcap));
        float sum[2] = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162* xp = reinterpret_cast<const __nv_bfloat162*>(&raw[q]);
            uint4 packed;
            uint32_t* pk = reinterpret_cast<uint32_t*>(&packed);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float v0 = clamp_act(__low2float(xp[i]), clamped), v1 = clamp_act(__high2float(xp[i]), clamped);
                if ((mw[q] >> (2 * i)) & 1u) v0 = 0.f;
                if ((mw[q] >> (2 * i + 1)) & 1u) v1 = 0.f;
                v0 = __half2float(__float2half_rn(v0));
                v1 = __half2float(__float2half_rn(v1));
                sum[q >> 1] += v0 + v1;
                const __half2 hv = __floats2half2_rn(v0 * sc[q & 1][i & 1], v1 * sc[q & 1][i & 1]);
                pk[i] = *reinterpret_cast<const uint32_t*>(&hv);
            }
            *reinterpret_cast<uint4*>(out + (8 * (q >> 1) + o + 4 * (q & 1)) * 128 + rr * 16) = packed;
        }
        if (fold) {   // sums of the unscaled values per quantization group: [group][row 8] fp32 behind the tile
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 8);
                sum[h] += __shfl_xor_sync(0xffffffffu, sum[h], 16);
            }
            float* so = reinterpret_cast<float*>(out + TC_TILE_BYTES);
            if (o == 0) so[rr] = G == 128 ? sum[0] + sum[1] : sum[0];
            if (o == 1 && G == 64) so[8 + rr] = sum[1];
        }
    }
    if (sw) {
        // cached channels, an octet of columns per thread (see gather_row for the order of the columns)
        const int P = L->P, P_pad = L->P_pad;
        const int32_t* ci = L->cache_idx + (long long)e * P;
        uint8_t* xp = reinterpret_cast<uint8_t*>(ws.xsig);
        for (int oc = (threadIdx.x >> 3) + 32 * blockIdx.y; oc < P_pad >> 3; oc += 32 * gridDim.y) {
            const int pq = oc >> 2, co = oc & 3;   // group of 32 columns, octet in it
            uint4 packed = make_uint4(0u, 0u, 0u, 0u);
            __half* hv = reinterpret_cast<__half*>(&packed);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int kp = 8 * (co & 1) + i;
                const int pj = pq * 32 + (co >> 1) * 16 + 2 * (kp >> 2) + (kp & 1) + ((kp & 2) ? 8 : 0);
                if (t >= 0 && pj < P) {
                    const int ch = ci[pj];
                    if ((mask[ch >> 5] >> (ch & 31)) & 1u)
                        hv[i] = __float2half_rn(clamp_act(__bfloat162float(xr[ch]), clamped));
                }
            }
            *reinterpret_cast<uint4*>(xp + xpool_off(pq, row0, ws.Rcap) + co * 128 + rr * 16) = packed;
        }
    }
    if (clamped && ws.status) atomicOr(ws.status, STATUS_RANGE);
}

// Small batches: routing, permutation and gather in ONE launch (three launches cost more than their work when the
// whole forward takes tens of microseconds).  One CTA per physical row; every CTA repeats the routing and the
// counting sort of all T * k pairs in shared memory (a few hundred pairs at most), then gathers its own row; CTA 0
// also writes the routing outputs and the row tables the later kernels read.  Same results as the three kernels.
constexpr int FRONT_MAX_PAIRS = 96;
constexpr int FRONT_BATCHES = FRONT_MAX_PAIRS / 32;
__global__ void __launch_bounds__(256) front_kernel(const LayerDev* __restrict__ L, WsDev ws,
                                                    const __nv_bfloat16* __restrict__ x,
                                                    const float* __restrict__ logits, int E, int Es, int k, int renorm) {
    __shared__ int s_idx[FRONT_MAX_PAIRS];
    __shared__ float s_w[FRONT_MAX_PAIRS];
    __shared__ int s_rank[FRONT_MAX_PAIRS];
    __shared__ int s_hist[FRONT_BATCHES][MAX_EXPERTS];
    __shared__ int s_count[MAX_EXPERTS + 1], s_off[MAX_EXPERTS + 1], s_pad[MAX_EXPERTS + 1];
    __shared__ int s_row_e, s_row_t;
    // No early start for the next kernel: a streaming CTA has nine warps, seven of which a quarter of an SM's registers
    // holds, so three of them fit only if their odd warps fall on different quarters.  CTAs that settled beside this
    // kernel's took other places, and the third waited for the first two to end, 70 us later, on 20 of 148 SMs (8 and 16
    // tokens of 4096: 166 and 4 x 180 us, 157 and 4 x 174 without; 64 tokens of 512: 28 and 25.5).
    pdl_wait();
    const int T = ws.T, n_pairs = T * k, kk = k + Es;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = warp; t < T; t += 8) topk_token(logits + (long long)t * E, lane, E, k, renorm, t, s_idx, s_w);
    for (int i = threadIdx.x; i < FRONT_BATCHES * E; i += blockDim.x) s_hist[i / E][i % E] = 0;
    if (threadIdx.x == 0) { s_row_e = -1; s_row_t = -1; }
    __syncthreads();
    // counting sort (pair i = t*k + j ascends in t: the stable order), one warp per 32 pairs: a pair's rank is the number
    // of its expert's pairs in the batches before its own, plus those on lower lanes
    const unsigned same = __match_any_sync(0xffffffffu, threadIdx.x < n_pairs ? s_idx[threadIdx.x] : -1);
    const int below = __popc(same & ((1u << lane) - 1));
    if (threadIdx.x < n_pairs && below == 0) s_hist[warp][s_idx[threadIdx.x]] = __popc(same);
    __syncthreads();
    for (int e = threadIdx.x; e < E + Es; e += blockDim.x) {
        int c = e < E ? 0 : T;
        if (e < E) {
#pragma unroll
            for (int b = 0; b < FRONT_BATCHES; ++b) c += s_hist[b][e];
        }
        s_count[e] = c;
    }
    if (threadIdx.x < n_pairs) {
        int r = below;
        for (int b = 0; b < warp; ++b) r += s_hist[b][s_idx[threadIdx.x]];
        s_rank[threadIdx.x] = r;
    }
    __syncthreads();
    if (warp == 0) {
        int run = 0, run_pad = 0;
        for (int e0 = 0; e0 < E + Es; e0 += 32) {
            const int e = e0 + lane;
            const int c = e < E + Es ? s_count[e] : 0;
            int v = c, vp = (c + 7) & ~7;
#pragma unroll
            for (int dd = 1; dd < 32; dd <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, dd), up = __shfl_up_sync(0xffffffffu, vp, dd);
                if (lane >= dd) {
                    v += u;
                    vp += up;
                }
            }
            if (e < E + Es) {
                s_off[e] = run + v - c;
                s_pad[e] = run_pad + vp - ((c + 7) & ~7);
            }
            run += __shfl_sync(0xffffffffu, v, 31);
            run_pad += __shfl_sync(0xffffffffu, vp, 31);
        }
        if (lane == 0) {
            s_off[E + Es] = run;
            s_pad[E + Es] = run_pad;
        }
    }
    __syncthreads();
    const int row = blockIdx.x;
    // whose row is this: the expert whose padded segment holds it, then the pair of that expert with this rank
    for (int e = threadIdx.x; e < E + Es; e += blockDim.x)
        if (row >= s_pad[e] && row < s_pad[e + 1]) s_row_e = e;
    __syncthreads();
    const int my_e = s_row_e;
    if (my_e >= 0) {
        const int r = row - s_pad[my_e];
        if (my_e < E) {
            for (int i = threadIdx.x; i < n_pairs; i += blockDim.x)
                if (s_idx[i] == my_e && s_rank[i] == r) s_row_t = i / k;
        } else if (threadIdx.x == 0 && r < T) {
            s_row_t = r;
        }
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x < 4) ws.status[4 + threadIdx.x] = 0;   // work-queue counters of the streaming launches
        // the outputs and tables of the route and scan kernels
        for (int i = threadIdx.x; i < n_pairs; i += blockDim.x) {
            const int e = s_idx[i], r = s_rank[i], t = i / k, j = i - t * k;
            ws.topk_idx[i] = e;
            ws.topk_w[i] = s_w[i];
            ws.perm[s_off[e] + r] = i;
            ws.pos[t * kk + j] = s_pad[e] + r;
            ws.row_token[s_pad[e] + r] = t;
            ws.row_expert[s_pad[e] + r] = e;
        }
        for (int e = threadIdx.x; e <= E + Es; e += blockDim.x) {
            ws.offsets[e] = s_off[e];
            ws.off_pad[e] = s_pad[e];
            if (e < E + Es) ws.counts[e] = s_count[e];
        }
        for (int e = threadIdx.x; e < E; e += blockDim.x) {
            const int c = s_count[e], po = s_pad[e];
            for (int r = c; r < ((c + 7) & ~7); ++r) {
                ws.row_token[po + r] = -1;
                ws.row_expert[po + r] = e;
            }
        }
        for (int sx = 0; sx < Es; ++sx) {
            const int po = s_pad[E + sx];
            const int padded = (T + 7) & ~7;
            for (int t = threadIdx.x; t < padded; t += blockDim.x) {
                if (t < T) ws.pos[t * kk + k + sx] = po + t;
                ws.row_token[po + t] = t < T ? t : -1;
                ws.row_expert[po + t] = E + sx;
            }
        }
    }
    __syncthreads();
    if (my_e < 0) return;
    gather_row(L, ws, x, row, s_row_t, my_e, s_pad[my_e],
               s_count[my_e] > ws.tc_min ? LAY_TILES : LAY_ROWS, warp, 8);
}

// x and the logits of a call on page-locked host buffers, over PCIe into the staging buffers: one launch that the front
// kernel follows by its programmatic launch, where two copies on the copy engine each add a hand-over between engine and
// SMs.  Bound by PCIe; every thread has its loads in flight at once.  Not launched programmatically itself: nothing of
// it runs beside an earlier kernel.
__global__ void __launch_bounds__(256) upload_kernel(const uint4* __restrict__ xh, uint4* __restrict__ xd, long long nx,
                                                     const float* __restrict__ lh, float* __restrict__ ld, long long nl) {
    pdl_trigger();
    const long long i0 = (long long)blockIdx.x * 256 + threadIdx.x, step = (long long)gridDim.x * 256;
    for (long long i = i0; i < nl; i += step) ld[i] = lh[i];
    for (long long i = i0; i < nx; i += 4 * step) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * step < nx) v[u] = xh[i + u * step];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * step < nx) xd[i + u * step] = v[u];
    }
}

// grid (T, ceil(d / 1024)): each thread owns four output columns of one token.  KS > 0: every expert's result is in KS
// copies of ypart (the K splits, known to the compiler, no lookups in front of their loads: 8 tokens of 4096 in 8 splits
// 6.0 -> 5.2 us); 0: any forward, the first copies of U of a token's rows (U divides their number) loaded at once.
template <int KS, int U>
__global__ void __launch_bounds__(256) combine_kernel(WsDev ws, int d, int k, int Es, void* __restrict__ y,
                                                      int y_f32, long long split_stride, int n_experts) {
    pdl_prologue();
    if (*ws.status & STATUS_TIMEOUT) return;  // the FFN kernels started nothing: leave y alone
    const int t = blockIdx.x;
    const int kk = k + Es;
    const int c = (blockIdx.y * blockDim.x + threadIdx.x) * 4;
    if (c >= d) return;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if constexpr (KS > 0) {
#pragma unroll 2
        for (int j = 0; j < kk; ++j) {
            const float* src = ws.ypart + (long long)ws.pos[t * kk + j] * d + c;
            const float w = (j < k) ? ws.topk_w[t * k + j] : 1.0f;
            float4 v[KS];
#pragma unroll
            for (int sp = 0; sp < KS; ++sp) v[sp] = *reinterpret_cast<const float4*>(src + sp * split_stride);
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int sp = 0; sp < KS; ++sp) {
                s[0] += v[sp].x; s[1] += v[sp].y; s[2] += v[sp].z; s[3] += v[sp].w;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = fmaf(w, s[i], acc[i]);
        }
    }
    for (int j0 = KS > 0 ? kk : 0; j0 < kk; j0 += U) {
        int r[U];
        float4 s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = ws.pos[t * kk + j0 + u];
#pragma unroll
        for (int u = 0; u < U; ++u) s[u] = *reinterpret_cast<const float4*>(ws.ypart + (long long)r[u] * d + c);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + u;
            const float w = (j < k) ? ws.topk_w[t * k + j] : 1.0f;
            const int e = ws.row_expert[r[u]];
            const int ns = (ws.counts[e] > ws.tc_min) ? 1 : ws.ksplit;  // the tensor-core path does not split K
            for (int sp = 1; sp < ns; ++sp) {
                const float4 v = *reinterpret_cast<const float4*>(
                    ypart_row(ws, sp, split_stride, e, n_experts, r[u], ws.off_pad[e], d) + c);
                s[u].x += v.x; s[u].y += v.y; s[u].z += v.z; s[u].w += v.w;
            }
            acc[0] = fmaf(w, s[u].x, acc[0]);
            acc[1] = fmaf(w, s[u].y, acc[1]);
            acc[2] = fmaf(w, s[u].z, acc[2]);
            acc[3] = fmaf(w, s[u].w, acc[3]);
        }
    }
    if (y_f32) {
        *reinterpret_cast<float4*>((float*)y + (long long)t * d + c) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    } else {
        __nv_bfloat162 a = __floats2bfloat162_rn(acc[0], acc[1]), b = __floats2bfloat162_rn(acc[2], acc[3]);
        uint2 o;
        o.x = *reinterpret_cast<uint32_t*>(&a);
        o.y = *reinterpret_cast<uint32_t*>(&b);
        *reinterpret_cast<uint2*>((__nv_bfloat16*)y + (long long)t * d + c) = o;
    }
}

cudaError_t launch_route(const float* logits, int T, int E, int k, int renorm, int32_t* idx, float* w,
                         cudaStream_t st) {
    return launch_pdl(route_kernel, dim3((unsigned)((T + 7) / 8)), dim3(256), 0, st, logits, T, E, k, renorm, idx, w);
}
cudaError_t launch_route_gemm(const void* x, const void* w_router, const float* bias, int T, int d, int E, int k,
                              int renorm, float* logits_out, int32_t* idx, float* w, cudaStream_t st) {
    // Two tokens a CTA until that fills the SMs several times over, then four (the part sums of four take 34 KB).
    if (T <= 1200)
        return launch_pdl(route_gemm_kernel<2>, dim3((unsigned)((T + 1) / 2)), dim3(256), 0, st, (const __nv_bfloat16*)x,
                          (const __nv_bfloat16*)w_router, bias, T, d, E, k, renorm, logits_out, idx, w);
    return launch_pdl(route_gemm_kernel<4>, dim3((unsigned)((T + 3) / 4)), dim3(256), 0, st, (const __nv_bfloat16*)x,
                      (const __nv_bfloat16*)w_router, bias, T, d, E, k, renorm, logits_out, idx, w);
}
cudaError_t launch_scan(const WsDev& ws, int E, int Es, int k, cudaStream_t st) {
    const int batches = (ws.T * k + 31) / 32;  // one warp per segment of whole 32-pair batches
    const int warps = batches < 8 ? 8 : (batches > 32 ? 32 : batches);  // >= 8: the per-expert loops want threads
    // from 2048 pairs on eight CTAs of 32 warps
    return launch_pdl(scan_kernel, dim3(batches >= 64 ? 8u : 1u), dim3((unsigned)(warps * 32)), 0, st, ws, E, Es, k);
}
cudaError_t launch_gather(const LayerDev* L, const WsDev& ws, const void* x, int d, int n_sms, cudaStream_t st) {
    if (ws.fold || ws.tc_min != 0x7fffffff) {
        // A group's chunks are cut over as many CTAs as it takes to have five per SM (at most one chunk a warp): 43
        // groups of 4096 15.6 -> 11.3 us, 258 21 -> 14.8; 2114 groups of 2048 cut in two 39 -> 45.
        const int groups = (ws.Rpad + 7) / 8, ny = std::max(1, std::min(d / KC / 8, (n_sms * 5 + groups - 1) / groups));
        return launch_pdl(gather_group_kernel, dim3((unsigned)groups, (unsigned)ny), dim3(256), 0, st, L, ws,
                          (const __nv_bfloat16*)x);
    }
    return launch_pdl(gather_kernel, dim3((unsigned)ws.Rpad), dim3(256), 0, st, L, ws, (const __nv_bfloat16*)x);
}
// Beyond this the three kernels are faster: top-2 of 8 experts, 20, 24, 32, 48, 64 tokens of 4096: 172, 173, 210, 237, 245 us a
// pass with this kernel, 180, 180, 210, 234, 241 with three (512-wide: 24 and 32 tokens 26 and 27, 32 and 31; 64: 31, 28);
// top-6 of 64: 8, 16, 20 tokens 53.8, 65.8, 75 and 57.1, 65.5, 70.
bool front_fits(int T, int k) { return T <= 32 && T * k <= FRONT_MAX_PAIRS; }
cudaError_t launch_front(const LayerDev* L, const WsDev& ws, const void* x, const float* logits, int E, int Es, int k,
                         int renorm, cudaStream_t st) {
    return launch_pdl(front_kernel, dim3((unsigned)ws.Rpad), dim3(256), 0, st, L, ws, (const __nv_bfloat16*)x, logits, E,
                      Es, k, renorm);
}
cudaError_t launch_upload(const void* xh, void* xd, long long x_bytes, const float* lh, float* ld, long long n_logits,
                          int n_sms, cudaStream_t st) {
    const long long nx = x_bytes / 16;
    const unsigned ctas = (unsigned)std::max(1ll, std::min(4ll * n_sms, (nx + 255) / 256));
    upload_kernel<<<ctas, 256, 0, st>>>((const uint4*)xh, (uint4*)xd, nx, lh, ld, n_logits);
    return cudaGetLastError();
}
cudaError_t launch_combine(const WsDev& ws, int d, int k, int Es, void* y, int y_f32, long long split_stride,
                           int n_experts, cudaStream_t st) {
    const bool uniform = ws.tc_min == 0x7fffffff && !ws.ysmall;
    auto kernel = uniform && ws.ksplit == 8   ? combine_kernel<8, 1>
                  : uniform && ws.ksplit == 4 ? combine_kernel<4, 1>
                  : uniform && ws.ksplit == 2 ? combine_kernel<2, 1>
                  : uniform && ws.ksplit == 1 ? combine_kernel<1, 1>
                                              : (k + Es) % 4 == 0         ? combine_kernel<0, 4>
                  : (k + Es) % 2 == 0         ? combine_kernel<0, 2>
                                              : combine_kernel<0, 1>;
    return launch_pdl(kernel, dim3((unsigned)ws.T, (unsigned)((d + 1023) / 1024)), dim3(256), 0, st, ws, d, k, Es, y, y_f32,
                      split_stride, n_experts);
}

}  // namespace dyn

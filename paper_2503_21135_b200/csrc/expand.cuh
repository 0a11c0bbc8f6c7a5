// Code expansion shared by the FFN kernels: packed codes of one atom -> fp16 A-operand register pairs.
// MAGIC = 0          : a field masked in place is the fp16 subnormal q * 2^(o-24)   (one AND per pair)
// MAGIC = 0x64006400 : the pair is (1024 + q * 2^o) in both halves                  (one AND-OR per pair)
// See layout.cuh for the field positions and the matching power-of-two scale of the activations.
#pragma once
#include "common.cuh"
#include "layout.cuh"

namespace dyn {

// Packed codes of one atom for one half chunk (64 k = 4 MMA steps), per lane, plus the shifted copies.
template <int BITS>
struct Codes;
template <>
struct Codes<2> { uint32_t w[2], ws[2]; };
template <>
struct Codes<3> { uint32_t w[2], x[2]; };  // W(jh); W2 or, for the upper half chunk, its >> 8 (other views where they are used:
                                           // kept in registers they made the fold kernel spill)
template <>
struct Codes<4> { uint32_t w[4], ws[4]; };
template <>
struct Codes<8> { uint32_t w[8]; };
template <>
struct Codes<6> { uint32_t w[4], ws[4], t[2][4]; };  // low-nibble words and their >> 8; four copies of the high-bit words

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Bits of a under the mask, of b elsewhere: one LOP3.  (As a & mask | b & ~mask the compiler takes the spread fields of 3-bit
// codes apart again under their own masks: a layer of 3-bit experts 161 -> 157 us at 8 tokens, 193 -> 189 at 24.)
__device__ __forceinline__ uint32_t bits_of(uint32_t mask, uint32_t a, uint32_t b) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xCA;" : "=r"(r) : "r"(mask), "r"(a), "r"(b));
    return r;
}

template <int BITS>
__device__ __forceinline__ void load_codes(Codes<BITS>& c, const uint8_t* atom, int lane, int half) {
    if constexpr (BITS == 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(atom + half * 512 + lane * 16);
        c.w[0] = v.x; c.w[1] = v.y; c.w[2] = v.z; c.w[3] = v.w;
#pragma unroll
        for (int i = 0; i < 4; ++i) c.ws[i] = c.w[i] >> 8;
    } else if constexpr (BITS == 8) {
        const uint4 v0 = *reinterpret_cast<const uint4*>(atom + (2 * half) * 512 + lane * 16);
        const uint4 v1 = *reinterpret_cast<const uint4*>(atom + (2 * half + 1) * 512 + lane * 16);
        c.w[0] = v0.x; c.w[1] = v0.y; c.w[2] = v0.z; c.w[3] = v0.w;
        c.w[4] = v1.x; c.w[5] = v1.y; c.w[6] = v1.z; c.w[7] = v1.w;
    } else if constexpr (BITS == 6) {
        const uint4 v = *reinterpret_cast<const uint4*>(atom + half * 512 + lane * 16);
        c.w[0] = v.x; c.w[1] = v.y; c.w[2] = v.z; c.w[3] = v.w;
#pragma unroll
        for (int i = 0; i < 4; ++i) c.ws[i] = c.w[i] >> 8;
        const uint2 hb = *reinterpret_cast<const uint2*>(atom + 1024 + lane * 16 + half * 8);
        const uint32_t hw[2] = {hb.x, hb.y};
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            const uint32_t sw = prmt(hw[rh], 0u, 0x2301u);   // bytes of each 16-bit half swapped
            c.t[rh][0] = hw[rh];
            c.t[rh][1] = hw[rh] >> 2;
            c.t[rh][2] = sw;
            c.t[rh][3] = sw >> 2;
        }
    } else if constexpr (BITS == 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(atom + lane * 16 + half * 8);
        c.w[0] = v.x; c.w[1] = v.y;
        c.ws[0] = v.x >> 10; c.ws[1] = v.y >> 10;
    } else {
        const uint2 v = *reinterpret_cast<const uint2*>(atom + lane * 16 + half * 8);
        const uint2 x = *reinterpret_cast<const uint2*>(atom + 512 + lane * 8);
        c.w[0] = v.x; c.w[1] = v.y;
        c.x[0] = half ? x.x >> 8 : x.x; c.x[1] = half ? x.y >> 8 : x.y;
    }
}

// A-fragment registers of step S4 (0..3) of the loaded half chunk: fp16 pairs q * 2^(o-24).
template <int BITS, int S4, uint32_t MAGIC = 0u>
__device__ __forceinline__ void expand(const Codes<BITS>& c, uint32_t (&a)[4]) {
    if constexpr (BITS == 4) {
        constexpr int jj = S4 >> 1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int phi = 2 * (S4 & 1) + h;
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
                const uint32_t src = (phi < 2) ? c.w[rh * 2 + jj] : c.ws[rh * 2 + jj];
                a[rh + 2 * h] = (src & (0x000F000Fu << (4 * (phi & 1)))) | MAGIC;
            }
        }
    } else if constexpr (BITS == 6) {
        constexpr int jj = S4 >> 1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int phi = 2 * (S4 & 1) + h;
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
                const uint32_t lo = (phi < 2) ? c.w[rh * 2 + jj] : c.ws[rh * 2 + jj];
                a[rh + 2 * h] = (lo & (0x000F000Fu << (4 * h))) | ((c.t[rh][S4] & (0x00300030u << (4 * h))) | MAGIC);
            }
        }
    } else if constexpr (BITS == 8) {
        const uint32_t w0 = c.w[(S4 >> 1) * 4 + 2 * (S4 & 1)], w1 = c.w[(S4 >> 1) * 4 + 2 * (S4 & 1) + 1];
        a[0] = prmt(w0, MAGIC ? 0x64646464u : 0u, 0x4140u);
        a[1] = prmt(w0, MAGIC ? 0x64646464u : 0u, 0x4342u);
        a[2] = prmt(w1, MAGIC ? 0x64646464u : 0u, 0x4140u);
        a[3] = prmt(w1, MAGIC ? 0x64646464u : 0u, 0x4342u);
    } else if constexpr (BITS == 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int phi = 2 * S4 + h;
#pragma unroll
            for (int rh = 0; rh < 2; ++rh)
                a[rh + 2 * h] = ((phi <= 4) ? (c.w[rh] & (0x00030003u << (2 * phi)))
                                            : (c.ws[rh] & (0x00030003u << ((2 * phi - 10) & 31)))) | MAGIC;
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int phi = 2 * S4 + h;
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
                const uint32_t w = c.w[rh], x = c.x[rh];
                const uint32_t src = phi < 4 ? (h ? w >> 6 : w)
                                             : (h ? bits_of(0x00880088u, w, bits_of(0x00440044u, w >> 9, x << 1)) : x);
                a[rh + 2 * h] = (src & (0x00070007u << (2 * (phi & 3)))) | MAGIC;
            }
        }
    }
}

// The packed words of one atom that a lane owns (both half chunks), as they lie in shared memory: 4, 6, 8, 12 or 16.
template <int BITS>
__device__ __forceinline__ void load_raw(uint32_t (&w)[16], uint32_t atom, int lane) {
    auto put = [&](int i, uint4 v) {
        w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
    };
    put(0, lds128(atom + lane * 16));
    if constexpr (BITS == 3) {
        const uint2 hb = lds64(atom + 512 + lane * 8);
        w[4] = hb.x; w[5] = hb.y;
    }
    if constexpr (BITS >= 4) put(4, lds128(atom + 512 + lane * 16));
    if constexpr (BITS >= 6) put(8, lds128(atom + 1024 + lane * 16));
    if constexpr (BITS == 8) put(12, lds128(atom + 1536 + lane * 16));
}
template <int BITS, int HALF>
__device__ __forceinline__ void codes_of(Codes<BITS>& c, const uint32_t (&w)[16]) {
    if constexpr (BITS == 2) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            c.w[i] = w[2 * HALF + i];
            c.ws[i] = c.w[i] >> 10;
        }
    } else if constexpr (BITS == 3) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            c.w[i] = w[2 * HALF + i];
            c.x[i] = HALF ? w[4 + i] >> 8 : w[4 + i];
        }
    } else if constexpr (BITS == 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) c.w[i] = w[8 * HALF + i];
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c.w[i] = w[4 * HALF + i];
            c.ws[i] = c.w[i] >> 8;
        }
        if constexpr (BITS == 6) {
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
                const uint32_t hw = w[8 + 2 * HALF + rh], sw = prmt(hw, 0u, 0x2301u);   // bytes of each half swapped
                c.t[rh][0] = hw;
                c.t[rh][1] = hw >> 2;
                c.t[rh][2] = sw;
                c.t[rh][3] = sw >> 2;
            }
        }
    }
}

// In-place bit offset o of the code of (MMA step S4 of a half chunk, k pair h): see layout.cuh.
template <int BITS>
__host__ __device__ constexpr int code_offset(int s4, int h) {
    const int phi = 2 * s4 + h;
    return BITS == 2 ? (phi <= 4 ? 2 * phi : 2 * phi - 10) : BITS == 3 ? 2 * (phi & 3) : (BITS == 4 || BITS == 6) ? 4 * h : 0;
}

}  // namespace dyn

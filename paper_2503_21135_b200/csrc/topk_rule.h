// Order in which the router's top-k takes the logits of a token, as unsigned integers: larger value first, -0 equal to
// +0, a NaN behind every number (-infinity included).  Plain functions, compiled for host and device alike.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define DYN_HD __host__ __device__ __forceinline__
#else
#define DYN_HD static inline
#endif

namespace dyn {

// No logit has key 0: it marks a candidate that is taken, or a place behind the last expert, so that every round of a
// selection of k <= E experts finds one that is neither, whatever the logits are.
constexpr uint32_t TOPK_TAKEN = 0u, TOPK_NAN = 1u;

DYN_HD uint32_t topk_key(float v) {
    const float z = v + 0.f;
    uint32_t b;
    memcpy(&b, &z, 4);
    if ((b & 0x7fffffffu) > 0x7f800000u) return TOPK_NAN;
    return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
// The value of a key; a NaN for TOPK_NAN.
DYN_HD float topk_value(uint32_t k) {
    const uint32_t b = k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu);
    float v;
    memcpy(&v, &b, 4);
    return v;
}

}  // namespace dyn

// The decision table of the bf16 compress kernels: what both compress files need to agree on which rows it serves.
#pragma once
#include <stdint.h>

#include "tq.h"

namespace tq {

constexpr uint32_t kLutBinade = 128;       // patterns per sign and binade
constexpr uint32_t kLutBinades = 64;       // evaluated binades, at most
constexpr uint32_t kLutMostTop = 0x61FFu;  // largest pattern with an entry: 4 * (2^15 + 0x61FF + 1) bytes of shared memory, 226 KB

// A row whose alpha has a larger pattern (2^69 and more) is served as 2^-64 times its values, whose patterns are this much lower: what
// that takes below the normal numbers lies far below the evaluated patterns, which are decided like zero.  Host parameters only: with device
// parameters, where the host cannot choose the kernel, such rows are left to the element-wise kernels (the factor in the common kernel: 124 M x 8
// 522 -> 532 us with 16 levels, 525 -> 604 with 4; the lifted form beside it, inlined or in a function: 506 -> 532 and 574).
__host__ __device__ inline uint32_t lut_lift(uint32_t top) { return top > kLutMostTop ? kLutBinade * kLutBinades : 0u; }

// What the decision depends on besides the value; the tables stay where they are.
struct LutRule {
    float alpha;
    uint32_t num_levels;
    const float* levels;
    const float* inv_width;
};

// X = k * 2^16 + min(T, 2^16) for a gradient value g: the decision of the quantizer equation up to the
// random draw.  One IEEE operation per step (the build disables contraction on both sides), so host and
// device agree bit for bit.
__host__ __device__ inline uint32_t decision_x(float g, const LutRule& q) {
    const uint32_t s = q.num_levels - 1;
    const float t = fminf(fmaxf(g, -q.alpha), q.alpha);      // NaN -> -alpha, +-Inf -> +-alpha
    uint32_t k = 0;
    for (uint32_t j = 1; j + 1 <= s; ++j)                     // largest j <= s - 1 with l_j <= t
        if (q.levels[j] <= t) k = j;
    const float p = (t - q.levels[k]) * q.inv_width[k];
    const float tf = p * 65536.0f;
    const uint32_t T = !(tf > 0.0f) ? 0u : (tf >= 65536.0f ? 65536u : static_cast<uint32_t>(rintf(tf)));
    return k * 65536u + T;
}

__host__ __device__ inline float bf16_pattern_value(uint32_t pattern16) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(pattern16 << 16);
#else
    union { uint32_t u; float f; } c;
    c.u = pattern16 << 16;
    return c.f;
#endif
}

// Smallest bf16 pattern whose value is >= alpha (alpha positive and finite); at most 0x7F80 (+Inf).
__host__ __device__ inline uint32_t top_pattern(float alpha) {
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(alpha);
#else
    union { float f; uint32_t u; } c;
    c.f = alpha;
    const uint32_t u = c.u;
#endif
    uint32_t p = u >> 16;
    if ((p << 16) < u) ++p;
    return p;
}

// Whether a window of n patterns per sign, the last one `top`, holds all that differ in their decision: either it reaches
// down to zero, or the decision at +-base equals that of everything smaller (it is monotone in the value).  *base receives the
// window's first pattern.
__host__ __device__ inline bool lut_window_fits(const LutRule& q, uint32_t top, uint32_t n, uint32_t* base) {
    if (top < n) { *base = 0; return true; }
    *base = top - (n - 1);
    return decision_x(bf16_pattern_value(*base | 0x8000u), q) == decision_x(bf16_pattern_value(*base), q);
}

// Device-resident parameters: a row goes through the table kernel when its record is usable and the largest window
// serves it; the element-wise kernels evaluate the same rule and leave exactly those rows alone.
__host__ __device__ inline LutRule lut_rule(const tq_params_t& p, uint32_t bits) { return LutRule{p.alpha, 1u << bits, p.levels, p.inv_width}; }
__host__ __device__ inline bool lut_usable(const tq_params_t& p, uint32_t bits) {
    return p.alpha > 0.0f && p.bits == bits && !(p.flags & TQ_FLAG_INVALID) && top_pattern(p.alpha) <= kLutMostTop;
}
__host__ __device__ inline bool lut_serves_record(const tq_params_t& p, uint32_t bits) {
    uint32_t base;
    return lut_usable(p, bits) && lut_window_fits(lut_rule(p, bits), top_pattern(p.alpha), kLutBinade * kLutBinades, &base);
}

}  // namespace tq
